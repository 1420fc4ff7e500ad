"""The inclusion apply's dense products (step tasks over ranges of the
inputs) against the same operators multiplied out with torch: one segment to
several 64-output blocks, input ranges that do not divide the cells, more
right-hand sides than one pass; and the operators themselves against the
entries of the volume operator, for segment centres placed on cell centres."""
import numpy as np
import pytest

from paper_2210_02698_gb300 import workloads as W
from tests._common import gpu_op, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import build
    build.build()


@pytest.mark.parametrize("N,ns,nrhs", [(10, 1, 1), (19, 65, 3), (33, 200, 9), (40, 31, 16), (24, 130, 35), (12, 1300, 2)])
def test_inclusion_equals_its_operators(N, ns, nrhs):
    import torch
    from paper_2210_02698_gb300 import binding
    w = W.small_workload(W.LENS, N, N / 8, nrhs)
    op = gpu_op(w, precision=binding.HB_FP64)
    cen, ln = W.circle_segments((0.47, 0.52), 0.3, ns) if ns > 2 else (np.array([[0.31, 0.47]]), np.array([0.01]))
    op.set_curve(cen, ln, W.LENS.n(cen[:, 0], cen[:, 1]))
    nv = w.grid.Nv
    S = torch.empty((ns, ns), dtype=torch.complex128, device="cuda")   # column-major: S[j, i]
    V, U = torch.empty((nv, ns), dtype=S.dtype, device="cuda"), torch.empty((ns, nv), dtype=S.dtype, device="cuda")
    op.curve_operators(S, V, U)
    s = to_dev(W.complex_normal_sources(nv, nrhs, 3))
    free, u = torch.empty_like(s), torch.empty_like(s)
    op.apply_dense(s, free, nrhs)
    op.apply_inclusion(s, u, nrhs, v2v_dense=True)
    torch.cuda.synchronize()
    want = op.h ** 2 * torch.linalg.solve(S.T, (s @ V).T).T @ U
    # both sides solve with K^{s2s} (condition below 1e4) in 64 bits
    assert float(torch.linalg.norm(u - free - want) / torch.linalg.norm(want)) < 1e-11
    op.close()


def test_operators_at_cell_centres_equal_the_entries():
    import torch
    from paper_2210_02698_gb300 import binding
    N = 21
    w = W.small_workload(W.LENS, N, N / 8, 1)
    op = gpu_op(w, precision=binding.HB_FP64)
    nv = w.grid.Nv
    at = np.sort(np.random.default_rng(4).choice(nv, 70, replace=False))
    x, z = w.grid.centroids()
    ln = np.linspace(0.01, 0.02, len(at))
    op.set_curve(np.stack([x[at], z[at]], 1), ln, np.full(len(at), 1.05))
    V = torch.empty((nv, len(at)), dtype=torch.complex128, device="cuda")
    U = torch.empty((len(at), nv), dtype=torch.complex128, device="cuda")
    S = torch.empty((len(at), len(at)), dtype=torch.complex128, device="cuda")
    op.curve_operators(S, V, U)
    K = torch.empty((nv, nv), dtype=torch.complex128, device="cuda")
    op.entries(np.arange(nv), np.arange(nv), K)   # K[j, i] = K_ij
    torch.cuda.synchronize()
    a = torch.from_numpy(at).cuda()
    w_ = torch.from_numpy(ln).cuda()
    off = torch.ones((nv, len(at)), dtype=torch.bool, device="cuda")
    off[a, torch.arange(len(at), device="cuda")] = False   # a point against itself is singular
    for got, want, m in ((V, K[:, a], off), (U, K[a] * w_[:, None], off.T), (S, -K[a][:, a] * w_[:, None], off[a].T)):
        # tau^2 to a few 1e-16 at distances of a cell (0.048) and more: omega 1e-15 / 0.1 in the phase
        assert float((got - want)[m].abs().max() / want[m].abs().max()) < 1e-12
    op.close()
