"""Inclusions whose segments differ widely in length.  The surface operators
carry the lengths (columns of K^{s2v} as w_j, rows of the inverse of K^{s2s}
as 1 / w_i), so products that keep a fixed number of bits below a block's
largest value lose those of the others: the field of the inclusion is compared
with the same operators solved and multiplied out by torch in 64 bits, without
the lengths' scale (K^{s2s} = G W, K^{s2v} = H W: the field is H G^{-1} Y)."""
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


def graded_circle(ns, ratio, geometric):
    """ns segments of a circle whose lengths grow by `ratio` from one end to the
    other; geometric: the chords themselves, else equal chords with those lengths."""
    step = ratio ** (np.arange(ns) / (ns - 1.0))
    t = np.concatenate([[0.0], np.cumsum(step)]) * (2 * np.pi / step.sum())
    if not geometric:
        t = np.linspace(0.0, 2 * np.pi, ns + 1)
    p = np.stack([0.48 + 0.3 * np.cos(t), 0.51 + 0.3 * np.sin(t)], axis=1)
    cen, ln = 0.5 * (p[1:] + p[:-1]), np.hypot(*(p[1:] - p[:-1]).T)
    return cen, (ln if geometric else 0.02 * step / ratio)


@pytest.mark.parametrize("ratio,geometric,ns,nrhs", [(1.0, True, 200, 3), (1e4, True, 200, 3), (1e6, False, 200, 3),
                                                     (1e9, False, 131, 19)])
def test_lengths_of_any_ratio_keep_64_bits(ratio, geometric, ns, nrhs):
    import torch
    from paper_2210_02698_gb300 import binding
    N = 24
    w = W.small_workload(W.LENS, N, N / 8, nrhs)
    op = gpu_op(w, precision=binding.HB_FP64)
    cen, ln = graded_circle(ns, ratio, geometric)
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
    wd = torch.from_numpy(ln).cuda()[:, None]
    G, H = S / wd, U / wd
    want = op.h ** 2 * torch.linalg.solve(G.T, (s @ V).T).T @ H
    # the two solves with G and the sums: a few roundings times the condition number
    bound = 8 * float(torch.linalg.cond(G)) * 2.0 ** -53
    err = float(torch.linalg.norm(u - free - want) / torch.linalg.norm(want))
    print(f"ratio {ratio:g}: error {err:.2e}, bound {bound:.2e}")
    assert err < bound
    op.close()


@pytest.mark.parametrize("ratio", [1.0, 1e3])
def test_compressed_operators_of_a_graded_curve(ratio):
    import torch
    from paper_2210_02698_gb300 import binding
    N, ns = 40, 256
    w = W.small_workload(W.LENS, N, N / 8, 2)
    op = gpu_op(w, precision=binding.HB_FP64, eps=1e-10)
    cen, ln = graded_circle(ns, ratio, True)
    op.set_curve(cen, ln, W.LENS.n(cen[:, 0], cen[:, 1]))
    s = to_dev(W.complex_normal_sources(w.grid.Nv, 2, 5))
    free, dense, bf = torch.empty_like(s), torch.empty_like(s), torch.empty_like(s)
    op.apply_dense(s, free, 2)
    op.apply_inclusion(s, dense, 2, v2v_dense=True)
    op.curve_compress(16)
    op.apply_inclusion(s, bf, 2, v2v_dense=True)
    torch.cuda.synchronize()
    # K^{s2v}'s columns are decomposed with their lengths, to eps of the largest
    err = float(torch.linalg.norm(bf - dense) / torch.linalg.norm(dense - free))
    print(f"ratio {ratio:g}: compressed against dense {err:.2e}")
    assert err < 100 * 1e-10 * ratio
    op.close()
