"""The FP64 apply's step tasks (integer digits on the tensor cores) against
the oracle's numpy products over the saved factors: output and input counts
off the 8-tiles and past the 64 outputs of a CTA, both row groupings of
right-hand sides and the pass limit, right-hand sides of very different
scales; values that are not finite reach the outputs as they do in plain
sums."""
import numpy as np
import pytest

from paper_2210_02698_gb300 import workloads as W
from tests._common import from_dev, gpu_op, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import build
    build.build()


@pytest.mark.parametrize("N,leaf,nrhs", [(8, 64, 1), (13, 3, 2), (24, 150, 8), (30, 29, 9), (40, 64, 16), (36, 700, 17),
                                         (21, 1, 33)])
def test_applies_equal_the_products(tmp_path, N, leaf, nrhs):
    import torch
    from oracle.factor_file import FactorFile
    from paper_2210_02698_gb300 import binding
    w = W.small_workload(W.LENS, N, N / 8, nrhs, leaf=leaf)
    op = gpu_op(w, precision=binding.HB_FP64)
    op.build()
    op.save(tmp_path / "f")
    F = FactorFile(tmp_path / "f")
    s = W.complex_normal_sources(w.grid.Nv, nrhs, 9)
    s[:, 0] *= 1e-200
    if nrhs > 1:
        s[:, 1] = 0
        s[N // 2, 1] = 1e200
    s_dev = to_dev(s)
    for fn, ref in ((op.apply, F.apply), (op.apply_adjoint, F.apply_adjoint)):
        u = torch.full_like(s_dev, float("nan"))
        fn(s_dev, u, nrhs)
        torch.cuda.synchronize()
        got, want = from_dev(u), ref(s)
        # both sides round every one of the ~10 chained products and the ~10 sums at 2^-53 of sums of up to 700 terms
        for k in range(nrhs):
            assert np.linalg.norm((got[:, k] - want[:, k]) / np.abs(want[:, k]).max()) <= 1e-13 * np.linalg.norm(
                want[:, k] / np.abs(want[:, k]).max())
    op.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("nrhs", [3, 12])
def test_values_that_are_not_finite(bad, nrhs):
    import torch
    from paper_2210_02698_gb300 import binding
    w = W.small_workload(W.GRADIENT, 24, 3, nrhs, leaf=32)
    op = gpu_op(w, precision=binding.HB_FP64)
    op.build()
    s_dev = to_dev(W.complex_normal_sources(w.grid.Nv, nrhs, 9))
    clean, u = torch.empty_like(s_dev), torch.empty_like(s_dev)
    for fn in (op.apply, op.apply_adjoint):
        fn(s_dev, clean, nrhs)
        t = s_dev.clone()
        t[1, 100] = complex(bad, 0.0)
        fn(t, u, nrhs)
        torch.cuda.synchronize()
        assert not torch.isfinite(torch.view_as_real(u[1])).all(-1).any()   # every output reads every input
        rest = [k for k in range(nrhs) if k != 1]
        # the finite columns take the plain sums in the tasks that hold the bad one: rounding only
        assert float(torch.linalg.norm(u[rest] - clean[rest]) / torch.linalg.norm(clean[rest])) < 1e-13
    op.close()
