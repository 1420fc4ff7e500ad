"""A right-hand side's result does not depend on the others of its pass: with a
column that is not finite, or too small for the digit products, beside it, every
other column keeps its bits (FP64 and matrix-free applies, forward and adjoint,
one and two tiles of right-hand sides), and the column itself is what it is
alone."""
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


@pytest.mark.parametrize("nrhs,at", [(3, 1), (16, 0), (21, 18)])
@pytest.mark.parametrize("kind", ["nan", "inf", "tiny"])
def test_other_columns_keep_their_bits(nrhs, at, kind):
    import torch
    from paper_2210_02698_gb300 import binding
    N = 28
    w = W.small_workload(W.LENS, N, N / 8, nrhs)
    op = gpu_op(w, precision=binding.HB_FP64)
    op.build()
    s = to_dev(W.complex_normal_sources(w.grid.Nv, nrhs, 11))
    odd = s.clone()
    if kind == "tiny":
        odd[at] *= 2.0 ** -1000
    else:
        odd[at, 37] = float(kind)
    others = [r for r in range(nrhs) if r != at]
    for f in (op.apply, op.apply_adjoint, op.apply_dense, op.apply_dense_adjoint):
        want, got, alone = torch.empty_like(s), torch.empty_like(s), torch.empty_like(s[:1])
        f(s, want, nrhs)
        f(odd, got, nrhs)
        f(odd[at:at + 1].clone(), alone, 1)
        torch.cuda.synchronize()
        assert torch.equal(got[others], want[others])
        if kind == "tiny":
            assert torch.equal(got[at], alone[0])
            # 2^-1000 is exact; what falls below the normal numbers is 2^-50 of the rest and less
            assert float(torch.linalg.norm(got[at] * 2.0 ** 1000 - want[at]) / torch.linalg.norm(want[at])) < 1e-12
        else:
            assert not bool(torch.isfinite(torch.view_as_real(got[at])).all())
    op.close()
