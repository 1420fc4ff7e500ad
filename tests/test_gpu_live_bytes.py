"""Device memory a handle holds: the FP64 step lists only where FP64 applies are
made, and the operands of the inclusion's dense products only for the products
that remain after its operators are compressed."""
import gc

import pytest

from paper_2210_02698_gb300 import workloads as W
from tests._common import gpu_op, rel_l2, from_dev, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import build
    build.build()


def _live():
    from paper_2210_02698_gb300 import binding
    gc.collect()
    return binding.device_alloc_cap(-1)


def test_mixed_handles_hold_no_fp64_steps():
    import torch
    from paper_2210_02698_gb300 import binding
    w = W.small_workload(W.LENS, 40, 5, 3)
    s = to_dev(W.complex_normal_sources(w.grid.Nv, 3, 5))
    live, held, out = _live(), {}, {}
    for prec in (binding.HB_FP64, binding.HB_MIXED_BF16X3):
        op = gpu_op(w, precision=prec)
        op.build()
        held[prec] = _live() - live
        op.set_precision(binding.HB_FP64)   # the steps of a mixed handle are made by the first FP64 apply
        u, a = torch.empty_like(s), torch.empty_like(s)
        op.apply_adjoint(s, a, 3)
        op.apply(s, u, 3)
        torch.cuda.synchronize()
        out[prec] = (u, a)
        op.close()
        assert _live() == live
    assert held[binding.HB_MIXED_BF16X3] < held[binding.HB_FP64]
    for x, y in zip(*out.values()):
        assert torch.equal(x, y)


def test_compressed_curve_gives_its_operands_back():
    import torch
    from paper_2210_02698_gb300 import binding
    w = W.small_workload(W.LENS, 48, 6, 2)
    op = gpu_op(w, precision=binding.HB_FP64)
    cen, ln = W.circle_segments((0.5, 0.5), 0.3, 256)
    live, ns, nv = _live(), 256, w.grid.Nv
    op.set_curve(cen, ln, W.LENS.n(cen[:, 0], cen[:, 1]))
    s = to_dev(W.complex_normal_sources(nv, 2, 5))
    dense, bf = torch.empty_like(s), torch.empty_like(s)
    op.apply_inclusion(s, dense, 2, v2v_dense=True)
    op.curve_compress(16)
    op.apply_inclusion(s, bf, 2, v2v_dense=True)
    torch.cuda.synchronize()
    assert rel_l2(from_dev(bf), from_dev(dense)) < 1e-4
    # LU and inverse, the butterflies, a segment's tables, the operands of the
    # inverse (its inputs and at most five ranges of outputs), and 2 MB of lists and vectors
    entries = sum(op.curve_info(k)[2] for k in (0, 1))
    most = 16 * (2 * ns * ns + entries) + (48 * 256 + 256) * ns + 256 * 6 * ns + (2 << 20)
    assert _live() - live < most
    op.close()
