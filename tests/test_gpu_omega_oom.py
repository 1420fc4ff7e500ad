"""hb_set_omega when memory runs out, and the memory it keeps: a move that
cannot be made returns HB_ERR_OOM and leaves the handle at its frequency (the
matrix-free apply gives the same bits), a retry with room equals a fresh handle,
and a graph of a matrix-free apply captured before a move still reads what it
read (the Hankel rows a handle has used stay until it is destroyed)."""
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


def _dense(op, s):
    import torch
    u = torch.empty_like(s)
    op.apply_dense(s, u, s.shape[0])
    torch.cuda.synchronize()
    return u


def test_failed_move_keeps_the_frequency():
    import gc
    from paper_2210_02698_gb300 import binding
    import torch
    N = 24
    w, w2 = W.small_workload(W.LENS, N, 3, 2), W.small_workload(W.LENS, N, 40, 2)
    s = to_dev(W.complex_normal_sources(w.grid.Nv, 2, 5))
    gc.collect()
    op, fresh = gpu_op(w, precision=binding.HB_FP64), gpu_op(w2, precision=binding.HB_FP64)
    try:
        before, want = _dense(op, s), _dense(fresh, s)
        live = binding.device_alloc_cap(-1)
        binding.device_alloc_cap(live + 8192)   # room for the quadrature, not for more Hankel rows
        with pytest.raises(binding.HBError) as e:
            op.set_omega(w2.omega)
        assert e.value.status == binding.HB_ERR_OOM
        assert binding.device_alloc_cap(-1) == live
        assert torch.equal(_dense(op, s), before)
        binding.device_alloc_cap(0)
        op.set_omega(w2.omega)
        assert torch.equal(_dense(op, s), want)
        # back and forth: nothing more is taken
        live = binding.device_alloc_cap(-1)
        for o in (w.omega, w2.omega, w.omega):
            op.set_omega(o)
        assert binding.device_alloc_cap(-1) == live
        assert torch.equal(_dense(op, s), before)
    finally:
        binding.device_alloc_cap(0)
        op.close()
        fresh.close()


def test_graph_of_an_earlier_frequency():
    import torch
    from paper_2210_02698_gb300 import binding
    N = 20
    w = W.small_workload(W.LENS, N, 3, 1)
    op = gpu_op(w, precision=binding.HB_FP64)
    nv = w.grid.Nv
    at = nv // 2 + 3
    s = torch.zeros((1, nv), dtype=torch.complex128, device="cuda")
    s[0, at] = 1.0 + 2.0j
    want, u = _dense(op, s), torch.empty_like(s)
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=st):
        op.apply_dense(s, u, 1, st)
    for waves in (10, 20, 40):
        op.set_omega(W.small_workload(W.LENS, N, waves, 1).omega)
    u.zero_()
    g.replay()
    torch.cuda.synchronize()
    off = torch.arange(nv, device="cuda") != at   # the self terms are the handle's, at its present frequency
    assert float((u - want)[0, off].abs().max() / want[0, off].abs().max()) < 1e-13
    op.close()
