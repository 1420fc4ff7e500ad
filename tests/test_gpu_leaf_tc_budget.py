"""The tensor-core leaf launch may begin while earlier depths still run; its
wait budget counts from the moment they are done.  With the wait self-test on,
every depth launch is held up by a whole budget, and the leaf launch behind
them must not run out of its own while it waits for them: the outputs are those
of an apply without the self-test (launched call by call, and from a graph,
where the launches follow one another closest)."""
import pytest

from paper_2210_02698_gb300 import workloads as W
from tests._common import gpu_op, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nrhs", [(32, 2), (48, 2), (64, 20)])
@pytest.mark.parametrize("graph", [False, True])
def test_leaf_launch_outlives_held_up_depths(N, nrhs, graph):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import binding
    w = W.small_workload(W.GRADIENT, N, N / 8, nrhs)
    s = to_dev(W.complex_normal_sources(w.grid.Nv, nrhs, 23))
    op = gpu_op(w, precision=binding.HB_MIXED_BF16X3, barrier_cycles=1 << 20, autotune=3)
    op.build()
    want, got = torch.empty_like(s), torch.zeros_like(s)
    for f in (op.apply, op.apply_adjoint):
        f(s, want, nrhs)
        torch.cuda.synchronize()
        op.set_wait_selftest(True)
        if graph:
            g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            with torch.cuda.graph(g, stream=st):
                f(s, got, nrhs, st)
            g.replay()
        else:
            f(s, got, nrhs)
        torch.cuda.synchronize()
        op.set_wait_selftest(False)
        with pytest.raises(binding.HBError) as e:   # the self-test's own wait ran out
            f(s, got.clone(), nrhs)
        assert e.value.status == binding.HB_ERR_TIMEOUT
        assert torch.equal(got, want)
    op.close()
