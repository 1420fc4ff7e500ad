"""The table builder where the sources alone fill the chip (one lane per mesh
point instead of four): equal to the oracle's FP64 builder bit for bit, with
sources that repeat and a count that is no multiple of anything the launch
is cut by."""
import numpy as np
import pytest

from paper_2210_02698_gb300 import workloads as W
from tests.test_gpu_sweep import _case, _oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("medium,ns", [(W.LENS, 403), (W.GRADIENT, 1217)])
def test_many_sources_equal_the_oracle_bitwise(medium, ns):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import build
    build.build()
    from paper_2210_02698_gb300 import binding
    mesh, n, px, pz, _, _ = _case(medium, 4, 1 / 20, [0])
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    assert ns * mesh[0] > 256 * nsm                 # past the bound of four lanes per point
    mesh, n, px, pz, s, tin = _case(medium, 4, 1 / 20, [(7 * k) % 16 for k in range(16)])
    want = _oracle(mesh, n, px, pz, s, tin, 3, 1e-12)
    at = np.arange(ns) % 16
    got = binding.sweep_tables(*mesh, n, px, pz, s[at], np.ascontiguousarray(tin[at]), 3, 1e-12)
    for g, w in zip(got[:3], want[:3]):
        assert np.array_equal(g, w[:, at])
    assert np.array_equal(got[3], want[3][at])
