"""Batches of equal matrices, decomposed by one CTA each, by clusters of two, of
four and of eight as their number asks for: the bits of each matrix alone."""
import numpy as np
import pytest

from paper_2210_02698_gb300 import workloads as W
from tests.test_gpu_id_teams import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [40, 76, 110, 152, 304])   # 8, 2, 4, 1 and 1 CTAs a matrix on 152 SMs
def test_equal_matrices(count):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import build
    build.build()
    mats = [W.random_id_matrices(1, 90, 41, 41, 0.6, 70 + k)[0].T for k in range(3)]
    got = _run((mats * count)[:count], 1e-6)
    for k, a in enumerate(mats):
        r, skel, V = _run([a], 1e-6)[0]
        for other in (got[k], got[k + (count - 1 - k) // 3 * 3]):
            assert other[0] == r and np.array_equal(other[1], skel) and np.array_equal(other[2], V)
