"""The interpolative decompositions of matrices on both sides of the size a
cluster of CTAs takes over at, mixed in one call, against the oracle's CPQR:
ranks, pivot orders and the interpolation; a matrix decomposes to the same
bits alone and in company (a launch of one CTA per matrix, of clusters of
eight and of four)."""
import numpy as np
import pytest

from paper_2210_02698_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (31, 33), (32, 32), (40, 26), (7, 200), (513, 2), (300, 65), (64, 64), (33, 31), (1100, 17)]


def _run(mats, eps):
    import torch
    from paper_2210_02698_gb300 import binding
    m, n = [a.shape[0] for a in mats], [a.shape[1] for a in mats]
    off = np.concatenate([[0], np.cumsum([a.size for a in mats])])
    flat = np.concatenate([np.asfortranarray(a).ravel(order="F") for a in mats])
    A = torch.from_numpy(flat).cuda()
    rank = torch.zeros(len(mats), dtype=torch.int32, device="cuda")
    skel = torch.zeros(sum(n), dtype=torch.int32, device="cuda")
    V = torch.zeros(sum(k * k for k in n), dtype=torch.complex128, device="cuda")
    binding.id_batch(A, m, n, off[:-1], eps, rank, skel, V)
    torch.cuda.synchronize()
    out, so, vo = [], 0, 0
    for b, k in enumerate(n):
        r = int(rank[b])
        v = V[vo:vo + k * k].cpu().numpy().reshape(k, k).T[:r]
        out.append((r, skel[so:so + r].cpu().numpy(), v.copy()))
        so, vo = so + k, vo + k * k
    return out


def test_decompositions_across_the_sizes():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from oracle import cpqr
    from paper_2210_02698_gb300 import build
    build.build()
    mats = [W.random_id_matrices(1, m, n, min(m, n), 0.6, 50 + k)[0].T for k, (m, n) in enumerate(SHAPES)]
    eps = 1e-6
    together = _run(mats, eps)
    many = _run(mats * 60, eps)   # past the launch size that takes clusters of four
    for k, a in enumerate(mats):
        r, skel, V = together[k]
        alone = _run([a], eps)[0]
        for other in (alone, many[k], many[k + 10 * 59]):
            assert other[0] == r and np.array_equal(other[1], skel) and np.array_equal(other[2], V)
        want = cpqr.cpqr_id(a, eps)
        assert r == len(want[0]) and np.array_equal(skel, want[0])
        # A = A[:, skel] V to the truncation (2-norm below eps |R_00| sqrt(n (n - r)) for a rank-revealing cut)
        assert np.linalg.norm(a - a[:, skel] @ V) <= 10 * eps * np.sqrt(a.shape[1]) * np.linalg.norm(a)
