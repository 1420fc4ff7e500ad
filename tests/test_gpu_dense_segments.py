"""The matrix-free apply on lines about the longest source segment (200 cells, in
tiles of 8): one segment, two, three, the last tile ragged, one and two tiles
of right-hand sides, against the product with the entries of hb_entries."""
import numpy as np
import pytest

from tests.test_gpu_dense_entries import _operator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,n_I,nrhs", [(144, 3, 16, 1), (145, 2, 5, 9), (199, 3, 16, 16), (200, 3, 16, 3),
                                            (201, 3, 16, 16), (401, 2, 8, 2)])
def test_long_lines_equal_the_entries(nx, ny, n_I, nrhs):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import build
    build.build()
    omega = 40.0
    op = _operator(nx, ny, n_I, omega)
    nv = nx * ny
    K = torch.empty((nv, nv), dtype=torch.complex128, device="cuda")   # column-major: K[j, i] = K_ij
    op.entries(np.arange(nv), np.arange(nv), K)
    g = torch.Generator(device="cuda").manual_seed(nv)
    s = torch.randn((nrhs, nv), dtype=torch.complex128, device="cuda", generator=g)
    u, a = torch.full_like(s, float("nan")), torch.full_like(s, float("nan"))
    op.apply_dense(s, u, nrhs)
    op.apply_dense_adjoint(s, a, nrhs)
    torch.cuda.synchronize()
    h2 = op.h ** 2
    # as in test_gpu_dense_entries: tau^2 to a few 1e-16 at distances of a cell and more
    tol = 2e-14 + 4e-15 * omega * (1.0 / (2.2 * op.h) + 1.6)
    for got, want in ((u, h2 * (s @ K)), (a, h2 * (s @ K.mH))):
        assert float(torch.linalg.norm(got - want) / torch.linalg.norm(want)) < tol
    op.close()
