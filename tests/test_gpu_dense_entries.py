"""The dense apply against the product with the entries hb_entries gives
(evaluated by the recurrence and the asymptotic series): line segments of
every shape (one cell, ragged, several per line), the padded orders of the
basis, arguments omega tau below the tabulated expansions, inside them and
past their end, and every right-hand-side grouping."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _operator(nx, ny, n_I, omega):
    from paper_2210_02698_gb300 import binding
    k = np.arange(1, n_I + 1)
    nodes = 0.5 - 0.5 * np.cos((2 * k - 1) * np.pi / (2 * n_I))
    x, z = np.tile(nodes, n_I), np.repeat(nodes, n_I)
    dx, dz = x[:, None] - x[None, :], z[:, None] - z[None, :]
    tau2 = 1.21 * (dx ** 2 + dz ** 2)
    v0 = 0.28 + 0.05 * (x[:, None] + z[None, :]) * (1 if n_I > 2 else 0)
    v1 = 0.3 - 0.1 * (z[:, None] + x[None, :])
    return binding.Operator((nx, ny), nodes, tau2, v0, v1, np.full(nx * ny, 1.1), omega, precision=binding.HB_FP64)


@pytest.mark.parametrize("nx,ny,n_I,omega,nrhs", [
    (1, 1, 3, 10.0, 1), (5, 3, 5, 0.02, 3), (16, 16, 3, 1.7, 2), (33, 4, 16, 60.0, 16), (70, 6, 16, 25.0, 5),
    (129, 2, 8, 400.0, 33), (40, 7, 9, 3000.0, 4), (64, 3, 3, 90.0, 8), (49, 20, 4, 31.0, 24)])
def test_dense_apply_equals_the_entries(nx, ny, n_I, omega, nrhs):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import build
    build.build()
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
    # tau^2 is known to a few 1e-16; the phase omega tau of the closest cells (tau >= 1.1 h) then to omega 1e-15 / (2 tau),
    # and omega tau itself rounds to 2e-16 of its value
    tol = 2e-14 + 4e-15 * omega * (1.0 / (2.2 * op.h) + 1.6)
    for got, want in ((u, h2 * (s @ K)), (a, h2 * (s @ K.mH))):
        assert float(torch.linalg.norm(got - want) / torch.linalg.norm(want)) < tol
    op.close()


@pytest.mark.parametrize("nrhs", [3, 18])
def test_right_hand_sides_outside_the_digits(nrhs):
    """Columns that are all zero, tiny (1e-300), huge, or hold a value that is
    not finite: the last fails the digits and the whole apply is summed in
    FP64; every column equals the product with the entries."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2210_02698_gb300 import build
    build.build()
    op = _operator(20, 9, 6, 17.0)
    nv = 180
    K = torch.empty((nv, nv), dtype=torch.complex128, device="cuda")
    op.entries(np.arange(nv), np.arange(nv), K)
    g = torch.Generator(device="cuda").manual_seed(5)
    s = torch.randn((nrhs, nv), dtype=torch.complex128, device="cuda", generator=g)
    s[0] = 0
    s[-1] *= 1e250
    for last in (1e-300, 1e-290, complex("nan"), complex("inf")):
        s[1] = torch.randn(nv, dtype=torch.complex128, device="cuda", generator=g)
        if np.isfinite(last):
            s[1] *= last
        else:
            s[1, 77] = last
        for fn, A in ((op.apply_dense, K), (op.apply_dense_adjoint, K.mH)):
            u = torch.full_like(s, 7.0)
            fn(s, u, nrhs)
            torch.cuda.synchronize()
            assert not u[0].any()
            for k in range(1, nrhs):
                if k == 1 and not np.isfinite(last):
                    assert not torch.isfinite(torch.view_as_real(u[1])).all(-1).any()
                    continue
                w = abs(last) if k == 1 else 1e250 if k == nrhs - 1 else 1.0
                want = op.h ** 2 * ((s[k] / w) @ A)
                # the entries: as above; a column at 1e-300 is summed in subnormals' neighbourhood, 1e-308 / 1e-300 of it
                tol = 1e-7 if w < 1e-280 else 1e-12
                assert float(torch.linalg.norm(u[k] / w - want) / torch.linalg.norm(want)) < tol
    op.close()
