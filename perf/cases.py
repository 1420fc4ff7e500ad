"""What is timed when this library's speed is looked at: its public calls, over the sizes and options they are used with.

Every case is one call (or the few calls that make one step) of the binding on a grid of nx x ny cells of the stored
media, 8 cells per wavelength across the grid unless `waves` says otherwise, the cluster tree, tolerance and proxy
options at their defaults.  The operator of a medium and grid is built once and kept, as a program keeps it that
applies it to one batch of sources after another; the sources (or residuals, curves, frequencies) are new for every
seed.  `exact` evaluates the same sums with torch in 64 bits, entry by entry, without the library.
"""
import functools
import math

import numpy as np
import torch

from paper_2210_02698_gb300 import binding

TABLES = {"homog": "tests/golden/tables/homog_n1_nI16.npz",
          "grad": "tests/golden/tables/grad_c1_g0.5_nI16.npz",
          "lens": "tests/golden/tables/lens_a0.1_w0.3_nI16.npz"}
DEV = "cuda"


# ---------------------------------------------------------------- cases ----
def listed():
    return [
        # The benchmark workload: a batch of 16 random sources through the compressed operator, mixed precision.
        dict(name="mixed_fwd_256", kind="apply", medium="grad", nx=256, ny=256, nrhs=16, prec="mixed", sources="normal"),
        # Many uneven sources (points, lines, bumps, wavepackets) in the lens medium: several passes over the factors.
        dict(name="mixed_fwd_256_many", kind="apply", medium="lens", nx=256, ny=256, nrhs=64, prec="mixed", sources="uneven"),
        # The adjoint on a grid that is neither square nor a power of two, with an odd number of right-hand sides.
        dict(name="mixed_adj_200x136", kind="adjoint", medium="lens", nx=200, ny=136, nrhs=3, prec="mixed", sources="normal"),
        # One step of a small source inversion (forward, misfit at receivers, its gradient by the adjoint): the
        # smallest calls, where launches count.
        dict(name="inversion_64", kind="step", medium="grad", nx=64, ny=64, nrhs=1, prec="mixed", sources="normal"),
        # The same operator in full precision, for users who need more than the mixed path's digits.
        dict(name="fp64_fwd_192", kind="apply", medium="grad", nx=192, ny=192, nrhs=16, prec="fp64", sources="normal"),
        dict(name="fp64_adj_120x88", kind="adjoint", medium="lens", nx=120, ny=88, nrhs=5, prec="fp64", sources="uneven"),
        # The matrix-free sum: no build, exact to rounding; the homogeneous 64 x 64 configuration with one source ...
        dict(name="dense_fwd_64", kind="dense", medium="homog", nx=64, ny=64, nrhs=1, prec="fp64", sources="bump"),
        # ... and the adjoint of a ragged grid for a batch.
        dict(name="dense_adj_144x100", kind="dense_adjoint", medium="lens", nx=144, ny=100, nrhs=16, prec="fp64", sources="uneven"),
        # Scattering by an inclusion whose surface operators are compressed: one batch of sources, the curve is kept.
        dict(name="inclusion_128", kind="inclusion", medium="grad", nx=128, ny=128, nrhs=8, prec="mixed", sources="normal", ns=512),
        # A new inclusion (one step of a shape search): its operators assembled and factored, then one batch.
        dict(name="curve_96", kind="curve", medium="lens", nx=96, ny=96, nrhs=2, prec="fp64", sources="normal", ns=300),
        # A new frequency (one step of a frequency sweep): the handle moved and rebuilt, then one batch.
        dict(name="rebuild_64", kind="rebuild", medium="lens", nx=64, ny=64, nrhs=2, prec="fp64", sources="normal"),
        # Tables of a medium without closed forms, by sweeping: one source per Chebyshev node.
        dict(name="tables_32", kind="tables", n_I=6, cells=32, max_iter=25),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "adjoint", "step", "apply64", "adjoint64", "dense", "dense_adjoint",
                       "inclusion", "curve", "rebuild", "tables"])
    if kind == "tables":
        return dict(kind="tables", n_I=rng.randint(3, 6), cells=rng.randint(24, 32), max_iter=rng.randint(12, 25))
    top = {"apply": 256, "adjoint": 256, "step": 192, "apply64": 192, "adjoint64": 192, "dense": 120,
           "dense_adjoint": 120, "inclusion": 128, "curve": 96, "rebuild": 64}[kind]
    many = {"apply": 64, "adjoint": 64, "step": 4, "apply64": 16, "adjoint64": 16, "dense": 16, "dense_adjoint": 16,
            "inclusion": 8, "curve": 8, "rebuild": 8}[kind]
    nx = _log(rng, 24, top)
    case = dict(kind=kind.replace("64", ""), medium=rng.choice(["grad", "lens", "homog"]), nx=nx,
                ny=max(16, int(nx * rng.uniform(0.5, 1.0))), nrhs=_log(rng, 1, many),
                prec="fp64" if "64" in kind or kind.startswith("dense") or kind == "rebuild" else "mixed",
                sources=rng.choice(["normal", "uneven"]))
    case["ny"] = min(case["nx"], case["ny"])
    if kind in ("inclusion", "curve"):
        case["ns"] = _log(rng, 64, 512 if kind == "inclusion" else 300)
    return case


# --------------------------------------------------------------- inputs ----
def _omega(case):
    return 2 * math.pi * case["nx"] / 8


def _n(medium, x, z):
    """Refractive index of the stored media."""
    if medium == "homog":
        return torch.ones_like(x)
    if medium == "grad":
        return 1.0 / (1.0 + 0.5 * z)
    return 1.0 + 0.1 * torch.exp(-((x - 0.5) ** 2 + (z - 0.5) ** 2) / 0.3 ** 2)


def _cells(case, device="cpu"):
    """Cell centres, natural order (x fastest)."""
    h = 1.0 / case["nx"]
    a = (torch.arange(case["nx"], dtype=torch.float64, device=device) + 0.5) * h
    b = (torch.arange(case["ny"], dtype=torch.float64, device=device) + 0.5) * h
    return a.repeat(case["ny"]), b.repeat_interleave(case["nx"])


@functools.lru_cache(maxsize=2)
def _tables(medium):
    with np.load(TABLES[medium]) as z:
        return tuple(np.ascontiguousarray(z[k]) for k in ("nodes", "tau2", "v0", "v1"))


@functools.lru_cache(maxsize=2)
def _operator(medium, nx, ny, prec, built, use):
    """`use` keeps handles apart that a case moves to another curve or frequency."""
    case = dict(nx=nx, ny=ny)
    x, z = _cells(case)
    op = binding.Operator((nx, ny), *_tables(medium), _n(medium, x, z).numpy(), _omega(case),
                          precision=binding.HB_FP64 if prec == "fp64" else binding.HB_MIXED_BF16X3)
    if built:
        op.build()
    return op


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _vectors(case, seed):
    """nrhs right-hand sides (one a row): complex Gaussian noise, a source bump, or quarters of point sources, line
    segments, Gaussian bumps and wavepackets."""
    g, R, h, omega = _gen(seed), case["nrhs"], 1.0 / case["nx"], _omega(case)
    nv = case["nx"] * case["ny"]
    if case["sources"] == "normal":
        return torch.randn((R, nv), dtype=torch.complex128, device=DEV, generator=g) * math.sqrt(2.0)
    x, z = _cells(case, DEV)
    top = case["ny"] * h
    u = torch.rand((R, 6), dtype=torch.float64, device=DEV, generator=g).cpu().tolist()
    s = torch.zeros((R, nv), dtype=torch.complex128, device=DEV)
    for k in range(R):
        kind = 2 if case["sources"] == "bump" else min(3, 4 * k // max(R, 4))
        cx, cz, dx, dz, e, f = u[k]
        if kind == 0:
            s[k, int(cz * case["ny"]) * case["nx"] + int(cx * case["nx"])] = 1.0 / h ** 2
        elif kind == 1:
            p, q = (0.1 + 0.8 * cx, (0.1 + 0.8 * cz) * top), (0.1 + 0.8 * dx, (0.1 + 0.8 * dz) * top)
            d = (q[0] - p[0], q[1] - p[1])
            t = (((x - p[0]) * d[0] + (z - p[1]) * d[1]) / (d[0] ** 2 + d[1] ** 2 + 1e-12)).clamp(0, 1)
            s[k] = torch.where(torch.hypot(x - p[0] - t * d[0], z - p[1] - t * d[1]) <= h / 2, 1.0 / h, 0.0)
        elif kind == 2:
            r2 = (x - 0.2 - 0.6 * cx) ** 2 + (z - (0.2 + 0.6 * cz) * top) ** 2
            s[k] = torch.exp(-r2 / (2 * (0.02 + 0.08 * dx) ** 2)) * complex(2 * e - 1, 2 * f - 1)
        else:
            th = 2 * math.pi * e
            r2 = (x - 0.5) ** 2 + (z - 0.5 * top) ** 2
            s[k] = torch.exp(-r2 / (2 * 0.15 ** 2) + 0.9j * omega * (x * math.cos(th) + z * math.sin(th)))
    return s


def _circle(case, seed):
    """A circular inclusion of ns segments inside the grid: centres (ns, 2), lengths, index at the centres."""
    r = np.random.default_rng(seed)
    top = case["ny"] / case["nx"]
    radius = r.uniform(0.18, 0.3) * top
    cx, cz = r.uniform(radius + 0.1, 0.9 - radius), r.uniform(radius + 0.1 * top, 0.9 * top - radius)
    t = np.linspace(0.0, 2 * math.pi, case["ns"] + 1)
    p = np.stack([cx + radius * np.cos(t), cz + radius * np.sin(t)], axis=1)
    cen, ln = 0.5 * (p[1:] + p[:-1]), np.hypot(*(p[1:] - p[:-1]).T)
    return cen, ln, _n(case["medium"], torch.from_numpy(cen[:, 0]), torch.from_numpy(cen[:, 1])).numpy()


def _receivers(case, seed):
    """Up to 256 receiver cells and the data measured there."""
    nv = case["nx"] * case["ny"]
    at = np.sort(np.random.default_rng(seed).choice(nv, size=min(256, nv // 4), replace=False))
    data = torch.randn((case["nrhs"], len(at)), dtype=torch.complex128, device=DEV, generator=_gen(seed + 1))
    return torch.from_numpy(at).to(DEV), 1e-2 * data


def _new_omega(case, seed):
    return _omega(case) * np.random.default_rng(seed).uniform(0.97, 1.0)


def _sweep_inputs(case, seed):
    """The mesh and the near-source series of a velocity-gradient medium c = 1 + g z, g from the seed."""
    g = np.random.default_rng(seed).uniform(0.35, 0.45)
    n_I, n1 = case["n_I"], case["cells"]
    h = 1.0 / n1
    k = max(int(math.ceil(0.3 / h)), 38)
    M, lo, w0, w1 = n1 + 1 + 2 * k, -k * h, k - 14, k + n1 + 14
    nodes = 0.5 - 0.5 * np.cos((2 * np.arange(1, n_I + 1) - 1) * np.pi / (2 * n_I))
    px, pz = np.tile(nodes, n_I), np.repeat(nodes, n_I)
    c = 1.0 + g * (lo + h * np.arange(M))
    s2 = np.zeros((n_I * n_I, 15))
    for i, z in enumerate(pz):
        cs = 1.0 + g * z
        for j in range(5):
            s2[i, j * (j + 1) // 2 + j] = (j + 1) * (-g / cs) ** j / cs ** 2
    return dict(mesh=(M, lo, h, w0, w1, 12, 12 + n1 + 4), n=np.repeat(1.0 / c[:, None], M, axis=1), px=px, pz=pz,
                src=np.arange(n_I * n_I, dtype=np.int32), s2=s2)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "tables":
        return dict(case=case, **_sweep_inputs(case, seed))
    s = _vectors(case, seed)
    op = _operator(case["medium"], case["nx"], case["ny"], case["prec"], kind not in ("dense", "dense_adjoint", "rebuild"),
                   kind if kind in ("inclusion", "curve", "rebuild") else "apply")
    st = dict(case=case, op=op, s=s, u=torch.empty_like(s))
    if kind == "step":
        st["at"], st["data"] = _receivers(case, seed)
    if kind == "inclusion":
        # the curve is the operator's: one per grid, the sources change
        if getattr(op, "curve_key", None) != case["ns"]:
            op.set_curve(*_circle(case, 5))
            op.curve_compress(16)
            op.curve_key = case["ns"]
    if kind == "curve":
        st["curve"] = _circle(case, seed)
    if kind == "rebuild":
        st["omega"] = _new_omega(case, seed)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "tables":
        taylor = binding.sweep_taylor(st["s2"])
        return binding.sweep_tables(*st["mesh"], st["n"], st["px"], st["pz"], st["src"], taylor, case["max_iter"], 1e-12)
    op, s, u, R = st["op"], st["s"], st["u"], case["nrhs"]
    stream = torch.cuda.current_stream()
    if kind == "apply":
        op.apply(s, u, R, stream)
    elif kind == "adjoint":
        op.apply_adjoint(s, u, R, stream)
    elif kind == "dense":
        op.apply_dense(s, u, R, stream)
    elif kind == "dense_adjoint":
        op.apply_dense_adjoint(s, u, R, stream)
    elif kind == "step":
        op.apply(s, u, R, stream)
        res = torch.zeros_like(u)
        res[:, st["at"]] = 2 * (u[:, st["at"]] - st["data"])
        grad = torch.empty_like(u)
        op.apply_adjoint(res, grad, R, stream)
        return u, grad
    elif kind == "inclusion":
        op.apply_inclusion(s, u, R, False, stream)
    elif kind == "curve":
        op.set_curve(*st["curve"])
        op.apply_inclusion(s, u, R, False, stream)
    else:
        op.set_omega(st["omega"])
        op.build()
        op.apply(s, u, R, stream)
        return u, op.rank_profile()
    return u


# ----------------------------------------------------------------- work ----
def _entries(nv):
    """Stored complex factor entries of the compressed operator: 2.5 to 3.4 N_v log2(N_v)^2 on the grids measured."""
    return 3.0 * nv * math.log2(nv) ** 2


def work(case):
    kind = case["kind"]
    if kind == "tables":
        M = case["cells"] + 1 + 2 * max(int(math.ceil(0.3 * case["cells"])), 38)
        Mw = case["cells"] + 29
        ns = case["n_I"] ** 2
        # the nonlinear solves: four orderings an iteration, about 700 operations a point (two WENO5 derivative pairs),
        # no fewer than 10 iterations each
        pts = 40 * (M * M + 2 * Mw * Mw)
        return {"bytes": 8 * M * M + 24 * ns * ns, "flops": 700.0 * pts * ns}
    nv, R = case["nx"] * case["ny"], case["nrhs"]
    vec = 32.0 * nv * R
    E = _entries(nv)
    if kind.startswith("dense"):
        # every entry: three 16-term contractions, one Hankel pair (about 40), 8 per right-hand side
        return {"bytes": vec, "flops": float(nv) * nv * (96 + 40 + 8 * R)}
    bpe = 8 if case["prec"] == "mixed" else 16
    if kind in ("apply", "adjoint"):
        return {"bytes": bpe * E + vec, "flops": 8 * E * R}
    if kind == "step":
        return {"bytes": 2 * (bpe * E + vec), "flops": 16 * E * R}
    if kind in ("inclusion", "curve"):
        ns = case["ns"]
        if kind == "inclusion":
            surf = 2 * _entries(nv) / 4
            return {"bytes": bpe * E + vec + 16 * (surf + ns * ns), "flops": 8 * R * (E + surf + ns * ns)}
        return {"bytes": bpe * E + vec + 32.0 * nv * ns, "flops": 8 * R * (E + 2 * nv * ns + ns * ns) + 2.0 * nv * ns * 136 + 16 / 3 * ns ** 3}
    # rebuild: sampled blocks of about 20 proxy rows a column, their decompositions, the factors written
    smp = 20 * E
    return {"bytes": 16 * E, "flops": 136 * smp + 8 * smp * 16}


# ---------------------------------------------------------------- exact ----
def _basis(nodes, x):
    d = x[:, None] - nodes[None, :]
    w = torch.stack([1.0 / torch.prod(torch.cat([nodes[k] - nodes[:k], nodes[k] - nodes[k + 1:]])) for k in range(len(nodes))])
    hit = d == 0
    q = w / torch.where(hit, torch.ones_like(d), d)
    out = q / q.sum(1, keepdim=True)
    return torch.where(hit.any(1, keepdim=True), hit.to(out.dtype), out)


def _tensor_basis(nodes, x, z):
    return (_basis(nodes, z)[:, :, None] * _basis(nodes, x)[:, None, :]).reshape(len(x), -1)


def _hankel_near(x):
    """J0 + i Y0 and J1 + i Y1 for 0 < x < 25: downward recurrence from order 80, normalised by J0 + 2 sum J_2k = 1,
    and Neumann's series for Y0 and Y1 = -Y0'."""
    up, cur = torch.zeros_like(x), torch.full_like(x, 1e-280)
    norm, y0, y1, j1 = (torch.zeros_like(x) for _ in range(4))
    for n in range(80, 0, -1):
        k = (n + 1) // 2
        if n % 2 == 0:
            norm, y0 = norm + 2 * cur, y0 + (-1) ** k * cur / k
        elif k > 1:
            y1 = y1 + (-1) ** k * (2 * k - 1) / (k * (k - 1)) * cur
        else:
            j1 = cur
        up, cur = cur, 2 * n / x * cur - up
        if n % 8 == 0:
            f = torch.where(cur.abs() > 1e150, 1e-150, 1.0).to(x.dtype)
            up, cur, norm, y0, y1 = (v * f for v in (up, cur, norm, y0, y1))
    norm = norm + cur
    j0, j1, y0, y1 = (v / norm for v in (cur, j1, y0, y1))
    ln = torch.log(x / 2) + 0.57721566490153286061
    y0 = 2 / math.pi * (ln * j0 - 2 * y0)
    y1 = 2 / math.pi * ((ln - 1) * j1 - j0 / x + y1)
    return torch.complex(j0, y0), torch.complex(j1, y1)


def _hankel(x):
    """H0 and H1 (first kind) of x > 0: the recurrence below 25, Hankel's expansion from there on."""
    y = x.clamp(min=25.0)
    e = torch.complex(torch.cos(y), torch.sin(y)) * torch.sqrt(1.0 / (math.pi * y))
    out = []
    for nu, turn in ((0, 1 - 1j), (1, -1 - 1j)):
        re, im, a = torch.ones_like(y), torch.zeros_like(y), torch.ones_like(y)
        for k in range(1, 21):
            a = a * ((4.0 * nu * nu - (2 * k - 1) ** 2) / (8.0 * k)) / y
            if k % 2:
                im = im + (1 - k % 4 // 2 * 2) * a
            else:
                re = re + (1 - k % 4) * a
        out.append(e * turn * torch.complex(re, im))
    near = x < 25.0
    small = x[near].clamp(min=1e-3)   # below the distance of any two cells or segments
    h0, h1 = _hankel_near(small)
    out[0][near], out[1][near] = h0, h1
    return out


def _green(case, omega, xo, zo, Gs):
    """g between the points (xo, zo) and the sources whose table contractions are Gs (3, N_I, n)."""
    nodes = torch.from_numpy(_tables(case["medium"])[0]).to(xo.device)
    t2, v0, v1 = torch.matmul(_tensor_basis(nodes, xo, zo)[None], Gs)
    tau = t2.clamp(min=0).sqrt()
    h0, h1 = _hankel((omega * tau).clamp(min=1e-12))
    c = math.sqrt(math.pi) / 2
    return 1j * c * v0 * h0 - (2j * c / omega) * tau * v1 * h1


def _contract(case, xs, zs):
    nodes, t2, v0, v1 = (torch.from_numpy(a).to(xs.device) for a in _tables(case["medium"]))
    return torch.stack([t2, v0, v1]) @ _tensor_basis(nodes, xs, zs).T


def _self_terms(case, omega, x, z):
    h = 1.0 / case["nx"]
    n0 = _n(case["medium"], x, z)
    gx, gw = (torch.from_numpy(a).to(x.device) for a in np.polynomial.legendre.leggauss(64))
    R = (0.5 * h * omega * n0)[:, None] / torch.cos(math.pi / 8 * (gx + 1))[None, :]
    val = math.pi / 8 * (gw * R * _hankel(R)[1]).sum(1)
    return 0.25j * (8 * val + 4j) / (n0 * omega) ** 2 / h ** 2


def _dense(case, omega, s, adjoint):
    """h^2 K s, or h^2 K^H s, of the uncompressed operator (one right-hand side a row)."""
    x, z = _cells(case, s.device)
    nv, h = len(x), 1.0 / case["nx"]
    Gs, diag = _contract(case, x, z), _self_terms(case, omega, x, z)
    out = torch.zeros_like(s)
    step = max(1, (1 << 24) // nv)
    for r0 in range(0, nv, step):
        r = torch.arange(r0, min(nv, r0 + step), device=s.device)
        K = _green(case, omega, x[r], z[r], Gs)
        K[r - r0, r] = diag[r]
        if adjoint:
            out += s[:, r] @ K.conj()
        else:
            out[:, r] = s @ K.T
    return h * h * out


def _with_curve(case, omega, s, curve):
    cen, ln, nseg = (torch.from_numpy(np.ascontiguousarray(a)).to(s.device) for a in curve)
    x, z = _cells(case, s.device)
    h = 1.0 / case["nx"]
    cx, cz = cen[:, 0].contiguous(), cen[:, 1].contiguous()
    Gc = _contract(case, cx, cz)
    S = -_green(case, omega, cx, cz, Gc) * ln[None, :]
    gamma = math.exp(0.57721566490153286061)
    i = torch.arange(len(ln), device=s.device)
    S[i, i] = -0.25j * ln * (1 + (2j / math.pi) * (torch.log(gamma * omega * nseg * ln / 4) - 1))
    Y = h * h * (_green(case, omega, cx, cz, _contract(case, x, z)) @ s.T)
    P = torch.linalg.solve(S, Y)
    return _dense(case, omega, s, False) + ((_green(case, omega, x, z, Gc) * ln[None, :]) @ P).T


def exact(case, seed):
    kind = case["kind"]
    if kind == "tables":
        return None   # the iterates of a fixed number of sweeps: no value but the scheme's own
    omega, s = _omega(case), _vectors(case, seed)
    if kind in ("apply", "dense"):
        return _dense(case, omega, s, False)
    if kind in ("adjoint", "dense_adjoint"):
        return _dense(case, omega, s, True)
    if kind == "step":
        at, data = _receivers(case, seed)
        u = _dense(case, omega, s, False)
        r = torch.zeros_like(u)
        r[:, at] = 2 * (u[:, at] - data)
        return u, _dense(case, omega, r, True)
    if kind == "inclusion":
        return _with_curve(case, omega, s, _circle(case, 5))
    if kind == "curve":
        return _with_curve(case, omega, s, _circle(case, seed))
    return _dense(case, _new_omega(case, seed), s, False), None
