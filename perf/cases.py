"""Cases that time the library through its Python entry points, as a program that uses it calls them.

Kinds of case (the `kind` of a case dict):
  solve   build the one-obstacle operator (fill + QR, or its truncated-SVD form) in a plan's workspace, form the
          incident data of W plane waves, apply A_0^+ and evaluate the far field in 64 directions;
  batch   the same for a plan of several obstacles of uneven size and both boundary conditions;
  apply   A_0^+ of a built operator on W sets of boundary data, then the far field;
  near    the sum over the eight phased nearest images at the ring nodes (A_else of eq. iter);
  field   the scattered potential (or its normal derivative) at target points and the far field;
  blocks  the periodizing blocks B~, Q and C of a unit cell;
  iter    one application of eq. iter's preconditioned periodic operator;
  pinv    the SVD of a periodizing matrix, the truncated solve and the fit Q xi of the solution.

Outputs are what the discrete problem determines: fields, boundary data, blocks and singular values. MFS
coefficients are not among them, because they are not unique to rounding (the modal blocks are ill conditioned).
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1506_05083_gb300 import axi

DEV = "cuda"
C128 = torch.complex128
N_DIRS = 64                       # far-field directions of a solve


def listed():
    return [
        # the smallest configuration: the sound-hard sphere of the closed-form check, one wave, native FP64
        dict(name="sphere", kind="solve", shape="polar", amp=0.0, k=2.0, M=72, N=60, P=32, q=128, tau=math.log(1 / 0.7),
             bc=0, split=False, tsvd=False, W=1),
        # a dielectric-like body (two fields, two proxy sets, 2M x 2N blocks) at odd sizes, native FP64
        dict(name="transmission", kind="solve", shape="polar", amp=0.1, k=8.3, M=134, N=111, P=72, q=0, tau=0.1,
             bc=1, split=False, tsvd=False, W=4),
        # the smooth sound-hard body, 16 waves, split precision
        dict(name="smooth", kind="solve", shape="polar", amp=0.1, k=10.0, M=216, N=180, P=120, q=0, tau=0.1,
             bc=0, split=True, tsvd=False, W=16),
        # the largest single obstacle: the thick-shell cup, 16 waves, split precision
        dict(name="cup", kind="solve", shape="cup", amp=0.0, k=25.0, M=432, N=360, P=180, q=1000, tau=0.05,
             bc=0, split=True, tsvd=False, W=16),
        # the operator in the form a periodic solve uses: truncated SVD per mode (1e-10)
        dict(name="tsvd", kind="solve", shape="polar", amp=0.1, k=8.0, M=144, N=120, P=60, q=0, tau=0.1,
             bc=0, split=True, tsvd=True, W=4),
        # several obstacles of uneven size, wavenumber and boundary condition in one plan
        dict(name="batch", kind="batch", n_obs=8, max_N=200, split=True, W=4),
        # many right-hand sides on existing factors
        dict(name="cup_apply", kind="apply", shape="cup", amp=0.0, k=25.0, M=432, N=360, P=180, q=1000, tau=0.05,
             bc=0, split=True, tsvd=False, W=64),
        # the near-image sum of the cup in its 13-wavelength lattice, as one step of a periodic solve calls it
        dict(name="near", kind="near", shape="cup", amp=0.0, k=25.0, M=432, N=360, P=180, tau=0.05, W=16, slices=7,
             ex=13 * 2 * math.pi / 25.0, ey=13 * 2 * math.pi / 25.0),
        # a picture of the scattered field: potential on a grid of targets, and the far field
        dict(name="field", kind="field", shape="polar", amp=0.1, k=10.0, M=216, N=180, P=120, tau=0.1, T=4096, deriv=False, W=4),
        # setting up a periodic problem: the blocks of a cell around a k = 12 body
        dict(name="blocks", kind="blocks", shape="polar", amp=0.1, k=12.0, M=208, N=173, P=90, tau=0.1, m1=16, n0=7, p=24,
             ex=13 * 2 * math.pi / 25.0, ey=13 * 2 * math.pi / 25.0),
        # one Krylov step of such a periodic problem (a k = 12 cup), 8 right-hand sides
        dict(name="iter", kind="iter", shape="cup", amp=0.0, k=12.0, M=208, N=173, P=90, tau=0.05, m1=16, n0=7, p=24, W=8,
             ex=13 * 2 * math.pi / 25.0, ey=13 * 2 * math.pi / 25.0),
        # the SVD of a periodizing matrix (12 x 12 nodes a face) and the truncated solve with it
        dict(name="pinv", kind="pinv", k=10.0, m1=12, n0=5, p=16, W=8, ex=13 * 2 * math.pi / 25.0, ey=13 * 2 * math.pi / 25.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _body(rng, lo, hi, bc=0):
    """A body of N proxies: resolved wavenumber, M = ceil(1.2 N), an even P of any factors."""
    N = int(round(_log(rng, lo, hi)))
    return dict(shape="polar", amp=round(rng.uniform(0.05, 0.1), 3), k=round(N / 15 * rng.uniform(0.5, 1.0), 3),
                M=int(math.ceil(1.2 * N)), N=N, P=2 * int(round(min(120, max(8, N / 3 * rng.uniform(0.6, 1.2))))), tau=0.1)


def _lattice(rng, body):
    """Periods of 1.25 to 4 times the body's largest possible diameter, square more often than not."""
    dia = 2 * (1 + 4 * body["amp"])
    ex = round(dia * _log(rng, 1.25, 4.0), 3)
    return dict(ex=ex, ey=ex if rng.random() < 0.6 else round(dia * _log(rng, 1.25, 4.0), 3))


def draw(rng):
    kind = rng.choice(["solve", "solve", "tsvd", "batch", "apply", "near", "near", "field", "blocks", "iter", "pinv"])
    if kind == "solve":
        bc = rng.randrange(2)
        return dict(kind="solve", **_body(rng, 32, 160 if bc else 320), q=0, bc=bc, split=rng.random() < 0.6, tsvd=False,
                    W=int(round(_log(rng, 1, 32))))
    if kind == "tsvd":
        return dict(kind="solve", **_body(rng, 24, 120), q=0, bc=0, split=rng.random() < 0.5, tsvd=True, W=int(round(_log(rng, 1, 16))))
    if kind == "batch":
        return dict(kind="batch", n_obs=rng.randint(2, 8), max_N=rng.randint(70, 200), split=rng.random() < 0.7, W=rng.randint(1, 8))
    if kind == "apply":
        return dict(kind="apply", **_body(rng, 32, 320), q=0, bc=0, split=rng.random() < 0.7, tsvd=False, W=int(round(_log(rng, 1, 64))))
    if kind == "near":
        direct = rng.random() < 0.25
        body = _body(rng, 24, 60 if direct else 320)
        return dict(kind="near", **body, **_lattice(rng, body), W=int(round(_log(rng, 1, 4 if direct else 16))),
                    slices=0 if direct else rng.choice([6, 7]))
    if kind == "field":
        return dict(kind="field", **_body(rng, 32, 200), T=int(round(_log(rng, 16, 8192))), deriv=rng.random() < 0.4,
                    W=int(round(_log(rng, 1, 8))))
    if kind in ("blocks", "iter", "pinv"):
        # a cell of 1.25 to 1.6 diameters with the Rayleigh-Bloch set and degree its wavenumber asks for, and enough wall nodes
        body = _body(rng, 24, 130)
        dia = 2 * (1 + 4 * body["amp"])
        ex = round(dia * rng.uniform(1.25, 1.6), 3)
        ey = ex if rng.random() < 0.6 else round(dia * rng.uniform(1.25, 1.6), 3)
        n0, p = int(math.ceil(body["k"] / math.pi)) + 1, int(1.5 * body["k"]) + 6
        m1 = 6
        while 8 * m1 * m1 < 1.2 * ((p + 1) ** 2 + 2 * math.pi / 4 * n0 * n0 * ex * ey + 8 * n0):
            m1 += 2
        cell = dict(ex=ex, ey=ey, m1=m1, n0=n0, p=p)
        if kind == "pinv":
            return dict(kind=kind, k=body["k"], **cell, W=rng.randint(1, 16))
        more = dict(W=rng.randint(1, 8)) if kind == "iter" else {}
        return dict(kind=kind, **body, **cell, **more)
    raise ValueError(kind)


# ---------------------------------------------------------------- inputs

def _directions(rng, n):
    th, ph = rng.uniform(0, math.pi / 2, n), rng.uniform(0, 2 * math.pi, n)
    return np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)


def _sphere_points(rng, n):
    v = rng.standard_normal((n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _cuda(x):
    return torch.tensor(x, device=DEV)


def _obstacle(case, rng):
    polar = case["shape"] == "polar"
    params = [1.0] + [case["amp"] * float(a) for a in rng.uniform(-1, 1, 4)] if polar else [0.2, math.pi / 2]
    bc = case.get("bc", 0)
    return SimpleNamespace(shape=axi.SHAPE_POLAR if polar else axi.SHAPE_CUP, params=params, k=case["k"], M=case["M"], N=case["N"],
                           P=case["P"], q=case.get("q", 0), tau=case["tau"], bc=bc, k_minus=1.5 * case["k"] if bc else 0.0)


def _batch_obstacles(case, rng):
    """Sizes and wavenumbers belong to the case, the bodies' shapes to the seed."""
    sizes = np.random.default_rng(case["n_obs"] * 1000 + case["max_N"])
    obs = []
    for i in range(case["n_obs"]):
        bc = int(i % 3 == 2)
        N = int(sizes.integers(40, case["max_N"] // (2 if bc else 1) + 10))
        obs.append(_obstacle(dict(shape="polar", amp=0.1, k=float(N / 15 * sizes.uniform(0.5, 1.0)), M=math.ceil(1.2 * N), N=N,
                                  P=int(sizes.choice([32, 64, 72, 90, 120])), tau=0.1, bc=bc), rng))
    return obs


def _prec(case):
    return (axi.PREC_SPLIT_BF16 if case.get("split") else axi.PREC_FP64) | (axi.PLAN_TSVD if case.get("tsvd") else 0)


def _data(case, seed):
    """Everything of a case that comes from the seed, on the host."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    d = SimpleNamespace()
    if kind == "pinv":
        # a cell whose height the seed chooses, and the unknowns whose discrepancies are the right-hand sides
        d.obs, d.z0 = [_obstacle(PINV_BODY, rng)], 2.2 * rng.uniform(0.95, 1.05)
        cols = axi.q_shape(_cell(case))[1]
        d.x = rng.standard_normal((case["W"], cols)) + 1j * rng.standard_normal((case["W"], cols))
        return d
    d.obs = _batch_obstacles(case, rng) if kind == "batch" else [_obstacle(case, rng)]
    W = case.get("W", 1)
    d.dirs = _directions(rng, W)
    d.xh = _sphere_points(rng, N_DIRS)
    if kind in ("near", "field"):
        # coefficients of a field that decays over the modes, as a solve gives
        P, N = case["P"], case["N"]
        n = np.minimum(np.arange(P), P - np.arange(P))
        c = rng.standard_normal((W, P, N)) + 1j * rng.standard_normal((W, P, N))
        d.coef = c * np.exp(-n / (P / 8.0))[None, :, None]
    if kind == "field":
        d.normals = _sphere_points(rng, case["T"])
        d.targets = _sphere_points(rng, case["T"]) * rng.uniform(1.8, 4.0, (case["T"], 1))
    return d


def _rho_max(case):
    return 1.2 if case.get("shape") == "cup" else 1.0 + 4 * case.get("amp", 0.1)


#: the body whose handle a pinv case fills Q with (Q depends on its wavenumber alone)
PINV_BODY = dict(shape="polar", amp=0.1, k=3.0, M=40, N=32, P=16, tau=0.1)


def _bloch():
    """The incident direction that sets a cell's Bloch phases: the case's own, since the number of Rayleigh-Bloch waves
    depends on it."""
    return _directions(np.random.default_rng(5), 1)


def _cell(case, z0=None):
    k, d = case["k"], _bloch()[0]
    z0 = _rho_max(case) + case["ex"] / 4 if z0 is None else z0
    return axi.Cell(k * d[0], k * d[1], case["ex"], case["ey"], z0, case["m1"], case["n0"], case["p"])


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(kind=kind, case=case)
    d = _data(case, seed)
    specs = [axi.spec_from_obstacle(ob) for ob in d.obs]
    if kind == "pinv":
        s.op = axi.Operator([axi.spec_from_obstacle(_obstacle(dict(PINV_BODY, k=case["k"]), np.random.default_rng(seed)))])
        s.Q = s.op.q_matrix(_cell(case, d.z0))
        s.b = _cuda(d.x) @ s.Q
        return s
    if kind == "iter":
        s.op = axi.Operator(specs, prec=axi.PREC_SPLIT_BF16 | axi.PLAN_TSVD)
    else:
        s.op = axi.Operator(specs, prec=_prec(case))
    s.dirs, s.xh = _cuda(d.dirs), _cuda(d.xh)
    if kind in ("near", "field"):
        s.coef = _cuda(d.coef)
    if kind == "field":
        s.targets, s.normals = _cuda(d.targets), _cuda(d.normals)
    if kind == "apply":
        s.f = s.op.incident(s.dirs)
    if kind in ("blocks", "iter"):
        s.cell = _cell(case)
    if kind == "iter":
        s.C = s.op.c_block(s.cell)
        s.US = s.op.q_matrix(s.cell)
        s.V, s.sigma, _ = axi.svd_jacobi(s.US)
        _, s.bt = s.op.btilde(case["p"])
        # smooth boundary data: the incident data of W waves; every image carries the cell's Bloch phases
        s.g = s.op.incident(s.dirs)
        s.bloch = _cuda(np.repeat(_bloch(), case["W"], 0))
    return s


def run(s):
    case, kind = s.case, s.kind
    if kind in ("solve", "batch"):
        s.op.refactor()
        out = []
        for i in range(len(s.op.specs)):
            coef = s.op.apply(s.op.incident(s.dirs, obs=i), obs=i)
            out.append(s.op.eval_field(coef, s.xh, axi.EVAL_FAR_FIELD, obs=i))
        return out
    if kind == "apply":
        return s.op.eval_field(s.op.apply(s.f), s.xh, axi.EVAL_FAR_FIELD)
    if kind == "near":
        return axi.near_image_sum(s.op, s.coef, (case["ex"], case["ey"]), s.dirs, slices=case["slices"])
    if kind == "field":
        how = axi.EVAL_NORMAL_DERIV if case["deriv"] else axi.EVAL_POTENTIAL
        return [s.op.eval_field(s.coef, s.targets, how, normals=s.normals), s.op.eval_field(s.coef, s.xh, axi.EVAL_FAR_FIELD)]
    if kind == "blocks":
        return [s.op.btilde(case["p"])[1], s.op.q_matrix(s.cell), s.op.c_block(s.cell)]
    if kind == "iter":
        return axi.periodic_iter_apply(s.op, s.g, (case["ex"], case["ey"]), s.bloch, s.C, s.US, s.V, s.sigma, s.bt, case["p"],
                                       near_slices=7)
    US = s.Q.clone()
    V, sigma, _ = axi.svd_jacobi(US)
    xi = axi.svd_solve(US, V, sigma, s.b)
    return [torch.sort(sigma, descending=True).values, axi.matvec_c128(s.Q, xi)]


def work(case):
    """Inputs and outputs once; arithmetic of the dense factorisations, applications and products, and an FFT per transform."""
    kind = case["kind"]
    W = case.get("W", 1)

    def solve(M, N, P, bc, build=True):
        r, c = (2 * M, 2 * N) if bc else (M, N)
        D = P // 2 + 1
        fl = W * P * (16.0 * r * c - 4.0 * c * c) / 1.0
        if build:
            fl += D * (8.0 * r * c * c - 8.0 / 3.0 * c ** 3)
        return fl, 16.0 * (6 * N + 4 * M + W * N_DIRS) + (0 if build else 16.0 * (D * r * c + W * r * P))
    if kind in ("solve", "apply"):
        fl, by = solve(case["M"], case["N"], case["P"], case.get("bc", 0), kind == "solve")
        return dict(flops=fl, bytes=by)
    if kind == "batch":
        both = [solve(o.M, o.N, o.P, o.bc) for o in _batch_obstacles(case, np.random.default_rng(0))]
        return dict(flops=sum(f for f, _ in both), bytes=sum(b for _, b in both))
    if kind == "pinv":
        m, n, _ = axi.q_shape(_cell(case))
        return dict(flops=4 * (4.0 * m * n * n + 8.0 * n ** 3) + 24.0 * W * m * n, bytes=16.0 * (m * n + 2 * W * m) + 8 * n)
    M, N, P = case["M"], case["N"], case["P"]
    fft = 5.0 * P * math.log2(P)
    if kind == "near":
        return dict(flops=W * (M + N) * fft, bytes=16.0 * W * P * (M + N))
    if kind == "field":
        T = case["T"]
        return dict(flops=W * (N * fft + 8.0 * (T + N_DIRS) * N), bytes=16.0 * W * (N * P + T + N_DIRS) + 48.0 * T)
    rows, cols, _ = axi.q_shape(_cell(case))
    c_entries, bt = rows * P * N, M * (case["p"] + 1) ** 2 / 2
    if kind == "blocks":
        return dict(flops=2.0 * c_entries, bytes=16.0 * (c_entries + rows * cols) + 8 * bt)
    fl = solve(M, N, P, 0, False)[0] + 8.0 * W * (c_entries + rows * cols + cols * cols)
    return dict(flops=fl, bytes=16.0 * (c_entries + rows * cols + cols * cols + 2 * W * M * P + (P // 2 + 1) * M * N) + 8 * bt)


# ---------------------------------------------------------------- the same in plain numpy and torch, 64 bits

def _erf(z):
    """erf(x + iy) for |y| <= 1: the Taylor series about x, erf^(n+1)(x) = (2/sqrt pi) (-1)^n H_n(x) e^{-x^2}."""
    z = np.asarray(z, dtype=complex)
    x, h = z.real, 1j * z.imag
    s = np.array([math.erf(v) for v in x.ravel()]).reshape(x.shape).astype(complex)
    g = 2 / math.sqrt(math.pi) * np.exp(-x * x)
    h0, h1, f = np.ones_like(x), 2 * x, h.copy()
    for n in range(80):
        s = s + (-1) ** n * h0 * g * f
        h0, h1 = h1, 2 * x * h1 - 2 * (n + 1) * h0
        f = f * h / (n + 2)
    return s


def _curve(ob, t):
    """zeta = z + i rho and its derivative at real or complex t."""
    t = np.asarray(t, dtype=complex)
    if ob.shape == axi.SHAPE_POLAR:
        r = sum(a * np.cos(j * t) for j, a in enumerate(ob.params))
        dr = -sum(a * j * np.sin(j * t) for j, a in enumerate(ob.params))
        e = np.exp(1j * t)
        return r * e, (dr + 1j * r) * e
    a, b = ob.params
    x = t - math.pi / 2
    er, g = _erf(x / a), np.exp(-(x / a) ** 2)
    r, dr = 1 - a * er, -2 / math.sqrt(math.pi) * g
    c = 2 * (1 - (b - a) / math.pi)
    e = np.exp(1j * (b - a + c * (a / math.sqrt(math.pi) * g + x * er)))
    return r * e, (dr + 1j * r * c * er) * e


def _geometry(ob):
    tm, tj = (np.arange(ob.M) + 0.5) * math.pi / ob.M, (np.arange(ob.N) + 0.5) * math.pi / ob.N
    zt = _curve(ob, np.linspace(0, math.pi, 4096))[0]
    z, r = zt.real, zt.imag
    sgn = 1.0 if np.sum(z[:-1] * r[1:] - z[1:] * r[:-1]) + z[-1] * r[0] - z[0] * r[-1] > 0 else -1.0
    ze, dz = _curve(ob, tm)
    nu = -1j * sgn * dz / np.abs(dz)
    yi, yx = _curve(ob, tj + 1j * sgn * ob.tau)[0], _curve(ob, tj - 1j * sgn * ob.tau)[0]
    return (np.stack([ze.imag, ze.real, nu.imag, nu.real], 1), np.stack([yi.imag, yi.real], 1), np.stack([yx.imag, yx.real], 1))


def _modal(k, coll, src, P, deriv):
    """A_n, n = 0 .. P/2, of the ring potentials by the trapezoid rule on enough nodes: [D][M][N]."""
    a = np.arccosh(1 + ((coll[:, None, 0] - src[None, :, 0]) ** 2 + (coll[:, None, 1] - src[None, :, 1]) ** 2)
                   / (2 * coll[:, None, 0] * src[None, :, 0])).min()
    q = int(math.ceil(max(2 * P, 38 / a + P / 2) / 40) * 40)
    phi = torch.arange(q, device=DEV, dtype=torch.float64) * (2 * math.pi / q)
    c, s = _cuda(coll), _cuda(src)
    out = torch.empty(P // 2 + 1, coll.shape[0], src.shape[0], device=DEV, dtype=C128)
    step = max(1, int(3e7 / (q * src.shape[0])))
    for i in range(0, coll.shape[0], step):
        m = c[i:i + step, :, None, None]
        dx, dy, dz = m[:, 0] - s[:, 0, None] * torch.cos(phi), -s[:, 0, None] * torch.sin(phi), m[:, 1] - s[:, 1, None]
        R = torch.sqrt(dx * dx + dy * dy + dz * dz)
        e = torch.polar(1 / (4 * math.pi * R), k * R)
        if deriv:
            e = (m[:, 2] * dx + m[:, 3] * dz) / R ** 2 * torch.complex(-torch.ones_like(R), k * R) * e
        out[:, i:i + step] = torch.movedim(torch.fft.fft(e, dim=2)[:, :, :P // 2 + 1], 2, 0) / q
    return out


def _nodes(rz, P):
    phi = np.arange(P) * 2 * math.pi / P
    return np.stack([rz[:, :1] * np.cos(phi), rz[:, :1] * np.sin(phi), np.broadcast_to(rz[:, 1:2], (len(rz), P))], -1)


def _strengths(coef):
    """[W][P][N] -> [W][N P] point strengths."""
    return torch.fft.ifft(coef, dim=1).transpose(1, 2).reshape(coef.shape[0], -1)


def _far(k, src, coef, xh):
    y = _cuda(_nodes(src, coef.shape[1]).reshape(-1, 3))
    K = torch.polar(torch.full((xh.shape[0], y.shape[0]), 1 / (4 * math.pi), device=DEV, dtype=torch.float64), -k * (xh @ y.T))
    return _strengths(coef) @ K.T


def _kernel(k, dx, dy, dz, n=None):
    R = torch.sqrt(dx * dx + dy * dy + dz * dz)
    e = torch.polar(1 / (4 * math.pi * R), k * R)
    if n is None:
        return e
    return (n[0] * dx + n[1] * dy + n[2] * dz) / (R * R) * torch.complex(-torch.ones_like(R), k * R) * e


def _incident(ob, coll, dirs):
    x, nu = _cuda(_nodes(coll[:, :2], ob.P)), _cuda(_nodes(coll[:, 2:], ob.P))
    u = torch.exp(1j * ob.k * torch.einsum("mlc,wc->wml", x, dirs))
    du = 1j * ob.k * torch.einsum("mlc,wc->wml", nu, dirs) * u
    return torch.cat([-u, -du], 1) if ob.bc else -du


def _exact_solve(ob, dirs, xh, tsvd):
    coll, src, srcx = _geometry(ob)
    A = _modal(ob.k, coll, src, ob.P, True)
    if ob.bc:
        A = torch.cat([torch.cat([_modal(ob.k, coll, src, ob.P, False), -_modal(ob.k_minus, coll, srcx, ob.P, False)], 2),
                       torch.cat([A, -_modal(ob.k_minus, coll, srcx, ob.P, True)], 2)], 1)
    f = torch.fft.fft(_incident(ob, coll, dirs), dim=2) / ob.P                    # [W][rows][P]
    W, P, D = f.shape[0], ob.P, ob.P // 2 + 1
    coef = torch.zeros(W, P, ob.N, device=DEV, dtype=C128)
    for n in range(D):
        idx = sorted({n, (P - n) % P})
        B = f[:, :, idx].permute(1, 0, 2).reshape(A.shape[1], -1)
        if tsvd:
            U, sv, Vh = torch.linalg.svd(A[n], full_matrices=False)
            keep = sv >= 1e-10 * sv[0]
            x = Vh[keep].conj().T @ ((U[:, keep].conj().T @ B) / sv[keep][:, None])
        else:
            Q, R = torch.linalg.qr(A[n])
            x = torch.linalg.solve_triangular(R, Q.conj().T @ B, upper=True)
        coef[:, idx] = x[:ob.N].reshape(ob.N, W, len(idx)).permute(1, 2, 0)
    return _far(ob.k, src, coef, xh)


def _exact_near(case, ob, d):
    """The eight images one by one where the lattice has no symmetry; with e_x = e_y and 4 | P a quarter turn of targets,
    sources and image leaves the kernel as it is, so two images serve all eight."""
    coll, src, _ = _geometry(ob)
    P, k, ex, ey = ob.P, ob.k, case["ex"], case["ey"]
    sig = _strengths(_cuda(d.coef)).reshape(case["W"], -1, P)
    x, nu, y = (_cuda(a.reshape(-1, 3)) for a in (_nodes(coll[:, :2], P), _nodes(coll[:, 2:], P), _nodes(src, P)))
    W, M = sig.shape[0], ob.M
    sym = ex == ey and P % 4 == 0
    images = [(1, 0), (1, 1)] if sym else [(a, b) for a in (-1, 0, 1) for b in (-1, 0, 1) if a or b]
    turns = 4 if sym else 1
    cols = torch.cat([torch.roll(sig, -r * (P // 4), dims=2).reshape(W, -1) for r in range(turns)], 0)
    U = torch.zeros(W, M, P, device=DEV, dtype=C128)
    step = max(1, int(6e7 / y.shape[0]))
    for a, b in images:
        c = torch.cat([cols @ _kernel(k, *(x[i:i + step, None, q] - y[None, :, q] - (a * ex, b * ey, 0.0)[q] for q in range(3)),
                                      [nu[i:i + step, None, q] for q in range(3)]).T for i in range(0, M * P, step)], 1)
        for r in range(turns):
            ph = np.exp(1j * k * (d.dirs[:, 0] * a * ex + d.dirs[:, 1] * b * ey))
            U += _cuda(ph)[:, None, None] * torch.roll(c[r * W:(r + 1) * W].reshape(W, M, P), r * (P // 4), dims=2)
            a, b = -b, a
    return U.reshape(W, -1)


def _exact_q(k, cell):
    """Q of eq. full: spherical waves j_l Y_lm and one Cartesian derivative at the wall nodes, then the Rayleigh-Bloch waves."""
    p, m1, ex, ey, z0 = cell.p, cell.m1, cell.ex, cell.ey, cell.z0
    al, be = np.exp(1j * cell.kx * ex), np.exp(1j * cell.ky * ey)
    g = np.polynomial.legendre.leggauss(m1)[0]
    ga, gb = (v.ravel() for v in np.meshgrid(g, g, indexing="ij"))

    def waves(x, y, z, axis):
        x, y, z = np.broadcast_arrays(x, y, z)
        rho, r = np.hypot(x, y), np.sqrt(x * x + y * y + z * z)
        t, ct, st = k * r, z / r, rho / r
        top = p + int(t.max()) + 60
        f = np.zeros((top + 2, len(t)))
        f[top] = 1e-280                                                     # the minimal solution, upside down
        for l in range(top, 0, -1):
            f[l - 1] = (2 * l + 1) / t * f[l] - f[l + 1]
            big = np.abs(f[l - 1]) > 1e250
            f[l - 1:, big] *= 1e-250
        j0, j1 = np.sin(t) / t, np.sin(t) / t ** 2 - np.cos(t) / t
        f = f * np.where(np.abs(j0) >= np.abs(j1), j0 / f[0], j1 / f[1])
        val, der = (np.zeros(((p + 1) ** 2, len(t)), dtype=complex) for _ in range(2))
        pmm = np.full(len(t), math.sqrt(1 / (4 * math.pi)))
        for m in range(p + 1):
            if m:
                pmm = -math.sqrt((2 * m + 1) / (2 * m)) * st * pmm
            prev, cur = np.zeros(len(t)), pmm
            for l in range(m, p + 1):
                if l > m:
                    a = math.sqrt((4 * l * l - 1) / (l * l - m * m))
                    b = math.sqrt(((l - 1) ** 2 - m * m) / (4 * (l - 1) ** 2 - 1)) if l > m + 1 else 0.0
                    prev, cur = cur, a * (ct * cur - b * prev)
                c = math.sqrt((2 * l + 1) * (l - m) * (l + m) / (2 * l - 1)) if l > m else 0.0
                dth = (l * ct * cur - c * prev) / st
                dj = k * ((f[l - 1] - (l + 1) / t * f[l]) if l else -f[1])
                E = ((x + 1j * y) / rho) ** m
                dr, dt, dp = dj * cur, f[l] * dth / r, 1j * m * f[l] * cur / (r * st)
                h = dr * st + dt * ct
                w = (h * x / rho - dp * y / rho, h * y / rho + dp * x / rho, dr * ct - dt * st)[axis]
                for sg in ((m, -m) if m else (0,)):
                    v, d = f[l] * cur * E, w * E
                    val[l * l + l + sg], der[l * l + l + sg] = (v, d) if sg >= 0 else ((-1) ** m * v.conj(), (-1) ** m * d.conj())
        return val, der
    L, R = (waves(s * ex / 2, ey / 2 * ga, z0 * gb, 0) for s in (-1, 1))
    B, F = (waves(ex / 2 * ga, s * ey / 2, z0 * gb, 1) for s in (-1, 1))
    T, Dn = (waves(ex / 2 * ga, ey / 2 * gb, s * z0, 2) for s in (1, -1))
    S = np.concatenate([R[0] - al * L[0], R[1] - al * L[1], F[0] - be * B[0], F[1] - be * B[1], *T, *Dn], 1)
    top, bot = [], []
    nr = m1 * m1
    for m, n in axi.q_modes(cell):
        kx, ky = cell.kx + 2 * math.pi * m / ex, cell.ky + 2 * math.pi * n / ey
        ikz = 1j * np.sqrt(complex(k * k - kx * kx - ky * ky))
        e = np.exp(1j * (kx * ex / 2 * ga + ky * ey / 2 * gb))
        top.append(np.concatenate([np.zeros(4 * nr), -e, -ikz * e, np.zeros(2 * nr)]))
        bot.append(np.concatenate([np.zeros(6 * nr), -e, ikz * e]))
    return _cuda(np.concatenate([S, np.array(top + bot).reshape(-1, 8 * nr)], 0))


def _exact_c(case, ob):
    """C by its definition, without the near images that cancel between the walls of a pair."""
    cell = _cell(case)
    _, src, _ = _geometry(ob)
    P, k, ex, ey, z0, m1 = ob.P, ob.k, cell.ex, cell.ey, cell.z0, cell.m1
    y = _cuda(_nodes(src, P))                                                      # [N][P][3]
    al, be = np.exp(1j * cell.kx * ex), np.exp(1j * cell.ky * ey)
    g = np.polynomial.legendre.leggauss(m1)[0]
    ga, gb = (v.ravel() for v in np.meshgrid(g, g, indexing="ij"))

    def rows(images, axis):
        val = torch.zeros(m1 * m1, ob.N, P, device=DEV, dtype=C128)
        der = torch.zeros_like(val)
        for w, p in images:
            pt = _cuda(np.stack(np.broadcast_arrays(*p), -1).astype(float))
            for i in range(0, m1 * m1, 32):
                dv = [pt[i:i + 32, None, None, q] - y[None, :, :, q] for q in range(3)]
                one = [torch.ones_like(dv[0]) if q == axis else torch.zeros_like(dv[0]) for q in range(3)]
                val[i:i + 32] += complex(w) * torch.fft.ifft(_kernel(k, *dv), dim=2)
                der[i:i + 32] += complex(w) * torch.fft.ifft(_kernel(k, *dv, one), dim=2)
        return [v.permute(2, 1, 0).reshape(P * ob.N, -1) for v in (val, der)]
    i3 = (-1, 0, 1)
    lr = [(be ** b * c, (x, ey / 2 * ga - b * ey, z0 * gb)) for b in i3 for c, x in ((1 / al, 1.5 * ex), (-al ** 2, -1.5 * ex))]
    bf = [(al ** a * c, (ex / 2 * ga - a * ex, yy, z0 * gb)) for a in i3 for c, yy in ((1 / be, 1.5 * ey), (-be ** 2, -1.5 * ey))]
    td = [[(al ** a * be ** b, (ex / 2 * ga - a * ex, ey / 2 * gb - b * ey, z)) for a in i3 for b in i3] for z in (z0, -z0)]
    return torch.cat(rows(lr, 0) + rows(bf, 1) + rows(td[0], 2) + rows(td[1], 2), 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "iter":
        return None                                # a chain of every other case
    d = _data(case, seed)
    if kind == "pinv":
        A = _exact_q(case["k"], _cell(case, d.z0)).T
        U, sv, _ = torch.linalg.svd(A, full_matrices=False)
        U = U[:, sv > 1e-10 * sv[0]]
        return [sv, (U @ (U.conj().T @ (A @ _cuda(d.x).T))).T]
    dirs, xh = _cuda(d.dirs), _cuda(d.xh)
    if kind in ("solve", "batch"):
        return [_exact_solve(ob, dirs, xh, case.get("tsvd", False)) for ob in d.obs]
    ob = d.obs[0]
    if kind == "apply":
        return _exact_solve(ob, dirs, xh, False)
    if kind == "near":
        return _exact_near(case, ob, d)
    if kind == "blocks":
        return [None, _exact_q(case["k"], _cell(case)), _exact_c(case, ob)]
    _, src, _ = _geometry(ob)
    coef, x, nu = _cuda(d.coef), _cuda(d.targets), _cuda(d.normals)
    y, sig = _cuda(_nodes(src, ob.P).reshape(-1, 3)), _strengths(coef)
    step = max(1, int(6e7 / y.shape[0]))
    u = torch.cat([sig @ _kernel(ob.k, *(x[i:i + step, None, q] - y[None, :, q] for q in range(3)),
                                 [nu[i:i + step, None, q] for q in range(3)] if case["deriv"] else None).T
                   for i in range(0, case["T"], step)], 1)
    return [u, _far(ob.k, src, coef, xh)]
