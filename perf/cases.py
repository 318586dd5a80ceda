"""The calls whose speed matters to a user of the lattice Boltzmann library, as cases that can be timed and compared.

Each case is one call sequence through the package's public entry points (Lattice, Refinement and the body
constructors), on a state that a user's program would hold.  The families:

  box       bodiless stream + collide: the method itself, on the smallest boxes (latency), on ragged ones (odd row
            lengths, one- and two-sided faces), with each stabilizer
  setup     initial fields on the device -> populations, and the global sums that a run's monitor reads
  sphere    the two-way coupled sedimenting sphere between no-slip walls (Sec. 4.1 of arXiv 1608.04658)
  airfoil   the plunging airfoil with inflow, outflow and far field (Sec. 4.2)
  swimmer   the self-propelled, deforming anguilliform swimmer (Sec. 4.3)
  adjoint   the gradient of a held swimmer's mean thrust (forward run and reverse sweep)
  refined   the plunging airfoil on a two-level grid (Sec. 4.2)

exact() is a restatement of the step in plain torch, FP64, written from the equations in include/lbm.h; it uses none of
the library's code.
"""
import math
import random

import numpy as np
import torch

import paper_1608_04658_gb300 as lbm

DEV = "cuda"
Q = 27
C = [(i // 9 - 1, (i // 3) % 3 - 1, i % 3 - 1) for i in range(Q)]
W = [(8 / 27, 2 / 27, 1 / 54, 1 / 216)[sum(map(abs, c))] for c in C]
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
# floating point operations of one node update (moments, product-form equilibrium, entropic scalar products, relaxation)
FLOPS = 650
PERIODIC, WALL, EQ, OUTFLOW = 0, 1, 2, 3
FACES = {"periodic": (0,) * 6, "walls": (1, 1, 1, 1, 0, 0), "tunnel": (2, 3, 2, 2, 0, 0)}


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest run of the test suite (a 32^3 Taylor-Green box): launches and latency
        dict(name="box_32_fp32", kind="box", nx=32, ny=32, nz=32, storage="fp32", gamma="analytic", faces="periodic", steps=20),
        # an odd row length, as a box sized by a body gives it, in 16-bit storage
        dict(name="box_ragged_bf16", kind="box", nx=161, ny=97, nz=83, storage="bf16", gamma="analytic", faces="periodic", steps=5),
        # the exact stabilizer (the benchmark's fp32_exact_gamma variant) between walls
        dict(name="box_exact_fp32", kind="box", nx=256, ny=192, nz=128, storage="fp32", gamma="exact", faces="walls", steps=2),
        # setting a run up and reading its global sums (what run_logged records)
        dict(name="setup_256_fp32", kind="setup", nx=256, ny=256, nz=256, storage="fp32"),
        # the reduced sedimenting sphere of the long-run drag test: the body's chain of small kernels
        dict(name="sphere_small_fp16", kind="sphere", nx=32, ny=32, nz=64, D=8.0, storage="fp16", steps=20),
        # the benchmark's sedimenting sphere, and its FP64 form (the reference of the storage comparison)
        dict(name="sphere_fp32", kind="sphere", nx=128, ny=128, nz=256, D=16.0, storage="fp32", steps=10),
        dict(name="sphere_fp64", kind="sphere", nx=128, ny=128, nz=256, D=16.0, storage="fp64", steps=2),
        # the benchmark's plunging airfoil, 16-bit storage
        dict(name="airfoil_fp16", kind="airfoil", nx=1024, ny=512, nz=64, chord=128.0, storage="fp16", steps=4),
        # the headline workload in FP32 and in 16 bits
        dict(name="swimmer_fp32", kind="swimmer", nx=768, ny=256, nz=256, L=128.0, free=1, storage="fp32", steps=4),
        dict(name="swimmer_fp16", kind="swimmer", nx=768, ny=256, nz=256, L=128.0, free=1, storage="fp16", steps=4),
        # the benchmark's differentiated swimmer (a shorter horizon)
        dict(name="adjoint_fp32", kind="adjoint", nx=256, ny=128, nz=128, L=64.0, storage="fp32", horizon=36),
        # the benchmark's two-level airfoil
        dict(name="refined_airfoil_fp32", kind="refined", nx=512, ny=256, nz=32, chord=128.0, storage="fp32", steps=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case of the same families; sizes spread over the logarithm of each family's range, odd ones included."""
    case = _drawn(rng)
    if "steps" in case:
        case["steps"] = max(1, min(case["steps"], int(1.2e8 / (case["nx"] * case["ny"] * case["nz"]))))
    return case


def _drawn(rng):
    kind = rng.choice(["box", "box", "box", "setup", "sphere", "sphere", "airfoil", "swimmer", "adjoint", "refined"])
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    if kind == "box":
        dims = [_log(rng, 16, 320) for _ in range(3)]
        gamma = rng.choice(["analytic", "analytic", "analytic", "lbgk", "exact"])
        return dict(kind=kind, nx=dims[0], ny=dims[1], nz=dims[2], storage=rng.choice([storage, storage, "fp64"]), gamma=gamma,
                    faces=rng.choice(list(FACES)), steps=rng.randint(2, 20))
    if kind == "setup":
        return dict(kind=kind, nx=_log(rng, 32, 300), ny=_log(rng, 32, 300), nz=_log(rng, 32, 300), storage=rng.choice([storage, "fp64"]))
    if kind == "sphere":
        D = round(math.exp(rng.uniform(math.log(6.0), math.log(24.0))), 2)
        n = [int(D * rng.uniform(3.5, 7.0)) for _ in range(2)] + [int(D * rng.uniform(6.0, 12.0))]
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], D=D, storage=rng.choice([storage, storage, "fp64"]), steps=rng.randint(3, 12))
    if kind == "airfoil":
        c = round(math.exp(rng.uniform(math.log(32.0), math.log(128.0))), 2)
        return dict(kind=kind, nx=int(c * rng.uniform(4.0, 8.0)), ny=int(c * rng.uniform(2.5, 4.0)), nz=_log(rng, 8, 64), chord=c,
                    storage=storage, steps=rng.randint(2, 6))
    if kind == "swimmer":
        L = round(math.exp(rng.uniform(math.log(32.0), math.log(100.0))), 2)
        return dict(kind=kind, nx=int(L * rng.uniform(3.0, 6.0)), ny=int(L * rng.uniform(1.5, 2.2)), nz=int(L * rng.uniform(1.2, 2.2)), L=L,
                    free=rng.choice([1, 1, 7]), storage=storage, steps=rng.randint(2, 8))
    if kind == "adjoint":
        L = round(math.exp(rng.uniform(math.log(24.0), math.log(60.0))), 2)
        return dict(kind=kind, nx=int(L * rng.uniform(2.2, 4.0)), ny=int(L * rng.uniform(1.2, 2.0)), nz=int(L * rng.uniform(1.2, 2.0)), L=L,
                    storage=rng.choice(["fp32", "fp32", "fp16"]), horizon=rng.randint(6, 36))
    c = round(math.exp(rng.uniform(math.log(32.0), math.log(100.0))), 2)
    return dict(kind=kind, nx=int(c * rng.uniform(3.0, 4.0)), ny=int(c * rng.uniform(1.8, 2.4)), nz=_log(rng, 6, 24), chord=c,
                storage=storage, steps=rng.randint(2, 4))


# ------------------------------------------------------------------------------------------------ inputs
def _flow(dims, seed, base, amp, origin=(0, 0, 0), h=1.0, period=None):
    """rho (nz, ny, nx) and u (nz, ny, nx, 3), float32 on the device: a uniform stream plus smooth random vortices of
    amplitude `amp` over `period` lattice units (the box), node j of axis a at origin[a] + h j."""
    rng = random.Random(seed)
    period = period or dims
    u = torch.empty((dims[2], dims[1], dims[0], 3), dtype=torch.float32, device=DEV)
    rho = torch.ones((dims[2], dims[1], dims[0]), dtype=torch.float32, device=DEV)

    def wave(a):
        k, ph = 2 * math.pi * rng.choice([1, 2]) / period[a], rng.uniform(0, 2 * math.pi)
        x = origin[a] + h * torch.arange(dims[a], dtype=torch.float64, device=DEV)
        return torch.sin(k * x + ph).float()

    def mode():
        x, y, z = wave(0), wave(1), wave(2)
        return z[:, None, None] * y[None, :, None] * x[None, None, :]

    for a in range(3):
        u[..., a] = float(base[a]) + amp * mode()
    rho += 0.1 * amp * mode()
    return rho, u


def _mesh(L):
    """The swimmer's closed triangulated surface (Sec. 4.3): elliptic cross sections along the centre line; rest[v] =
    (s, dy, dz), triangles counter-clockwise from outside, head vertex first, tail-cap vertex last."""
    # 150 sections as in the paper; coarser on bodies shorter than the benchmark's smallest, as the tests' swimmers are
    segments, ring = (150, 64) if L >= 64 else (int(2 * L), max(16, int(0.66 * L)))
    s = L * np.arange(1, segments + 1) / segments
    wh = sb = 0.04 * L
    st, wt = 0.95 * L, 0.01 * L
    w = np.where(s < sb, np.sqrt(np.clip(2 * wh * s - s * s, 0, None)),
                 np.where(s < st, wh - (wh - wt) * ((s - sb) / (st - sb)) ** 2, np.clip(wt * (L - s) / (L - st), 0, None)))
    a, b = 0.51 * L, 0.08 * L
    hgt = b * np.sqrt(np.clip(1 - ((s - a) / a) ** 2, 0, None))
    phi = 2 * np.pi * (np.arange(ring) + 0.5) / ring
    body = np.stack(np.broadcast_arrays(s[:, None], w[:, None] * np.cos(phi), hgt[:, None] * np.sin(phi)), -1).reshape(-1, 3)
    rest = np.concatenate([[[0.0, 0.0, 0.0]], body, [[L, 0.0, 0.0]]])
    j = np.arange(ring)
    jn = (j + 1) % ring
    k = ring * np.arange(segments - 1)[:, None]
    p, q, r, t = 1 + k + j, 1 + k + jn, 1 + k + ring + j, 1 + k + ring + jn
    last = 1 + ring * (segments - 1)
    tris = np.concatenate([np.stack([np.zeros(ring, int), 1 + jn, 1 + j], -1),
                           np.stack([p, q, t], -1).reshape(-1, 3), np.stack([p, t, r], -1).reshape(-1, 3),
                           np.stack([np.full(ring, len(rest) - 1), last + j, last + jn], -1)])
    x = np.linspace(0, L, 20001)
    wx = np.where(x < sb, np.sqrt(np.clip(2 * wh * x - x * x, 0, None)),
                  np.where(x < st, wh - (wh - wt) * ((x - sb) / (st - sb)) ** 2, np.clip(wt * (L - x) / (L - st), 0, None)))
    mass = float(np.trapezoid(np.pi * wx * b * np.sqrt(np.clip(1 - ((x - a) / a) ** 2, 0, None)), x))
    return rest, tris.astype(np.int32), mass


def _thickness():
    """Half-thickness coefficients of the 8.5 % airfoil (maximum at a quarter chord, closed trailing edge)."""
    x, a0 = 0.25, 0.126
    A = np.array([[x, x ** 2, x ** 3, x ** 4], [1, 2 * x, 3 * x ** 2, 4 * x ** 3], [1, 1, 1, 1], [1, 2, 3, 4.0]])
    a = np.linalg.solve(A, [0.0425 - a0 * math.sqrt(x), -0.5 * a0 / math.sqrt(x), -a0, -0.10 - 0.5 * a0])
    return (a0, *map(float, a))


def _airfoil(le, chord, u_inf):
    al = math.radians(4.0)
    return dict(kind="airfoil", le=le, chord=chord, ca=math.cos(al), sa=math.sin(al), h_amp=0.05 * chord,
                h_omega=2 * 3.93 * u_inf / chord, camber_m=0.015, camber_p=0.35, thick=_thickness())


def _setting(case, seed):
    """What the workload is made of: viscosity, faces, body and flow, each as in the paper's section (see the module's
    text) with the body placed off the lattice planes by the seed."""
    rng = random.Random(seed * 7919 + 5)
    kind, dims = case["kind"], (case["nx"], case["ny"], case["nz"])
    off = [rng.uniform(0.05, 0.45) for _ in range(3)]
    if kind in ("box", "setup"):
        faces = FACES[case.get("faces", "periodic")]
        base = (0.05, 0.0, 0.0) if case.get("faces") == "tunnel" else (0.0, 0.0, 0.0)
        return dict(nu=0.005, faces=faces, u_face=base, base=base, amp=0.05 if faces == FACES["periodic"] else 0.01, body=None)
    if kind == "sphere":
        D, ut = case["D"], 0.04
        X = (dims[0] / 2 - 0.5 + off[0], dims[1] / 2 - 0.5 + off[1], 0.75 * dims[2] + off[2])
        g = 3.0 * ut ** 2 * 1.1 / (4.0 * D * 0.5)
        return dict(nu=ut * D / 100.0, faces=FACES["walls"], u_face=(0.0,) * 3, base=(0.0,) * 3, amp=0.002,
                    body=dict(kind="sphere", X=X, R=D / 2, U=(0.0, 0.0, -ut), g=(0.0, 0.0, -g), rho_ratio=1.5))
    if kind == "airfoil":
        c, ui = case["chord"], 0.05
        return dict(nu=ui * c / 40000.0, faces=FACES["tunnel"], u_face=(ui, 0.0, 0.0), base=(ui, 0.0, 0.0), amp=0.002,
                    body=_airfoil((dims[0] / 4 + off[0], dims[1] / 2 + off[1]), c, ui))
    if kind == "refined":
        # the block spans z and holds the airfoil, in fine lattice units; the coarse level takes half the viscosity
        c, ui = case["chord"], 0.05
        lo = (int(0.1875 * dims[0]), dims[1] // 4, 0)
        hi = (lo[0] + max(8, int(0.5 * dims[0])) - 1, dims[1] - dims[1] // 4 - 1, dims[2])
        return dict(nu=0.5 * ui * c / 40000.0, faces=FACES["tunnel"], u_face=(ui, 0.0, 0.0), base=(ui, 0.0, 0.0), amp=0.002, lo=lo, hi=hi,
                    body=_airfoil(((hi[0] - lo[0]) * 0.5 + off[0], float(hi[1] - lo[1]) + off[1]), c, ui))
    L, period = case["L"], 4000.0
    rest, tris, mass = _mesh(L)
    if kind == "adjoint":
        X = (dims[0] / 2 - L / 2 + off[0], dims[1] / 2 + off[1], dims[2] / 2 + off[2])
    elif case["free"] & 6:  # X is the centre of mass
        X = (dims[0] / 2 + off[0], dims[1] / 2 + off[1], dims[2] / 2 + off[2])
    else:
        X = (min(round(2 * dims[0] / 3), dims[0] - math.ceil(L) - 12) + off[0], dims[1] / 2 + off[1], dims[2] / 2 + off[2])
    return dict(nu=(L * L / period) / 7142.0, faces=FACES["periodic"], u_face=(0.0,) * 3, base=(0.0,) * 3, amp=0.002,
                body=dict(kind="swimmer", X=X, rest=rest, tris=tris, L=L, amp=0.125, wavelength=L, period=period, mass=mass,
                          free=0 if kind == "adjoint" else case["free"], t0=float(rng.randint(0, 3999))))


def _geometry(b):
    if b["kind"] == "sphere":
        return lbm.sphere(b["X"], b["R"], U=b["U"], free=True, rho_ratio=b["rho_ratio"], g=b["g"])
    if b["kind"] == "airfoil":
        return lbm.airfoil(b["le"], b["chord"], b["ca"], b["sa"], b["h_amp"], b["h_omega"], b["camber_m"], b["camber_p"], b["thick"])
    return lbm.swimmer(b["X"], b["rest"], b["tris"], b["L"], b["amp"], b["wavelength"], b["period"], free=int(b["free"]), mass=b["mass"], t0=b["t0"])


_GAMMA = {"analytic": lbm.GAMMA_ANALYTIC, "exact": lbm.GAMMA_EXACT, "lbgk": lbm.GAMMA_LBGK}


def prepare(case, seed):
    """The lattice with its body and its initial state (and for `setup` the initial fields)."""
    s, dims = _setting(case, seed), (case["nx"], case["ny"], case["nz"])
    lat = lbm.Lattice(dims, s["nu"], storage=case["storage"], faces=s["faces"], u_face=s["u_face"], gamma_mode=_GAMMA[case.get("gamma", "analytic")])
    rho, u = _flow(dims, seed, s["base"], s["amp"])
    st = dict(case=case, lat=lat)
    if case["kind"] == "setup":
        return dict(st, rho=rho, u=u)
    # nodes inside the body hold no defined state: zeros there, so that whole outputs can be compared
    lat.f_b.zero_()
    if case["kind"] == "refined":
        ref = lbm.Refinement(lat, s["lo"], s["hi"])
        ref.fine.f_b.zero_()
        ref.fine.set_geometry(_geometry(s["body"]))
        lat.init_state(rho, u)
        ref.fine.init_state(*_flow(ref.fine.shape, seed, s["base"], s["amp"], s["lo"], 0.5, dims))
        ref.init()
        return dict(st, ref=ref)
    if s["body"] is not None:
        lat.set_geometry(_geometry(s["body"]))
    lat.init_state(rho, u)
    return st


def _typed(v, like):
    """Numbers summed from the populations, in the populations' own type: they are no more exact than these."""
    return torch.tensor([float(x) for x in v], dtype=torch.float64).to(like.dtype)


def _body_out(lat):
    b = lat.body()
    return dict(pose=_typed([*b["X"], *b["U"]], lat.f), force=_typed([*b["F"], *b["M"]], lat.f),
                counts=np.array([b["n_boundary"], b["n_uncovered"], b["n_links"]], dtype=np.int64))


def run(state):
    case, lat = state["case"], state["lat"]
    kind = case["kind"]
    if kind == "box":
        lat.step(case["steps"])
        return dict(f=lat.f)
    if kind == "setup":
        lat.init_state(state["rho"], state["u"])
        return dict(f=lat.f, totals=lat.totals())
    if kind == "adjoint":
        out = lat.adjoint(case["horizon"], (-1.0, 0.0, 0.0), want_lambda0=True)
        g = out["lambda_0"]
        return dict(f=lat.f, J=_typed([out["J"]], g), dJ=_typed(out["dJ_dtheta"], g), lambda_0=g)
    if kind == "refined":
        state["ref"].step(case["steps"])
        fine = state["ref"].fine
        return dict(f=lat.f, fine=fine.f, **_body_out(fine))
    lat.step(case["steps"])
    return dict(f=lat.f, **_body_out(lat))


def work(case):
    """Each population read once and written once a step; a reversed step reads the state and the adjoint and writes the
    adjoint."""
    N, es = case["nx"] * case["ny"] * case["nz"], BYTES[case["storage"]]
    if case["kind"] == "setup":
        return dict(bytes=N * (16 + 2 * Q * es), flops=N * 250)
    if case["kind"] == "adjoint":
        r = 8 if case["storage"] == "fp64" else 4
        return dict(bytes=case["horizon"] * N * Q * (2 * es + es + 2 * r), flops=case["horizon"] * N * 3 * FLOPS)
    if case["kind"] == "refined":
        s = _setting(case, 0)
        fine = [2 * (h - l) + (0 if l == 0 else 2) for l, h in zip(s["lo"], s["hi"])]
        m = [h - l - (0 if l == 0 else 1) for l, h in zip(s["lo"], s["hi"])]
        n = N - int(np.prod(m)) + 2 * int(np.prod(fine))
        return dict(bytes=case["steps"] * n * 2 * Q * es, flops=case["steps"] * n * FLOPS)
    return dict(bytes=case["steps"] * N * 2 * Q * es, flops=case["steps"] * N * FLOPS)


# ------------------------------------------------------------------------------------------------ the same in 64 bits
def _feq(drho, rho, u):
    """Shifted entropic equilibrium f^eq(rho, u) - W rho0, (27, ...); u (3, ...)."""
    fac = []
    for a in range(3):
        S = torch.sqrt(1 + 3 * u[a] ** 2)
        B = (2 * u[a] + S) / (1 - u[a])
        sig = 3 * u[a] ** 2 / (S + 1)
        fac.append(((1 - sig) / B - 1, -sig, (1 - sig) * B - 1))  # e(c) = phi(c) - 1
    out = []
    for i, c in enumerate(C):
        x, y, z = (fac[a][c[a] + 1] for a in range(3))
        xy = x + y + x * y
        out.append(W[i] * (drho + rho * (xy + z + xy * z)))
    return torch.stack(out)


def _moments(g):
    m = [g.sum(0)] + [sum(C[i][a] * g[i] for i in range(Q) if C[i][a]) for a in range(3)]
    return m[0], torch.stack(m[1:])


def _stress(d):
    return [sum(C[i][a] * C[i][b] * d[i] for i in range(Q) if C[i][a] * C[i][b]) for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]


def _shear(i, P):
    """Shear part of direction i: the deviatoric second moments of P on the D3Q27 directions."""
    nx, ny = P[0] - P[2], P[1] - P[2]
    c = C[i]
    n = sum(map(abs, c))
    if n == 1:
        return (2 * nx - ny) / 6 if c[0] else (2 * ny - nx) / 6 if c[1] else -(nx + ny) / 6
    if n == 2:
        return (c[0] * c[1] * P[3] + c[0] * c[2] * P[4] + c[1] * c[2] * P[5]) / 4
    return torch.zeros_like(P[0])


def _collide(g, beta, rho0, gamma):
    """KBC collision (Eqs. kineticEq, kbc_relax, feq_min and the stabilizer) of shifted populations g (27, ...)."""
    drho, j = _moments(g)
    rho = rho0 + drho
    geq = _feq(drho, rho, j / rho)
    d = g - geq
    P = _stress(d)
    ds = torch.stack([_shear(i, P) for i in range(Q)])
    dh = d - ds
    feq = geq + torch.tensor(W, dtype=g.dtype, device=g.device).view(-1, *[1] * (g.dim() - 1)) * rho0
    sh, hh = (ds * dh / feq).sum(0), (dh * dh / feq).sum(0)
    two = torch.full_like(sh, 2.0)
    if gamma == "lbgk":
        gam = two
    else:
        ok = hh > 1e-300
        gam = torch.where(ok, 1 / beta - (2 - 1 / beta) * sh / torch.where(ok, hh, torch.ones_like(hh)), two)
        if gamma == "exact":
            e, B = (dh - (2 * beta - 1) * ds) / feq, beta * dh / feq
            for _ in range(12):  # Newton from the analytic value
                x = 1 + e - gam * B
                slope = (dh * B / x).sum(0)
                gam = torch.where(ok, gam + (dh * torch.log(x)).sum(0) / torch.where(ok, slope, torch.ones_like(slope)), two)
    return g - beta * (2 * ds + gam * dh)


class _Exact:
    """The whole step in FP64 torch.  States are (27, nz, ny, nx) shifted populations in two buffers that alternate."""

    def __init__(self, dims, s, gamma, body=None, rho0=1.0):
        self.n, self.faces, self.gamma, self.rho0 = dims, s["faces"], gamma, rho0
        self.nu = s["nu"]
        self.beta = 1 / (6 * self.nu + 1)
        uf = torch.tensor(s["u_face"], dtype=torch.float64, device=DEV)
        self.g_face = _feq(torch.zeros((), dtype=torch.float64, device=DEV), torch.full((), rho0, dtype=torch.float64, device=DEV), uf)
        self.W = torch.tensor(W, dtype=torch.float64, device=DEV)
        self.c = torch.tensor(C, device=DEV)
        self.keep = None  # nodes that the step leaves alone (the refined block)
        self.b = dict(body) if body else None
        if self.b:
            self._body_start()
            self.solid = self._inside()

    # ---- streaming
    def _axis(self, a, c, lo=0, hi=None):
        """Source indices of the pulls of component c along axis a, and the kind of each (0 node, 1 EQ, 2 wall)."""
        n = self.n[a]
        i = torch.arange(lo, n if hi is None else hi, device=DEV) - c
        kind = torch.zeros_like(i)
        for out, face in ((i < 0, self.faces[2 * a]), (i >= n, self.faces[2 * a + 1])):
            if face in (WALL, EQ):
                kind[out] = 2 if face == WALL else 1
        return (i % n if self.faces[2 * a] == PERIODIC else i.clamp(0, n - 1)), kind

    def pulled(self, S, z0, z1):
        out = []
        for i, c in enumerate(C):
            (x, kx), (y, ky), (z, kz) = self._axis(0, c[0]), self._axis(1, c[1]), self._axis(2, c[2], z0, z1)
            v = S[i][z][:, y][:, :, x]
            if any(self.faces[2 * a + k] in (WALL, EQ) for a in range(3) for k in (0, 1)):
                kind = torch.maximum(torch.maximum(kz[:, None, None], ky[None, :, None]), kx[None, None, :])
                v = torch.where(kind == 2, S[26 - i][z0:z1], torch.where(kind == 1, self.g_face[i], v))
            out.append(v)
        return torch.stack(out)

    def step(self, a, b):
        """a (state at t, refilled in place) -> b."""
        if self.b:
            self._advance()
            was, self.solid = self.solid, self._inside()
            self._refill(a, was)
        per = max(1, 1_500_000 // (self.n[0] * self.n[1]))
        for z0 in range(0, self.n[2], per):
            z1 = min(self.n[2], z0 + per)
            v = _collide(self.pulled(a, z0, z1), self.beta, self.rho0, self.gamma)
            off = torch.zeros(v.shape[1:], dtype=torch.bool, device=DEV)
            if self.b:
                off |= self.solid[z0:z1]
            if self.keep is not None:
                off |= self.keep[z0:z1]
            b[:, z0:z1] = torch.where(off, b[:, z0:z1], v)
        if self.b:
            self._boundary(a, b)

    # ---- body motion and marks
    def _body_start(self):
        b = self.b
        b["F"], b["M"] = np.zeros(3), np.zeros(3)
        if b["kind"] == "airfoil":
            b["t"], b["y0"] = 0.0, b["le"][1]
            b["X"], b["U"] = np.array([b["le"][0], b["le"][1], 0.0]), np.array([0.0, b["h_amp"] * b["h_omega"], 0.0])
            return
        b["X"] = np.array(b["X"])
        b["U"] = np.array(b.get("U", (0.0, 0.0, 0.0)))
        if b["kind"] == "sphere":
            b["mass"] = b["rho_ratio"] * self.rho0 * math.pi * (2 * b["R"]) ** 3 / 6
        else:
            b["t"] = b["t0"]
            b["rest"] = torch.tensor(b["rest"], device=DEV)
            b["tri"] = torch.tensor(b["tris"], device=DEV).long()
            self._pose()

    def _midline(self, s, t):
        b = self.b
        A = b["amp"] * b["L"] * (s / b["L"] + 0.03125) / 1.03125
        return A * torch.sin(2 * math.pi * (s / b["wavelength"] - t / b["period"]))

    def _rate(self, s, t):
        return (self._midline(s, t + 1) - self._midline(s, t - 1)) / 2

    def _pose(self):
        b = self.b
        s, dy, dz = b["rest"].unbind(1)
        b["P"] = torch.stack([b["X"][0] + s, b["X"][1] + self._midline(s, b["t"]) + dy, b["X"][2] + dz], 1)
        b["V"] = torch.stack([b["U"][0] + 0 * s, b["U"][1] + self._rate(s, b["t"]), b["U"][2] + 0 * s], 1)

    def _advance(self):
        b = self.b
        if b["kind"] == "airfoil":
            b["t"] += 1
            b["X"] = np.array([b["X"][0], b["y0"] + b["h_amp"] * math.sin(b["h_omega"] * b["t"]), 0.0])
            b["U"] = np.array([0.0, b["h_amp"] * b["h_omega"] * math.cos(b["h_omega"] * b["t"]), 0.0])
        elif b["kind"] == "sphere":
            acc = b["F"] / b["mass"] + (1 - 1 / b["rho_ratio"]) * np.array(b["g"])
            b["X"] = b["X"] + b["U"]
            b["U"] = b["U"] + acc
            for a in range(3):
                if self.faces[2 * a] == PERIODIC:
                    b["X"][a] %= self.n[a]
        else:
            if b["free"]:
                f = np.array([b["F"][0] / b["mass"], 0.0, 0.0])
                b["X"] = b["X"] + np.array([b["U"][0], 0.0, 0.0])
                b["U"] = b["U"] + f
            b["t"] += 1
            self._pose()

    def _offset(self, a, p):
        """Displacement of lattice coordinates p from the body's reference point (nearest image of a sphere)."""
        b = self.b
        if b["kind"] == "airfoil" and a == 2:
            return p.double()
        d = p.double() - b["X"][a]
        if b["kind"] == "sphere" and self.faces[2 * a] == PERIODIC:
            n = self.n[a]
            d = torch.where(d > n / 2, d - n, torch.where(d < -n / 2, d + n, d))
        return d

    def _in_airfoil(self, x, y):
        b = self.b
        dx, dy = x - b["X"][0], y - b["X"][1]
        xi, eta = (dx * b["ca"] - dy * b["sa"]) / b["chord"], (dx * b["sa"] + dy * b["ca"]) / b["chord"]
        m, p, t = b["camber_m"], b["camber_p"], b["thick"]
        yc = torch.where(xi < p, m / p ** 2 * (2 * p * xi - xi * xi), m / (1 - p) ** 2 * (1 - 2 * p + 2 * p * xi - xi * xi))
        th = t[0] * torch.sqrt(xi.clamp(min=0)) + xi * (t[1] + xi * (t[2] + xi * (t[3] + xi * t[4])))
        return (xi >= 0) & (xi <= 1) & ((eta - yc).abs() < th)

    def _inside(self):
        b, (nx, ny, nz) = self.b, self.n
        x, y, z = (torch.arange(v, device=DEV) for v in self.n)
        if b["kind"] == "sphere":
            d = [self._offset(a, p) ** 2 for a, p in enumerate((x, y, z))]
            return d[0][None, None] + d[1][None, :, None] + d[2][:, None, None] < b["R"] ** 2
        if b["kind"] == "airfoil":
            return self._in_airfoil(x.double()[None, :], y.double()[:, None])[None].expand(nz, ny, nx).contiguous()
        # swimmer: parity of the surface crossings beyond a node along +x, column by column
        P = b["P"][b["tri"]]  # (nt, 3 vertices, 3)
        lo, hi = torch.ceil(P[..., 1:].amin(1)).long(), torch.floor(P[..., 1:].amax(1)).long()
        count = torch.zeros(nz, ny, nx + 1, dtype=torch.int32, device=DEV)
        spread = (hi - lo).clamp(min=-1).amax(0) + 1

        def edge(u, v, yy, zz):
            """Signed area value of edge u -> v evaluated from its lower-index vertex, zero counted positive there."""
            iu, iv = b["tri"][:, u], b["tri"][:, v]
            sw = iu > iv
            A, B = torch.where(sw[:, None], P[:, v], P[:, u]), torch.where(sw[:, None], P[:, u], P[:, v])
            val = (B[:, 1] - A[:, 1]) * (zz - A[:, 2]) - (B[:, 2] - A[:, 2]) * (yy - A[:, 1])
            sg = torch.where(val >= 0, 1, -1)
            return torch.where(sw, -val, val), torch.where(sw, -sg, sg)

        for ky in range(int(spread[0])):
            for kz in range(int(spread[1])):
                yi, zi = lo[:, 0] + ky, lo[:, 1] + kz
                yy, zz = yi.double(), zi.double()
                (e0, s0), (e1, s1), (e2, s2) = edge(1, 2, yy, zz), edge(2, 0, yy, zz), edge(0, 1, yy, zz)
                den = e0 + e1 + e2
                hit = (s0 == s1) & (s1 == s2) & (den != 0) & (yi <= hi[:, 0]) & (zi <= hi[:, 1])
                xc = (e0 * P[:, 0, 0] + e1 * P[:, 1, 0] + e2 * P[:, 2, 0])[hit] / den[hit]
                at = torch.ceil(xc).long().clamp(0, nx)  # nodes x < at lie before the crossing
                count.index_put_((zi[hit], yi[hit], at), torch.ones_like(at, dtype=torch.int32), accumulate=True)
        beyond = count.flip(2).cumsum(2).flip(2)
        return (beyond[..., 1:] % 2) == 1

    # ---- nodes at the body
    def _near(self, n, sign, clamp):
        """Flat indices (27, len(n)) of n + sign c_i; -1 through a non-periodic face (an outflow face clamps if asked)."""
        nx, ny, nz = self.n
        p = [n % nx, (n // nx) % ny, n // (nx * ny)]
        gone = torch.zeros((Q, len(n)), dtype=torch.bool, device=DEV)
        q = []
        for a in range(3):
            v = p[a][None] + sign * self.c[:, a][:, None]
            for out, face in ((v < 0, self.faces[2 * a]), (v >= self.n[a], self.faces[2 * a + 1])):
                if face != PERIODIC and not (clamp and face == OUTFLOW):
                    gone |= out
            q.append(v % self.n[a] if self.faces[2 * a] == PERIODIC else v.clamp(0, self.n[a] - 1))
        at = q[0] + nx * (q[1] + ny * q[2])
        return torch.where(gone, -1, at), p

    def _state_at(self, S, at):
        """rho and u (3) of the nodes `at` (any shape; -1 gives node 0)."""
        g = S.view(Q, -1)[:, at.clamp(min=0)]
        drho, j = _moments(g)
        return self.rho0 + drho, j / (self.rho0 + drho)

    def _gradient(self, u, ok, uc):
        """du[a][b] by central, one-sided or no differences over the neighbours x +- e_b; u (3, 27, m)."""
        du = [[None] * 3 for _ in range(3)]
        for b, st in enumerate((9, 3, 1)):
            op, om = ok[13 + st], ok[13 - st]
            for a in range(3):
                up, um = u[a, 13 + st], u[a, 13 - st]
                du[a][b] = torch.where(op & om, (up - um) / 2, torch.where(op, up - uc[a], torch.where(om, uc[a] - um, torch.zeros_like(up))))
        return du

    def _grad(self, rho, u, du):
        """Shifted Grad distribution (Eqs. grad, pressure, pressure2), (27, m)."""
        k = rho / (6 * self.beta)
        T = [[rho * u[a] * u[b] - k * (du[a][b] + du[b][a]) for b in range(3)] for a in range(3)]
        tr = (T[0][0] + T[1][1] + T[2][2]) / 3
        out = []
        for i, c in enumerate(C):
            cu = sum(c[a] * u[a] for a in range(3))
            cc = sum(c[a] * c[b] * T[a][b] for a in range(3) for b in range(3))
            out.append(W[i] * ((rho - self.rho0) + 3 * rho * cu + 4.5 * (cc - tr)))
        return torch.stack(out)

    def _refill(self, S, was):
        n = torch.nonzero((was & ~self.solid).reshape(-1)).flatten()
        if not len(n):
            return
        at, p = self._near(n, 1, False)
        ok = (at >= 0) & ~was.reshape(-1)[at.clamp(min=0)]
        ok[13] = False
        rho_n, u_n = self._state_at(S, at)
        cnt = ok.sum(0)
        rho = torch.where(cnt > 0, (rho_n * ok).sum(0) / cnt.clamp(min=1), self.rho0)
        b = self.b
        u = torch.tensor(b["U"], device=DEV)[:, None].expand(3, len(n)).clone()
        if b["kind"] == "swimmer":
            u[1] += self._rate((p[0].double() - b["X"][0]).clamp(0, b["L"]), b["t"])
        S.view(Q, -1)[:, n] = self._grad(rho, u, self._gradient(u_n, ok, u))

    def _links(self, x, y, z, d):
        """Fraction q and wall velocity (3) of the links from nodes (x, y, z) along -c_d."""
        b, c = self.b, self.c[d]
        U = torch.tensor(b["U"], device=DEV)[:, None].expand(3, len(d))
        if b["kind"] == "sphere":
            o = torch.stack([self._offset(a, p) for a, p in enumerate((x, y, z))], 1)
            cc, cd, dd = (c * c).sum(1), (c * o).sum(1), (o * o).sum(1)
            return (cd - torch.sqrt((cd * cd - cc * (dd - b["R"] ** 2)).clamp(min=0))) / cc, U
        if b["kind"] == "airfoil":
            lo, hi = torch.zeros(len(d), dtype=torch.float64, device=DEV), torch.ones(len(d), dtype=torch.float64, device=DEV)
            for _ in range(50):
                mid = (lo + hi) / 2
                inn = self._in_airfoil(x - mid * c[:, 0], y - mid * c[:, 1])
                lo, hi = torch.where(inn, lo, mid), torch.where(inn, mid, hi)
            return (lo + hi) / 2, U
        # swimmer: first triangle crossed, p - s c = A + u e1 + v e2
        P, V = b["P"][b["tri"]], b["V"][b["tri"]]
        A, e1, e2 = P[:, 0], P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]
        q, uw = torch.empty(len(d), dtype=torch.float64, device=DEV), torch.empty((3, len(d)), dtype=torch.float64, device=DEV)
        p = torch.stack([x, y, z], 1).double()
        normal = torch.linalg.cross(e1, e2)
        for k in range(0, len(d), 512):
            w = slice(k, k + 512)
            c0 = c[w].double()
            D = c0 @ normal.T
            r = p[w][:, None, :] - A[None]
            # det(r, e2, c) = c . (r x e2), det(e1, r, c) = c . (e1 x r)
            cr = torch.linalg.cross(c0[:, None, :].expand_as(r), r)
            uu, vv, ss = (cr * e2[None]).sum(2) / D, -(cr * e1[None]).sum(2) / D, (r * normal[None]).sum(2) / D
            ok = (D != 0) & (uu >= 0) & (vv >= 0) & (uu + vv <= 1) & (ss >= 0) & (ss <= 1)
            s, t = torch.where(ok, ss, 2.0).min(1)
            none = s > 1.5
            at = torch.arange(len(t), device=DEV)
            bu, bv = uu[at, t], vv[at, t]
            vel = (1 - bu - bv)[:, None] * V[t, 0] + bu[:, None] * V[t, 1] + bv[:, None] * V[t, 2]
            mid = torch.tensor(b["U"], device=DEV)[None].repeat(len(t), 1)
            mid[:, 1] += self._rate((p[w][:, 0] - 0.5 * c0[:, 0] - b["X"][0]).clamp(0, b["L"]), b["t"])
            q[w] = torch.where(none, 0.5, s)
            uw[:, w] = torch.where(none[:, None], mid, vel).T
        return q, uw

    def _boundary(self, S, out):
        solid = self.solid.reshape(-1)
        near = torch.zeros_like(self.solid)
        for i, c in enumerate(C):
            if i == 13:
                continue
            ix = [self._axis(a, c[a]) for a in range(3)]
            src = self.solid[ix[2][0]][:, ix[1][0]][:, :, ix[0][0]]
            cut = (ix[2][1][:, None, None] > 0) | (ix[1][1][None, :, None] > 0) | (ix[0][1][None, None, :] > 0)
            near |= src & ~cut
        n = torch.nonzero((near & ~self.solid).reshape(-1)).flatten()
        src, (x, y, z) = self._near(n, -1, True)
        miss = (src >= 0) & solid[src.clamp(min=0)]
        miss[13] = False
        at, _ = self._near(n, 1, False)
        ok = (at >= 0) & ~solid[at.clamp(min=0)]
        _, u_n = self._state_at(S, at)
        # known pulls (the walls and equilibrium faces of the box as in streaming)
        own = S.view(Q, -1)[:, n]
        F = torch.where(src >= 0, torch.gather(S.view(Q, -1), 1, src.clamp(min=0)), torch.zeros_like(own))
        if bool((src < 0).any()):
            wall = torch.zeros_like(miss)
            for a, p in enumerate((x, y, z)):
                v = p[None] - self.c[:, a][:, None]
                for gone, face in ((v < 0, self.faces[2 * a]), (v >= self.n[a], self.faces[2 * a + 1])):
                    if face == WALL:
                        wall |= gone
            F = torch.where(src < 0, torch.where(wall, own.flip(0), self.g_face[:, None]), F)
        d, m = torch.nonzero(miss, as_tuple=True)
        q, uw = self._links(x[m], y[m], z[m], d)
        fbb = own.flip(0)
        dyn = torch.zeros_like(F)
        dyn[d, m] = 6 * self.W[d] * self.rho0 * (self.c[d].T * uw).sum(0)
        ut = torch.zeros((3, Q, len(n)), dtype=torch.float64, device=DEV)
        fluid = ok[d, m]
        ut[:, d, m] = torch.where(fluid, (q * u_n[:, d, m] + uw) / (1 + q), uw)
        rho_t = self.rho0 + torch.where(miss, fbb, F).sum(0) + dyn.sum(0)
        u_t = ut.sum(1) / miss.sum(0)
        F = torch.where(miss, self._grad(rho_t, u_t, self._gradient(u_n, ok, u_n[:, 13])), F)
        # momentum exchange (Sec. 4.1)
        c = self.c[d].T.double()
        fo, fi = fbb[d, m] + self.W[d] * self.rho0, F[d, m] + self.W[d] * self.rho0
        dF = (-c - uw) * fo - (c - uw) * fi
        r = torch.stack([self._offset(a, p[m]) for a, p in enumerate((x, y, z))]) - q * c
        self.b["F"] = dF.sum(1).cpu().numpy()
        self.b["M"] = torch.linalg.cross(r, dF, dim=0).sum(1).cpu().numpy()
        out.view(Q, -1)[:, n] = _collide(F, self.beta, self.rho0, self.gamma)

    def answer(self, like):
        b = self.b
        # the counts are whole numbers of the library's own bookkeeping: no value in 64 bits
        return dict(pose=torch.tensor([*b["X"], *b["U"]]), force=torch.tensor([*b["F"], *b["M"]]), counts=None)


def _start(dims, fields):
    rho, u = fields
    a = _feq(rho.double() - 1.0, rho.double(), u.double().permute(3, 0, 1, 2))
    return a


def _exact_refined(case, seed, s):
    dims = (case["nx"], case["ny"], case["nz"])
    lo, hi = s["lo"], s["hi"]
    full = [False, False, True]
    m = [h - l for l, h in zip(lo, hi)]
    fdims = tuple(2 * dims[a] if full[a] else 2 * m[a] + 2 for a in range(3))
    co = _Exact(dims, s, "analytic")
    fi = _Exact(fdims, dict(nu=2 * s["nu"], faces=FACES["periodic"], u_face=(0.0,) * 3), "analytic", s["body"])
    c = [_start(dims, _flow(dims, seed, s["base"], s["amp"]))]
    f = [_start(fdims, _flow(fdims, seed, s["base"], s["amp"], lo, 0.5, dims))]
    c.append(torch.zeros_like(c[0]))
    f.append(torch.zeros_like(f[0]))
    E = [dims[a] if full[a] else m[a] + 1 for a in range(3)]   # coarse nodes of the block
    Ef = [2 * E[a] if full[a] else 2 * m[a] + 1 for a in range(3)]
    block = (slice(None), *(slice(lo[a], lo[a] + E[a]) for a in (2, 1, 0)))

    def shell(sizes, inset):
        """Mask of a box whose `inset` outer layers along the closed axes are set."""
        k = torch.zeros(sizes[2], sizes[1], sizes[0], dtype=torch.bool, device=DEV)
        for dim, a in ((0, 2), (1, 1), (2, 0)):
            if not full[a]:
                k.narrow(dim, 0, inset)[:] = True
                k.narrow(dim, sizes[a] - inset, inset)[:] = True
        return k

    skip = torch.zeros(dims[2], dims[1], dims[0], dtype=torch.bool, device=DEV)
    skip[tuple(slice(lo[a] + (0 if full[a] else 1), lo[a] + (E[a] if full[a] else m[a])) for a in (2, 1, 0))] = True
    co.keep = skip
    ends = torch.zeros(fdims[2], fdims[1], fdims[0], dtype=torch.bool, device=DEV)
    ends[tuple(slice(0, Ef[a]) for a in (2, 1, 0))] = shell(Ef, 1)
    pad = torch.ones_like(ends)
    pad[tuple(slice(0, Ef[a]) for a in (2, 1, 0))] = False
    fi.keep = ends | pad
    ring = shell(E, 2) & ~shell(E, 1)  # the coarse layer inside the block's surface

    def moments(g):
        drho, j = _moments(g)
        u = j / (1 + drho)
        return torch.stack([drho, *u, *_stress(g - _feq(drho, 1 + drho, u))])

    def rebuild(M, k):
        u = M[1:4]
        P = [[M[4], M[7], M[8]], [M[7], M[5], M[9]], [M[8], M[9], M[6]]]
        g = _feq(M[0], 1 + M[0], u)
        tr = (M[4] + M[5] + M[6]) / 3
        return torch.stack([g[i] + W[i] * 4.5 * k * (sum(C[i][a] * C[i][b] * P[a][b] for a in range(3) for b in range(3)) - tr) for i in range(Q)])

    def fill(buf, M):
        at = []
        for a in range(3):
            j = torch.arange(Ef[a], device=DEV)
            at.append((j // 2, (j // 2 + j % 2) % E[a] if full[a] else j // 2 + j % 2))
        for dim, a in ((3, 0), (2, 1), (1, 2)):
            M = (M.index_select(dim, at[a][0]) + M.index_select(dim, at[a][1])) / 2
        k = shell(Ef, 1)
        v = _collide(rebuild(M[:, k], co.beta / (2 * fi.beta)), fi.beta, 1.0, "analytic")
        buf[:, ends] = v

    Mt = moments(c[0][block])
    fill(f[0], Mt)
    for _ in range(case["steps"]):
        F = co.pulled(c[0], 0, dims[2])[block]
        Mn = moments(F)
        del F
        fill(f[1], (Mt + Mn) / 2)
        co.step(c[0], c[1])
        fi.step(f[0], f[1])
        G = fi.pulled(f[1], 0, fdims[2])[(slice(None), *(slice(0, 2 * E[a] if full[a] else 2 * m[a] + 1, 2) for a in (2, 1, 0)))]
        part = c[1][block]
        part[:, ring] = _collide(rebuild(moments(G[:, ring]), 2 * fi.beta / co.beta), co.beta, 1.0, "analytic")
        c[1][block] = part
        del G, part
        fill(f[0], Mn)
        fi.step(f[1], f[0])
        c.reverse()
        Mt = Mn
    return dict(f=c[0], fine=f[0], **fi.answer(None))


@torch.no_grad()
def exact(case, seed):
    """run()'s outputs in 64 bits.  None for the adjoint (a taped FP64 run of its horizon takes more than 20 seconds) and
    for the swimmer that turns (the same, by the moments of its mesh)."""
    kind = case["kind"]
    if kind == "adjoint" or case.get("free", 0) & 6:
        return None
    s, dims = _setting(case, seed), (case["nx"], case["ny"], case["nz"])
    if kind == "refined":
        return _exact_refined(case, seed, s)
    a = _start(dims, _flow(dims, seed, s["base"], s["amp"]))
    if kind == "setup":
        drho, j = _moments(a)
        rho = 1 + drho
        return dict(f=a, totals=torch.stack([rho.sum(), *(j[k].sum() for k in range(3)), ((j ** 2).sum(0) / (2 * rho)).sum()]))
    e = _Exact(dims, s, case.get("gamma", "analytic"), s["body"])
    b = torch.zeros_like(a)
    for _ in range(case["steps"]):
        e.step(a, b)
        a, b = b, a
    return dict(f=a) if s["body"] is None else dict(f=a, **e.answer(a))
