"""The work that a user of this framework has it do, as cases that can be timed and compared.

A case is a stretch of a simulation between two snapshots (steps of a resident solver, then the state
that the steps left), a tick of a served batch of shots, or one misfit gradient of an inversion.  A
solver keeps its grid, material and state on the device, as a user's program does; ``run`` advances it
through the public entry points and returns the whole state or gradient.

Families (``case["family"]``)
  stretch    2-D leapfrog or RK4 steps: ``model`` names the grid, medium and data (below)
  batch      resident shots of mixed sizes advanced together by the batch's persistent kernel
  gradient   misfit gradient with respect to the density and the stiffness
  block3d    3-D leapfrog steps on one curvilinear block

2-D models
  topography two stacked blocks under a hilly free surface, tilted VTI, welded interface, Robin sides,
             Ricker point force at the surface
  shot       one curvilinear block, smooth random pair stiffness, free top, displacement elsewhere,
             Ricker point force inside
  forced     ``blocks`` x ``blocks`` curvilinear blocks welded together, time-harmonic body force and
             traction data on the outer faces; with one block displacement data on every face
  survey     the shot's grid with a smooth tilted VTI medium and the source near the surface

``exact`` restates the scheme in plain torch in 64 bits: first derivatives with the summation-by-parts
property, the narrow second derivative as D b D - H^-1 R(b), the boundary and interface terms, leapfrog,
RK4, and reverse-mode differentiation for the gradient.
"""
import math

import numpy as np
import torch

DEV = "cuda"
BASIS = [("sin", 1.0), ("cos", 1.0), ("sin", 2.0), ("cos", 2.0)]


# ----------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the headline run: a hilly-surface section at full resolution, ten steps between two looks
        dict(name="topography_4001x2001_f32", family="stretch", model="topography", n1=4001, n2=2001, order=6,
             precision="fp32", integrator="leapfrog", stencil="narrow", steps=10),
        # one forward shot of ordinary size as a server steps it: graph-replayed ticks
        dict(name="shot_1001_f32_graph", family="stretch", model="shot", n1=1001, n2=1001, order=6,
             precision="fp32", integrator="graph", stencil="narrow", steps=64),
        # the smallest shot of a served mix, on its own: every step is a few small launches
        dict(name="shot_201_f32", family="stretch", model="shot", n1=201, n2=201, order=6,
             precision="fp32", integrator="leapfrog", stencil="narrow", steps=40),
        # the smallest accuracy run: boundary data on all faces and a body force, in double precision
        dict(name="forced_101_f64_order4", family="stretch", model="forced", n1=101, n2=101, order=4, blocks=1,
             precision="fp64", integrator="leapfrog", stencil="narrow", steps=40),
        # a multiblock accuracy run in double precision
        dict(name="forced_4x401_f64", family="stretch", model="forced", n1=401, n2=401, order=6, blocks=2,
             precision="fp64", integrator="leapfrog", stencil="narrow", steps=8),
        # the paper's integrator on a section of ordinary size
        dict(name="rk4_topography_2001x1001_f32", family="stretch", model="topography", n1=2001, n2=1001, order=6,
             precision="fp32", integrator="rk4", stencil="narrow", steps=4),
        # a convergence study with the paper's integrator: double precision, fourth order, odd sizes
        dict(name="rk4_shot_161x243_f64_order4", family="stretch", model="shot", n1=161, n2=243, order=4,
             precision="fp64", integrator="rk4", stencil="narrow", steps=10),
        # the wide-stencil operator of the narrow/wide comparison
        dict(name="wide_topography_2001x1001_f32", family="stretch", model="topography", n1=2001, n2=1001, order=6,
             precision="fp32", integrator="leapfrog", stencil="wide", steps=10),
        # a tick of continuous batching: a dozen resident shots of mixed sizes
        dict(name="batch_12_shots_f32", family="batch", shots=12, lo=201, hi=1201, order=6, steps=32),
        # one gradient of an inversion on a survey-sized block (a short record: the work is the same per step)
        dict(name="gradient_501_f32", family="gradient", n1=501, n2=501, order=6, precision="fp32", steps=64,
             receivers=48, layout="voigt6"),
        # the 3-D operator on a block of ordinary size, ragged in every direction
        dict(name="block3d_160x151x144_f32", family="block3d", n1=160, n2=151, n3=144, order=6, precision="fp32",
             steps=300),
        # a small 3-D block in double precision at fourth order (accuracy checks of the 3-D operator)
        dict(name="block3d_64x61x57_f64_order4", family="block3d", n1=64, n2=61, n3=57, order=4, precision="fp64",
             steps=40),
    ]


def _size(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: FP32 sixth-order stretches most often, as in use."""
    kind = rng.choice(["stretch", "stretch", "stretch", "rk4", "wide", "fp64", "fp64", "batch", "gradient", "3d", "3d64"])
    order = rng.choice([6, 6, 6, 4, 2])
    if kind in ("stretch", "rk4", "wide"):
        model = rng.choice(["topography", "shot", "shot", "forced"])
        c = dict(family="stretch", model=model, n1=_size(rng, 101, 2401), n2=_size(rng, 101, 1601), order=order,
                 precision="fp32", integrator="rk4" if kind == "rk4" else "leapfrog",
                 stencil="wide" if kind == "wide" else "narrow", steps=rng.randrange(4, 33))
        if model == "forced":
            c["blocks"] = rng.choice([1, 2])
            c["n1"] = c["n2"] = _size(rng, 101, 901)
        elif kind == "stretch" and rng.random() < 0.4:
            c.update(integrator="graph", steps=2 * rng.randrange(2, 17))
        return c
    if kind == "fp64":
        model = rng.choice(["forced", "shot", "topography"])
        c = dict(family="stretch", model=model, n1=_size(rng, 61, 601), n2=_size(rng, 61, 601), order=order,
                 precision="fp64", integrator=rng.choice(["leapfrog", "leapfrog", "rk4"]),
                 stencil=rng.choice(["narrow", "narrow", "narrow", "wide"]), steps=rng.randrange(4, 13))
        if model == "forced":
            c["blocks"] = rng.choice([1, 2])
            c["n2"] = c["n1"]
        return c
    if kind == "batch":
        lo = _size(rng, 101, 501)
        return dict(family="batch", shots=rng.randrange(3, 13), lo=lo, hi=lo + rng.randrange(1, 701), order=order,
                    steps=16 * rng.randrange(1, 4))
    if kind == "gradient":
        return dict(family="gradient", n1=_size(rng, 101, 501), n2=_size(rng, 101, 501), order=order,
                    precision=rng.choice(["fp32", "fp32", "fp64"]), steps=rng.randrange(24, 65),
                    receivers=rng.randrange(4, 65), layout=rng.choice(["voigt6", "pair10"]))
    big = kind == "3d"
    return dict(family="block3d", n1=_size(rng, 30, 150 if big else 64), n2=_size(rng, 30, 150 if big else 64),
                n3=_size(rng, 30, 140 if big else 64), order=order, precision="fp32" if big else "fp64",
                steps=rng.randrange(20, 101) if big else rng.randrange(5, 31))


def work(case):
    """Per step every node reads its displacement, its previous level or increment, its coefficients
    and 1/(rho J) once and writes what the step changes once (a step needs the step before it, so
    nothing carries over but what the chip holds): words per node below.  The floating-point
    operations are those of the stencils."""
    f, q = case["family"], case["order"] // 2
    es = 4 if case.get("precision", "fp32") == "fp32" else 8
    flops2 = 8 * 3 * q + 28 + 6 * q * (4 * q) + 16 * q   # four derivatives and their divergence, edge weights, edges
    if f == "block3d":
        n = case["n1"] * case["n2"] * case["n3"]
        flops3 = 18 * 3 * q + 9 * 18 + 3 * (2 * q + 1) * (3 * 4 * q + 18)
        return {"bytes": n * 58 * es * case["steps"], "flops": n * flops3 * case["steps"]}
    if f == "batch":
        n = sum(s * s for s in _sides(case))
        return {"bytes": n * 19 * es * case["steps"], "flops": n * flops2 * case["steps"]}
    n = case["n1"] * case["n2"]
    if f == "gradient":
        # a forward and an adjoint step per level (the adjoint steps two levels), both levels read again
        # for the gradient; the gradient's products cost about one more step's arithmetic
        return {"bytes": n * es * case["steps"] * (19 + 17 + 4), "flops": n * flops2 * 3 * case["steps"]}
    n *= {"topography": 2, "forced": case.get("blocks", 1) ** 2}.get(case["model"], 1)
    words, passes = (19 if es == 4 else 17), case["steps"]
    if case["integrator"] == "rk4":
        # a stage reads its input, the coefficients and 1/(rho J) and what its combination takes, and
        # writes the next input and its acceleration: 86 words over the four stages
        words, passes = 86 / 4, 4 * case["steps"]
    if case["model"] == "forced":
        words += 8
    if case["stencil"] == "wide":
        flops2 = 8 * 3 * q + 28 + 4 * 3 * q
    return {"bytes": n * words * es * passes, "flops": n * flops2 * passes}


def _sides(case):
    k, lo, hi = case["shots"], case["lo"], case["hi"]
    return [int(round(lo + (hi - lo) * i / max(1, k - 1))) for i in range(k)]


# ------------------------------------------------------------------------------------------ the inputs
class _Field:
    """A block in plain tensors: X (d, ...), rho, pair planes M[p][q] of C_IJKL (p = d I + J, q = d K + L,
    entries shared where equal), faces, forcing (2, K, ...)."""

    def __init__(self, X, rho, M, faces, forcing=None):
        self.X, self.rho, self.M, self.faces, self.forcing = X, rho, M, faces, forcing


def _waves(rng, X, modes=3, kmax=3.0):
    """A smooth field in [0, 1] of low Fourier modes of the coordinates."""
    f = 0.0
    for _ in range(modes):
        arg = float(rng.uniform(0, 2 * math.pi))
        for x in X:
            arg = arg + float(rng.uniform(-kmax, kmax)) * math.pi * x
        f = f + torch.sin(arg)
    return 0.5 + 0.5 / modes * f


def _lin(n):
    return torch.arange(n, device=DEV, dtype=torch.float64) / (n - 1)


def _grid2(n1, n2):
    return _lin(n1)[None, :].expand(n2, n1), _lin(n2)[:, None].expand(n2, n1)


def _vti2(scale, tilt, rho=2.3, vp=3.5, vs=2.0, eps=0.2, delta=0.1):
    """Pair planes of a tilted VTI stiffness: the Voigt matrix scaled by ``scale``, turned by ``tilt``."""
    c33, c55 = rho * vp * vp, rho * vs * vs
    c11 = c33 * (1 + 2 * eps)
    c13 = math.sqrt(2 * delta * c33 * (c33 - c55) + (c33 - c55) ** 2) - c55
    V, v = [[c11, c13, 0.0], [c13, c33, 0.0], [0.0, 0.0, c55]], [0, 2, 2, 1]
    c, s = torch.cos(tilt), torch.sin(tilt)
    R = [[c, -s], [s, c]]
    Rp = [[R[p // 2][a // 2] * R[p % 2][a % 2] for a in range(4)] for p in range(4)]
    T = [[sum(Rp[p][a] * V[v[a]][v[b]] for a in range(4) if V[v[a]][v[b]]) for b in range(4)] for p in range(4)]
    M = [[None] * 4 for _ in range(4)]
    for p in range(4):
        for q in range(p, 4):
            M[p][q] = M[q][p] = scale * sum(T[p][b] * Rp[q][b] for b in range(4))
    return M, c11


def _pair_random(rng, X):
    """Smooth random stiffness with major symmetry only: entries in [0, 1], four more on the diagonal."""
    M = [[None] * 4 for _ in range(4)]
    for p in range(4):
        for q in range(p, 4):
            M[p][q] = M[q][p] = _waves(rng, X) + (4.0 if p == q else 0.0)
    return M


def _edge(a, f):
    """Face f (0: x1=0, 1: x1=1, 2: x2=0, ...) of a tensor whose last axis is x1."""
    return a.select(a.dim() - 1 - f // 2, 0 if f % 2 == 0 else -1)


def _steepest(X, h):
    """min over the nodes of sigma_min(dX/dx) (a coarse sample: the maps are smooth)."""
    d = X.shape[0]
    st = [max(1, n // (150 if d == 2 else 30)) for n in X.shape[1:]]
    Xs = X[(slice(None),) + tuple(slice(None, None, s) for s in st)]
    sp = [s * h[d - 1 - k] for k, s in enumerate(st)]
    G = torch.stack([torch.stack(torch.gradient(Xs[I], spacing=sp)) for I in range(d)])
    return float(torch.linalg.svdvals(G.reshape(d, d, -1).permute(2, 0, 1)).min())


def _model2(case, seed):
    """(blocks, time basis, sources, dt) of a 2-D case; a source is (block, (x1, x2), direction, amplitude,
    peak frequency, t0)."""
    rng = np.random.default_rng([20031, seed])
    n1, n2, model = case["n1"], case["n2"], case.get("model", "survey")
    h = (1.0 / (n1 - 1), 1.0 / (n2 - 1))
    basis, sources, blocks = [], [], []
    if model == "topography":
        W = D = 8.0
        xs, am, wd = rng.uniform(0.1, 0.9, 5) * W, rng.uniform(0.02, 0.06, 5) * D, rng.uniform(0.06, 0.14, 5) * W
        x1, x2 = _grid2(n1, n2)
        hx = sum(float(a) * torch.exp(-((W * x1 - float(c)) / float(w)) ** 2) for a, c, w in zip(am, xs, wd))
        state = rng.bit_generator.state
        for b in range(2):
            rng.bit_generator.state = state                  # the medium is one function of the position
            yb, yt = (0.0 * hx, D / 2 + 0.5 * hx) if b == 0 else (D / 2 + 0.5 * hx, D + hx)
            X = torch.stack([W * x1, yb + x2 * (yt - yb)])
            tilt = (math.pi / 3) * (_waves(rng, X / W) - 0.5)
            scale = 0.9 + 0.2 * _waves(rng, X / W)
            M, c11 = _vti2(scale, tilt)
            faces = []
            for f in range(4):
                if f == 3 - b:
                    faces.append(dict(kind="interface", nbr=(1 - b, 2 + b)))
                elif b == 1 and f == 3:
                    faces.append(dict(kind="robin"))
                else:
                    m = f // 2                               # U = n C n / depth
                    faces.append(dict(kind="robin", U=torch.stack([_edge(M[2 * m + j][2 * m + l], f) / D
                                                                   for j, l in ((0, 0), (0, 1), (1, 1))])))
            blocks.append(_Field(X, 2.3 * scale, M, faces))
        sources = [(1, (0.5, 1.0), (0.0, -1.0), 1.0, 8.0, 0.125)]
        speed = math.sqrt(c11 / 2.3)
    elif model in ("shot", "survey"):
        x1, x2 = _grid2(n1, n2)
        a1, a2 = (float(v) for v in rng.uniform(0.02, 0.05, 2))
        X = torch.stack([x1 + a1 * torch.sin(2 * math.pi * x2) * torch.sin(math.pi * x1),
                         x2 + a2 * torch.sin(math.pi * x2) * torch.sin(2 * math.pi * x1)])
        if model == "shot":
            M, rho, speed = _pair_random(rng, (x1, x2)), 1 + _waves(rng, (x1, x2)), math.sqrt(8.0)
            at, peak = tuple(float(v) for v in rng.uniform(0.3, 0.7, 2)), 4.0
        else:
            scale = 0.9 + 0.2 * _waves(rng, X)
            M, c11 = _vti2(scale, (math.pi / 4) * (_waves(rng, X) - 0.5))
            rho, speed, at, peak = 2.3 * scale, math.sqrt(c11 / 2.3), (0.5, 0.95), 15.0
        blocks = [_Field(X, rho, M, [dict(kind="displacement")] * 3 + [dict(kind="robin")])]
        sources = [(0, at, (0.0, -1.0), 1.0, peak, 1.0 / peak)]
    else:
        nb, basis = case["blocks"], BASIS
        state = rng.bit_generator.state
        xi1, xi2 = _grid2(n1, n2)
        for b in range(nb * nb):
            bx, by = b % nb, b // nb
            rng.bit_generator.state = state
            x, y = (bx + xi1) / nb, (by + xi2) / nb
            bump = 0.05 * torch.sin(2 * math.pi * x) * torch.sin(2 * math.pi * y)
            X = torch.stack([x + bump, y + bump])
            M, rho = _pair_random(rng, X), 1 + _waves(rng, X)
            harm = torch.stack([_waves(rng, X) - 0.5 for _ in range(8)]).reshape(2, 4, n2, n1)
            faces = []
            for f in range(4):
                outer = (bx == 0, bx == nb - 1, by == 0, by == nb - 1)[f]
                if outer:
                    faces.append(dict(kind="displacement" if nb == 1 else "robin", g=_edge(harm, f).contiguous()))
                else:
                    faces.append(dict(kind="interface", nbr=(b + (-1, 1, -nb, nb)[f], f ^ 1)))
            blocks.append(_Field(X, rho, M, faces, forcing=10.0 * harm))
        speed = math.sqrt(8.0)
    slow = min(_steepest(b.X, h) for b in blocks)
    # the paper steps RK4 at a CFL number of 0.4 to 0.5, leapfrog takes 0.25 to 0.3
    cfl = 0.4 if case.get("integrator") == "rk4" else 0.25
    return blocks, basis, sources, cfl * min(h) * slow / speed


def _start(case, seed, blocks, dt):
    """A smooth displacement and velocity per block, a wave in motion; returned as (u_prev, u_cur) levels, or (u, v) for RK4,
    in the precision of the case."""
    rng = np.random.default_rng([20032, seed])
    kind = torch.float32 if case.get("precision", "fp32") == "fp32" else torch.float64
    state, out = rng.bit_generator.state, []
    for b in blocks:
        rng.bit_generator.state = state                      # one function of the position
        d = b.X.shape[0]
        Xn = b.X / max(1.0, float(b.X.abs().max()))
        # waves of a few Hz (a survey's 15 Hz are shorter and faster): the velocity is omega times as large
        kmax, omega = (10.0, 60.0) if case["family"] == "gradient" else (3.0, 25.0)
        u = torch.stack([2 * _waves(rng, Xn, kmax=kmax) - 1 for _ in range(d)])
        v = omega * torch.stack([2 * _waves(rng, Xn, kmax=kmax) - 1 for _ in range(d)])
        out.append((u.to(kind), v.to(kind)) if case.get("integrator") == "rk4" else ((u - dt * v).to(kind), u.to(kind)))
    return out


def _host(t):
    return t.to(torch.float64).cpu().numpy()


def _problem(case, blocks, basis, sources):
    import workloads as W
    made = []
    for b in blocks:
        planes = {id(b.M[p][q]): b.M[p][q] for p in range(4) for q in range(p, 4)}
        host = {k: _host(v) for k, v in planes.items()}
        C = np.empty((4, 4) + tuple(b.rho.shape))
        for p in range(4):
            for q in range(4):
                C[p, q] = host[id(b.M[p][q])]
        faces = []
        for f in b.faces:
            take = {k: _host(f[k]) for k in ("U", "g") if k in f}
            faces.append(W.Face(f["kind"], nbr=f["nbr"] + (False,) if "nbr" in f else None, **take))
        made.append(W.Block(X=_host(b.X), rho=_host(b.rho), C=C.reshape((2, 2, 2, 2) + tuple(b.rho.shape)), faces=faces,
                            forcing=None if b.forcing is None else _host(b.forcing)))
    src = [W.PointSource(block=k, x_ref=x, direction=d, amplitude=a, alpha_p=p, t0=t) for k, x, d, a, p, t in sources]
    return W.Problem(case["family"], case["order"], made, time_basis=list(basis), sources=src,
                     stencil=case.get("stencil", "narrow"))


def _pitched(u):
    """A device field (2, N2, N1) in rows of a multiple of 16 bytes, as sbp_set_state_device takes it."""
    n1 = u.shape[-1]
    buf = torch.zeros(u.shape[:-1] + ((n1 + 3) // 4 * 4,), dtype=u.dtype, device=u.device)
    buf[..., :n1] = u
    return buf


def _load(S, b, prev, cur):
    prev, cur = _pitched(prev), _pitched(cur)
    S.sbp_set_state_device(b, prev.data_ptr(), cur.data_ptr(), cur.shape[-1], 0.0)
    torch.cuda.synchronize()                                 # the borrowed buffers may go


def _solver(case, seed):
    """A solver with its problem and state set, and the step size."""
    from paper_2003_12811_gb300 import Solver
    blocks, basis, sources, dt = _model2(case, seed)
    S = Solver(_problem(case, blocks, basis, sources), case.get("precision", "fp32"))
    start = _start(case, seed, blocks, dt)
    if case.get("integrator") == "rk4":
        S.sbp_set_state_rk4([_host(u) for u, _ in start], [_host(v) for _, v in start], 0.0)
    else:
        for b, (prev, cur) in enumerate(start):
            _load(S, b, prev, cur)
    return S, dt


def _receivers(case):
    n1, n2, k = case["n1"], case["n2"], case["receivers"]
    at = sorted({int(round((0.05 + 0.9 * i / max(1, k - 1)) * (n1 - 1))) for i in range(k)})
    return [(0, i, n2 - 1) for i in at]


def _observed(case, seed, nrec):
    """Traces of the size of the field, as a survey brings them: a smooth function of time and receiver."""
    rng = np.random.default_rng([20033, seed])
    t, r = np.arange(case["steps"])[:, None], np.arange(nrec)[None, :]
    k = rng.uniform(0.02, 0.08, (2, 2))
    ph = rng.uniform(0, 2 * np.pi, 2)
    return np.ascontiguousarray(np.stack([0.5 * np.sin(k[j, 0] * t + k[j, 1] * r + ph[j]) for j in range(2)], axis=-1))


def _model3(case, seed):
    """(block, dt) of a 3-D case: a deformed box with a hilly top, tilted transversely isotropic medium."""
    rng = np.random.default_rng([20034, seed])
    n = (case["n1"], case["n2"], case["n3"])
    x1, x2, x3 = _lin(n[0])[None, None, :], _lin(n[1])[None, :, None], _lin(n[2])[:, None, None]
    a = [float(v) for v in rng.uniform(-0.04, 0.04, 6)]
    sin, cos, pi = torch.sin, torch.cos, math.pi
    full = (n[2], n[1], n[0])
    X = torch.stack([t.expand(full) for t in (
        x1 + a[0] * sin(pi * x2) * sin(pi * x3) + a[1] * x1 * (1 - x1) * x2,
        1.2 * x2 + a[2] * sin(pi * x1) * cos(pi * x3) + a[3] * x2 * (1 - x2) * x3,
        0.9 * x3 + (a[4] * sin(2 * pi * x1) * sin(pi * x2) + a[5] * cos(pi * x1 + 0.3) * x2) * x3)])
    x = (x1, x2, x3)
    rho = (0.8 + 0.4 * _waves(rng, x)).expand(full)
    vp, vs = 1.7 + 0.6 * _waves(rng, x), 0.95 + 0.3 * _waves(rng, x)
    c33, c44 = rho * vp * vp, rho * vs * vs
    c11, c66 = 1.3 * c33, 1.2 * c44
    c13 = torch.sqrt((c33 - c44) * (1.16 * c33 - c44)) - c44
    # the stiffness is linear in the five moduli: the rotated pattern of each
    pats = {}
    for name, entries in (("11", {(0, 0): 1, (1, 1): 1, (0, 1): 1}), ("13", {(0, 2): 1, (1, 2): 1}), ("33", {(2, 2): 1}),
                          ("44", {(3, 3): 1, (4, 4): 1}), ("66", {(5, 5): 1, (0, 1): -2})):
        V = np.zeros((6, 6))
        for (i, j), v in entries.items():
            V[i, j] = V[j, i] = v
        pats[name] = V
    ang = rng.uniform(-0.6, 0.6, 3)

    def turn(t, axis):
        c_, s_ = math.cos(t), math.sin(t)
        return np.array([[c_, -s_, 0], [s_, c_, 0], [0, 0, 1]] if axis == 2 else [[c_, 0, s_], [0, 1, 0], [-s_, 0, c_]])
    R = turn(ang[0], 2) @ turn(ang[1], 1) @ turn(ang[2], 2)
    v6 = [[0, 5, 4], [5, 1, 3], [4, 3, 2]]
    M = [[None] * 9 for _ in range(9)]
    rot = []
    for V in pats.values():
        T = np.array([[[[V[v6[i][j], v6[k][l]] for l in range(3)] for k in range(3)] for j in range(3)] for i in range(3)])
        rot.append(np.einsum("ia,jb,kc,ld,abcd->ijkl", R, R, R, R, T).reshape(9, 9))
    for p in range(9):
        for q in range(p, 9):
            M[p][q] = M[q][p] = sum(float(r[p, q]) * m for r, m in zip(rot, (c11, c13, c33, c44, c66)))
    blk = _Field(X, rho, M, [dict(kind="displacement")] * 5 + [dict(kind="robin")])
    h = [1.0 / (v - 1) for v in n]
    dt = 0.2 * min(h) * _steepest(X, h) / (2.3 * math.sqrt(1.3))
    return blk, dt


def _sized(case, side, k):
    """The k-th shot of a batch as a case of its own."""
    return dict(family="stretch", model="shot", n1=side, n2=side, order=case["order"], precision="fp32",
                integrator="leapfrog", stencil="narrow")


def prepare(case, seed):
    f = case["family"]
    if f == "stretch":
        S, dt = _solver(case, seed)
        return dict(case=case, S=S, dt=dt)
    if f == "batch":
        from paper_2003_12811_gb300 import Batch
        made = [_solver(_sized(case, s, k), 1000 * seed + k) for k, s in enumerate(_sides(case))]
        # the batch goes before its solvers where a state is dropped
        return dict(case=case, batch=Batch(case["order"], case["shots"]), solvers=[S for S, _ in made], dts=[d for _, d in made])
    if f == "gradient":
        S, dt = _solver(case, seed)
        rec = _receivers(case)
        S.sbp_set_receivers(rec)
        blocks, _, _, _ = _model2(case, seed)
        prev, cur = _start(case, seed, blocks, dt)[0]
        return dict(case=case, S=S, dt=dt, observed=_observed(case, seed, len(rec)), prev=_pitched(prev), cur=_pitched(cur))
    from paper_2003_12811_gb300 import Solver3D
    blk, dt = _model3(case, seed)
    faces = ["traction" if a["kind"] == "robin" else a["kind"] for a in blk.faces]
    S = Solver3D(_host(blk.X), faces, order=case["order"], precision=case["precision"])
    n3, step = case["n3"], 32                                # planes at a time, as for a medium that is read in parts
    for k in range(0, n3, step):
        part = torch.stack([blk.M[p][q][k:k + step] for p in range(9) for q in range(p, 9)])
        S.sbp3_set_material(k, part.shape[1], _host(blk.rho[k:k + step]), _host(part))
    prev, cur = _start(case, seed, [blk], dt)[0]
    S.set_state(_host(prev), _host(cur))
    return dict(case=case, S=S, dt=dt)


# ------------------------------------------------------------------------------------------- one pass
def _fields(S, which):
    """The named fields of every block as device tensors."""
    out = []
    for b, blk in enumerate(S.problem.blocks):
        n1 = blk.N1
        buf = torch.empty((2, blk.N2, (n1 + 3) // 4 * 4), device=DEV, dtype=torch.float64 if S.precision == 0 else torch.float32)
        S.sbp_get_field_device(b, which, buf.data_ptr(), buf.shape[-1])
        out.append(buf[..., :n1])
    return out


def run(state):
    case = state["case"]
    f = case["family"]
    if f == "stretch":
        S, n, dt = state["S"], case["steps"], state["dt"]
        if case["integrator"] == "rk4":
            S.sbp_step_rk4(n, dt)
            return {"u": _fields(S, 1), "v": _fields(S, 3)}
        if case["integrator"] == "graph":
            S.sbp_step_graph(n, dt)
        else:
            S.sbp_step(n, dt)
        return {"prev": _fields(S, 0), "cur": _fields(S, 1)}
    if f == "batch":
        B = state["batch"]
        slots = [B.sbp_batch_add(S, case["steps"], dt) for S, dt in zip(state["solvers"], state["dts"])]
        for _ in range(case["steps"] // 16):
            B.sbp_batch_step(16)
        B.sbp_batch_poll()
        for slot in slots:
            B.sbp_batch_remove(slot)
        return {"cur": [_fields(S, 1)[0] for S in state["solvers"]]}
    if f == "gradient":
        from paper_2003_12811_gb300 import binding
        S, kind = state["S"], np.float32 if case["precision"] == "fp32" else np.float64
        S.sbp_set_state_device(0, state["prev"].data_ptr(), state["cur"].data_ptr(), state["cur"].shape[-1], 0.0)
        layout = binding.C_VOIGT6 if case["layout"] == "voigt6" else binding.C_PAIR10
        phi, rho, C = S.sbp_misfit_gradient(case["steps"], state["dt"], state["observed"], layout=layout)
        return {"misfit": kind(phi), "rho": rho[0].astype(kind), "C": C[0].astype(kind)}
    S, kind = state["S"], torch.float32 if case["precision"] == "fp32" else torch.float64
    S.step(case["steps"], state["dt"])
    prev, cur = S.state()
    return {"prev": torch.from_numpy(prev).to(kind), "cur": torch.from_numpy(cur).to(kind)}


# --------------------------------------------------------------------------- the same in plain torch
# h H D on the boundary rows, the norm weights H / h there and the interior coefficients, per order
def _table(order):
    a = {2: [1 / 2], 4: [2 / 3, -1 / 12], 6: [3 / 4, -3 / 20, 1 / 60]}[order]
    hw = {2: [1 / 2], 4: [17 / 48, 59 / 48, 43 / 48, 49 / 48],
          6: [13649 / 43200, 12013 / 8640, 2711 / 4320, 5359 / 4320, 7877 / 8640, 43801 / 43200]}[order]
    up = {2: {(0, 1): 1 / 2},
          4: {(0, 1): 59 / 96, (0, 2): -1 / 12, (0, 3): -1 / 32, (1, 2): 59 / 96, (2, 3): 59 / 96, (2, 4): -1 / 12,
              (3, 4): 2 / 3, (3, 5): -1 / 12},
          6: {(0, 1): 104009 / 172800, (0, 2): 30443 / 259200, (0, 3): -33311 / 86400, (0, 4): 5621 / 28800,
              (0, 5): -601 / 20736, (1, 2): -311 / 51840, (1, 3): 6743 / 5760, (1, 4): -24337 / 34560,
              (1, 5): 36661 / 259200, (2, 3): -2231 / 5184, (2, 4): 41287 / 51840, (2, 5): -7333 / 28800,
              (3, 4): 4147 / 17280, (3, 5): 25427 / 259200, (3, 6): 1 / 60, (4, 5): 342523 / 518400, (4, 6): -3 / 20,
              (4, 7): 1 / 60, (5, 6): 3 / 4, (5, 7): -3 / 20, (5, 8): 1 / 60}}[order]
    nb = len(hw)
    Q = np.zeros((nb, {2: 2, 4: 6, 6: 9}[order]))
    Q[0, 0] = -0.5
    for (i, j), v in up.items():
        Q[i, j] = v
        if j < nb:
            Q[j, i] = -v
    return a, np.array(hw), Q / np.array(hw)[:, None]


# the remainder R(b): c_alpha and the averaging offsets of b around the centre of the alpha-th difference
_REMAINDER = {2: {2: (1 / 4, [0])}, 4: {3: (1 / 18, [0, 1]), 4: (1 / 144, [0])},
              6: {4: (1 / 80, [-1, 0, 1]), 5: (1 / 600, [0, 1]), 6: (1 / 3600, [0])}}


class _Line:
    """The one-dimensional operators along one direction (axis -1-i of a field)."""

    def __init__(self, order, n, h, i):
        a, hw, Db = _table(order)
        self.a, self.n, self.h, self.i, self.order, self.nb = a, n, h, i, order, len(hw)
        self.Db = torch.tensor(Db, device=DEV)
        H = np.ones(n)
        H[:len(hw)], H[n - len(hw):] = hw, hw[::-1]
        self.H = h * torch.tensor(H, device=DEV)

    def along(self, v, like):
        """A line vector broadcast over a field."""
        return v.reshape([-1 if k == like.dim() - 1 - self.i else 1 for k in range(like.dim())])

    def D(self, u, axis=None):
        ax = u.dim() - 1 - self.i if axis is None else axis
        nb, nc, n = self.nb, self.Db.shape[1], self.n
        mid = 0.0
        for k, c in enumerate(self.a, 1):
            mid = mid + c * (u.narrow(ax, nb + k, n - 2 * nb) - u.narrow(ax, nb - k, n - 2 * nb))
        lo = torch.tensordot(self.Db, u.narrow(ax, 0, nc), dims=([1], [ax])).movedim(0, ax)
        hi = torch.tensordot(self.Db, u.narrow(ax, n - nc, nc).flip(ax), dims=([1], [ax])).movedim(0, ax)
        return torch.cat([lo, mid, -hi.flip(ax)], ax) / self.h

    def remainder(self, avg, u):
        """H^-1 R(b) u with the averages of b."""
        ax = u.dim() - 1 - self.i
        out = 0.0
        for alpha, (c, _) in _REMAINDER[self.order].items():
            y = avg[alpha] * torch.diff(u, n=alpha, dim=ax)
            shape = list(y.shape)
            shape[ax] = alpha
            z = torch.zeros(shape, dtype=y.dtype, device=y.device)
            out = out + (c / self.h ** 2) * (-1) ** alpha * torch.diff(torch.cat([z, y, z], ax), n=alpha, dim=ax)
        return out / self.along(self.H, u)

    def averages(self, b):
        """The averages of b that R(b) weights its differences with, times the norm at their centres."""
        ax, out = b.dim() - 1 - self.i, {}
        for alpha, (_, offs) in _REMAINDER[self.order].items():
            rows, c0 = self.n - alpha, alpha // 2
            if alpha % 2 == 0:
                hc = self.H[c0:c0 + rows]
            else:
                hc = 0.5 * (self.H[c0:c0 + rows] + self.H[c0 + 1:c0 + 1 + rows])
            mean = sum(b.narrow(ax, c0 + o, rows) for o in offs) / len(offs)
            out[alpha] = mean * self.along(hc, mean)
        return out


class _Block:
    """The spatial operator of one block: A u = sum_ik DD_ik(c_ijkl) u_l and what the faces add."""

    def __init__(self, field, order, wide, rho=None, M=None):
        X, d = field.X, field.X.shape[0]
        self.f, self.d, self.wide = field, d, wide
        self.n = [X.shape[d - i] for i in range(d)]          # nodes along x_1, x_2, ...
        self.line = [_Line(order, self.n[i], 1.0 / (self.n[i] - 1), i) for i in range(d)]
        G = [[self.line[i].D(X[I]) for I in range(d)] for i in range(d)]
        if d == 2:
            J = G[0][0] * G[1][1] - G[0][1] * G[1][0]
            F = [[G[1][1] / J, -G[0][1] / J], [-G[1][0] / J, G[0][0] / J]]
        else:
            cof = lambda i, I: (G[(i + 1) % 3][(I + 1) % 3] * G[(i + 2) % 3][(I + 2) % 3]  # noqa: E731
                                - G[(i + 1) % 3][(I + 2) % 3] * G[(i + 2) % 3][(I + 1) % 3])
            J = sum(G[0][I] * cof(0, I) for I in range(3))
            F = [[cof(i, I) / J for i in range(3)] for I in range(3)]
        self.G, self.J, self.F = G, J, F
        self.material(field.rho if rho is None else rho, field.M if M is None else M)

    def material(self, rho, M):
        d, F, J = self.d, self.F, self.J
        self.w = 1.0 / (rho * J)
        c = {}
        for i in range(d):
            for j in range(d):
                for k in range(d):
                    for l in range(d):
                        if (k, l, i, j) in c:
                            c[i, j, k, l] = c[k, l, i, j]
                            continue
                        s = 0.0
                        for I in range(d):
                            for K in range(d):
                                s = s + F[I][i] * M[d * I + j][d * K + l] * F[K][k]
                        c[i, j, k, l] = J * s
        self.c = c
        self.avg = {}
        if not self.wide:
            for i in range(d):
                for j in range(d):
                    for l in range(j, d):
                        self.avg[i, j, l] = self.avg[i, l, j] = self.line[i].averages(c[i, j, i, l])

    def volume(self, u):
        """The volume terms and the fluxes s_ij = c_ijkl D_k u_l."""
        d = self.d
        g = [[self.line[k].D(u[l]) for l in range(d)] for k in range(d)]
        s = [[sum(self.c[i, j, k, l] * g[k][l] for k in range(d) for l in range(d)) for j in range(d)] for i in range(d)]
        r = []
        for j in range(d):
            rj = sum(self.line[i].D(s[i][j]) for i in range(d))
            if not self.wide:
                rj = rj - sum(self.line[i].remainder(self.avg[i, j, l], u[l]) for i in range(d) for l in range(d))
            r.append(rj)
        return r, s

    def jump(self, r, f, w, half):
        """Adds half H^-1 T^T P w of the jump w on face f to r."""
        d, m = self.d, f // 2
        nu, L = (-1.0 if f % 2 == 0 else 1.0), self.line[m]
        ax = d - 1 - m                                       # the normal axis of a field
        at = (lambda a: _edge(a, f))
        nc = L.Db.shape[1]
        row = L.Db[0] if f % 2 == 0 else -L.Db[0].flip(0)    # the face's row of h D
        hh = L.H[:nc] if f % 2 == 0 else L.H[self.n[m] - nc:]
        spread = row / L.h / hh
        h0 = float(L.H[0])
        for j in range(d):
            amp = half * nu * sum(at(self.c[m, l, m, j]) * w[l] for l in range(d))
            part = r[j].narrow(ax, 0 if f % 2 == 0 else self.n[m] - nc, nc)
            shape = [nc if k == ax else 1 for k in range(d)]
            part += spread.reshape(shape) * amp.unsqueeze(ax)
            face = at(r[j])
            for k in range(d):
                if k == m:
                    continue
                b = half * nu * sum(at(self.c[m, l, k, j]) * w[l] for l in range(d))
                # H^-1 D^T H b = H^-1 (e_N e_N^T - e_0 e_0^T) b - D b along direction k on the face
                axk = d - 1 - k - (1 if d - 1 - k > ax else 0)
                t = -self.line[k].D(b, axk)
                hk = float(self.line[k].H[0])
                t.select(axk, 0).sub_(b.select(axk, 0) / hk)
                t.select(axk, -1).add_(b.select(axk, -1) / hk)
                face += t / h0

    def traction(self, s, f):
        m = f // 2
        nu = -1.0 if f % 2 == 0 else 1.0
        return [nu * _edge(s[m][j], f) for j in range(self.d)]


class _Scheme:
    def __init__(self, blocks, order, wide=False, basis=(), sources=(), **material):
        self.B = [_Block(b, order, wide, **material) for b in blocks]
        self.basis, self.order = basis, order
        self.src = []
        q = order // 2
        for k, x, direction, amp, peak, t0 in sources:
            B, nodes, wts = self.B[k], [], []
            for i in range(2):
                n, h = B.n[i], B.line[i].h
                lo = max(0, min(int(math.floor(x[i] / h)) - q + 1, n - 2 * q))
                at = np.arange(lo, lo + 2 * q)
                wt = [np.prod([(x[i] - at[c] * h) / ((at[a] - at[c]) * h) for c in range(2 * q) if c != a]) for a in range(2 * q)]
                nodes.append(lo)
                wts.append(torch.tensor(wt, device=DEV) / B.line[i].H[lo:lo + 2 * q])
            self.src.append((k, nodes, wts[1][:, None] * wts[0][None, :], direction, amp, peak, t0))

    def accel(self, us, t, data=True):
        T = [math.sin(w * t) if k == "sin" else math.cos(w * t) for k, w in self.basis]
        harm = lambda g: sum(a * g[:, k] for k, a in enumerate(T))   # noqa: E731
        vol = [B.volume(u) for B, u in zip(self.B, us)]
        out = []
        for b, B in enumerate(self.B):
            r, s = vol[b]
            d, u = B.d, us[b]
            for f, face in enumerate(B.f.faces):
                m = f // 2
                h0 = float(B.line[m].H[0])
                uf = [_edge(u[l], f) for l in range(d)]
                cn = lambda A, j, l, g: _edge(A.c[g // 2, j, g // 2, l], g)   # noqa: E731
                if face["kind"] == "robin":
                    tau = B.traction(s, f)
                    jh = None
                    if "U" in face or "g" in face:
                        k = 1 - m
                        jh = torch.sqrt(_edge(B.G[k][0], f) ** 2 + _edge(B.G[k][1], f) ** 2)
                    g = harm(face["g"]) if "g" in face and data else None
                    for j in range(d):
                        v = tau[j]
                        if "U" in face:
                            v = v + jh * sum(face["U"][j + l] * uf[l] for l in range(d))
                        if g is not None:
                            v = v - jh * g[j]
                        _edge(r[j], f).sub_(v / h0)
                elif face["kind"] == "displacement":
                    w = uf
                    if "g" in face and data:
                        g = harm(face["g"])
                        w = [uf[l] - g[l] for l in range(d)]
                    B.jump(r, f, w, 1.0)
                    for j in range(d):
                        _edge(r[j], f).sub_((d / h0) / h0 * sum(cn(B, j, l, f) * w[l] for l in range(d)))
                else:
                    nb, nf = face["nbr"]
                    V = self.B[nb]
                    hv = float(V.line[nf // 2].H[0])
                    w = [uf[l] - _edge(us[nb][l], nf) for l in range(d)]
                    B.jump(r, f, w, 0.5)
                    tu, tv = B.traction(s, f), V.traction(vol[nb][1], nf)
                    for j in range(d):
                        z = sum((d / 4) * (cn(B, j, l, f) / h0 + cn(V, j, l, nf) / hv) * w[l] for l in range(d))
                        _edge(r[j], f).sub_((z + 0.5 * (tu[j] + tv[j])) / h0)
            if data and B.f.forcing is not None:
                fo = harm(B.f.forcing)
                r = [r[j] + B.J * fo[j] for j in range(d)]
            out.append(r)
        if data:
            for k, (l1, l2), wt, direction, amp, peak, t0 in self.src:
                z = (math.pi * peak * (t - t0)) ** 2
                ric = amp * (1 - 2 * z) * math.exp(-z)
                for j in range(2):
                    if direction[j]:
                        out[k][j][l2:l2 + wt.shape[0], l1:l1 + wt.shape[1]] += direction[j] * ric * wt
        return [torch.stack([B.w * rj for rj in r]) for B, r in zip(self.B, out)]

    def leapfrog(self, prev, cur, dt, steps, t=0.0):
        for _ in range(steps):
            a = self.accel(cur, t)
            prev, cur = cur, [2 * c - p + dt * dt * x for p, c, x in zip(prev, cur, a)]
            t += dt
        return prev, cur

    def rk4(self, u, v, dt, steps, t=0.0):
        def go(x, y, c):
            return [p + c * q for p, q in zip(x, y)]
        for _ in range(steps):
            a1 = self.accel(u, t)
            v2 = go(v, a1, dt / 2)
            a2 = self.accel(go(u, v, dt / 2), t + dt / 2)
            v3 = go(v, a2, dt / 2)
            a3 = self.accel(go(u, v2, dt / 2), t + dt / 2)
            v4 = go(v, a3, dt)
            a4 = self.accel(go(u, v3, dt), t + dt)
            u = [x + dt / 6 * (p + 2 * q + 2 * r + s) for x, p, q, r, s in zip(u, v, v2, v3, v4)]
            v = [x + dt / 6 * (p + 2 * q + 2 * r + s) for x, p, q, r, s in zip(v, a1, a2, a3, a4)]
            t += dt
        return u, v


def _exact_stretch(case, seed):
    blocks, basis, sources, dt = _model2(case, seed)
    S = _Scheme(blocks, case["order"], case["stencil"] == "wide", basis, sources)
    start = _start(case, seed, blocks, dt)
    a, b = [x.double() for x, _ in start], [y.double() for _, y in start]
    if case["integrator"] == "rk4":
        u, v = S.rk4(a, b, dt, case["steps"])
        return {"u": u, "v": v}
    prev, cur = S.leapfrog(a, b, dt, case["steps"])
    return {"prev": prev, "cur": cur}


def _exact_gradient(case, seed):
    from torch.utils.checkpoint import checkpoint
    blocks, basis, sources, dt = _model2(case, seed)
    b = blocks[0]
    if case["layout"] == "voigt6":
        at = [(0, 0), (0, 3), (0, 1), (3, 3), (1, 3), (1, 1)]
        v = [0, 2, 2, 1]
        order6 = {(0, 0): 0, (0, 1): 1, (0, 2): 2, (1, 1): 3, (1, 2): 4, (2, 2): 5}
        C = torch.stack([b.M[p][q] for p, q in at]).requires_grad_(True)
        M = [[C[order6[min(v[p], v[q]), max(v[p], v[q])]] for q in range(4)] for p in range(4)]
    else:
        tri = [(p, q) for p in range(4) for q in range(p, 4)]
        C = torch.stack([b.M[p][q] for p, q in tri]).requires_grad_(True)
        M = [[C[tri.index((min(p, q), max(p, q)))] for q in range(4)] for p in range(4)]
    rho = b.rho.clone().requires_grad_(True)
    rec = _receivers(case)
    at1, at2 = torch.tensor([r[1] for r in rec], device=DEV), torch.tensor([r[2] for r in rec], device=DEV)
    obs = torch.from_numpy(_observed(case, seed, len(rec))).to(DEV)
    S = _Scheme(blocks, case["order"], False, basis, sources, rho=rho, M=M)
    B = S.B[0]
    keys = sorted(B.c)
    # the transformed coefficients and 1 / (rho J) are the leaves of the time loop; what they get goes on to C and rho
    uniq = {id(B.c[k]): B.c[k] for k in keys}
    outer = list(uniq.values()) + [B.w]
    inner = [x.detach().requires_grad_(True) for x in outer]
    where = {i: n for n, i in enumerate(uniq)}

    def one(prev, cur, n, *c):
        B.c = {k: c[where[ids[k]]] for k in keys}
        B.w = c[-1]
        B.avg = {}
        for i in range(2):
            for j in range(2):
                for l in range(j, 2):
                    B.avg[i, j, l] = B.avg[i, l, j] = B.line[i].averages(B.c[i, j, i, l])
        new = 2 * cur - prev + dt * dt * S.accel([cur], n * dt)[0]
        e = new[:, at2, at1].T - obs[n]
        return new, 0.5 * dt * (e * e).sum()
    ids = {k: id(B.c[k]) for k in keys}
    prev, cur = (x.double() for x in _start(case, seed, blocks, dt)[0])
    phi = 0.0
    for n in range(case["steps"]):
        new, part = checkpoint(one, prev, cur, n, *inner, use_reentrant=False)
        prev, cur, phi = cur, new, phi + part
    got = torch.autograd.grad(phi, inner)
    gC, grho = torch.autograd.grad(outer, [C, rho], got)
    return {"misfit": phi.detach(), "rho": grho, "C": gC}


def exact(case, seed):
    f = case["family"]
    if f == "gradient":
        return _exact_gradient(case, seed)
    with torch.no_grad():
        if f == "stretch":
            return _exact_stretch(case, seed)
        if f == "batch":
            return {"cur": [_exact_stretch(dict(_sized(case, s, k), steps=case["steps"]), 1000 * seed + k)["cur"][0]
                            for k, s in enumerate(_sides(case))]}
        blk, dt = _model3(case, seed)
        S = _Scheme([blk], case["order"])
        prev, cur = (x.double() for x in _start(case, seed, [blk], dt)[0])
        prev, cur = S.leapfrog([prev], [cur], dt, case["steps"])
        return {"prev": prev[0], "cur": cur[0]}
