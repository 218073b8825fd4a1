"""The work that users of this framework have it do, as measurable cases.

Each case goes through the public binding: whole calls (``Solver.advance``,
``Solver.advance_steps``, ``Batch.advance_steps``) and the single layers they
are made of (``Solver.rk_stage``, ``Solver.reconstruct_fluxes``), on device
buffers, in both precisions, with both designed orders, in one, two and three
dimensions, from the paper's 200-cell advection run to 512^3 cells.

Inputs are drawn from the seed alone, on the GPU.  ``exact`` evaluates the
scheme (arXiv 2108.12742) in 64-bit torch arithmetic, written from the paper
as window values and undivided differences; it uses nothing of the package.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

import paper_2108_12742_gb300 as eno

GAMMA, DELTA, CFL = 1.4, 1e-5, 0.5
DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _case(kind, shape, system="euler", order=5, precision="fp32", bc="transmissive", **more):
    nx, ny, nz = (tuple(shape) + (1, 1))[:3]
    return dict(kind=kind, ndim=len(shape), nx=nx, ny=ny, nz=nz, system=system, order=order,
                precision=precision, bc=bc, **more)


def listed():
    def named(name, *a, **k):
        return dict(name=name, **_case(*a, **k))

    return [
        # the paper's Sec. 4.1 accuracy run: 401 steps of 200 cells, all launch latency
        named("advect1d-200", "run", (200,), system="advection", precision="fp64", bc="periodic",
              t_end=2.0),
        # one output interval of a 1D shock-tube program, N = 2000 (about a hundred steps)
        named("euler1d-2000", "run", (2000,), precision="fp64", t_end=0.0125),
        # the batched workload: thousands of uneven 1D problems in one call
        named("batch-4096", "batch", (16384,), nprob=4096, nmin=256, steps=2),
        # the same on a small set, all FP64, seventh order
        named("batch-300-fp64", "batch", (6000,), order=7, precision="fp64", nprob=300, nmin=100,
              steps=3),
        # the headline workload: one time step of 4096^2 four-quadrant flow per call
        named("euler2d-4096", "steps", (4096, 4096), steps=1),
        # the same flow in full double precision, the default precision of a Solver
        named("euler2d-2048-fp64", "steps", (2048, 2048), precision="fp64", steps=1),
        # the size of the paper's 2D Riemann figures, seventh order, developed fronts, with the
        # grid-wide re-decision pass the interface recommends for such flows
        named("riemann2d-800-ao7", "stage", (800, 800), order=7, redecide="grid"),
        # a small ragged plane stepped by a program with its own Runge-Kutta loop
        named("euler2d-130x75", "stage", (130, 75), order=5),
        # interface fluxes and stencil choices of a ragged plane, both axes (diagnostics, coupling)
        named("fluxes2d-1000x777", "flux", (1000, 777), order=5),
        # spectral analysis of the scheme: every mode of a 4096-cell grid as one row, x fluxes
        named("spectrum-4096", "flux", (4096, 2048), system="advection", order=7,
              precision="fp64", bc="periodic"),
        # the 3D blast at full size, seventh order, periodic: one Runge-Kutta stage
        named("blast3d-512", "stage", (512, 512, 512), order=7, bc="periodic"),
        # a small 3D box in double precision, odd extents
        named("blast3d-97-fp64", "steps", (97, 80, 63), precision="fp64", bc="periodic", steps=1),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("run", "run", "batch", "stage", "stage", "steps", "flux"))
    order = rng.choice((5, 5, 7))
    bc = rng.choice(("periodic", "transmissive"))
    prec = rng.choice(("fp32", "fp64"))
    if kind == "run":  # 1D programs, run to an output time
        if rng.random() < 0.5:
            return _case("run", (size(25, 400),), system="advection", order=order,
                         precision="fp64", bc="periodic", t_end=rng.choice((0.5, 1.0, 2.0)))
        n = size(200, 4000)
        return _case("run", (n,), order=order, precision="fp64", bc=bc, t_end=25.0 / n)
    if kind == "batch":
        return _case("batch", (size(1000, 16384),), order=order, precision=prec, bc="transmissive",
                     nprob=size(64, 4096), nmin=size(50, 500), steps=rng.choice((1, 2)))
    ndim = rng.choice((2, 2, 3))
    if ndim == 2:
        shape = (size(96, 4096), size(64, 3072))
    else:
        shape = (size(40, 320), size(32, 256), size(24, 256))
    if kind == "flux":
        system = rng.choice(("euler", "euler", "advection"))
        return _case("flux", shape, system=system, order=order, precision=prec, bc=bc)
    if kind == "steps" and ndim == 2:
        bc = "transmissive"  # the quadrant flow
    case = _case(kind, shape, order=order, precision=prec, bc=bc)
    if kind == "steps":
        case["steps"] = 1
    elif prec == "fp32" and ndim == 2 and rng.random() < 0.4:
        case["redecide"] = "grid"
    return case


# ------------------------------------------------------------------ inputs

def _grids(c):
    ax = []
    for d, n in enumerate((c["nx"], c["ny"], c["nz"])):
        x = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
        ax.append(x.reshape([-1 if k == 2 - d else 1 for k in range(3)]))
    return ax  # x, y, z broadcastable to (nz, ny, nx)


def _conserved(rho, vel, p):
    ke = sum(v * v for v in vel) * 0.5 * rho
    return torch.stack(torch.broadcast_tensors(rho, *[rho * v for v in vel], p / (GAMMA - 1) + ke))


def _modes(rng, ax, n, kmax, ndim):
    """A smooth random field of max |value| about 1: n Fourier modes of up to kmax periods."""
    s = 0.0
    for _ in range(n):
        k = [int(rng.integers(-kmax, kmax + 1)) for _ in range(ndim)]
        ph = float(rng.uniform(0, 2 * math.pi))
        s = s + torch.sin(sum(2 * math.pi * kd * x for kd, x in zip(k, ax)) + ph)
    return s / n


def _quadrants(c, rng, width):
    """Four-quadrant Riemann states (rho, p in [0.1, 1.5], u, v in [-1, 1]) behind wavy fronts
    `width` cells thick (0: jumps, as at the start of a run; 1 to 2: as the scheme carries
    them), over smooth waves."""
    ax = _grids(c)
    x, y, z = ax
    q = rng.uniform(size=(4, 4))
    split = rng.uniform(0.4, 0.6, size=2)
    a, k, ph = rng.uniform(0.01, 0.05, 2), rng.integers(1, 5, 2), rng.uniform(0, 6.28, 2)

    def side(r, n):
        r = r * n
        return torch.sigmoid(2 * r / width) if width else (r >= 0).double()

    sx = side(x - split[0] - a[0] * torch.sin(2 * math.pi * float(k[0]) * y + ph[0]), c["nx"])
    sy = side(y - split[1] - a[1] * torch.sin(2 * math.pi * float(k[1]) * x + ph[1]), c["ny"])
    w = ((1 - sx) * (1 - sy), sx * (1 - sy), (1 - sx) * sy, sx * sy)
    rho, p, u, v = (sum(wi * float(lo + (hi - lo) * t) for wi, t in zip(w, q[:, i]))
                    for i, (lo, hi) in enumerate(((0.1, 1.5), (0.1, 1.5), (-1, 1), (-1, 1))))
    m = [_modes(rng, ax, 5, 4, 2) for _ in range(4)]
    vel = [u + 0.2 * m[2], v + 0.2 * m[3]][:c["ndim"]]
    return _conserved(rho * (1 + 0.2 * m[0]), vel, p * (1 + 0.2 * m[1]))


def _blast(c, rng, width):
    """Density waves and a pressure sphere, p = 10 inside and 1 outside, in a moving gas."""
    ax = _grids(c)
    ctr, rad = rng.uniform(0.3, 0.7, 3), rng.uniform(0.1, 0.2)
    r = sum((x - float(x0)) ** 2 for x, x0 in zip(ax, ctr)).sqrt()
    t = (float(rad) - r) * min(c["nx"], c["ny"], c["nz"])
    p = 1 + 9 * (torch.sigmoid(2 * t / width) if width else (t >= 0).double())
    vel = [0.3 * _modes(rng, ax, 3, 2, 3) for _ in range(3)]
    return _conserved(1 + 0.3 * _modes(rng, ax, 8, 3, 3), vel, p)


def _sizes(c):
    """Log-uniform problem lengths in nmin..nx, the same for every seed of a case."""
    rng = np.random.default_rng([c["nprob"], c["nmin"], c["nx"]])
    lo, hi = math.log(c["nmin"]), math.log(c["nx"])
    return np.rint(np.exp(rng.uniform(lo, hi, size=c["nprob"]))).astype(np.int64)


def _tubes(sizes, rng):
    """1D Riemann data of each problem on [0, 1] (rho, p in [0.1, 1], u in [-1, 1], jump in
    [0.3, 0.7]) with a density wave rho (1 + 0.2 sin k pi x), k in 3..8, on one side."""
    n = len(sizes)
    draws = np.column_stack([rng.uniform(0.1, 1, (n, 4)), rng.uniform(-1, 1, (n, 2)),
                             rng.uniform(0.3, 0.7, n), rng.integers(3, 9, n),
                             rng.integers(0, 2, n), sizes, np.cumsum(sizes) - sizes])
    reps = torch.from_numpy(np.asarray(sizes)).to(DEV)
    rl, rr, pl, pr, ul, ur, x0, k, on, m, off = torch.from_numpy(draws).to(DEV).repeat_interleave(
        reps, dim=0).T
    x = (torch.arange(len(x0), dtype=torch.float64, device=DEV) - off + 0.5) / m
    left = x < x0
    rho = torch.where(left, rl, rr)
    rho = torch.where(left == (on == 0), rho * (1 + 0.2 * torch.sin(k * math.pi * x)), rho)
    return _conserved(rho, [torch.where(left, ul, ur)], torch.where(left, pl, pr))


def _input(c, seed):
    """(state as the binding takes it, problem sizes of a batch)."""
    rng = np.random.default_rng([seed, c["nx"], c["ny"], c["nz"]])
    if c["kind"] == "batch":
        sizes = _sizes(c)
        return _tubes(sizes, rng).contiguous(), sizes
    shape = (c["nz"], c["ny"], c["nx"])
    if c["system"] == "advection":
        if c["ndim"] == 1:  # the sine wave, at a random phase
            x = 2 * _grids(c)[0] - 1 + float(rng.uniform(-1, 1))
            u = torch.sin(math.pi * x)
        else:  # row k holds mode k of the line
            k = torch.arange(c["ny"], dtype=torch.float64, device=DEV).reshape(1, -1, 1)
            j = torch.arange(c["nx"], dtype=torch.float64, device=DEV).reshape(1, 1, -1)
            u = torch.cos(2 * math.pi * torch.remainder((k + 1) * j, c["nx"]) / c["nx"]
                          + float(rng.uniform(0, 6.28))) + 0 * _grids(c)[2]
        return u.broadcast_to(shape).reshape((1,) + shape).contiguous(), None
    if c["ndim"] == 1:
        return _tubes([c["nx"]], rng).reshape((3,) + shape).contiguous(), None
    # a step starts from jumps like a run does, one layer meets developed fronts
    make = _quadrants if c["ndim"] == 2 else _blast
    width = 0.0 if c["kind"] == "steps" else float(rng.uniform(1.0, 2.0))
    return make(c, rng, width).broadcast_to((c["ndim"] + 2,) + shape).contiguous(), None


def _domain(c):
    lo = -1.0 if c["system"] == "advection" else 0.0
    return (lo,) * c["ndim"], (1.0,) * c["ndim"]


def _dx(c):
    lo, hi = _domain(c)
    return [(h - a) / n for a, h, n in zip(lo, hi, (c["nx"], c["ny"], c["nz"]))]


def prepare(case, seed):
    c = case
    U, sizes = _input(c, seed)
    kw = dict(system=eno.EULER if c["system"] == "euler" else eno.SCALAR_ADVECTION,
              order=c["order"], bc=eno.PERIODIC if c["bc"] == "periodic" else eno.TRANSMISSIVE,
              precision=eno.FP32_BULK if c["precision"] == "fp32" else eno.FP64)
    st = dict(case=c, U=U)
    if c["kind"] == "batch":
        st["solver"] = s = eno.Batch(sizes, 0.0, 1.0, **kw)
    else:
        shape = (c["nx"], c["ny"], c["nz"])[:c["ndim"]]
        st["solver"] = s = eno.Solver(shape, *_domain(c), **kw)
        if c.get("redecide") == "grid":
            s.set_redecide(eno.REDECIDE_GRID)
    if c["kind"] == "flux":
        st["F"] = [torch.empty(s.face_shape(d), dtype=torch.float64, device=DEV)
                   for d in _flux_axes(c)]
        st["idx"] = [torch.empty((s.nv, 2) + s.face_shape(d)[1:], dtype=torch.int8, device=DEV)
                     for d in _flux_axes(c)]
    else:
        st["out"] = torch.empty_like(U)
    if c["kind"] in ("flux", "stage"):  # layers: the context holds the state they work on
        if c["kind"] == "stage":
            st["dt"] = _dt(U, _dx(c))
        s.init_state(U)
    return st


def _flux_axes(c):
    return (0,) if c["system"] == "advection" else tuple(range(c["ndim"]))


def run(state):
    c, s = state["case"], state["solver"]
    if c["kind"] == "flux":
        for k, d in enumerate(_flux_axes(c)):
            s.reconstruct_fluxes(d, want_idx=True, out=state["F"][k], idx_out=state["idx"][k])
        return {"F": state["F"], "idx": state["idx"]}
    if c["kind"] == "stage":  # U1 = U^n + dt L(U^n)
        s.rk_stage(0, state["dt"])
        return s.get_stage_state(1, state["out"])
    s.init_state(state["U"])
    if c["kind"] == "run":
        s.advance(c["t_end"], cfl=CFL)
    else:
        s.advance_steps(c["steps"], cfl=CFL)
    return s.get_state(state["out"])


# -------------------------------------------------------------------- work

def work(case):
    """Bytes: the state read once and the results written once.  Flops: the method's count of
    operations per cell and axis of a stage (flux, splitting, Roe eigen-system, projection of the
    window, indicators and choice for both signs, back-projection)."""
    c = case
    nv = c["ndim"] + 2 if c["system"] == "euler" else 1
    cells = c["nx"] * c["ny"] * c["nz"]
    if c["kind"] == "batch":
        cells = int(_sizes(c).sum())
    seven = 1.7 if c["order"] == 7 else 1.0
    per = {1: 70, 3: 760, 4: 1150, 5: 1200}[nv] * seven
    if c["kind"] == "flux":
        axes = len(_flux_axes(c))
        return {"bytes": cells * (8 * nv + axes * (8 * nv + 2 * nv)), "flops": per * cells * axes}
    stages = 1 if c["kind"] == "stage" else 3 * c.get("steps", 0)
    if c["kind"] == "run":
        speed = 1.0 if c["system"] == "advection" else 1.5
        stages = 3 * c["t_end"] * speed / (CFL * _dx(c)[0])
    return {"bytes": 16 * nv * cells, "flops": per * cells * c["ndim"] * stages}


# ------------------------------------------------------------ 64-bit values

STENCILS = [(0, 0), (0, 1), (-1, 1), (-2, 1), (-1, 2), (-2, 2), (-3, 2), (-2, 3), (-3, 3)]


def _weights(l, r):
    """Weights of cells l..r in the value at the right face of cell 0 (exact fractions)."""
    k, s, out = r - l + 1, -l, []
    for j in range(k):
        t = Fraction(0)
        for m in range(j + 1, k + 1):
            den = math.prod(m - i for i in range(k + 1) if i != m)
            num = sum(math.prod(s - q + 1 for q in range(k + 1) if q not in (m, i))
                      for i in range(k + 1) if i != m)
            t += Fraction(num, den)
        out.append(float(t))
    return out


def _select(w, order):
    """The chosen candidate's value at the right face of cell 0, and its number; w(i) is the
    quantity in cell i of the window."""
    def diff(a, b):  # undivided difference over cells a..b
        n = b - a
        return sum(((-1) ** (n - i) * math.comb(n, i)) * w(a + i) for i in range(n + 1))

    cand = STENCILS[:6 if order == 5 else 9]
    IS = []
    for l, r in cand:
        if l == r:
            d = [(w(i + 1) - w(i)).abs() for i in range(-2, 2)]
            IS.append(0.5 * torch.minimum(d[1] + d[0], d[2] + d[3]))
        else:
            IS.append(torch.minimum(diff(l - 1, r).abs(), diff(l, r + 1).abs()))
    pick = torch.zeros_like(IS[0], dtype=torch.int8)
    best = IS[0].clone()
    for i, v in enumerate(IS):  # the smallest, equal ones to the higher number
        m = v <= best
        best[m], pick[m] = v[m], i
    for i, v in enumerate(IS):  # the highest one at or below the threshold
        pick[v <= DELTA] = i
    val = torch.zeros_like(best)
    for i, (l, r) in enumerate(cand):
        t = sum(b * w(l + m) for m, b in enumerate(_weights(l, r)))
        val = torch.where(pick == i, t, val)
    return val, pick


def _flux_of(q):
    if len(q) == 1:
        return q.clone()
    u = q[1] / q[0]
    p = (GAMMA - 1) * (q[-1] - 0.5 * (q[1:-1] ** 2).sum(0) / q[0])
    F = q * u
    F[1] += p
    F[-1] += p * u
    return F


def _ghosts(n, G, bc):
    """Cells of a line of n with G ghosts on each side."""
    i = np.arange(-G, n + G)
    return i % n if bc == "periodic" else np.clip(i, 0, n - 1)


def _line_fluxes(q, order, alpha):
    """Interface fluxes (nv, lines, n + 1) and choices (nv, 2, lines, n + 1) of lines of n cells
    and G ghosts on each side, q (nv, lines, n + 2 G), momentum along the line first."""
    G = order // 2 + 2
    n = q.shape[-1] - 2 * G
    F = _flux_of(q)
    split = (0.5 * (F + alpha * q), 0.5 * (F - alpha * q))
    nv = len(q)

    def at(a, i):  # cells i + G - 1 + face
        return a[..., G - 1 + i:G + i + n]

    def both(vec):
        out, picks = 0.0, []
        for s, f in enumerate(split):
            seen = {}

            def w(i, f=f, s=s, seen=seen):
                if i not in seen:
                    x = at(f, i if s == 0 else 1 - i)
                    seen[i] = x[0] if vec is None else sum(a * b for a, b in zip(vec, x)
                                                           if a is not None)
                return seen[i]
            v, k = _select(w, order)
            out = out + v
            picks.append(k)
        return out, torch.stack(picks)

    if nv == 1:
        f, k = both(None)
        return f[None], k[None]
    # Roe average and eigenvectors of the faces
    rt = q[0].sqrt()
    p = (GAMMA - 1) * (q[-1] - 0.5 * (q[1:-1] ** 2).sum(0) / q[0])
    H, vel = (q[-1] + p) / q[0], q[1:-1] / q[0]
    wl = at(rt, 0) / (at(rt, 0) + at(rt, 1))

    def mean(a):
        return wl * at(a, 0) + (1 - wl) * at(a, 1)

    H, vel = mean(H), [mean(v) for v in vel]
    q2 = sum(v * v for v in vel)
    c2 = (GAMMA - 1) * (H - 0.5 * q2)
    c, one = c2.sqrt(), torch.ones_like(c2)
    b1, u = (GAMMA - 1) / c2, vel[0]
    b2 = 0.5 * q2 * b1
    total, picks = torch.zeros((nv,) + u.shape, dtype=u.dtype, device=u.device), []
    for v in range(nv):
        if v in (0, nv - 1):
            s = 1.0 if v == 0 else -1.0
            left = [0.5 * (b2 + s * u / c), 0.5 * (-b1 * u - s / c)]
            left += [-0.5 * b1 * t for t in vel[1:]] + [0.5 * b1]
            right = [one, u - s * c] + vel[1:] + [H - s * u * c]
        elif v == 1:
            left = [1 - b2] + [b1 * t for t in vel] + [-b1]
            right = [one] + vel + [0.5 * q2]
        else:
            left = [-vel[v - 1]] + [one if i == v else None for i in range(1, nv)]
            right = [one if i == v else None for i in range(nv - 1)] + [vel[v - 1]]
        w, k = both(left)
        picks.append(k)
        for i, r in enumerate(right):
            if r is not None:
                total[i] += r * w
    return total, torch.stack(picks)


def _axis(U, d, c, alpha, want):
    """Fluxes and choices (want "F"), or -(F_{j+1/2} - F_{j-1/2})/dx (want "L"), of axis d."""
    nv = len(U)
    perm = list(range(nv))
    if nv > 2:
        nd = nv - 2
        perm[1:-1] = [1 + (d + i) % nd for i in range(nd)]
    V = U.movedim(3 - d, 3)
    lead, n = V.shape[1:3], V.shape[3]
    V = V.reshape(nv, -1, n)
    wide = n + (1 if want == "F" else 0)
    out = torch.empty((nv, V.shape[1], wide), dtype=U.dtype, device=U.device)
    idx = torch.empty((nv, 2, V.shape[1], wide), dtype=torch.int8, device=U.device) \
        if want == "F" else None
    lines = max(1, (1 << 22) // n)
    ext = torch.from_numpy(_ghosts(n, c["order"] // 2 + 2, c["bc"])).to(U.device)
    for a in range(0, V.shape[1], lines):
        F, k = _line_fluxes(V[perm, a:a + lines][..., ext], c["order"], alpha)
        if want == "F":
            out[perm, a:a + lines] = F
            idx[:, :, a:a + lines] = k
        else:
            out[perm, a:a + lines] = (F[..., :-1] - F[..., 1:]) / _dx(c)[d]
    out = out.reshape((nv,) + lead + (wide,)).movedim(3, 3 - d)
    if want == "F":
        return out, idx.reshape((nv, 2) + lead + (wide,)).movedim(4, 4 - d)
    return out


def _alpha(U):
    if len(U) == 1:
        return [1.0] * 3
    p = (GAMMA - 1) * (U[-1] - 0.5 * (U[1:-1] ** 2).sum(0) / U[0])
    cs = (GAMMA * p / U[0]).sqrt()
    return [float(((U[i] / U[0]).abs() + cs).max()) for i in range(1, len(U) - 1)]


def _dt(U, dx):
    return CFL / sum(a / h for a, h in zip(_alpha(U), dx))


def _rhs(U, c, alpha):
    return sum(_axis(U, d, c, alpha[d], "L") for d in range(c["ndim"]))


def _step(U, dt, rhs):
    U1 = U + dt * rhs(U)
    U2 = 0.75 * U + 0.25 * (U1 + dt * rhs(U1))
    return U / 3 + 2 / 3 * (U2 + dt * rhs(U2))


def exact(case, seed):
    c = case
    U, sizes = _input(c, seed)
    if c["kind"] == "flux":
        got = [_axis(U, d, c, _alpha(U)[d], "F") for d in _flux_axes(c)]
        return {"F": [f for f, _ in got], "idx": [None for _ in got]}
    if c["kind"] == "stage":
        return U + _dt(U, _dx(c)) * _rhs(U, c, _alpha(U))
    if c["kind"] == "batch":
        return _batch_steps(U, sizes, c)
    if c["kind"] == "run":
        return _steps(U.cpu(), c)
    return _steps(U, c)


def _steps(U, c):
    t, k = 0.0, 0
    while t < c.get("t_end", math.inf) and k < c.get("steps", 1 << 30):
        alpha = _alpha(U)
        dt = _dt(U, _dx(c))
        last = t + dt >= c.get("t_end", math.inf)
        U = _step(U, c["t_end"] - t if last else dt, lambda V: _rhs(V, c, alpha))
        t, k = c["t_end"] if last else t + dt, k + 1
    return U


def _batch_steps(U, sizes, c):
    """Every problem with its own alpha and time step: one line of all problems, each with its
    ghosts."""
    G, dev = c["order"] // 2 + 2, U.device
    off = np.cumsum(sizes) - sizes
    ext = np.concatenate([o + _ghosts(int(n), G, c["bc"]) for o, n in zip(off, sizes)])
    own = np.concatenate([np.arange(n) + o + 2 * G * i for i, (o, n) in enumerate(zip(off, sizes))])
    ext, own = (torch.from_numpy(a).to(dev) for a in (ext, own))
    prob = torch.arange(len(sizes), device=dev).repeat_interleave(
        torch.from_numpy(np.asarray(sizes)).to(dev))
    dx = (1.0 / torch.from_numpy(np.asarray(sizes)).to(dev).double())
    for _ in range(c["steps"]):
        p = (GAMMA - 1) * (U[2] - 0.5 * U[1] ** 2 / U[0])
        s = (U[1] / U[0]).abs() + (GAMMA * p / U[0]).sqrt()
        alpha = torch.zeros_like(dx).scatter_reduce_(0, prob, s, "amax")
        dt, acell = CFL * dx / alpha, alpha[prob][ext]

        def rhs(V):
            F = _line_fluxes(V[:, None, ext], c["order"], acell)[0][:, 0]
            return (F[:, own] - F[:, own + 1]) / dx[prob]

        U = _step(U, dt[prob], rhs)
    return U
