"""Performance cases of the Poisson solver: the calls its users make, over the sizes they make them at.

A case is a dict of plain values; ``prepare`` turns it into a plan (or plans, or a serving engine) and
seeded inputs on the GPU, ``run`` makes one pass through the public entry points of
``paper_2106_03583_gb300.snac`` and returns the computed fields, and ``exact`` gives the same fields
from plain 64-bit linear algebra (tensor-product eigenvectors, or conjugate gradients where the
blocks do not fill a rectangle).

Kinds of case
  solve    one solve of one problem to a relative residual, from a zero guess (a new pressure field)
           or from the previous time step's solution (``guess`` "warm")
  batch    independent mixed-precision problems solved together (``snac.solve_batch``)
  engine   a burst of requests to a resident serving engine, host arrays in and out
  pencil   one rank's forward transform and backward update in a solve sharded by wavenumber
"""
import math
import random

import numpy as np
import torch

from paper_2106_03583_gb300 import inputs, snac

# z boundary pairs of Table 1 of the paper, and one-dimensional wall kinds
PAIRS = ("PP", "NN", "DD", "ND", "DN")
# The named problems are solved to the repository's usual relative residual of 1e-10. Random ones may
# amplify a residual several times in the solution, so they are solved to a tenth of it: each field is
# then determined to 1e-10 or so, whatever path the iteration takes.
TIGHT = 1e-11


def _solve(name, layout, nx, ny, nz, precision, **kw):
    c = {"name": name, "kind": "solve", "layout": layout, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
         "lx": 1.0, "ly": 1.0, "xfac": 0.0, "yfac": 0.0, "zpair": "PP", "walls": "DDNN", "rhs": "divergence",
         "tol": 1e-10, "guess": "zero", "shift": 0.0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest grid of the serving range: launches and host round trips count
        _solve("small 32^3 mixed", "1", 32, 32, 32, "mixed", zpair="NN", walls="DNNN", rhs="uniform"),
        # the repository's small parity problem (64 x 64 x 32), full precision
        _solve("c64 fp64", "1", 64, 64, 32, "fp64", rhs="uniform"),
        # the 2x2-block workload: Neumann walls, singular, y clustered, 6.7e7 cells
        _solve("mb2x2 mixed", "2x2", 512, 512, 256, "mixed", lx=2.0, ly=2.0, yfac=1.5, zpair="NN", walls="NNNN"),
        _solve("mb2x2 fp64", "2x2", 512, 512, 256, "fp64", lx=2.0, ly=2.0, yfac=1.5, zpair="NN", walls="NNNN"),
        # the benchmark's channel: 2.7e8 cells, the largest single problem
        _solve("chan mixed", "1", 1024, 512, 512, "mixed", lx=2.0, yfac=2.0),
        # a pressure solve inside a time loop: half-scale channel, warm start, full precision
        _solve("chan/2 step fp64", "1", 512, 256, 256, "fp64", lx=2.0, yfac=2.0, guess="warm"),
        # an L-shaped duct of three blocks (re-entrant corner): the multi-block geometry of the method
        _solve("L duct mixed", "L", 512, 512, 128, "mixed", zpair="NN", walls="DNNN"),
        # the paper's four-block T junction (Table 2), refined, both plane axes clustered, n_z = 96
        _solve("T junction fp64", "T", 320, 160, 96, "fp64", lx=4.0, ly=2.0, xfac=1.0, yfac=1.0, walls="DNNN"),
        # a duct clustered along both plane axes; sizes that are not powers of two, Dirichlet-Neumann
        # along z
        _solve("duct ragged mixed", "1", 336, 192, 150, "mixed", xfac=1.3, yfac=2.0, zpair="DN", walls="DNNN"),
        # many independent problems at once, 32^3 .. 256 x 256 x 128, one to four blocks
        {"name": "batch 16 mixed", "kind": "batch", "count": 16, "mix": 3},
        # a burst of requests to the serving engine, both precisions
        {"name": "engine 12", "kind": "engine", "count": 12, "mix": 5, "workers": 4},
        # one rank of a sharded solve: 20011 columns of a 576-plane field (an odd pencil width)
        {"name": "pencil 576", "kind": "pencil", "ncols": 20011, "nz": 576, "zpair": "NN"},
    ]


def _halvings_fit(layout, nx, ny):
    """Whether the multigrid of this plane can coarsen down to a coarsest plane of at most 256 cells."""
    rects = _rects(layout, nx, ny)
    while True:
        cells = sum((b - a) * (d - c) for a, b, c, d in rects)
        if cells <= 64:
            return True
        if any(v % 2 for r in rects for v in r) or any(b - a < 4 or d - c < 4 for a, b, c, d in rects):
            return cells <= 256
        rects = [tuple(v // 2 for v in r) for r in rects]


def _log_choice(rng, values, lo, hi):
    """One of the values in [lo, hi], uniform over the logarithm."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((v for v in values if lo <= v <= hi), key=lambda v: abs(math.log(v / t)))


_PLANE = sorted(m << k for m in (1, 3, 5, 7) for k in range(3, 11) if 24 <= m << k <= 1024)
_LENGTH = sorted({2 * 2 ** a * 3 ** b * 5 ** c * 7 ** d for a in range(9) for b in range(4) for c in range(3)
                  for d in range(2) if 16 <= 2 * 2 ** a * 3 ** b * 5 ** c * 7 ** d <= 576})


def draw(rng):
    kind = rng.choice(["solve"] * 8 + ["batch", "engine", "pencil"])
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(6, 20), "mix": rng.randrange(1 << 20)}
    if kind == "engine":
        return {"kind": kind, "count": rng.randint(6, 14), "mix": rng.randrange(1 << 20), "workers": 4}
    if kind == "pencil":
        return {"kind": kind, "ncols": int(math.exp(rng.uniform(math.log(1000), math.log(60000)))) | 1,
                "nz": _log_choice(rng, _LENGTH, 32, 576), "zpair": rng.choice(PAIRS)}
    while True:
        layout = rng.choice(["1", "1", "1x2", "2x1", "2x2", "L", "T"])
        nx, ny = _log_choice(rng, _PLANE, 24, 1024), _log_choice(rng, _PLANE, 24, 1024)
        if layout == "T":
            nx, ny = 2 * ny, ny
        nz = _log_choice(rng, _LENGTH, 16, 576)
        if 16384 <= nx * ny * nz <= 1 << 25 and nx <= 1024 and _halvings_fit(layout, nx, ny):
            break
    ly = rng.choice([1.0, 2.0])   # cells of the mean grid: square, or twice as wide as high, or half
    return {"kind": "solve", "layout": layout, "nx": nx, "ny": ny, "nz": nz,
            "precision": rng.choice(["mixed", "mixed", "fp64"]), "lx": ly * nx / ny * rng.choice([0.5, 1.0, 1.0, 2.0]),
            "ly": ly,
            "xfac": rng.choice([0.0, 0.0, round(rng.uniform(0.5, 1.5), 2)]),
            "yfac": rng.choice([0.0, round(rng.uniform(0.5, 2.0), 2)]), "zpair": rng.choice(PAIRS),
            "walls": "".join(rng.choice("DN") for _ in range(4)), "rhs": rng.choice(["divergence", "uniform"]),
            "tol": TIGHT, "guess": rng.choice(["zero", "zero", "warm"]),
            "shift": rng.choice([0.0, 0.0, 0.0, -40.0])}


# ---- geometry and inputs ----

def _rects(layout, nx, ny):
    """Block rectangles (x0, x1, y0, y1) of a layout on an nx x ny bounding box."""
    hx, hy = nx // 2, ny // 2
    if layout == "1":
        return [(0, nx, 0, ny)]
    if layout == "1x2":
        return [(0, hx, 0, ny), (hx, nx, 0, ny)]
    if layout == "2x1":
        return [(0, nx, 0, hy), (0, nx, hy, ny)]
    if layout == "L":
        return [(0, hx, 0, hy), (hx, nx, 0, hy), (0, hx, hy, ny)]
    if layout == "2x2":
        return [(0, hx, 0, hy), (hx, nx, 0, hy), (0, hx, hy, ny), (hx, nx, hy, ny)]
    if layout == "T":   # a row of three blocks under one block above the middle one
        qx = nx // 4
        return [(0, 2 * qx, 0, hy), (2 * qx, 3 * qx, 0, hy), (3 * qx, nx, 0, hy), (2 * qx, 3 * qx, hy, ny)]
    raise ValueError(layout)


def _geometry(c):
    """Face coordinates, block rectangles and blocks of a solve case."""
    xf = inputs.tanh_faces(c["nx"], 0, c["xfac"], 0.0, c["lx"])
    yf = inputs.tanh_faces(c["ny"], 0, c["yfac"], 0.0, c["ly"])
    zf = np.linspace(0.0, 1.0, c["nz"] + 1)
    rects = _rects(c["layout"], c["nx"], c["ny"])
    walls = dict(zip(("x-", "x+", "y-", "y+"), c["walls"]))
    blocks = inputs.make_blocks(xf, yf, zf, rects, walls, (c["zpair"][0], c["zpair"][1]), inner_wall="N")
    return xf, yf, zf, rects, blocks


def _singular(c):
    return c["shift"] == 0.0 and c["zpair"] in ("PP", "NN") and not _has_dirichlet(c)


def _has_dirichlet(c):
    nx, ny = c["nx"], c["ny"]
    walls = c["walls"]
    return any((r[0] == 0 and walls[0] == "D") or (r[1] == nx and walls[1] == "D") or (r[2] == 0 and walls[2] == "D") or
               (r[3] == ny and walls[3] == "D") for r in _rects(c["layout"], nx, ny))


def _rhs(c, gen):
    """A right-hand side on the GPU, blocks concatenated, [z][y][x]: uniform noise in [-1, 1], or the
    divergence of a random-phase velocity field with a k^-5/3 spectrum (zero on the walls), unit RMS."""
    xf, yf, zf, rects, blocks = _geometry(c)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    dev = {"dtype": torch.float64, "device": "cuda"}
    w = [torch.tensor(np.diff(v), **dev) for v in (zf, yf, xf)]
    if c["rhs"] == "uniform":
        parts = [2.0 * torch.rand(nz, y1 - y0, x1 - x0, generator=gen, **dev) - 1.0 for x0, x1, y0, y1 in rects]
    else:
        parts = [torch.zeros(nz, y1 - y0, x1 - x0, **dev) for x0, x1, y0, y1 in rects]
        k2 = (torch.fft.fftfreq(nz, 1.0 / nz, **dev)[:, None, None] ** 2 +
              torch.fft.fftfreq(ny, 1.0 / ny, **dev)[None, :, None] ** 2 +
              torch.fft.rfftfreq(nx, 1.0 / nx, **dev)[None, None, :] ** 2)
        amp = torch.where(k2 > 0, k2.clamp(min=1.0) ** (-11.0 / 12.0), torch.zeros_like(k2))
        del k2
        for axis in range(3):   # the face velocity along x, y, z (value i = lower face of cell i)
            spec = torch.polar(amp, 2.0 * math.pi * torch.rand(amp.shape, generator=gen, **dev))
            u = torch.fft.irfftn(spec, s=(nz, ny, nx))
            del spec
            u /= u.square().mean().sqrt()
            for b, (x0, x1, y0, y1) in enumerate(rects):
                d = 2 - axis
                ub = u[:, y0:y1, x0:x1]
                n = (c["nx"], c["ny"], nz)[axis]
                hi = ((x1, y1, nz)[axis]) % n
                top = u.narrow(d, hi, 1)
                top = top[:, y0:y1] if axis == 0 else top[:, :, x0:x1] if axis == 1 else top[:, y0:y1, x0:x1]
                faces = torch.cat([ub, top], dim=d)
                for side, at in ((0, 0), (1, faces.shape[d] - 1)):
                    if blocks[b]["bc"][axis][side] in "DN":
                        faces.narrow(d, at, 1).zero_()
                wd = np.diff((xf, yf, zf)[axis])[((x0, y0, 0)[axis]):((x1, y1, nz)[axis])]
                shape = [1, 1, 1]
                shape[d] = -1
                parts[b] += faces.diff(dim=d) / torch.tensor(wd, **dev).reshape(shape)
            del u
        rms = math.sqrt(sum(float(q.square().sum()) for q in parts) / sum(q.numel() for q in parts))
        for q in parts:
            q /= rms
    if _singular(c):   # compatible: no volume-weighted mean
        for _ in range(2):
            s = v = 0.0
            for q, (x0, x1, y0, y1) in zip(parts, rects):
                a = w[1][y0:y1, None] * w[2][None, x0:x1]
                s += float((q.sum(0) * a).sum())
                v += float(a.sum()) * nz
            for q in parts:
                q -= s / v
    return blocks, torch.cat([q.reshape(-1) for q in parts])


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _mix(c):
    """The problems of a batch or an engine burst: sizes, layouts, walls and pairs as in the repository's
    random problems (powers of two, 32^3 upwards, cubic cells), drawn from the case's own seed."""
    rng = random.Random(c["mix"])
    out = []
    for _ in range(c["count"]):
        nx, ny, nz = 2 ** rng.randint(5, 8), 2 ** rng.randint(5, 8), 2 ** rng.randint(5, 7)
        out.append(_solve("", rng.choice(["1", "1x2", "2x1", "L", "2x2"]), nx, ny, nz, "mixed", lx=nx / 64.0, ly=ny / 64.0,
                          zpair=rng.choice(PAIRS), walls="".join(rng.choice("DN") for _ in range(4)),
                          rhs="uniform" if c["kind"] == "batch" else "divergence", tol=TIGHT))
    if c["kind"] == "engine":
        for q in out:
            q["precision"] = rng.choice(["mixed", "mixed", "fp64"])
    return out


def _problem(c, seed):
    blocks, f = _rhs(c, _generator(seed))
    plan = snac.Plan(blocks, precision=c["precision"], shift=c["shift"])
    return blocks, f, plan


def _step_rhs(c, seed):
    """The right-hand sides of two successive time steps: the second differs by a tenth."""
    gen = _generator(seed)
    blocks, f0 = _rhs(c, gen)
    _, df = _rhs(c, gen)
    return blocks, f0, f0 + 0.1 * df


def _pencil_blocks(c):
    n = c["nz"]
    return inputs.make_blocks(np.linspace(0, 1, 17), np.linspace(0, 1, 17), np.linspace(0, 1, n + 1), [(0, 16, 0, 16)],
                              {"x-": "D", "x+": "D", "y-": "N", "y+": "N"}, (c["zpair"][0], c["zpair"][1]))


def _pencil_input(c, seed):
    gen = _generator(seed)
    x = torch.randn(c["nz"], c["ncols"], generator=gen, dtype=torch.float64, device="cuda")
    p0 = torch.randn(c["nz"], c["ncols"], generator=gen, dtype=torch.float64, device="cuda")
    return x, p0


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        if case["guess"] == "zero":
            _, f, plan = _problem(case, seed)
            return {"case": case, "plan": plan, "f": f, "p": torch.zeros_like(f)}
        blocks, f0, f = _step_rhs(case, seed)
        plan = snac.Plan(blocks, precision=case["precision"], shift=case["shift"])
        p0 = torch.zeros_like(f)
        plan.solve(f0, p0, tol=case["tol"])   # the previous time step
        return {"case": case, "plan": plan, "f": f, "p0": p0, "p": torch.empty_like(f)}
    if kind == "batch":
        mix = [_problem(c, 1000 * seed + k) for k, c in enumerate(_mix(case))]
        return {"case": case, "plans": [m[2] for m in mix], "f": [m[1] for m in mix],
                "p": [torch.zeros_like(m[1]) for m in mix]}
    if kind == "engine":
        mix = _mix(case)
        reqs = []
        for k, c in enumerate(mix):
            blocks, f = _rhs(c, _generator(1000 * seed + k))
            reqs.append((blocks, f.cpu().numpy(), c["tol"], c["precision"]))
        eng = snac.Engine(workers=case["workers"], hbm_budget=50e9)
        state = {"case": case, "engine": eng, "requests": reqs}
        run(state)   # a serving process keeps the plans of recurring grids resident
        return state
    plan = snac.Plan(_pencil_blocks(case), precision="fp64")
    x, p0 = _pencil_input(case, seed)
    return {"case": case, "plan": plan, "x": x, "modes": torch.empty_like(x), "p0": p0, "p": torch.empty_like(x)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        p = state["p"]
        if case["guess"] == "zero":
            p.zero_()
        else:
            p.copy_(state["p0"])
        state["plan"].solve(state["f"], p, tol=case["tol"])
        return {"p": p}
    if kind == "batch":
        for p in state["p"]:
            p.zero_()
        snac.solve_batch(state["plans"], state["f"], state["p"], tol=TIGHT)
        return list(state["p"])
    if kind == "engine":
        eng = state["engine"]
        tickets = [eng.submit(blocks, f, tol=tol, precision=precision) for blocks, f, tol, precision in state["requests"]]
        return [eng.wait(t)[0] for t in tickets]
    state["p"].copy_(state["p0"])
    state["plan"].pencil_forward(state["x"], state["modes"])
    state["plan"].pencil_backward_update(state["modes"], state["p"])
    return {"modes": state["modes"], "p": state["p"]}


def _cells(c):
    return c["nz"] * sum((x1 - x0) * (y1 - y0) for x0, x1, y0, y1 in _rects(c["layout"], c["nx"], c["ny"]))


def work(case):
    """Bytes: the right-hand side and the guess read, the solution written (each once). Flops: two
    transforms along z, one sweep of the plane operator per cell and the 3-D residual that decides."""
    if case["kind"] == "pencil":
        n = case["nz"] * case["ncols"]
        return {"bytes": 40.0 * n, "flops": 5.0 * n * math.log2(case["nz"])}
    probs = [case] if case["kind"] == "solve" else _mix(case)
    return {"bytes": sum(24.0 * _cells(c) for c in probs),
            "flops": sum(_cells(c) * (5.0 * math.log2(c["nz"]) + 30.0) for c in probs)}


# ---- the same results from plain 64-bit linear algebra ----

def _axis(w, lo, hi, w_lo, w_hi):
    """Symmetric second-difference matrix K = W A of one axis (numpy): ends "D", "N", "P", or "B" with
    the width of the connected cell (its coupling enters the diagonal)."""
    n = len(w)
    K = np.zeros((n, n))
    for i in range(n - 1):
        g = 1.0 / (0.5 * (w[i] + w[i + 1]))
        K[i, i] -= g
        K[i + 1, i + 1] -= g
        K[i, i + 1] += g
        K[i + 1, i] += g
    for i, kind, wn in ((0, lo, w_lo), (n - 1, hi, w_hi)):
        if kind == "D":
            K[i, i] -= 2.0 / w[i]
        elif kind == "B":
            K[i, i] -= 1.0 / (0.5 * (w[i] + wn))
    if lo == "P":
        g = 1.0 / (0.5 * (w[0] + w[-1]))
        K[0, 0] -= g
        K[-1, -1] -= g
        K[0, -1] += g
        K[-1, 0] += g
    return K


def _eigen(K, w):
    """A = W^-1 K = B diag(lam) F with F = Q^T W^1/2 and B = W^-1/2 Q, on the GPU."""
    r = np.sqrt(w)
    lam, q = torch.linalg.eigh(torch.tensor(K / r[:, None] / r[None, :]))
    lam, q, r = lam.cuda(), q.cuda(), torch.tensor(r).cuda()
    return lam, q.T * r[None, :], q / r[:, None]


def _apply_axes(x, mz, my, mx):
    x = torch.matmul(x, mx.T)
    x = torch.matmul(my, x)
    return torch.matmul(mz, x.reshape(x.shape[0], -1)).reshape(x.shape)


def _tensor_solver(axes, shift, singular):
    """x -> A^-1 x for A = Az + Ay + Ax + shift on one rectangle; axes: (K, w) of z, y, x."""
    (lz, fz, bz), (ly, fy, by), (lx, fx, bx) = (_eigen(K, w) for K, w in axes)
    d = lz[:, None, None] + ly[None, :, None] + lx[None, None, :] + shift
    if singular:
        d.view(-1)[torch.argmin(d.abs()).item()] = math.inf

    def solve(x):
        return _apply_axes(_apply_axes(x, fz, fy, fx) / d, bz, by, bx)
    return solve


def _exact_solve(c, f):
    xf, yf, zf, rects, blocks = _geometry(c)
    wx, wy, wz = np.diff(xf), np.diff(yf), np.diff(zf)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    zaxis = (_axis(wz, c["zpair"][0], c["zpair"][1], 0.0, 0.0), wz)
    parts, o = [], 0
    for x0, x1, y0, y1 in rects:
        n = nz * (y1 - y0) * (x1 - x0)
        parts.append(f[o:o + n].reshape(nz, y1 - y0, x1 - x0))
        o += n
    wl = c["walls"]
    if c["layout"] not in ("L", "T"):
        g = torch.empty(nz, ny, nx, dtype=torch.float64, device="cuda")
        for q, (x0, x1, y0, y1) in zip(parts, rects):
            g[:, y0:y1, x0:x1] = q
        axes = (zaxis, (_axis(wy, wl[2], wl[3], 0.0, 0.0), wy), (_axis(wx, wl[0], wl[1], 0.0, 0.0), wx))
        u = _tensor_solver(axes, c["shift"], _singular(c))(g)
        return torch.cat([u[:, y0:y1, x0:x1].reshape(-1) for x0, x1, y0, y1 in rects])
    # conjugate gradients on the volume-weighted operator, each block's own tensor solve as preconditioner
    solvers, mats, vols = [], [], []
    for b, (x0, x1, y0, y1) in enumerate(rects):
        bc = blocks[b]["bc"]
        ax = (_axis(wx[x0:x1], *bc[0], wx[x0 - 1], wx[x1 % nx]), wx[x0:x1])
        ay = (_axis(wy[y0:y1], *bc[1], wy[y0 - 1], wy[y1 % ny]), wy[y0:y1])
        solvers.append(_tensor_solver((zaxis, ay, ax), c["shift"], False))
        mats.append([torch.tensor(K / w[:, None]).cuda() for K, w in (zaxis, ay, ax)])
        vols.append(torch.tensor(wz[:, None, None] * wy[None, y0:y1, None] * wx[None, None, x0:x1]).cuda())

    def face(q, axis, side):
        d = 2 - axis
        return q.narrow(d, 0 if side == 0 else q.shape[d] - 1, 1)

    def stencil(x, m, d):   # the tridiagonal m along dimension d, by its three diagonals (plus the wrap)
        shape = [1, 1, 1]
        shape[d] = -1
        n = x.shape[d]
        y = x * m.diagonal().reshape(shape)
        y.narrow(d, 1, n - 1).add_(x.narrow(d, 0, n - 1) * m.diagonal(-1).reshape(shape))
        y.narrow(d, 0, n - 1).add_(x.narrow(d, 1, n - 1) * m.diagonal(1).reshape(shape))
        if n > 2 and float(m[0, -1]) != 0.0:
            y.narrow(d, 0, 1).add_(x.narrow(d, n - 1, 1) * m[0, -1])
            y.narrow(d, n - 1, 1).add_(x.narrow(d, 0, 1) * m[-1, 0])
        return y

    def apply(xs):   # -V (A + shift) x
        out = []
        for b, x in enumerate(xs):
            y = stencil(x, mats[b][0], 0) + stencil(x, mats[b][1], 1) + stencil(x, mats[b][2], 2) + c["shift"] * x
            for axis in range(2):
                w = (wx, wy)[axis]
                lo, hi = rects[b][2 * axis], rects[b][2 * axis + 1]
                for side in range(2):
                    if blocks[b]["bc"][axis][side] != "B":
                        continue
                    wi, wn = (w[lo], w[lo - 1]) if side == 0 else (w[hi - 1], w[hi])
                    face(y, axis, side).add_(face(xs[blocks[b]["nbr"][axis][side]], axis, 1 - side),
                                             alpha=1.0 / (0.5 * (wi + wn) * wi))
            out.append(-vols[b] * y)
        return out

    def dot(a, b):
        return sum(float((p * q).sum()) for p, q in zip(a, b))

    total = sum(float(v.sum()) for v in vols)
    x = [torch.zeros_like(q) for q in parts]
    r = [-v * q for v, q in zip(vols, parts)]
    r0 = math.sqrt(dot(r, r))
    p, rz = None, 0.0
    for _ in range(400):
        if math.sqrt(dot(r, r)) <= 1e-14 * r0:
            break
        z = [-s(q / v) for s, q, v in zip(solvers, r, vols)]
        old, rz = rz, dot(r, z)
        p = z if p is None else [a + (rz / old) * b for a, b in zip(z, p)]
        ap = apply(p)
        a = rz / dot(p, ap)
        for k in range(len(x)):
            x[k] += a * p[k]
            r[k] -= a * ap[k]
    if _singular(c):
        mean = dot(x, vols) / total
        x = [q - mean for q in x]
    return torch.cat([q.reshape(-1) for q in x])


def _transform_matrix(pair, n):
    """The unnormalised real-to-real transform of Table 1 as a matrix (half-complex order for PP)."""
    j, k = np.meshgrid(np.arange(n), np.arange(n))
    if pair == "PP":
        return np.where(k <= n // 2, np.cos(2 * np.pi * (j * k % n) / n), -np.sin(2 * np.pi * (j * (n - k) % n) / n))
    if pair == "NN":
        return 2 * np.cos(np.pi * ((2 * j + 1) * k % (4 * n)) / (2 * n))
    if pair == "DD":
        return 2 * np.sin(np.pi * ((2 * j + 1) * (k + 1) % (4 * n)) / (2 * n))
    a = np.pi * ((2 * j + 1) * (2 * k + 1) % (8 * n)) / (4 * n)
    return 2 * np.cos(a) if pair == "ND" else 2 * np.sin(a)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        f = _rhs(case, _generator(seed))[1] if case["guess"] == "zero" else _step_rhs(case, seed)[2]
        return {"p": _exact_solve(case, f)}
    if kind in ("batch", "engine"):
        out = [_exact_solve(c, _rhs(c, _generator(1000 * seed + k))[1]) for k, c in enumerate(_mix(case))]
        return [p.cpu().numpy() for p in out] if kind == "engine" else out
    x, p0 = _pencil_input(case, seed)
    return {"modes": torch.matmul(torch.tensor(_transform_matrix(case["zpair"], case["nz"])).cuda(), x), "p": p0 + x}
