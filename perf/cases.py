"""The measured work of the 2D-FC library: what a program has it do, call by call.

A program makes a plan for a domain and a grid once and keeps it; then it passes fields
through the plan.  `prepare` makes the plan (kept between states, as such a program keeps
it) and the fields, on the GPU; `run` is one call, or the few calls that belong together.

Kinds of case (`kind`):
  spectrum   extension + DFT of n_f fields: `form` "grid" (fields on the whole grid),
             "compact" (at the domain's points only), "complex" (complex fields), "split"
             (the extension and its DFT as two calls, both results used)
  group      several domains in one call (a plan group)
  poisson    a Poisson solve with Dirichlet data
  interior   one large step of the Fourier Forwarding interior propagator
  forward    the whole Fourier Forwarding solve, one large step of 8 n_c small ones:
             `mode` 0 full U_FC, 1 small squares, 2 small squares in double-float

`exact` restates the method in plain torch and numpy in 64 bits, from the formulas of
arXiv 2010.03901: geometry, FC matrices, matching values, blend, strip interpolation, DFT.
"""
import decimal
import functools
import math

import numpy as np
import torch

from paper_2010_03901_gb300 import fc2d

F64 = torch.float64
C, Z, N_OS, N_R, M_F = 27, 12, 20, 6, 20  # the paper's continuation parameters
N_C = 8                                   # cells a wave crosses in a large step
STAR_SIZES = (256, 384, 512, 640, 768, 1024, 1536, 2048)


def _dev():
    return torch.device("cuda:0")


# ---------------------------------------------------------------------------- cases
def listed():
    return [
        # The smallest call: the unit disk at 128^2, one field, double.  Launches count.
        {"name": "disk128_fp64", "kind": "spectrum", "form": "grid", "domain": "disk",
         "nx": 128, "ny": 128, "x0": -1.5, "y0": -1.5, "h": 3.0 / 128, "B": 256, "k1": 0.015,
         "n_f": 1, "precision": "fp64", "bdry": True},
        # A small ragged grid (2^5 5 x 2^4 3^2) and a few fields; the program wants the
        # extended field itself and its spectrum.
        {"name": "kite160x144_split_fp64", "kind": "spectrum", "form": "split",
         "domain": "kite", "nx": 160, "ny": 144, "x0": -3.17, "y0": -2.63, "h": 0.0366,
         "B": 320, "k1": 0.0366, "n_f": 3, "precision": "fp64", "bdry": True},
        # An ordinary grid in the mixed form, the field given at the domain's points only.
        {"name": "star1024_compact_mixed", "kind": "spectrum", "form": "compact",
         "domain": "star", "a": 0.3, "k": 5, "nx": 1024, "ny": 1024, "x0": -1.1955,
         "y0": -1.3, "h": 2.6 / 1024, "B": 2048, "k1": 0.0013, "n_f": 1,
         "precision": "mixed", "bdry": True},
        # The paper's kind of grid (1728 x 1200 = 2^6 3^3 x 2^4 3 5^2), a complex field
        # without boundary values (Remark 3.2 II), double.
        {"name": "kite1728x1200_complex_fp64", "kind": "spectrum", "form": "complex",
         "domain": "kite", "nx": 1728, "ny": 1200, "n_f": 1, "precision": "fp64",
         "bdry": False},
        # The headline: the kite at 4096^2 with 8192 normals, one field, mixed form...
        {"name": "kite4096_mixed", "kind": "spectrum", "form": "grid", "domain": "kite",
         "nx": 4096, "ny": 4096, "x0": -1.776, "y0": -1.53, "h": 3.06 / 4096, "B": 8192,
         "k1": 3.06 / 4096, "n_f": 1, "precision": "mixed", "bdry": True},
        # ... and in double, the library's default precision.
        {"name": "kite4096_fp64", "kind": "spectrum", "form": "grid", "domain": "kite",
         "nx": 4096, "ny": 4096, "x0": -1.776, "y0": -1.53, "h": 3.06 / 4096, "B": 8192,
         "k1": 3.06 / 4096, "n_f": 1, "precision": "fp64", "bdry": True},
        # Many uneven domains at once: eight stars of 256^2 .. 2048^2, 32 fields each.
        {"name": "stars8_mixed", "kind": "group", "sizes": "256,384,512,640,768,1024,1536,2048",
         "shape_seed": 4, "n_f": 32, "precision": "mixed"},
        # Poisson on the star at 1024^2.
        {"name": "poisson_star1024", "kind": "poisson", "domain": "star", "a": 0.3, "k": 5,
         "nx": 1024, "ny": 1024, "x0": -1.1955, "y0": -1.3, "h": 2.6 / 1024, "B": 2048,
         "k1": 0.0013, "d": 5, "n_f": 1},
        # One interior step of the wave solver at 2048^2 (fourth order, d = 4, M = 7).
        {"name": "interior_kite2048", "kind": "interior", "domain": "kite", "nx": 2048,
         "ny": 2048, "B": 4096, "d": 4, "n_f": 1},
        # The whole wave solver, full U_FC at every small step, driven by boundary data
        # (plane waves), 8 solutions at 1024^2.
        {"name": "forward_full_kite1024", "kind": "forward", "mode": 0, "domain": "kite",
         "nx": 1024, "ny": 1024, "B": 2048, "d": 4, "n_f": 8, "driven": True},
        # The same solver with the small squares, pulses away from a reflecting boundary,
        # 8 solutions at 2048^2.
        {"name": "forward_squares_kite2048", "kind": "forward", "mode": 1, "domain": "kite",
         "nx": 2048, "ny": 2048, "B": 4096, "d": 4, "n_f": 8, "driven": False},
        # The largest: 32 solutions at 2048^2, squares in double-float.
        {"name": "forward_squares_df_kite2048", "kind": "forward", "mode": 2,
         "domain": "kite", "nx": 2048, "ny": 2048, "B": 4096, "d": 4, "n_f": 32,
         "driven": False},
    ]


def _smooth(lo, hi):
    return [n for n in range(lo + lo % 2, hi + 1, 2)
            if functools.reduce(lambda m, q: _strip_factor(m, q), (2, 3, 5), n) == 1]


def _strip_factor(m, q):
    while m % q == 0:
        m //= q
    return m


def _size(rng, lo, hi):
    """An even size 2^a 3^b 5^c near a log-uniform draw; every third one a power of two."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if rng.random() < 1 / 3:
        p = 2 ** round(math.log2(x))
        if lo <= p <= hi:
            return p
    return min(_smooth(lo, hi), key=lambda n: abs(n - x))


def _fields(rng, most, points):
    """A number of fields, log-uniform, so that n_f * points stays within `most` points."""
    top = max(1, min(32, int(most // points)))
    return max(1, int(round(math.exp(rng.uniform(0, math.log(top))))))


def _domain(rng, smallest):
    kind = rng.choice(("disk", "kite", "star")) if smallest >= 256 else rng.choice(("disk", "kite"))
    if kind == "star":
        return {"domain": "star", "a": round(rng.uniform(0.1, 0.3), 3), "k": rng.randint(3, 5)}
    return {"domain": kind}


def draw(rng):
    kind = rng.choice(("spectrum", "spectrum", "spectrum", "group", "poisson", "interior",
                       "forward"))
    if kind == "spectrum":
        nx = _size(rng, 128, 4096)
        ny = _size(rng, max(128, nx // 2), min(4096, 2 * nx))
        form = rng.choice(("grid", "grid", "compact", "complex", "split"))
        n_f = _fields(rng, 4096 * 4096 // (2 if form == "complex" else 1), nx * ny)
        return dict(_domain(rng, min(nx, ny)), kind=kind, form=form, nx=nx, ny=ny, n_f=n_f,
                    precision=rng.choice(("fp64", "mixed")), bdry=rng.random() < 0.75)
    if kind == "group":
        sizes = [_size(rng, 256, 2048) for _ in range(rng.randint(2, 6))]
        n_f = _fields(rng, 20e6, sum(n * n for n in sizes))
        return {"kind": kind, "sizes": ",".join(map(str, sizes)), "n_f": n_f,
                "shape_seed": rng.randrange(1000), "precision": rng.choice(("mixed", "mixed", "fp64"))}
    if kind == "poisson":
        n = _size(rng, 256, 1024)
        return dict(_domain(rng, n), kind=kind, nx=n, ny=n, d=rng.choice((5, 5, 10)), n_f=1)
    if kind == "interior":
        n = _size(rng, 256, 2048)
        return dict(_domain(rng, n), kind=kind, nx=n, ny=n, d=rng.choice((4, 5)),
                    n_f=_fields(rng, 2048 * 2048, n * n))
    mode = rng.choice((0, 1, 2))
    if mode == 0:
        n = _size(rng, 256, 1024)
        n_f = _fields(rng, 1024 * 1024 * 8, n * n)
    else:
        n = _size(rng, 960, 2048)
        n_f = _fields(rng, 2048 * 8, n)
    return {"kind": kind, "mode": mode, "domain": rng.choice(("disk", "kite")), "nx": n, "ny": n,
            "d": 4, "n_f": n_f, "driven": rng.random() < 0.5}


# ---------------------------------------------------------------------------- domains
def _curve(case):
    """Trigonometric coefficients (cx, sx, cy, sy) of the counter-clockwise curve."""
    if case["domain"] == "disk":
        return np.array([[0.0, 1.0], [0.0, 0.0], [0.0, 0.0], [0.0, 1.0]])
    if case["domain"] == "kite":  # x = cos t + 0.65 cos 2t - 0.65, y = 1.5 sin t
        return np.array([[-0.65, 1.0, 0.65], [0.0] * 3, [0.0] * 3, [0.0, 1.5, 0.0]])
    a, k = case["a"], case["k"]   # r = 1 + a cos k t
    cv = np.zeros((4, k + 2))
    cv[0, 1] += 1.0
    cv[3, 1] += 1.0
    cv[0, k + 1] += a / 2
    cv[0, k - 1] += a / 2
    cv[3, k + 1] += a / 2
    cv[3, k - 1] -= a / 2
    return cv


def _xy(cv, t, der=0):
    """The curve's point (or a derivative) at the parameters t."""
    k = np.arange(cv.shape[1]).reshape(-1, *([1] * np.ndim(t)))
    ph = k * t + der * math.pi / 2
    c, s = k ** der * np.cos(ph), k ** der * np.sin(ph)
    return (np.tensordot(cv[0], c, 1) + np.tensordot(cv[1], s, 1),
            np.tensordot(cv[2], c, 1) + np.tensordot(cv[3], s, 1))


@functools.lru_cache(maxsize=None)
def _outline(key):
    """Bounding box, perimeter, area and smallest radius of curvature of a curve."""
    cv = np.array(key)
    t = 2 * math.pi * np.arange(8192) / 8192
    (x, y), (xp, yp), (xq, yq) = _xy(cv, t), _xy(cv, t, 1), _xy(cv, t, 2)
    v = np.hypot(xp, yp)
    area = float(np.mean(x * yp - y * xp)) * math.pi
    rho = 1.0 / np.max(np.abs(xp * yq - yp * xq) / v ** 3)
    return x.min(), x.max(), y.min(), y.max(), float(np.mean(v)) * 2 * math.pi, area, rho


def _setting(case):
    """(curve, (x0, y0, h, nx, ny), parameters) of a case.  Without a box of its own the
    grid is laid around the curve's bounding box, a fraction of a cell off its centre (so
    that no grid line touches a symmetric curve), and the strip of width C k1 ends about 4
    cells inside it; k1 is h unless the strip would pass half the smallest radius of
    curvature."""
    cv = _curve(case)
    x0, x1, y0, y1, length, _, rho = _outline(tuple(map(tuple, cv)))
    nx, ny, d = case["nx"], case["ny"], case.get("d", 5)
    prm = {"d": d, "M": d + 3}
    if "h" in case:
        grid = (case["x0"], case["y0"], case["h"], nx, ny)
        prm.update(B=case["B"], k1=case["k1"])
        return cv, grid, prm
    cap = (rho if case["domain"] == "star" else min(rho, 1.0)) / (2 * C)
    room = [(x1 - x0, nx - 8 - 2 * C), (y1 - y0, ny - 8 - 2 * C)]
    h = max(w / n if n > 0 else math.inf for w, n in room)
    k1 = h
    if h > cap:
        k1 = cap
        h = max((x1 - x0 + 2 * C * k1) / (nx - 8), (y1 - y0 + 2 * C * k1) / (ny - 8))
    h, k1 = float(h), float(k1)
    prm.update(k1=k1, B=case.get("B", 32 * math.ceil(length / h / 32)))
    return cv, (float(0.5 * (x0 + x1 - nx * h) + 0.31 * h), float(0.5 * (y0 + y1 - ny * h) + 0.17 * h), h,
                nx, ny), prm


def _stars(case):
    """The domains of a group: stars r = 1 + a cos k t, a in [0.1, 0.3], k in 3..7, the
    more concave ones on the larger grids."""
    rng = np.random.default_rng(case["shape_seed"])
    sizes = sorted(int(n) for n in case["sizes"].split(","))
    shapes = [{"domain": "star", "a": float(0.1 + 0.2 * rng.random()), "k": int(rng.integers(3, 8))}
              for _ in sizes]
    shapes.sort(key=lambda s: -_outline(tuple(map(tuple, _curve(s))))[6])
    return [dict(s, nx=n, ny=n) for s, n in zip(shapes, sizes)]


# ---------------------------------------------------------------------------- fields
def _rng(case, seed):
    return np.random.default_rng([seed, case["nx"], case["ny"]] if "nx" in case else [seed, 1])


def _centres(cv, rng, n, margin):
    """n points of the domain at least `margin` from the curve."""
    px, py = _xy(cv, 2 * math.pi * np.arange(1024) / 1024)
    qx, qy = np.roll(px, -1), np.roll(py, -1)
    got = np.zeros((0, 2))
    while len(got) < n:
        p = np.stack([rng.uniform(px.min(), px.max(), 256), rng.uniform(py.min(), py.max(), 256)], 1)
        x, y = p[:, :1], p[:, 1:]
        span = (py > y) != (qy > y)
        cross = span & (x < (qx - px) * (y - py) / np.where(qy == py, 1.0, qy - py) + px)
        ok = (cross.sum(1) % 2 == 1) & (np.hypot(x - px, y - py).min(1) >= margin)
        got = np.concatenate([got, p[ok]])
    return got[:n]


def _blobs(cv, rng, n_f, terms, w0, w1, margin=0.0):
    """n_f sums of `terms` Gaussians: amplitudes N(0, 1), widths in [w0, w1]."""
    ctr = _centres(cv, rng, n_f * terms, margin).reshape(n_f, terms, 2)
    return [torch.tensor(v, dtype=F64, device=_dev()) for v in
            (rng.standard_normal((n_f, terms)), ctr[..., 0], ctr[..., 1],
             rng.uniform(w0, w1, (n_f, terms)))]


def _blobs_on(blobs, x, y):
    """Gaussian sums at every (x[i], y[i])."""
    a, cx, cy, w = (v[..., None] for v in blobs)
    return (a * torch.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2 * w * w))).sum(1)


def _blobs_grid(blobs, xs, ys):
    """Gaussian sums on a tensor grid, [n_f][ny][nx]."""
    a, cx, cy, w = (v[..., None] for v in blobs)
    gx, gy = (torch.exp(-((s - c) ** 2) / (2 * w * w)) for s, c in ((xs, cx), (ys, cy)))
    return torch.einsum("fky,fkx->fyx", a * gy, gx)


def _waves(rng, n_f):
    """Plane waves cos(kappa (x cos s + y sin s + t) + phi), kappa near 10."""
    v = np.stack([rng.uniform(8, 12, n_f), rng.uniform(0, 2 * math.pi, n_f),
                  rng.uniform(0, 2 * math.pi, n_f)])
    return torch.tensor(v, dtype=F64, device=_dev())


def _waves_on(wv, x, y, t, rate=False):
    k, s, phi = (v.reshape(-1, *([1] * max(x.ndim, y.ndim))) for v in wv)
    ph = k * (x * torch.cos(s) + y * torch.sin(s) + t) + phi
    return -k * torch.sin(ph) if rate else torch.cos(ph)


def _product(rng):
    """u = sin(p x + s) e^(q y), with Laplacian (q^2 - p^2) u."""
    p, q, s = rng.uniform(1.5, 2.5), rng.uniform(0.4, 1.2), rng.uniform(0, 2 * math.pi)
    return (lambda x, y: torch.sin(p * x + s) * torch.exp(q * y)), q * q - p * p


def _axes(grid):
    x0, y0, h, nx, ny = grid
    return (x0 + h * torch.arange(nx, dtype=F64, device=_dev()),
            y0 + h * torch.arange(ny, dtype=F64, device=_dev()))


# ---------------------------------------------------------------------------- prepare, run
@functools.lru_cache(maxsize=None)
def _plan_of(key, grid, prm, mixed):
    return fc2d.fc2d_plan(np.array(key), grid, dict(prm), fc2d.FC2D_MIXED if mixed else fc2d.FC2D_FP64)


def _plan(case, mixed):
    cv, grid, prm = _setting(case)
    plan = _plan_of(tuple(map(tuple, cv)), grid, tuple(sorted(prm.items())), mixed)
    return cv, grid, plan


def _boundary(plan):
    return [torch.tensor(v, dtype=F64, device=_dev()) for v in plan.fc2d_boundary_points().T.copy()]


@functools.lru_cache(maxsize=None)
def _group_of(plans):
    return fc2d.fc2d_group_create(plans)


def prepare(case, seed):
    kind, n_f = case["kind"], case["n_f"]
    rng = _rng(case, seed)
    mixed = case.get("precision") == "mixed"
    out_t = torch.float32 if mixed else F64
    new = lambda *shape: torch.zeros(shape, dtype=out_t, device=_dev())  # noqa: E731
    if kind == "group":
        made = [_plan(c, mixed) for c in _stars(case)]
        state = {"kind": kind, "group": _group_of(tuple(p for _, _, p in made)),
                 "n_f": [n_f] * len(made), "f": [], "b": [], "out": []}
        for cv, grid, plan in made:
            blobs = _blobs(cv, rng, n_f, 16, 0.1, 0.3)
            state["f"].append(_blobs_grid(blobs, *_axes(grid)))
            state["b"].append(_blobs_on(blobs, *_boundary(plan)))
            state["out"].append(new(n_f, grid[4], grid[3] // 2 + 1, 2))
        return state
    cv, grid, plan = _plan(case, mixed)
    nx, ny = grid[3], grid[4]
    xs, ys = _axes(grid)
    bx, by = _boundary(plan)
    state = {"kind": kind, "plan": plan, "n_f": n_f}
    if kind == "spectrum":
        form = case["form"]
        parts = 2 if form == "complex" else 1
        blobs = _blobs(cv, rng, n_f * parts, 16, 0.1, 0.3)
        state.update(form=form, f=_blobs_grid(blobs, xs, ys), b=_blobs_on(blobs, bx, by) if case["bdry"] else None)
        if form == "compact":
            at = torch.tensor(plan.fc2d_inside_points(), device=_dev())
            state["f"] = state["f"].reshape(n_f, -1)[:, at].contiguous()
        if form == "split":
            state["ext"] = new(n_f, ny, nx)
        state["out"] = new(n_f, ny, nx if form == "complex" else nx // 2 + 1, 2)
    elif kind == "poisson":
        u, factor = _product(rng)
        plan.fc2d_poisson_plan(0)
        gx, gy = torch.tensor(plan.fc2d_poisson_nodes().T.copy(), dtype=F64, device=_dev())
        state.update(f=factor * u(xs, ys[:, None])[None], b=factor * u(bx, by)[None], g=u(gx, gy)[None],
                     out=new(1, ny, nx), phi=new(1, len(gx)))
    elif kind == "interior":
        u, v = (_blobs(cv, rng, n_f, 32, 0.05, 0.05, 0.3) for _ in range(2))
        state.update(t=N_C * grid[2], u0=_blobs_grid(u, xs, ys), ub=_blobs_on(u, bx, by), v0=_blobs_grid(v, xs, ys),
                     vb=_blobs_on(v, bx, by), u=new(n_f, ny, nx), v=new(n_f, ny, nx))
    else:
        state.update(mode=case["mode"], u=new(n_f, ny, nx), v=new(n_f, ny, nx), g=None, gt=None)
        if case["driven"]:
            wv, dt = _waves(rng, n_f), grid[2] / 8
            at = lambda s, rate: _waves_on(wv, bx, by, s * dt, rate)  # noqa: E731
            state.update(u0=_waves_on(wv, xs, ys[:, None], 0.0), v0=_waves_on(wv, xs, ys[:, None], 0.0, True),
                         g=torch.stack([at(s, False) for s in range(8 * N_C + 1)]),
                         gt=torch.stack([at(s, True) for s in (0, 8 * N_C)]))
        else:
            pulse = _blobs(cv, rng, n_f, 1, 0.05, 0.05, 0.35)
            state.update(u0=_blobs_grid(pulse, xs, ys), v0=new(n_f, ny, nx))
    return state


def run(state):
    kind, n_f = state["kind"], state["n_f"]
    if kind == "group":
        state["group"].fc2d_group_extend_coeffs(n_f, state["f"], state["b"], state["out"])
        return state["out"]
    plan = state["plan"]
    if kind == "spectrum":
        f, b, out = state["f"], state["b"], state["out"]
        if state["form"] == "compact":
            plan.fc2d_extend_coeffs_compact(n_f, f, b, out)
        elif state["form"] == "complex":
            plan.fc2d_extend_coeffs_complex(n_f, f, b, out)
        elif state["form"] == "split":
            plan.fc2d_extend(n_f, f, b, state["ext"])
            plan.fc2d_coeffs(n_f, state["ext"], out)
            return {"ext": state["ext"], "spectrum": out}
        else:
            plan.fc2d_extend_coeffs(n_f, f, b, out)
        return {"spectrum": out}
    if kind == "poisson":
        plan.fc2d_poisson(n_f, state["f"], state["b"], state["g"], state["out"], state["phi"])
        return {"u": state["out"], "phi": state["phi"]}
    if kind == "interior":
        plan.fc2d_wave_interior(n_f, 1.0, state["t"], state["u0"], state["ub"], state["v0"],
                                state["vb"], state["u"], state["v"])
    else:  # the solver advances u and u_t in place, from the kept initial data
        state["u"].copy_(state["u0"])
        state["v"].copy_(state["v0"])
        plan.fc2d_forward_wave(n_f, 1.0, N_C, 1, state["u"], state["v"], state["g"], state["gt"],
                               squares=state["mode"] > 0, double_float=state["mode"] == 2)
    return {"u": state["u"], "ut": state["v"]}


def work(case):
    """Each field read at the domain's points and each result written once; the DFTs
    (5/2 N log2 N for N reals), the continuation and, for Poisson, the boundary sums."""
    if case["kind"] == "group":
        parts = [work(dict(c, kind="spectrum", form="grid", n_f=case["n_f"], bdry=True,
                           precision=case["precision"])) for c in _stars(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    cv, (_, _, h, nx, ny), prm = _setting(case)
    length, area = _outline(tuple(map(tuple, cv)))[4:6]
    n, inside, n_f = nx * ny, area / h ** 2, case["n_f"]
    dft = 2.5 * n * math.log2(n)
    m, d = prm["M"], prm["d"]
    ext = prm["B"] * 2.0 * ((m - 1) * m + d * m + d * d + C * N_R * d) \
        + length * C * prm["k1"] / h ** 2 * 2.0 * (m * m + m)
    kind = case["kind"]
    if kind == "spectrum":
        parts = 2 if case["form"] == "complex" else 1
        size = 4 if case["precision"] == "mixed" else 8
        out = n * size * (2 if case["form"] == "split" else 1)
        return {"bytes": n_f * parts * (8.0 * inside + out), "flops": n_f * parts * (dft + ext)}
    if kind == "poisson":
        return {"bytes": n_f * 16.0 * inside, "flops": n_f * (2 * dft + ext + 8.0 * inside * nx)}
    if kind == "interior":
        return {"bytes": n_f * 16.0 * (inside + n), "flops": n_f * (4 * dft + 2 * ext)}
    # both spectra, U_FC and its derivative at the end, and 8 n_c small steps: of the band
    # (about 40 operator entries a point), and of the interface values: by a whole inverse
    # DFT, or from squares of 37 points along the band's inner edge
    band = 8 * N_C * length / h * (N_C + 2) * 80.0
    face = 8 * N_C * (dft if case["mode"] == 0 else length / h / 20 * 2.5 * 4096 * 12)
    return {"bytes": n_f * 32.0 * inside, "flops": n_f * (4 * dft + 2 * ext + band + face)}


# ---------------------------------------------------------------------------- exact
@functools.lru_cache(maxsize=None)
def _fc_matrices(d):
    """Q (d x d) and A_r (C n_r x d) of Section 2.2 in 60-digit arithmetic: the Gram
    polynomials of d points, each continued by the trigonometric polynomial that fits it on
    the oversampled points and zero on the far ones in the least-squares sense."""
    D = decimal.Decimal
    with decimal.localcontext(decimal.Context(prec=60)):
        atan = lambda n: sum((-1) ** k * D(1) / ((2 * k + 1) * D(n) ** (2 * k + 1)) for k in range(90))  # noqa: E731
        period = d + 2 * C + Z - 1
        den = 60 * period  # N_OS and N_R divide 60
        x = 2 * (16 * atan(5) - 4 * atan(239)) / den
        c1 = sum((-1) ** k * x ** (2 * k) / math.factorial(2 * k) for k in range(30))
        s1 = sum((-1) ** k * x ** (2 * k + 1) / math.factorial(2 * k + 1) for k in range(30))
        turn = [(D(1), D(0))]
        for _ in range(den - 1):
            c, s = turn[-1]
            turn.append((c * c1 - s * s1, s * c1 + c * s1))

        def basis(num):  # at the point num / 60
            w = [turn[m * num % den] for m in range(1, M_F + 1)]
            return [D(1)] + [v for cs in w for v in cs]

        def orthonormal(cols):
            q, r = [], []
            for v in cols:
                r.append([])
                for u in q:
                    p = sum(a * b for a, b in zip(u, v))
                    r[-1].append(p)
                    v = [b - p * a for a, b in zip(u, v)]
                p = sum(b * b for b in v).sqrt()
                r[-1].append(p)
                q.append([b / p for b in v])
            return q, r  # r[j][i], i <= j

        def solve(r, b):  # upper triangular
            y = list(b)
            for j in reversed(range(len(y))):
                y[j] /= r[j][j]
                for i in range(j):
                    y[i] -= r[j][i] * y[j]
            return y

        q, r = orthonormal([[D(i) ** j if j else D(1) for i in range(d)] for j in range(d)])
        near = [60 // N_OS * i for i in range(N_OS * (d - 1) + 1)]
        far = [60 // N_OS * i for i in range(N_OS * (d + C), N_OS * (d + C + Z - 1) + 1)]
        rows = [basis(v) for v in near + far]
        bq, br = orthonormal([list(col) for col in zip(*rows)])
        fine = [basis(60 * (d - 1) + 60 // N_R * v) for v in range(1, C * N_R + 1)]
        ar = np.zeros((C * N_R, d))
        for j in range(d):
            unit = solve(r, [D(int(i == j)) for i in range(d)])  # Gram polynomial j's coefficients
            gram = [sum(a * (D(v) / 60) ** i if i else a for i, a in enumerate(unit)) for v in near]
            coef = solve(br, [sum(a * b for a, b in zip(u, gram)) for u in bq])
            ar[:, j] = [float(sum(a * b for a, b in zip(row, coef))) for row in fine]
        return np.array([[float(q[j][i]) for j in range(d)] for i in range(d)]), ar


def _crossings(cv, axis, o, h, n, samples):
    """Crossings of the grid lines o + h i of coordinate `axis` (0: x, 1: y) with the curve,
    by line and then along it: (line, parameter sorted by the other coordinate, that)."""
    t = 2 * math.pi * np.arange(samples + 1) / samples
    v = _xy(cv, t)[axis]
    v[-1] = v[0]
    lo, hi = np.minimum(v[:-1], v[1:]), np.maximum(v[:-1], v[1:])
    first = np.maximum(np.ceil((lo - o) / h).astype(int) - 1, 0)
    span = np.minimum(np.ceil((hi - o) / h).astype(int) + 1, n) - first
    at = np.repeat(np.arange(samples), np.maximum(span, 0))
    start = np.cumsum(np.maximum(span, 0)) - np.maximum(span, 0)
    line = first[at] + np.arange(len(at)) - start[at]
    c = o + h * line
    use = (v[at] > c) != (v[at + 1] > c)
    at, line, c = at[use], line[use], c[use]
    a, b, up = t[at].copy(), t[at + 1].copy(), v[at] > c
    for _ in range(55):
        m = 0.5 * (a + b)
        same = (_xy(cv, m)[axis] > c) == up
        a, b = np.where(same, m, a), np.where(same, b, m)
    r = 0.5 * (a + b)
    other = _xy(cv, r)[1 - axis]
    order = np.lexsort((other, line))
    line, other = line[order], other[order]
    touch = np.zeros(len(line) + 1, bool)  # a line that only touches the curve
    touch[1:-1] = (np.diff(line) == 0) & (np.diff(other) < 1e-7 * n * h)
    keep = ~(touch[1:] | touch[:-1])
    return line[keep], other[keep]


class _Reference:
    """The extension of one domain, grid and order, in 64 bits."""

    def __init__(self, cv, grid, prm, bdry=True):
        self.cv, self.grid, self.prm, self.bdry = cv, grid, prm, bdry
        x0, y0, h, nx, ny = grid
        d, m, n_b, k1 = prm["d"], prm["M"], prm["B"], prm["k1"]
        self.xs, self.ys = x0 + h * np.arange(nx), y0 + h * np.arange(ny)
        self.cols = _crossings(cv, 0, x0, h, nx, 16 * n_b)
        self.rows = _crossings(cv, 1, y0, h, ny, 16 * n_b)
        # inside: between consecutive crossings of the row
        mark = np.zeros((ny, nx + 1), int)
        j, x = self.rows
        np.add.at(mark, (j[::2], np.searchsorted(self.xs, x[::2], "left")), 1)
        np.add.at(mark, (j[1::2], np.searchsorted(self.xs, x[1::2], "right")), -1)
        self.inside = np.cumsum(mark, 1)[:, :-1] > 0
        # strip: feet of the normals, from seeds laid out along the normals
        t = 2 * math.pi * np.arange(8 * n_b) / (8 * n_b)
        (bx, by), (tx, ty) = _xy(cv, t), _xy(cv, t, 1)
        v = np.hypot(tx, ty)
        seed = np.full((ny, nx), -1.0)
        for s in np.arange(0, C * k1 + 2 * h, 0.4 * min(h, k1)):
            i = np.rint((bx + s * ty / v - x0) / h).astype(int)
            j = np.rint((by - s * tx / v - y0) / h).astype(int)
            ok = (i >= 0) & (i < nx) & (j >= 0) & (j < ny)
            seed[j[ok], i[ok]] = t[ok]
        self.at = np.flatnonzero(((seed >= 0) & ~self.inside).ravel())
        th = seed.ravel()[self.at]
        qx, qy = self.xs[self.at % nx], self.ys[self.at // nx]
        for _ in range(12):
            (x, y), (xp, yp), (xq, yq) = (_xy(cv, th, der) for der in (0, 1, 2))
            th = th - ((x - qx) * xp + (y - qy) * yp) / (xp ** 2 + yp ** 2 + (x - qx) * xq + (y - qy) * yq)
        x, y = _xy(cv, th)
        eta = np.hypot(qx - x, qy - y)
        keep = (eta > 0) & (eta <= C * k1)
        self.at, th, eta = self.at[keep], np.mod(th[keep], 2 * math.pi), eta[keep]
        # interpolation onto the strip: M normals around the foot, M fine nodes around eta
        left = (m + 1) // 2 - 1
        p = np.floor(th * n_b / (2 * math.pi)).astype(int)
        u = eta * N_R / k1
        s = np.clip(np.floor(u).astype(int) - left, 0, C * N_R + 1 - m)
        nodes = np.arange(m)[None, :] + np.zeros((len(s), 1))
        self.w_theta = self._lagrange(nodes, th * n_b / (2 * math.pi) - (p - left))
        self.w_eta = self._lagrange(nodes, u - s)
        self.normal = np.mod(p[:, None] - left + np.arange(m), n_b)
        self.fine = s[:, None] + np.arange(m)
        self._matching()

    @staticmethod
    def _lagrange(nodes, t, used=None):
        """Lagrange weights of each row's nodes (of those `used`) at t."""
        w = np.ones(nodes.shape)
        for a in range(nodes.shape[1]):
            for b in range(nodes.shape[1]):
                if a != b:
                    f = (t - nodes[:, b]) / np.where(nodes[:, a] == nodes[:, b], 1.0, nodes[:, a] - nodes[:, b])
                    w[:, a] *= f if used is None else np.where(used[:, b], f, 1.0)
        return w if used is None else np.where(used, w, 0.0)

    def _matching(self):
        """Points and weights of the matching values of every normal (Section 3.2)."""
        x0, y0, h, nx, ny = self.grid
        d, m, n_b, k1 = (self.prm[k] for k in ("d", "M", "B", "k1"))
        t = 2 * math.pi * np.arange(n_b) / n_b
        (bx, by), (tx, ty) = _xy(self.cv, t), _xy(self.cv, t, 1)
        v = np.hypot(tx, ty)
        nrm = np.stack([ty / v, -tx / v])
        foot = np.stack([bx, by])
        self.foot = foot
        self.px, self.py = np.zeros((n_b, m - 1, m)), np.zeros((n_b, m - 1, m))
        self.pw, self.tk = np.zeros((n_b, m - 1, m)), np.zeros((n_b, m - 1))
        upright = np.abs(nrm[0]) >= np.abs(nrm[1]) * (1 - 2.0 ** -30)
        for axis, lines, o, along in ((0, self.cols, (x0, y0), ny), (1, self.rows, (y0, x0), nx)):
            at = np.flatnonzero(upright if axis == 0 else ~upright)
            b, c = foot[axis, at], foot[1 - axis, at]
            nb, nc = nrm[axis, at], nrm[1 - axis, at]
            xi = (b - 0.5 * h * nb - o[0]) / h
            i0 = np.where(nb > 0, np.floor(xi), np.ceil(xi)).astype(int)
            key = lines[0] * 64.0 + lines[1]
            for k in range(m - 1):
                line = i0 - np.where(nb > 0, 1, -1) * k
                coord = o[0] + h * line
                tk = (coord - b) / nb
                star = c + tk * nc
                e = np.searchsorted(key, line * 64.0 + star, "right") - 1
                lo, hi = lines[1][e], lines[1][e + 1]
                first, last = np.ceil((lo - o[1]) / h).astype(int), np.floor((hi - o[1]) / h).astype(int)
                if self.bdry:
                    first += (o[1] + h * first) - lo < 0.5 * h
                    last -= hi - (o[1] + h * last) < 0.5 * h
                ends = 1 if self.bdry else 0
                n = last - first + 1 + 2 * ends
                below = np.clip(np.floor((star - o[1]) / h).astype(int) - first + 1, 0, n - 2 * ends) + ends
                s = np.clip(below - (m + 1) // 2, 0, np.maximum(n - m, 0))
                idx = s[:, None] + np.arange(m)
                pos = o[1] + h * (first[:, None] + idx - ends)
                if self.bdry:
                    pos = np.where(idx == 0, lo[:, None], np.where(idx >= n[:, None] - 1, hi[:, None], pos))
                self.pw[at, k] = self._lagrange(pos, star, idx < n[:, None])
                self.px[at, k], self.py[at, k] = (coord[:, None], pos) if axis == 0 else (pos, coord[:, None])
                self.tk[at, k] = tk
        nodes = np.concatenate([np.zeros((n_b, 1)), self.tk], 1) if self.bdry else self.tk
        self.wn = np.stack([self._lagrange(nodes, (q - d + 1) * k1) for q in range(d)], 1)

    def extend(self, on_points, on_grid):
        """The extended fields: on_points(x, y) gives the fields [n_f][...] at points,
        on_grid the fields on the grid."""
        T = lambda a: torch.tensor(a, device=_dev())  # noqa: E731
        q, ar = (T(a) for a in _fc_matrices(self.prm["d"]))
        at = on_points(T(self.px).reshape(-1), T(self.py).reshape(-1))
        stars = (at.reshape(-1, *self.pw.shape) * T(self.pw)).sum(-1)
        if self.bdry:
            foot = on_points(T(self.foot[0]), T(self.foot[1]))
            stars = torch.cat([foot[..., None], stars], -1)
        match = torch.einsum("pqk,fpk->fpq", T(self.wn), stars)
        first = match[..., -1:]
        blend = torch.cat([first, torch.einsum("rk,fpk->fpr", ar, torch.einsum("qk,fpq->fpk", q, match))], -1)
        normal, fine = T(self.normal), T(self.fine)
        wt, we = T(self.w_theta), T(self.w_eta)
        out = torch.where(T(self.inside), on_grid, 0.0).reshape(len(on_grid), -1)
        for f in range(len(out)):
            v = blend[f][normal[:, :, None], fine[:, None, :]]
            out[f, T(self.at)] = torch.einsum("na,nab,nb->n", wt, v, we)
        return out.reshape(on_grid.shape)


@functools.lru_cache(maxsize=4)
def _reference_of(key, grid, prm, bdry):
    return _Reference(np.array(key), grid, dict(prm), bdry)


def _reference(case, bdry=True):
    cv, grid, prm = _setting(case)
    return _reference_of(tuple(map(tuple, cv)), grid, tuple(sorted(prm.items())), bdry)


def _spectrum(ext):
    return torch.view_as_real(torch.fft.rfft2(ext) / ext[0].numel())


def exact(case, seed):
    kind, n_f = case["kind"], case["n_f"]
    rng = _rng(case, seed)
    if kind == "group":
        out = []
        for c in _stars(case):
            ref = _reference(c)
            blobs = _blobs(ref.cv, rng, n_f, 16, 0.1, 0.3)
            out.append(_spectrum(ref.extend(lambda x, y: _blobs_on(blobs, x, y), _blobs_grid(blobs, *_axes(ref.grid)))))
        return out
    cv, grid, prm = _setting(case)
    xs, ys = _axes(grid)
    if kind == "spectrum":
        parts = 2 if case["form"] == "complex" else 1
        ref = _reference(case, case["bdry"])
        blobs = _blobs(cv, rng, n_f * parts, 16, 0.1, 0.3)
        ext = ref.extend(lambda x, y: _blobs_on(blobs, x, y), _blobs_grid(blobs, xs, ys))
        if case["form"] == "complex":
            return {"spectrum": torch.view_as_real(torch.fft.fft2(torch.complex(ext[0::2], ext[1::2])) / ext[0].numel())}
        return dict({"spectrum": _spectrum(ext)}, **({"ext": ext} if case["form"] == "split" else {}))
    ref = _reference(case)
    inside = torch.tensor(ref.inside, device=_dev())
    if kind == "poisson":  # the solution of the continuous problem; the density has no closed form
        u, _ = _product(rng)
        return {"u": torch.where(inside, u(xs, ys[:, None]), 0.0)[None], "phi": None}
    if kind == "forward" and case["driven"]:
        wv, t = _waves(rng, n_f), N_C * grid[2]
        return {"u": torch.where(inside, _waves_on(wv, xs, ys[:, None], t), 0.0),
                "ut": torch.where(inside, _waves_on(wv, xs, ys[:, None], t, True), 0.0)}
    # modal solution of the wave equation on the periodic box; a pulse of the whole solver
    # stays away from the boundary
    if kind == "interior":
        u, v = (_blobs(cv, rng, n_f, 32, 0.05, 0.05, 0.3) for _ in range(2))
        f, g = (ref.extend(lambda x, y, b=b: _blobs_on(b, x, y), _blobs_grid(b, xs, ys)) for b in (u, v))
    else:
        f = _blobs_grid(_blobs(cv, rng, n_f, 1, 0.05, 0.05, 0.35), xs, ys)
        g = torch.zeros_like(f)
    h, nx, ny = grid[2:]
    l = torch.arange(nx // 2 + 1, dtype=F64, device=_dev()) / (nx * h)
    m = torch.fft.fftfreq(ny, h, dtype=F64, device=_dev())
    w = 2 * math.pi * torch.sqrt(l ** 2 + m[:, None] ** 2)
    t = N_C * h
    sw = torch.where(w > 0, torch.sin(w * t) / torch.where(w > 0, w, 1.0), t)
    out = {"u": [], "ut": []}
    for a, b in zip(f, g):
        a, b = torch.fft.rfft2(a), torch.fft.rfft2(b)
        out["u"].append(torch.fft.irfft2(a * torch.cos(w * t) + b * sw, s=(ny, nx)))
        out["ut"].append(torch.fft.irfft2(b * torch.cos(w * t) - a * w * torch.sin(w * t), s=(ny, nx)))
    out = {k: torch.stack(v) for k, v in out.items()}
    return out if kind == "interior" else {k: torch.where(inside, v, 0.0) for k, v in out.items()}
