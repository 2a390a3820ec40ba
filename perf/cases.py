"""The workloads this framework is timed on, through its public entry points.

Five kinds of call, as a user's program makes them:

  noalloc   fmm.reinit_noalloc: a tiny level set, no handle, no device allocation
  reinit    Solver.reinit: signed distance to the zero set of a level set
  sources   Solver.solve: first arrivals of point sources
  grad      EikonalFn: travel times for a slowness field, and the gradient of a
            receiver loss with respect to the slowness
  batch     Batch.reinit: many uneven grids in one solve

Inputs follow the recipes of ``workloads`` (random spheres with a modulated
level set, random Fourier speed, uneven batches), drawn from the seed alone.
"""
import math

import numpy as np
import torch

from paper_1502_07303_gb300 import fmm, workloads

DEV = "cuda"
DTYPES = {"f32": torch.float32, "f64": torch.float64}
EXACT_CELLS = 18_000_000   # larger grids take too long in plain torch


def listed():
    return [
        # a small level set reinitialised by a caller that cannot allocate:
        # the smallest call, all launches and latency
        {"name": "noalloc_45x37x40_f32", "kind": "noalloc", "nx": 45, "ny": 37, "nz": 40,
         "dtype": "f32", "spheres": 3},
        # the method's reference instance: one point source in a 64^3 cube
        {"name": "point_64_f64", "kind": "sources", "nx": 64, "ny": 64, "nz": 64,
         "dtype": "f64", "sources": 1, "fourier": False},
        # reinitialisation inside a simulation step, ordinary size, both types
        {"name": "reinit_256_f32", "kind": "reinit", "nx": 256, "ny": 256, "nz": 256,
         "dtype": "f32", "spheres": 32, "width": 0.0, "order": 1, "ry": 1.0, "rz": 1.0},
        {"name": "reinit_256_f64", "kind": "reinit", "nx": 256, "ny": 256, "nz": 256,
         "dtype": "f64", "spheres": 32, "width": 0.0, "order": 1, "ry": 1.0, "rz": 1.0},
        # a narrow band around the front, as level-set codes keep it, on a
        # ragged grid (in double: in single precision the cells at the band's
        # rim change tags from run to run)
        {"name": "band_203x171x190_f64", "kind": "reinit", "nx": 203, "ny": 171, "nz": 190,
         "dtype": "f64", "spheres": 12, "width": 6.5, "order": 1, "ry": 1.0, "rz": 1.0},
        # cells of unequal sides on a ragged grid
        {"name": "aniso_227x150x301_f32", "kind": "reinit", "nx": 227, "ny": 150, "nz": 301,
         "dtype": "f32", "spheres": 16, "width": 0.0, "order": 1, "ry": 1.25, "rz": 0.8},
        # the second-order march
        {"name": "second_order_128_f64", "kind": "reinit", "nx": 128, "ny": 128, "nz": 128,
         "dtype": "f64", "spheres": 4, "width": 0.0, "order": 2, "ry": 1.0, "rz": 1.0},
        # travel times of several sources in a heterogeneous medium
        {"name": "speed_251x260x243_f32", "kind": "sources", "nx": 251, "ny": 260, "nz": 243,
         "dtype": "f32", "sources": 8, "fourier": True},
        # one step of a travel-time inversion: forward and backward, small and
        # full size (in double: in single precision the gradient jumps where
        # two arrivals meet and rounding picks the side)
        {"name": "grad_125x110x131_f64", "kind": "grad", "nx": 125, "ny": 110, "nz": 131,
         "dtype": "f64", "sources": 4, "receivers": 64},
        {"name": "grad_512_f64", "kind": "grad", "nx": 512, "ny": 512, "nz": 512,
         "dtype": "f64", "sources": 8, "receivers": 64},
        # many independent grids in one solve
        {"name": "batch_256_f32", "kind": "batch", "grids": 256, "lo": 32, "hi": 192,
         "dtype": "f32"},
        # the largest: signed distance to one sphere on 1.07e9 cells
        {"name": "sphere_1024_f64", "kind": "reinit", "nx": 1024, "ny": 1024, "nz": 1024,
         "dtype": "f64", "spheres": 1, "width": 0.0, "order": 1, "ry": 1.0, "rz": 1.0},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi):
        n = size(lo, hi)
        return {a: max(16, int(n * rng.uniform(0.7, 1.0))) for a in ("nx", "ny", "nz")}

    kind = rng.choice(["noalloc", "reinit", "reinit", "band", "second", "sources", "sources", "grad", "batch"])
    dt = rng.choice(["f32", "f64"])
    if kind == "noalloc":
        return {"kind": "noalloc", **box(24, 64), "dtype": dt, "spheres": rng.randint(1, 6)}
    if kind == "sources":
        return {"kind": "sources", **box(32, 500), "dtype": dt, "sources": rng.randint(1, 12),
                "fourier": rng.random() < 0.6}
    if kind == "grad":
        return {"kind": "grad", **box(32, 400), "dtype": "f64", "sources": rng.randint(1, 12),
                "receivers": rng.randint(16, 96)}
    if kind == "batch":
        lo = size(20, 64)
        return {"kind": "batch", "grids": size(6, 200), "lo": lo, "hi": lo + size(8, 128), "dtype": dt}
    unequal = rng.random() < 0.3
    case = {"kind": "reinit", **box(*((32, 140) if kind == "second" else (32, 700))),
            "dtype": dt, "spheres": size(1, 40), "width": 0.0, "order": 1,
            "ry": round(rng.uniform(0.6, 1.7), 2) if unequal else 1.0,
            "rz": round(rng.uniform(0.6, 1.7), 2) if unequal else 1.0}
    if kind == "second":
        case["order"] = 2
    if kind == "band":
        case.update(dtype="f64", width=round(rng.uniform(3.0, 14.0), 2))
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _shape(c):
    return (c["nz"], c["ny"], c["nx"])


def _cell(c):
    """Cell size of a case: one value, or (dx, dy, dz)."""
    h = workloads.spacing(_shape(c))
    if c.get("ry", 1.0) == 1.0 and c.get("rz", 1.0) == 1.0:
        return h
    return (h, h * c["ry"], h * c["rz"])


def _three(h):
    return (h, h, h) if np.isscalar(h) else h


def _level_set(shape, h, count, rng):
    """Random spheres inside the grid's own box: centres in [0.15, 0.85] of
    every side, radii 0.05 to 0.15 of the shortest side (one sphere: 0.2 to
    0.35), the level set of several modulated as in the workloads."""
    hx, hy, hz = _three(h)
    nz, ny, nx = shape
    ext = np.array([nx * hx, ny * hy, nz * hz])
    unit = workloads.draw_spheres(rng, count)
    if count == 1:
        unit = workloads.Spheres(rng.uniform(0.45, 0.55, (1, 3)), rng.uniform(0.2, 0.35, 1))
    sph = workloads.Spheres(unit.centres * ext[None, :], unit.radii * float(ext.min()))
    return workloads.spheres_phi0(shape, sph, h=h, modulate=count > 1, device=DEV)


def _batch_shapes(c):
    """Grid sizes of a batch: part of the case, not of the seed."""
    dims = np.random.default_rng([c["grids"], c["lo"], c["hi"]]).integers(c["lo"], c["hi"] + 1, size=(c["grids"], 3))
    return [tuple(int(v) for v in d) for d in dims]


def _cells(c):
    if c["kind"] == "batch":
        return sum(math.prod(s) for s in _batch_shapes(c))
    return c["nx"] * c["ny"] * c["nz"]


def _inputs(c, seed):
    """The arrays a case starts from, on the GPU in its dtype."""
    rng = np.random.default_rng([1502, int(seed)])
    dt = DTYPES[c["dtype"]]
    if c["kind"] == "batch":
        shapes = _batch_shapes(c)
        counts = rng.integers(1, 9, size=c["grids"])
        hs = [workloads.spacing(s) for s in shapes]
        phis = [_level_set(s, h, int(k), rng).to(dt).contiguous() for s, h, k in zip(shapes, hs, counts)]
        return {"shapes": shapes, "hs": hs, "phis": phis}
    shape, h = _shape(c), _cell(c)
    if c["kind"] in ("noalloc", "reinit"):
        return {"phi": _level_set(shape, h, c["spheres"], rng).to(dt).contiguous(), "h": h}
    if c["kind"] == "sources" and c["sources"] == 1:
        # the reference instance: the source at the centre cell, shifted a little by the seed
        d = rng.integers(-3, 4, size=3)
        src = np.array([[c["nx"] // 2 + d[0], c["ny"] // 2 + d[1], c["nz"] // 2 + d[2]]], np.int64)
    else:
        src = workloads.random_cells(rng, shape, c["sources"])
    out = {"h": h, "src": src, "speed": None}
    if c["kind"] == "grad" or c["fourier"]:
        modes = workloads.draw_fourier_modes(rng)
        F = workloads.fourier_speed(shape, modes, h=h, device=DEV)
        if c["kind"] == "grad":
            out["slowness"] = (1.0 / F).to(dt).contiguous()
            out["rec"] = workloads.random_cells(rng, shape, c["receivers"], exclude=src)
        else:
            out["speed"] = F.to(dt).contiguous()
    return out


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

def prepare(case, seed):
    c, x = case, _inputs(case, seed)
    dt = DTYPES[c["dtype"]]
    st = {"case": c, "x": x}
    if c["kind"] == "noalloc":
        st["T"] = torch.empty(_shape(c), dtype=dt, device=DEV)
        st["G"] = torch.empty(_shape(c), dtype=torch.uint8, device=DEV)
    elif c["kind"] == "reinit":
        h = _three(x["h"])[0]
        kw = {"width": c["width"] * h} if c["width"] else {}
        st["solver"] = fmm.Solver(_shape(c), x["h"], dtype=dt, accuracy=c["order"], **kw)
    elif c["kind"] == "sources":
        st["solver"] = fmm.Solver(_shape(c), x["h"], dtype=dt, speed=x["speed"], sources=x["src"])
    elif c["kind"] == "grad":
        st["solver"] = fmm.Solver(_shape(c), x["h"], dtype=dt, sources=x["src"], record_tape=True)
        st["s"] = x["slowness"].requires_grad_(True)
        st["rec"] = tuple(torch.as_tensor(x["rec"][:, a], device=DEV) for a in (2, 1, 0))
    else:
        st["solver"] = fmm.Batch(x["shapes"], x["hs"], dtype=dt)
        # one buffer for all grids' results, as a program that loops keeps it
        # (slices start on 256-byte boundaries)
        n = [(a * b * d + 255) // 256 * 256 for a, b, d in x["shapes"]]
        st["T"] = torch.zeros(sum(n), dtype=dt, device=DEV)
        st["G"] = torch.zeros(sum(n), dtype=torch.uint8, device=DEV)
        at = np.concatenate([[0], np.cumsum(n)])
        cut = [(int(at[g]), math.prod(s), s) for g, s in enumerate(x["shapes"])]
        st["Ts"] = [st["T"][a:a + m].view(s) for a, m, s in cut]
        st["Gs"] = [st["G"][a:a + m].view(s) for a, m, s in cut]
    return st


def run(state):
    c, x = state["case"], state["x"]
    if c["kind"] == "noalloc":
        T, G = fmm.reinit_noalloc(x["phi"], x["h"], state["T"], state["G"])
        return {"T": T, "tags": G}
    if c["kind"] == "reinit":
        T, G = state["solver"].reinit(x["phi"])
        return {"T": T, "tags": G}
    if c["kind"] == "sources":
        T, G = state["solver"].solve()
        return {"T": T, "tags": G}
    if c["kind"] == "grad":
        T = fmm.EikonalFn.apply(state["s"], state["solver"])
        loss = T[state["rec"]].sum()
        (g,) = torch.autograd.grad(loss, state["s"])
        return {"T": T.detach(), "loss": loss.detach(), "grad": g}
    state["solver"].reinit(x["phis"], state["Ts"], state["Gs"])
    return {"T": state["T"], "tags": state["G"]}


def work(case):
    c = case
    size = 8 if c["dtype"] == "f64" else 4
    n = float(_cells(c))
    # values in and out: a level set or a speed field if any, the solution; a
    # gradient step reads the slowness and writes the times and the gradient
    reads = 0 if c["kind"] == "sources" and not c["fourier"] else 1
    writes = 2 if c["kind"] == "grad" else 1
    tags = 0 if c["kind"] == "grad" else 1
    # one quadratic per cell (three axes: three comparisons, a sort, the
    # discriminant, a square root), and as much again for its derivative
    flops = 30.0 * n * (2 if c["kind"] == "grad" else 1)
    return {"bytes": n * (size * (reads + writes) + tags), "flops": flops}


# ---------------------------------------------------------------------------
# 64-bit values in plain torch
# ---------------------------------------------------------------------------

INF = float("inf")


def _shift(a, axis, step, fill):
    """b[i] = a[i + step] along a dimension, fill beyond the border."""
    b = torch.full_like(a, fill)
    n = a.shape[axis]
    if n > 1:
        src, dst = (slice(1, n), slice(0, n - 1)) if step > 0 else (slice(0, n - 1), slice(1, n))
        ix = [slice(None)] * 3
        ix[axis] = src
        jx = [slice(None)] * 3
        jx[axis] = dst
        b[tuple(jx)] = a[tuple(ix)]
    return b


def _front(phi, h):
    """Distances of the cells next to the zero set (sum_a d_a^-2)^(-1/2), d_a
    the smaller linear crossing distance along axis a; inf elsewhere."""
    pos = phi >= 0
    inv = torch.zeros_like(phi)
    zero = torch.zeros_like(pos)
    near = torch.zeros_like(pos)
    for axis, ha in ((2, h[0]), (1, h[1]), (0, h[2])):
        d = torch.full_like(phi, INF)
        for step in (1, -1):
            q = _shift(phi, axis, step, float("nan"))
            cross = torch.isfinite(q) & ((q >= 0) != pos)
            d = torch.where(cross, torch.minimum(d, phi / (phi - q) * ha), d)
        hit = torch.isfinite(d)
        near |= hit
        zero |= hit & (d == 0)
        inv = torch.where(hit & (d != 0), inv + 1.0 / (d * d), inv)
    T = torch.where(zero, torch.zeros_like(phi), 1.0 / torch.sqrt(inv))
    return torch.where(near, T, torch.full_like(phi, INF)), near


def _order(v, w):
    """Sort three values, their weights with them."""
    for a, b in ((0, 1), (1, 2), (0, 1)):
        sw = v[b] < v[a]
        v[a], v[b] = torch.where(sw, v[b], v[a]), torch.where(sw, v[a], v[b])
        if w is not None:
            w[a], w[b] = torch.where(sw, w[b], w[a]), torch.where(sw, w[a], w[b])
    return v, w


def _godunov(T, q, wts, width):
    """The root of sum_a w_a max(t - T_a, 0)^2 = q, T_a the smaller neighbour
    of axis a (none above width)."""
    known = T if width == INF else torch.where(T <= width, T, torch.full_like(T, INF))
    v = [torch.minimum(_shift(known, a, 1, INF), _shift(known, a, -1, INF)) for a in (2, 1, 0)]
    equal = wts == (1.0, 1.0, 1.0)
    w = None if equal else [torch.full_like(T, x) for x in wts]
    v, w = _order(v, w)
    w0, w1, w2 = (1.0, 1.0, 1.0) if equal else w
    m = v[0]
    ok = torch.isfinite(m)
    m = torch.where(ok, m, torch.zeros_like(m))
    u = (q / w0) ** 0.5 * torch.ones_like(m)
    d1 = v[1] - m
    two = d1 < u
    d1 = torch.where(two, d1, torch.zeros_like(d1))
    k = w0 + w1
    s = torch.sqrt(torch.clamp(k * q - w0 * w1 * d1 * d1, min=0.0))
    u = torch.where(two, (w1 * d1 + s) / k, u)
    d2 = v[2] - m
    three = two & (d2 < u)
    d2 = torch.where(three, d2, torch.zeros_like(d2))
    k = w0 + w1 + w2
    e = d1 - d2
    s = torch.sqrt(torch.clamp(k * q - w0 * w1 * d1 * d1 - w0 * w2 * d2 * d2 - w1 * w2 * e * e, min=0.0))
    u = torch.where(three, (w1 * d1 + w2 * d2 + s) / k, u)
    return torch.where(ok, m + u, torch.full_like(m, INF))


def _march(T, fix, q, wts, width=INF):
    """Iterate the upwind update from above until nothing changes."""
    for it in range(1, 64 * sum(T.shape)):
        new = torch.where(fix, T, torch.minimum(T, _godunov(T, q, wts, width)))
        if it % 16 == 0 and torch.equal(new, T):
            break
        T = new
    return T


def _tags(T, fix, width):
    t = torch.where(torch.isfinite(T), torch.where(T <= width, 2, 1), 0)
    return torch.where(fix, 3, t).to(torch.uint8)


def _exact_level_set(phi, h, width=INF):
    phi = phi.double()
    hx, hy, hz = _three(h)
    T, fix = _front(phi, (hx, hy, hz))
    T = _march(T, fix, hx * hx, (1.0, (hx / hy) ** 2, (hx / hz) ** 2), width)
    tags = _tags(T, fix, width)
    return torch.where((phi < 0) & torch.isfinite(T), -T, T), tags


def _exact_gradient(T, fix, s, h, lam0):
    """dL/ds: mu = lambda / D from the upwind sets, by repeated substitution
    down the arrivals until nothing changes."""
    vals, sides = [], []
    for axis in (2, 1, 0):
        lo, hi = _shift(T, axis, -1, INF), _shift(T, axis, 1, INF)
        vals.append(torch.minimum(lo, hi))
        sides.append(hi < lo)
    t = torch.stack(vals)
    used = t < T
    used &= ~fix
    D = torch.where(used, T - t, torch.zeros_like(t)).sum(0)
    inv = torch.where(D > 0, 1.0 / D, torch.zeros_like(D))
    # pull weights: cell p receives (T_q - T_p) mu_q from the cells q that use it
    parts = []
    for a, axis in enumerate((2, 1, 0)):
        drop = torch.where(used[a], T - t[a], torch.zeros_like(D)) * inv
        parts.append((axis, torch.where(sides[a], drop, torch.zeros_like(D)),
                      torch.where(sides[a], torch.zeros_like(D), drop)))
    lam = lam0.clone()
    for it in range(1, 64 * sum(T.shape)):
        new = lam0.clone()
        for axis, up, down in parts:
            new += _shift(lam * up, axis, -1, 0.0) + _shift(lam * down, axis, 1, 0.0)
        if it % 16 == 0 and torch.equal(new, lam):
            break
        lam = new
    return torch.where(fix, torch.zeros_like(lam), lam * inv * s * h * h)


def exact(case, seed):
    c = case
    # the second-order result depends on the order of acceptance: it has no
    # value of its own
    if _cells(c) > EXACT_CELLS or c.get("order", 1) == 2 or (c["kind"] == "batch" and c["grids"] > 24):
        return None
    x = _inputs(c, seed)
    if c["kind"] in ("noalloc", "reinit"):
        h = _three(x["h"])[0]
        T, G = _exact_level_set(x["phi"], x["h"], c["width"] * h if c.get("width") else INF)
        return {"T": T, "tags": G}
    if c["kind"] == "batch":
        Ts, Gs = [], []
        for phi, h, s in zip(x["phis"], x["hs"], x["shapes"]):
            pad = (-math.prod(s)) % 256
            T, G = _exact_level_set(phi, h)
            Ts.append(torch.cat([T.reshape(-1), T.new_zeros(pad)]))
            Gs.append(torch.cat([G.reshape(-1), G.new_zeros(pad)]))
        return {"T": torch.cat(Ts), "tags": torch.cat(Gs)}
    h = x["h"]
    T = torch.full(_shape(c), INF, dtype=torch.float64, device=DEV)
    fix = torch.zeros(_shape(c), dtype=torch.bool, device=DEV)
    i, j, k = (torch.as_tensor(x["src"][:, a], device=DEV) for a in range(3))
    T[k, j, i] = 0.0
    fix[k, j, i] = True
    if c["kind"] == "sources":
        q = h * h if x["speed"] is None else (h / x["speed"].double()) ** 2
        T = _march(T, fix, q, (1.0, 1.0, 1.0))
        return {"T": T, "tags": _tags(T, fix, INF)}
    s = x["slowness"].double()
    T = _march(T, fix, (h * s) ** 2, (1.0, 1.0, 1.0))
    rec = tuple(torch.as_tensor(x["rec"][:, a], device=DEV) for a in (2, 1, 0))
    lam0 = torch.zeros_like(T)
    lam0[rec] = 1.0
    return {"T": T, "loss": T[rec].sum(), "grad": _exact_gradient(T, fix, s, h, lam0)}
