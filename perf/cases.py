"""The work that a user has this library do, as measurable cases.

A case is one pass through the public entry points of
``paper_2402_18311_gb300.place`` on a seeded synthetic design: iterations of a
placement, a perturbation, an evaluation at a selection point, gradients or a
field.  ``prepare`` makes what a user's program holds before the call (the
design's handle, the positions on the GPU), ``run`` makes the call, ``work``
says what it cannot do without, and ``exact`` computes the same values in
64 bits with plain torch and numpy.

Designs have the shape of ``synth``'s: unit-height cells of width 1..4, fixed
macros, IO pads, and the net degrees 60% 2, 20% 3, 15% 4-10, 5% 11-50 and
0.1% up to several thousand pins.
"""
import math

import numpy as np
import torch

from paper_2402_18311_gb300 import place, synth

# Optimiser constants of place_default_params(), which every case keeps.
GAMMA_BASE, LAMBDA_ETA, ALPHA0, HPWL_REF = 4.0, 1e-3, 0.05, 0.3
MU_BASE, MU_LO, MU_HI = 1.1, 0.95, 1.05


def _case(kind, cells, nx, ny, **more):
    case = {"kind": kind, "cells": cells, "nx": nx, "ny": ny, "copies": 1, "iters": 0,
            "phase": "spread", "fixed_macros": 10, "movable_macros": 0, "weights": False,
            "stretch": False, "fillers": False}
    case.update(more)
    return case


# Iterations of one pass, counted from a reset.  Small differences of rounding
# grow with every iteration, and the faster the smaller gamma is: a spread
# cloud multiplies them by three to ten, the dense start hardly.
_ITERS = {"start": 10, "middle": 2, "spread": 2}


def listed():
    named = {
        # the smallest design (1k cells on 64 x 64 bins): launches and latency
        "place_1k": _case("place", 1000, 64, 64, iters=10, phase="start", fixed_macros=0),
        # a mixed-size 20k-cell design with the optional modes in use: fillers,
        # density stretching, net weights, movable macros with their own weight
        "place_20k_options": _case("place", 20011, 128, 128, iters=2, phase="middle",
                                   movable_macros=20, weights=True, stretch=True, fillers=True),
        # an ordinary design (ISPD 2005 sized) from its centred start
        "place_210k": _case("place", 210000, 512, 512, iters=10, phase="start"),
        # the headline size at the dense start of a placement ...
        "place_2m_start": _case("place", 2100000, 1024, 1024, iters=10, phase="start",
                                fixed_macros=60),
        # ... and once its cells have spread, where most iterations are spent
        "place_2m_spread": _case("place", 2100000, 1024, 1024, iters=2, fixed_macros=60),
        # 32 restarts of one design as one batched handle, each from its own start
        "restarts_32x210k": _case("place", 210000, 512, 512, copies=32, iters=2),
        # the Shuffle (all) perturbation of a batched handle's copies
        "shuffle_8x210k": _case("shuffle", 210000, 512, 512, copies=8),
        # the WireMask perturbation of a mixed-size design's 32 macros
        "wiremask_210k": _case("wiremask", 210000, 512, 512, movable_macros=32),
        # the exact HPWL and overflow at a selection point of a large design
        "evaluate_2m": _case("evaluate", 2100000, 1024, 1024, fixed_macros=60),
        # both gradients for a caller with its own optimiser; a non-square grid
        "gradients_495k": _case("gradients", 494716, 512, 1024),
        # the potential and the field on a ragged grid
        "field_ragged": _case("field", 30011, 368, 176),
        # the overflow for a caller that may not allocate; a ragged grid
        "overflow_noalloc": _case("noalloc", 500009, 768, 656),
    }
    return [dict(case, name=name) for name, case in named.items()]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, cells):
    """The power of two nearest sqrt(cells) within 64..1024 per side (one side
    sometimes doubled or halved), or, a quarter of the time, ragged sides."""
    side = min(max(2 ** round(math.log2(math.sqrt(cells))), 64), 1024)
    if rng.random() < 0.25:
        ragged = [min(max(16 * round(side * rng.uniform(0.6, 1.1) / 16), 48), 1024) for _ in "xy"]
        return ragged[0], ragged[1]
    other = min(max(int(side * rng.choice([0.5, 1, 1, 1, 2])), 64), 1024)
    return (side, other) if rng.random() < 0.5 else (other, side)


def draw(rng):
    kind = rng.choice(["place", "place", "place", "place", "shuffle", "wiremask", "evaluate",
                       "gradients", "field", "noalloc"])
    cells = _log_uniform(rng, 1000, 1500000) | 1
    nx, ny = _grid(rng, cells)
    more = {"phase": rng.choice(["start", "middle", "spread", "spread"]),
            "fixed_macros": rng.choice([0, 4, 10, 30])}
    if kind in ("place", "shuffle"):
        most = max(1, 1500000 // cells)
        more["copies"] = min(most, rng.choice([1, 1, 2, 5, 16, 32]), 1 << 23 >> (nx * ny).bit_length())
        more["copies"] = max(1, more["copies"])
    if kind == "place":
        more["iters"] = rng.randint(1, _ITERS[more["phase"]])
        more["weights"] = rng.random() < 0.25
        more["stretch"] = rng.random() < 0.2
        more["fillers"] = rng.random() < 0.2
    if kind in ("place", "wiremask", "gradients") and rng.random() < (1.0 if kind == "wiremask" else 0.3):
        more["movable_macros"] = rng.randint(4, 32)
    return _case(kind, cells, nx, ny, **more)


# ---- inputs -----------------------------------------------------------------

def _die(case):
    """Bins of a dyadic size, square within an eighth, such that the movable
    cells (mean area 2.5) and the macros leave a third of the die free."""
    area = case["cells"] * 2.5 + case["movable_macros"] * 40.0 ** 2 * 0.25
    free = 0.8 if case["fixed_macros"] else 1.0
    size = math.sqrt(area / 0.62 / free / (case["nx"] * case["ny"]))
    step = max(0.125, round(size * 8) / 8)
    return (0.0, 0.0, step * case["nx"], step * case["ny"])


def _positions(case, rng, w, h, die):
    """Lower-left corners of the movable cells: a placement's centred start,
    its middle (a cloud over a tenth of the die) or spread over the die."""
    n = w.shape[0]
    out = []
    for size, extent in ((w, die[2]), (h, die[3])):
        if case["phase"] == "spread":
            c = rng.random(n) * extent
        else:
            sigma = 1e-3 if case["phase"] == "start" else 0.1
            c = 0.5 * extent + sigma * extent * rng.standard_normal(n)
        out.append(np.clip(c - 0.5 * size, 0.0, extent - size).astype(np.float32))
    return out


def _design(case, seed):
    """The case's netlist, made from the seed."""
    rng = np.random.default_rng([seed, case["cells"], case["nx"]])
    n, die = case["cells"], _die(case)
    w = rng.integers(1, 5, n).astype(np.float32)
    h = np.ones(n, np.float32)
    movable = np.zeros(n, np.uint8)
    if case["movable_macros"]:
        at = rng.choice(n, case["movable_macros"], replace=False)
        top = max(4, int(min(64, 0.08 * min(die[2], die[3]))))
        w[at] = rng.integers(top // 4, top + 1, at.size)
        h[at] = rng.integers(top // 4, top + 1, at.size)
        movable[at] = 1
    # fixed macros on the cells of a lattice (a fifth of the die), 16 pads
    m = case["fixed_macros"]
    lattice = max(1, math.ceil(math.sqrt(m)))
    sx, sy = die[2] / lattice, die[3] / lattice
    spot = rng.permutation(lattice * lattice)[:m]
    scale = math.sqrt(0.2 * lattice * lattice / max(m, 1))
    fw = np.floor(np.maximum(1.0, sx * scale * rng.uniform(0.8, 1.0, m)))
    fh = np.floor(np.maximum(1.0, sy * scale * rng.uniform(0.8, 1.0, m)))
    fx = np.floor((spot % lattice) * sx + rng.random(m) * np.maximum(sx - fw, 0.0))
    fy = np.floor((spot // lattice) * sy + rng.random(m) * np.maximum(sy - fh, 0.0))
    k = (np.arange(4) + 0.5) / 4
    px = np.concatenate([k * die[2], k * die[2], np.zeros(4), np.full(4, die[2] - 1)])
    py = np.concatenate([np.zeros(4), np.full(4, die[3] - 1), k * die[3], k * die[3]])
    w = np.concatenate([w, fw, np.ones(16)]).astype(np.float32)
    h = np.concatenate([h, fh, np.ones(16)]).astype(np.float32)
    x, y = _positions(case, rng, w[:n], h[:n], die)
    x = np.concatenate([x, fx, px]).astype(np.float32)
    y = np.concatenate([y, fy, py]).astype(np.float32)
    is_macro = np.concatenate([movable, np.ones(m, np.uint8), np.zeros(16, np.uint8)])

    nets = int(n * 1.05)
    u = rng.random(nets)
    deg = np.where(u < 0.60, 2, 3)
    mid, long = (u >= 0.80) & (u < 0.95), u >= 0.95
    deg[mid] = rng.integers(4, 11, int(mid.sum()))
    deg[long] = rng.integers(11, 51, int(long.sum()))
    big = rng.choice(nets, round(1e-3 * nets), replace=False)
    deg[big] = np.exp(rng.uniform(math.log(51), math.log(max(52, min(5000, n // 4))), big.size))
    ptr = np.zeros(nets + 1, np.int64)
    np.cumsum(deg, out=ptr[1:])
    cell = rng.integers(0, w.size, int(ptr[-1]), dtype=np.int32)
    dx = rng.random(cell.size, dtype=np.float32) * w[cell]
    dy = rng.random(cell.size, dtype=np.float32) * h[cell]
    d = synth.Design(name="case", n_movable=n, w=w, h=h, x=x, y=y, net_ptr=ptr.astype(np.int32),
                     pin_cell=cell, pin_dx=dx, pin_dy=dy, die=die, nx=case["nx"], ny=case["ny"],
                     target_density=0.9, is_macro=is_macro)
    if case["weights"]:
        d.net_w = rng.choice(np.array([0.5, 1.0, 1.0, 2.0, 3.25], np.float32), nets)
    return d


def _starts(case, seed, d):
    """[copies, n_cells] start positions: the design's for the first copy, a
    fresh draw for each of the others where the copies are placed."""
    copies = case["copies"] if case["kind"] == "place" else 1
    x, y = np.tile(d.x, (copies, 1)), np.tile(d.y, (copies, 1))
    n = case["cells"]
    for c in range(1, copies):
        rng = np.random.default_rng([seed, c, 77])
        x[c, :n], y[c, :n] = _positions(case, rng, d.w[:n], d.h[:n], d.die)
    return x, y


def _frac_bits(d):
    """The fixed-point resolution: the largest F <= 24 that keeps coordinates
    below 2^30 and the total area below 2^62 units."""
    extent, area = max(d.die), float((d.w.astype(np.float64) * d.h).sum())
    return next(f for f in range(24, -1, -1)
                if extent * 2.0 ** f < 2.0 ** 30 and area * 4.0 ** f < 2.0 ** 62)


def _fillers(case, seed, d):
    """Size, count and start of the filler cells (none without the option)."""
    if not case["fillers"]:
        return 0.0, 0.0, np.zeros((2, 0), np.float32)
    s, n = 2.0 ** _frac_bits(d), case["cells"]
    plain = d.is_macro[:n] == 0
    size = [np.rint(np.rint(v[:n][plain].astype(np.float64) * s).mean()) / s for v in (d.w, d.h)]
    ox = np.minimum(d.x[n:] + d.w[n:].astype(np.float64), d.die[2]) - np.maximum(d.x[n:], 0.0)
    oy = np.minimum(d.y[n:] + d.h[n:].astype(np.float64), d.die[3]) - np.maximum(d.y[n:], 0.0)
    fixed = float((np.maximum(ox, 0.0) * np.maximum(oy, 0.0)).sum())
    t = float(np.float32(d.target_density))
    free = t * (d.die[2] * d.die[3] - fixed) - float((d.w[:n].astype(np.float64) * d.h[:n]).sum())
    count = int(max(0.0, free) // (size[0] * size[1]))
    rng = np.random.default_rng([seed, 5])
    at = [rng.random(count) * (d.die[2 + a] - size[a]) for a in (0, 1)]
    return size[0], size[1], np.asarray(at, np.float32)


class _State:
    """A design's handle and device buffers, released with the object."""

    def __init__(self):
        self.handle = None

    def __del__(self):
        if self.handle is not None:
            place.place_destroy(self.handle)


def prepare(case, seed):
    s = _State()
    s.case = case
    d = _design(case, seed)
    x, y = _starts(case, seed, d)
    s.x, s.y = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    s.seed = 1000 * seed + 17
    n, bins = case["cells"], case["nx"] * case["ny"]
    if case["kind"] == "noalloc":
        s.w, s.h = torch.from_numpy(d.w).cuda(), torch.from_numpy(d.h).cuda()
        s.xm, s.ym = s.x[0, :n].contiguous(), s.y[0, :n].contiguous()
        s.die, s.bins = d.die, (d.nx, d.ny, d.target_density)
        s.frac_bits = _frac_bits(d)
        s.fixed = _fixed_map(d).reshape(-1)
        s.overflow = torch.zeros(1, dtype=torch.float64, device="cuda")
        s.map = torch.zeros(bins, dtype=torch.int64, device="cuda")
        return s
    params = place.place_default_params(
        n_copies=case["copies"], tau_stop=-1.0, max_iters=1 << 30, stretch=int(case["stretch"]),
        fillers=int(case["fillers"]), macro_precond=2.0 if case["movable_macros"] else 1.0)
    s.handle = place.place_create(d, params)
    if case["kind"] in ("place", "shuffle", "wiremask"):
        s.ox = torch.empty((case["copies"], d.n_cells), device="cuda")
        s.oy = torch.empty_like(s.ox)
        s.fill = torch.from_numpy(_fillers(case, seed, d)[2]).cuda()
    elif case["kind"] == "gradients":
        s.grads = torch.empty((4, n), device="cuda")
    elif case["kind"] == "field":
        s.field = torch.empty((3, bins), device="cuda")
    if case["kind"] not in ("place", "shuffle", "wiremask"):
        place.place_set_positions(s.handle, -1, s.x[0], s.y[0])
    return s


def run(s):
    case, h, K = s.case, s.handle, s.case["copies"]
    kind = case["kind"]
    if kind == "noalloc":
        place.place_overflow_noalloc(s.xm, s.ym, s.w, s.h, case["cells"], s.die, s.bins,
                                     s.frac_bits, s.fixed, s.overflow, s.map)
        return {"overflow": s.overflow, "map": s.map}
    if kind == "evaluate":
        hpwl, overflow = np.empty(K), np.empty(K)
        place.place_eval_hpwl_overflow(h, hpwl, overflow)
        return {"hpwl": hpwl, "overflow": overflow}
    if kind == "gradients":
        wl = place.place_eval_wirelength(h, 0, _gamma(case), s.grads[0], s.grads[1])
        place.place_eval_density_grad(h, 0, s.grads[2], s.grads[3])
        return {"wl": wl, "grads": s.grads}
    if kind == "field":
        place.place_eval_field(h, 0, s.field[0], s.field[1], s.field[2])
        return {"field": s.field}
    if s.fill.shape[1]:
        place.place_set_fillers(h, -1, s.fill[0], s.fill[1])
    if s.x.shape[0] == 1:
        place.place_set_positions(h, -1, s.x[0], s.y[0])
    else:
        for c in range(K):
            place.place_set_positions(h, c, s.x[c], s.y[c])
    if kind == "shuffle":
        place.place_perturb(h, place.PLACE_SHUFFLE_ALL, 0.5, s.seed, -1)
    elif kind == "wiremask":
        place.place_perturb(h, place.PLACE_WIREMASK, 0.0, 0, -1)
    else:
        place.place_step(h, case["iters"])
    for c in range(K):
        place.place_get_positions(h, c, s.ox[c], s.oy[c])
    out = {"x": s.ox, "y": s.oy}
    if kind == "place":
        state = place.place_get_state(h, 0)
        out.update(iterations=state.iter, overflow=state.overflow, gamma=state.gamma,
                   density_weight=state.lambda_, hpwl=state.hpwl_wa)
    return out


def _pins(case):
    """Expected pins of the case's netlist."""
    top = max(52, min(5000, case["cells"] // 4))
    big = (top - 51) / math.log(top / 51)
    return int(case["cells"] * 1.05 * (0.6 * 2 + 0.2 * 3 + 0.15 * 7 + 0.05 * 30.5 + 1e-3 * big))


def work(case):
    n, G, P, K = case["cells"], case["nx"] * case["ny"], _pins(case), case["copies"]
    nets, kind = int(n * 1.05), case["kind"]
    netlist = 12 * P + 4 * nets
    solve = 7.5 * G * math.log2(G)  # one forward and two inverse 2-D cosine transforms
    if kind == "place":
        # per iteration: the netlist, the fixed map and the cells' sizes once;
        # per copy positions, both points and both gradients in and out
        one = netlist + 8 * G + 16 * n + K * (40 * n + 8 * G)
        return {"bytes": case["iters"] * one + K * 16 * n,
                "flops": case["iters"] * K * (80.0 * P + 60.0 * n + solve)}
    if kind in ("shuffle", "wiremask"):
        return {"bytes": K * 24 * n + 8 * n, "flops": 0}
    if kind == "evaluate":
        return {"bytes": netlist + 16 * n + 8 * G, "flops": 6.0 * P + 20.0 * n}
    if kind == "gradients":
        return {"bytes": netlist + 32 * n + 8 * G, "flops": 80.0 * P + 60.0 * n + solve}
    if kind == "field":
        return {"bytes": 16 * n + 20 * G, "flops": 20.0 * n + 1.4 * solve}
    return {"bytes": 16 * n + 16 * G, "flops": 20.0 * n}


# ---- the same values in 64 bits ---------------------------------------------

def _gamma(case):
    d = _die(case)
    return 2.0 * math.sqrt(d[2] / case["nx"] * d[3] / case["ny"])


def _quantised(d, *v):
    s = 2.0 ** _frac_bits(d)
    return [torch.round(a * s) for a in v]


def _each_bin(X, Y, W, H, d):
    """For the rectangles (in units of 2^-F): (rows, flat bin, overlap) of
    every bin that some of them cover, one bin offset at a time."""
    s = 2.0 ** _frac_bits(d)
    bw, bh = d.die[2] / d.nx * s, d.die[3] / d.ny * s
    ix, iy = torch.floor(X / bw), torch.floor(Y / bh)
    sx = (torch.ceil((X + W) / bw) - ix).clamp(min=0)
    sy = (torch.ceil((Y + H) / bh) - iy).clamp(min=0)
    rows = torch.arange(X.numel(), device=X.device)
    for kx in range(int(sx.max()) if X.numel() else 0):
        some = rows[sx > kx]
        for ky in range(int(sy[some].max())):
            r = some[sy[some] > ky]
            bx, by = ix[r] + kx, iy[r] + ky
            ox = torch.minimum(X[r] + W[r], (bx + 1) * bw) - torch.maximum(X[r], bx * bw)
            oy = torch.minimum(Y[r] + H[r], (by + 1) * bh) - torch.maximum(Y[r], by * bh)
            ok = (bx >= 0) & (bx < d.nx) & (by >= 0) & (by < d.ny) & (ox > 0) & (oy > 0)
            r, flat = r[ok], (bx * d.ny + by)[ok].long()
            yield r, flat, (ox * oy)[ok]


def _overlap_map(x, y, w, h, d, scale=None):
    """Overlap areas per bin (units of 2^-2F) of quantised rectangles."""
    X, Y, W, H = _quantised(d, x, y, w, h)
    M = torch.zeros(d.nx * d.ny, dtype=torch.float64, device=x.device)
    for r, flat, ov in _each_bin(X, Y, W, H, d):
        M.index_add_(0, flat, ov if scale is None else ov * scale[r])
    return M.reshape(d.nx, d.ny)


def _fixed_map(d):
    """The fixed cells' overlap areas per bin (whole units of 2^-2F)."""
    s, n, sides = 2.0 ** _frac_bits(d), d.n_movable, []
    for at, size, extent, count in ((d.x, d.w, d.die[2], d.nx), (d.y, d.h, d.die[3], d.ny)):
        edge = torch.arange(count + 1, dtype=torch.float64, device="cuda") * (extent / count * s)
        lo = torch.from_numpy(np.rint(at[n:].astype(np.float64) * s)).cuda()[:, None]
        hi = lo + torch.from_numpy(np.rint(size[n:].astype(np.float64) * s)).cuda()[:, None]
        sides.append((torch.minimum(hi, edge[1:]) - torch.maximum(lo, edge[:-1])).clamp(min=0).long())
    M = torch.zeros((d.nx, d.ny), dtype=torch.int64, device="cuda")
    for ox, oy in zip(*sides):
        M += ox[:, None] * oy[None, :]
    return M


def _stretched(d, w, h):
    """Shifts, sizes and density scale of cells narrower than sqrt(2) bins."""
    s = 2.0 ** _frac_bits(d)
    out = []
    for size, b in ((w, d.die[2] / d.nx), (h, d.die[3] / d.ny)):
        W = torch.round(size * s)
        W2 = torch.clamp(W, min=float(np.rint(math.sqrt(2.0) * b * s)))
        out += [torch.floor((W2 - W) / 2) / s, W2 / s]
    return out[0], out[2], out[1], out[3], (w * h) / (out[1] * out[3])


def _axis(n, size, device):
    k = torch.arange(n, dtype=torch.float64, device=device)
    arg = math.pi * k[:, None] * (k[None, :] + 0.5) / n
    c = torch.full((n,), 2.0 / n, dtype=torch.float64, device=device)
    c[0] = 1.0 / n
    return torch.cos(arg), torch.sin(arg), math.pi * k / (n * size), c


def _poisson(rho, d):
    Cx, Sx, wu, cu = _axis(d.nx, d.die[2] / d.nx, rho.device)
    Cy, Sy, wv, cv = _axis(d.ny, d.die[3] / d.ny, rho.device)
    a = (Cx @ rho @ Cy.T) * cu[:, None] * cv[None, :]
    den = wu[:, None] ** 2 + wv[None, :] ** 2
    den[0, 0] = 1.0
    b = a / den
    b[0, 0] = 0.0
    return (Cx.T @ b @ Cy, Sx.T @ (b * wu[:, None]) @ Cy, Cx.T @ (b * wv[None, :]) @ Sy)


def _wirelength(net, x, y, g, n):
    """WA wirelength, its gradient per movable cell, and the pins' HPWL."""
    total, hpwl, grads = 0.0, 0.0, []
    for v, off in ((x, net["dx"]), (y, net["dy"])):
        p = v[net["cell"]] + off
        big = torch.full((net["count"],), -1e300, dtype=torch.float64, device=p.device)
        mx = big.scatter_reduce(0, net["of"], p, "amax")
        mn = -big.scatter_reduce(0, net["of"], -p, "amax")
        grad = torch.zeros_like(p)
        value = mx - mn
        hpwl = hpwl + ((mx - mn) * net["w"]).sum()
        for sign, m in ((1.0, mx), (-1.0, mn)):
            q = p - m[net["of"]]
            e = torch.exp(sign * q / g)
            zero = torch.zeros(net["count"], dtype=torch.float64, device=p.device)
            s = zero.index_add(0, net["of"], e)
            r = zero.index_add(0, net["of"], q * e) / s
            value = value + sign * r
            grad += sign * e / s[net["of"]] * (1.0 + sign * (q - r[net["of"]]) / g)
        total = total + (value * net["w"]).sum()
        grad *= net["w"][net["of"]]
        zero = torch.zeros(x.numel(), dtype=torch.float64, device=p.device)
        grads.append(zero.index_add(0, net["cell"], grad)[:n])
    return total, grads[0], grads[1], hpwl


def _net(d):
    dev = "cuda"
    deg = torch.from_numpy(np.diff(d.net_ptr)).to(dev)
    net_w = getattr(d, "net_w", None)
    return {"cell": torch.from_numpy(d.pin_cell).to(dev).long(), "count": d.n_nets,
            "dx": torch.from_numpy(d.pin_dx).to(dev).double(),
            "dy": torch.from_numpy(d.pin_dy).to(dev).double(),
            "of": torch.repeat_interleave(torch.arange(d.n_nets, device=dev), deg),
            "w": torch.ones(d.n_nets, dtype=torch.float64, device=dev) if net_w is None
            else torch.from_numpy(net_w).to(dev).double()}


class _Exact:
    """The electrostatic placer of one copy in 64 bits."""

    def __init__(self, case, seed, d):
        up = lambda v: torch.from_numpy(np.asarray(v)).cuda().double()  # noqa: E731
        n = self.n = case["cells"]
        self.case, self.d, self.net = case, d, _net(d)
        fw, fh, self.fill = _fillers(case, seed, d)
        nf = self.fill.shape[1]
        self.w = torch.cat([up(d.w[:n]), torch.full((nf,), fw, dtype=torch.float64, device="cuda")])
        self.h = torch.cat([up(d.h[:n]), torch.full((nf,), fh, dtype=torch.float64, device="cuda")])
        self.fx, self.fy = up(d.x[n:]), up(d.y[n:])
        self.F = _fixed_map(d).double()
        s = 2.0 ** _frac_bits(d)
        self.bin = d.die[2] / d.nx * s * (d.die[3] / d.ny * s)
        self.t = float(np.float32(d.target_density))
        self.w_bin = math.sqrt(d.die[2] / d.nx * d.die[3] / d.ny)
        weight = 2.0 if case["movable_macros"] else 1.0
        macro = up(d.is_macro[:n])
        self.area = self.w * self.h
        self.area[:n] *= 1.0 + (weight - 1.0) * macro
        pins = torch.bincount(self.net["cell"], minlength=d.n_cells)[:n].double()
        self.pins = torch.cat([pins, torch.zeros(nf, dtype=torch.float64, device="cuda")])
        self.stretch = _stretched(d, self.w, self.h) if case["stretch"] else None

    def density(self, x, y):
        """Overflow and the field (psi, ex, ey) at movable corners x, y."""
        n, d = self.n, self.d
        M = _overlap_map(x[:n], y[:n], self.w[:n], self.h[:n], d)
        area = (self.w[:n] * self.h[:n]).sum() * 4.0 ** _frac_bits(d)
        tau = float((M - self.t * (self.bin - self.F)).clamp(min=0.0).sum() / area)
        if self.stretch:
            sx, sy, w, h, r = self.stretch
            M = _overlap_map(x - sx, y - sy, w, h, d, r)
        elif x.numel() > n:
            M = M + _overlap_map(x[n:], y[n:], self.w[n:], self.h[n:], d)
        return tau, _poisson((M + self.t * self.F) / self.bin, d)

    def gather(self, x, y, ex, ey):
        d = self.d
        w, h, r = self.w, self.h, None
        if self.stretch:
            sx, sy, w, h, r = self.stretch
            x, y = x - sx, y - sy
        unit = 4.0 ** -_frac_bits(d)
        out = torch.zeros((2, x.numel()), dtype=torch.float64, device=x.device)
        for rows, flat, ov in _each_bin(*_quantised(d, x, y, w, h), d):
            ov = ov * unit if r is None else ov * unit * r[rows]
            out[0].index_add_(0, rows, -ov * ex.reshape(-1)[flat])
            out[1].index_add_(0, rows, -ov * ey.reshape(-1)[flat])
        return out[0], out[1]

    def wirelength(self, x, y, gamma):
        n = self.n
        total, gx, gy, hpwl = _wirelength(self.net, torch.cat([x[:n], self.fx]),
                                          torch.cat([y[:n], self.fy]), gamma, n)
        none = torch.zeros(x.numel() - n, dtype=torch.float64, device=x.device)
        return float(total), torch.cat([gx, none]), torch.cat([gy, none]), float(hpwl)

    def place(self, x, y, iters):
        d = self.d
        x = torch.cat([x, torch.from_numpy(self.fill[0]).cuda().double()])
        y = torch.cat([y, torch.from_numpy(self.fill[1]).cuda().double()])
        clamp = lambda v, size, top: torch.minimum(v, top - size).clamp(min=0.0)  # noqa: E731
        fix = lambda p: torch.stack([clamp(p[0], self.w, d.die[2]), clamp(p[1], self.h, d.die[3])])  # noqa: E731
        gamma_of = lambda tau: GAMMA_BASE * self.w_bin * 10.0 ** (20.0 / 9.0 * tau - 11.0 / 9.0)  # noqa: E731
        v = fix(torch.stack([x, y]))
        u, a, g_old, v_old, hp_old = v, 1.0, None, None, 0.0
        gamma, lam, tau, hpwl = gamma_of(self.density(*v)[0]), 0.0, 0.0, 0.0
        dref = HPWL_REF * d.n_nets * self.w_bin
        for k in range(iters):
            tau, (_, ex, ey) = self.density(*v)
            gd = torch.stack(self.gather(*v, ex, ey))
            _, gwx, gwy, hpwl = self.wirelength(*v, gamma)
            gw = torch.stack([gwx, gwy])
            if k == 0:
                lam = LAMBDA_ETA * float(gw.abs().sum() / gd.abs().sum())
            g = (gw + lam * gd) / (self.pins + lam * self.area).clamp(min=1.0)
            if k == 0:
                alpha = ALPHA0 * self.w_bin / math.sqrt(float(g.square().sum()) / (2.0 * x.numel()))
            else:
                alpha = float((v - v_old).norm() / (g - g_old).norm())
                lam *= min(max(MU_BASE ** (1.0 - (hpwl - hp_old) / dref), MU_LO), MU_HI)
            a_next = (1.0 + math.sqrt(4.0 * a * a + 1.0)) / 2.0
            u_next = fix(v - alpha * g)
            v_next = fix(u_next + (a - 1.0) / a_next * (u_next - u))
            u, v_old, v, g_old, hp_old, a = u_next, v, v_next, g, hpwl, a_next
            gamma = gamma_of(tau)
        return v[0, :self.n], v[1, :self.n], tau, gamma, lam, hpwl


def _splitmix64(seed, count):
    """The first outputs of SplitMix64 started from the seed."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (np.arange(count, dtype=np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def exact(case, seed):
    if case["kind"] == "wiremask":
        return None  # an argmin over every corner of the grid for each macro in turn
    d = _design(case, seed)
    n, K = case["cells"], case["copies"]
    x, y = _starts(case, seed, d)
    if case["kind"] == "shuffle":
        # half of the cells, those of the lowest keys, take each other's centres
        X, Y = np.tile(x, (K, 1)).astype(np.float64), np.tile(y, (K, 1)).astype(np.float64)
        for c in range(K):
            picked = np.argsort(_splitmix64(1000 * seed + 17 + c, n), kind="stable")[:int(n / 2 + 0.5)]
            donor = np.sort(picked)
            for P, size, top, now in ((X, d.w, d.die[2], x[0]), (Y, d.h, d.die[3], y[0])):
                centre = now[donor].astype(np.float64) + 0.5 * size[donor]
                P[c, picked] = np.clip(centre - 0.5 * size[picked], 0.0, top - size[picked].astype(np.float64))
        return {"x": X, "y": Y}
    e = _Exact(case, seed, d)
    up = lambda v: torch.from_numpy(v).cuda().double()  # noqa: E731
    if case["kind"] == "place":
        X, Y, state = x.astype(np.float64), y.astype(np.float64), None
        for c in range(K):
            px, py, *scalars = e.place(up(x[c, :n]), up(y[c, :n]), case["iters"])
            X[c, :n], Y[c, :n] = px.cpu().numpy(), py.cpu().numpy()
            state = state or scalars
        return {"x": X, "y": Y, "iterations": None, "overflow": state[0], "gamma": state[1],
                "density_weight": state[2], "hpwl": state[3]}
    px, py = up(x[0, :n]), up(y[0, :n])
    if case["kind"] == "gradients":
        wl, gx, gy, _ = e.wirelength(px, py, _gamma(case))
        _, (_, ex, ey) = e.density(px, py)
        return {"wl": wl, "grads": torch.stack([gx, gy, *e.gather(px, py, ex, ey)])}
    tau, field = e.density(px, py)
    if case["kind"] == "field":
        return {"field": torch.stack([f.reshape(-1) for f in field])}
    if case["kind"] == "evaluate":
        return {"hpwl": np.array([e.wirelength(px, py, 1.0)[3]]), "overflow": np.array([tau])}
    return {"overflow": torch.tensor([tau], dtype=torch.float64), "map": None}
