"""The workloads this library is measured on: calls of the public Python API on
synthetic terrain, from one small tile to a 32768 x 32768 grid.

A case names a kind of call, its grid and its options; `prepare` draws the
terrain from the seed, `run` makes the call and `exact` computes the same
outputs in 64 bits with plain torch.
"""
import math

import torch

from paper_2606_12800_gb300 import api
from paper_2606_12800_gb300._lib import (FR_D4, FR_D8_LOWEST, FR_DINF, FR_EDGE_ROUTE,
                                         FR_SINK_SUMS_IN_WORKSPACE)

DX = 30.0  # grid spacing of every case (metres)
# neighbour offsets in code order E N W S NE NW SW SE
OFF = ((1, 0), (0, -1), (-1, 0), (0, 1), (1, -1), (-1, -1), (-1, 1), (1, 1))


def listed():
    return [
        # one small survey tile: a call is launches and latency
        {"name": "d8_tile", "kind": "d8", "ny": 160, "nx": 192, "beta": 2.0, "tilt": 0.01, "rain": True,
         "rule": "steepest", "edge_route": False},
        # a ragged clip of a DEM (odd width: no row is aligned)
        {"name": "d8_ragged", "kind": "d8", "ny": 1537, "nx": 2603, "beta": 2.1, "tilt": 0.0, "rain": True,
         "rule": "steepest", "edge_route": True},
        # an ordinary sheet with a rain field: codes, water, areas and the mass balance
        {"name": "d8_step", "kind": "d8_step", "ny": 4096, "nx": 4096, "beta": 2.0, "tilt": 0.01},
        # the largest grid: codes, unit-rain areas, mass balance
        {"name": "d8_area_large", "kind": "d8_area", "ny": 32768, "nx": 32768, "beta": 2.0, "tilt": 0.005},
        # depression filling before routing
        {"name": "fill", "kind": "fill", "ny": 4096, "nx": 4096, "beta": 2.0, "tilt": 0.01},
        # a depression-filled sheet (rivers cross the whole grid) with a rain field
        {"name": "filled_water", "kind": "filled", "ny": 4096, "nx": 4096, "beta": 2.0, "tilt": 0.01,
         "surface": "filled", "water": True},
        # drainage areas of a larger filled sheet
        {"name": "filled_area", "kind": "filled", "ny": 8192, "nx": 8192, "beta": 2.0, "tilt": 0.005,
         "surface": "filled", "water": False},
        # slope-split routing: a large sheet under unit rain
        {"name": "mfd_large", "kind": "mfd", "ny": 8192, "nx": 8192, "beta": 2.2, "tilt": 0.0, "p": 1.1,
         "split": "slope", "rain": False, "edge_route": False},
        # slope-split routing: a ragged clip with a rain field
        {"name": "mfd_ragged", "kind": "mfd", "ny": 777, "nx": 1333, "beta": 2.0, "tilt": 0.01, "p": 1.1,
         "split": "slope", "rain": True, "edge_route": True},
        # one training step through the autograd function: water, then both gradients
        {"name": "mfd_train", "kind": "train", "ny": 2048, "nx": 2048, "beta": 2.2, "tilt": 0.0, "p": 1.1},
        # the adjoint alone, of a loss over the sinks, on a large sheet
        {"name": "mfd_adjoint", "kind": "adjoint", "ny": 8192, "nx": 8192, "beta": 2.2, "tilt": 0.0, "p": 1.1},
        # many independent tiles of uneven size in one call
        {"name": "batch", "kind": "batch", "tiles": 32, "side_min": 64, "side_max": 2048, "beta": 2.1,
         "tilt": 0.01, "routing": "d8"},
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi):
    """Sides of a grid of about side^2 cells, aspect up to 2, odd or even."""
    side, a = _logu(rng, lo, hi), math.sqrt(_logu(rng, 0.5, 2.0))
    ny, nx = max(3, round(side * a)), max(3, round(side / a))
    step = rng.choice((1, 1, 4, 32))
    return ny, max(step, 3, nx // step * step)


def draw(rng):
    kind = rng.choice(("d8", "d8", "d8_step", "d8_area", "fill", "filled", "filled", "mfd", "mfd", "train",
                       "adjoint", "batch"))
    beta, tilt = round(rng.uniform(1.8, 2.3), 3), rng.choice((0.0, 0.005, 0.01))
    if kind == "batch":
        return {"kind": kind, "tiles": rng.randint(2, 32), "side_min": rng.randint(16, 100),
                "side_max": rng.randint(200, 2048), "beta": beta, "tilt": tilt, "routing": rng.choice(("d8", "mfd"))}
    lo, hi = {"d8": (48, 6000), "d8_step": (200, 6000), "d8_area": (1000, 24000), "fill": (64, 3000),
              "filled": (64, 4096), "mfd": (48, 6000), "train": (64, 3000), "adjoint": (200, 6000)}[kind]
    ny, nx = _grid(rng, lo, hi)
    c = {"kind": kind, "ny": ny, "nx": nx, "beta": beta, "tilt": tilt}
    if kind == "d8":
        c.update(rain=rng.random() < 0.7, rule=rng.choice(("steepest", "steepest", "lowest", "d4")),
                 edge_route=rng.random() < 0.5)
    elif kind == "filled":
        c.update(surface=rng.choice(("filled", "filled", "plane")), water=rng.random() < 0.5)
    elif kind == "mfd":
        c.update(p=rng.choice((1.0, 1.1, 1.1, 2.0, 4.5)), split=rng.choice(("slope", "slope", "slope", "dinf")),
                 rain=rng.random() < 0.5, edge_route=rng.random() < 0.5)
    elif kind in ("train", "adjoint"):
        c["p"] = rng.choice((1.0, 1.1, 1.1, 2.0))
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _terrain(ny, nx, beta, tilt, g):
    """Fractal surface of spectral slope beta, 1000 m of relief, a tilt down
    towards +x and a jitter of 0.1 mm."""
    ky = torch.fft.fftfreq(ny, device="cuda") * ny
    kx = torch.fft.fftfreq(nx, device="cuda") * nx
    amp = torch.sqrt(ky[:, None] ** 2 + kx[None, :] ** 2)
    amp[0, 0] = 1.0
    amp.pow_(-beta / 2.0)
    amp[0, 0] = 0.0
    m = torch.complex(torch.randn(ny, nx, generator=g, device="cuda"), torch.randn(ny, nx, generator=g, device="cuda"))
    m.mul_(amp)
    del amp
    z = torch.fft.ifft2(m).real.contiguous()
    del m
    lo, hi = z.min(), z.max()
    z.sub_(lo).mul_(1000.0 / (hi - lo).clamp_min(1e-30))
    z.add_((tilt * DX) * (nx - 1 - torch.arange(nx, device="cuda", dtype=torch.float32))[None, :])
    z.add_(torch.rand(ny, nx, generator=g, device="cuda"), alpha=1e-4)
    return z


def _d8_flags(c):
    return ((FR_EDGE_ROUTE if c.get("edge_route") else 0)
            | {"steepest": 0, "lowest": FR_D8_LOWEST, "d4": FR_D4}[c.get("rule", "steepest")])


def _mfd_flags(c):
    return (FR_EDGE_ROUTE if c.get("edge_route") else 0) | (FR_DINF if c.get("split") == "dinf" else 0)


def _side(c, i):
    """Side of tile i of a batch: log-uniform, spread evenly over the tiles."""
    return round(c["side_min"] * (c["side_max"] / c["side_min"]) ** (((i + 0.5) * 0.6180339887) % 1.0))


def prepare(case, seed):
    g, k = _gen(seed), case["kind"]
    s = {"case": case}
    if k == "batch":
        # clips of one surface: tiles of a region, sides log-uniform
        side = max(case["side_max"], 2048)
        z = _terrain(side, side, case["beta"], case["tilt"], g)
        cpu = torch.Generator().manual_seed(int(seed))
        s["dems"], s["rains"] = [], []
        for i in range(case["tiles"]):
            n = _side(case, i)
            oy, ox = (int(v) for v in torch.randint(0, side - n + 1, (2,), generator=cpu))
            s["dems"].append(z[oy:oy + n, ox:ox + n].contiguous())
            s["rains"].append(torch.rand(n, n, generator=g, device="cuda"))
        return s
    ny, nx = case["ny"], case["nx"]
    if case.get("surface") == "plane":
        x = torch.arange(nx, device="cuda", dtype=torch.float32)
        slope = 0.1 + 0.2 * torch.rand(1, generator=g, device="cuda")
        z = (slope * (nx - 1 - x))[None, :].expand(ny, nx).contiguous()
    else:
        z = _terrain(ny, nx, case["beta"], case["tilt"], g)
        if case.get("surface") == "filled":
            z, _ = api.fill(z)
    s["z"] = z
    if k in ("d8_step", "train") or case.get("rain") or case.get("water"):
        s["rain"] = torch.rand(ny, nx, generator=g, device="cuda")
    if k == "train":
        s["grad"] = torch.rand(ny, nx, generator=g, device="cuda")
        s["z"].requires_grad_(True)
        s["rain"].requires_grad_(True)
    if k == "adjoint":  # what the forward call left: mask and two-float water
        out = api.route_mfd(z, DX, case["p"], want_lo=True, want_mask=True)
        s["w"], s["w_lo"], s["mask"] = out["w"], out["w_lo"], out["mask"]
    return s


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "d8":
        o = api.route_d8(s["z"], DX, s.get("rain"), _d8_flags(c))
        return [o["w"], o["area"]]
    if k == "d8_step":
        d = api.receivers_d8(s["z"], DX)
        R = api.routing_d8(d)
        o = api.accumulate(R, s["rain"], want_w=True, want_area=True)
        mb = api.mass_balance(R, s["rain"], o["w"], None, o["area"], device=d.device)
        return [d, o["w"], o["area"], mb]
    if k == "d8_area":
        d = api.receivers_d8(s["z"], DX)
        R = api.routing_d8(d, FR_SINK_SUMS_IN_WORKSPACE)
        o = api.accumulate(R, None, want_w=False, want_area=True, device=d.device)
        mb = api.mass_balance(R, area=o["area"], device=d.device)
        return [d, o["area"], mb]
    if k == "fill":
        return [api.fill(s["z"])[0]]
    if k == "filled":
        o = api.route_d8(s["z"], DX, s.get("rain"), 0, want_w=c["water"], want_area=True)
        return [o["w"], o["area"]] if c["water"] else [o["area"]]
    if k == "mfd":
        return [api.route_mfd(s["z"], DX, c["p"], s.get("rain"), _mfd_flags(c))["w"]]
    if k == "train":
        w = api.RouteMFD.apply(s["z"], s["rain"], DX, c["p"])
        gz, gr = torch.autograd.grad(w, (s["z"], s["rain"]), s["grad"])
        return [w.detach(), gz, gr]
    if k == "adjoint":
        R = api.routing_mfd(s["mask"], s["z"], DX, c["p"])
        gr, gz = api.adjoint(R, s["w"], s["w_lo"], want_dz=True)
        return [gr, gz]
    outs = api.route_batch(s["dems"], s["rains"], kind=c["routing"], dx=DX)
    return [[o["route"], o["w"]] for o in outs]


def work(case):
    """Each input read once, each output written once; the operations are the
    comparisons and slopes of the receiver rule and the additions (D8: about 34
    per cell; slope split: eight powers and products, about 200; adjoint with
    the gradients, about 150)."""
    k = case["kind"]
    if k == "batch":
        n = sum(_side(case, i) ** 2 for i in range(case["tiles"]))
        return {"bytes": n * 13, "flops": n * (34 if case["routing"] == "d8" else 200)}
    n = case["ny"] * case["nx"]
    rain = 4 if case.get("rain") or case.get("water") else 0
    b, f = {"d8": (16 + rain, 34), "d8_step": (21, 40), "d8_area": (13, 34), "fill": (8, 9),
            "filled": (12 + (8 if case.get("water") else 0), 34), "mfd": (8 + rain, 200),
            # z, rain, gradient in; water and two gradients out
            "train": (24, 350),
            # z, mask and two-float water in; two gradients out
            "adjoint": (21, 150)}[k]
    return {"bytes": n * b, "flops": n * f}


# ------------------------------------------------------- 64-bit references
def _nbr(a, k, fill):
    """a at neighbour k of every cell, `fill` off the grid."""
    dx, dy = OFF[k]
    ny, nx = a.shape
    out = torch.full_like(a, fill)
    out[max(0, -dy):ny - max(0, dy), max(0, -dx):nx - max(0, dx)] = \
        a[max(0, dy):ny - max(0, -dy), max(0, dx):nx - max(0, -dx)]
    return out


def _edges_off(t, edge_route, value):
    if not edge_route:
        t[0, :] = t[-1, :] = value
        t[:, 0] = t[:, -1] = value
    return t


def _codes(z, rule, edge_route):
    """D8 codes by the rule in fp32 (255: none)."""
    best, code = torch.full_like(z, -1.0), torch.full_like(z, 255, dtype=torch.uint8)
    for k in range(4 if rule == "d4" else 8):
        d = z - _nbr(z, k, float("inf"))
        c = torch.tensor(1.0 / (DX if k < 4 else math.sqrt(2.0) * DX), dtype=torch.float32, device=z.device)
        s = d if rule == "lowest" else d * c
        take = (d > 0) & (s > best)
        best, code = torch.where(take, s, best), torch.where(take, torch.full_like(code, k), code)
    return _edges_off(code, edge_route, 255)


def _steps(nx, device):
    return torch.tensor([dy * nx + dx for dx, dy in OFF], device=device)


def _d8_water(code, rain):
    """Every cell's water in 64 bits: after round r each cell holds the water
    of all cells less than 2^r steps above it."""
    n = code.numel()
    k = code.reshape(-1).long()
    at = torch.arange(n, device=code.device)
    to = torch.where(k < 8, at + _steps(code.shape[1], code.device)[k.clamp_max(7)], n)
    to = torch.cat([to, to.new_full((1,), n)])  # n: past the end of a path
    w = torch.cat([rain.double().reshape(-1), rain.new_zeros(1, dtype=torch.float64)])
    while bool((to[:n] < n).any()):
        live = torch.nonzero(to[:n] < n).reshape(-1)
        w = w.index_add(0, to[live], w[live])
        to = to[to]
    return w[:n].reshape(code.shape)


def _fractions(z, c):
    """Fractions of every cell towards its eight neighbours in 64 bits."""
    ny, nx = z.shape
    edge = bool(c.get("edge_route"))
    if c.get("split") != "dinf":
        u = []
        for k in range(8):
            zn = _nbr(z, k, float("inf"))
            d = (z.double() - zn.double()) / (DX if k < 4 else math.sqrt(2.0) * DX)
            u.append(_edges_off(torch.where(zn < z, d.clamp_min(0) ** c["p"], torch.zeros_like(d)), edge, 0.0))
        s = sum(u)
        return [torch.where(s > 0, x / torch.where(s > 0, s, torch.ones_like(s)), torch.zeros_like(x)) for x in u]
    # D-infinity: the facet by fp32 slopes, the split of the angle in 64 bits
    c1 = torch.tensor(1.0 / DX, dtype=torch.float32, device=z.device)
    cd = torch.tensor(1.0 / (math.sqrt(2.0) * DX), dtype=torch.float32, device=z.device)
    best = torch.full_like(z, -1.0)
    facet, kind = torch.full_like(z, -1, dtype=torch.int8), torch.zeros_like(z, dtype=torch.int8)
    for i in range(8):
        kc, kd = ((i + 1) >> 1) & 3, 4 + (i >> 1)
        zc, zd = _nbr(z, kc, float("nan")), _nbr(z, kd, float("nan"))
        s1, s2, sd = (z - zc) * c1, (zc - zd) * c1, (z - zd) * cd
        inside = ~(torch.isnan(zc) | torch.isnan(zd))
        flat, steep = s2 <= 0, s2 >= s1
        kd_ = torch.where(flat, 0, torch.where(steep, 2, 1)).to(torch.int8)
        none = torch.full_like(z, -1.0)
        key = torch.where(flat, torch.where(s1 > 0, s1 * s1, none),
                          torch.where(steep, torch.where(sd > 0, sd * sd, none), s1 * s1 + s2 * s2))
        take = inside & (key > best)
        best, kind = torch.where(take, key, best), torch.where(take, kd_, kind)
        facet = torch.where(take, torch.full_like(facet, i), facet)
    _edges_off(facet, edge, -1)
    f = [torch.zeros_like(z, dtype=torch.float64) for _ in range(8)]
    for i in range(8):
        kc, kd = ((i + 1) >> 1) & 3, 4 + (i >> 1)
        zc, zd = _nbr(z, kc, 0.0).double(), _nbr(z, kd, 0.0).double()
        s1, s2 = z.double() - zc, zc - zd
        part = torch.atan2(s2, s1) * (4.0 / math.pi)
        part = torch.where(kind == 0, 0.0, torch.where(kind == 2, 1.0, part))
        f[kd] = torch.where(facet == i, part, f[kd])
        f[kc] = torch.where(facet == i, 1.0 - part, f[kc])
    return f


def _levels(f, nx):
    """The cells in levels: each cell after all its donors."""
    n, step = f[0].numel(), _steps(nx, f[0].device).tolist()
    fl = [x.reshape(-1) for x in f]
    wait = torch.zeros(n, dtype=torch.int32, device=f[0].device)
    for k in range(8):
        src = torch.nonzero(fl[k] > 0).reshape(-1)
        wait.index_add_(0, src + step[k], torch.ones_like(src, dtype=torch.int32))
    level, got = torch.nonzero(wait == 0).reshape(-1), []
    while level.numel():
        got.append(level)
        to = []
        for k in range(8):
            t = level[fl[k][level] > 0] + step[k]
            wait.index_add_(0, t, torch.full_like(t, -1, dtype=torch.int32))
            to.append(t)
        to = torch.cat(to)
        level = torch.unique(to[wait[to] == 0])
    return got


def _mfd_water(f, levels, rain):
    nx = rain.shape[1]
    fl, step, w = [x.reshape(-1) for x in f], _steps(nx, rain.device).tolist(), rain.double().reshape(-1).clone()
    for level in levels:
        for k in range(8):
            a = fl[k][level]
            src, a = level[a > 0], a[a > 0]
            w.index_add_(0, src + step[k], w[src] * a)
    return w.reshape(rain.shape)


def _mfd_grads(z, f, levels, w, gbar, p):
    """g = gbar + sum of f g over the receivers, and the gradient with
    respect to the elevations through the fractions."""
    ny, nx = z.shape
    fl, step, g = [x.reshape(-1) for x in f], _steps(nx, z.device).tolist(), gbar.reshape(-1).clone()
    n = g.numel()
    for level in reversed(levels):
        v = g[level]
        for k in range(8):
            a = fl[k][level]
            v = v + torch.where(a > 0, a * g[(level + step[k]).clamp(0, n - 1)], torch.zeros_like(a))
        g[level] = v
    g = g.reshape(ny, nx)
    mean = sum(f[k] * _nbr(g, k, 0.0) for k in range(8))
    dz = torch.zeros_like(g)
    for k in range(8):
        drop = z.double() - _nbr(z, k, float("inf")).double()
        on = f[k] > 0
        a = torch.where(on, p * w * (_nbr(g, k, 0.0) - mean) * f[k] / torch.where(on, drop, torch.ones_like(drop)),
                        torch.zeros_like(g))
        dz += a
        dz -= _nbr(a, k ^ 2, 0.0)
    return g, dz


def _filled(z):
    """max(z, the next fp32 value above the lowest neighbour) to its fixed
    point, on order-preserving integers."""
    b = z.contiguous().view(torch.int32)
    key = torch.where(b >= 0, b, -(b & 0x7FFFFFFF))  # -0.0 and 0.0 both 0
    top = torch.full_like(key, 0x7F800000)
    F = top.clone()
    F[0, :], F[-1, :], F[:, 0], F[:, -1] = key[0, :], key[-1, :], key[:, 0], key[:, -1]
    if min(z.shape) > 2:
        while True:
            before = F.clone()
            for _ in range(64):
                m = torch.minimum(torch.minimum(F[:, :-2], F[:, 1:-1]), F[:, 2:])
                low = torch.minimum(torch.minimum(m[:-2], m[1:-1]), m[2:])
                F[1:-1, 1:-1] = torch.minimum(F[1:-1, 1:-1], torch.maximum(key[1:-1, 1:-1], low + 1))
            if torch.equal(F, before):
                break
    out = torch.where(F >= 0, F, (-F) | -0x80000000).view(torch.float32)
    return torch.where(F == key, z, out).double()


def exact(case, seed):
    k = case["kind"]
    if k != "batch" and case["ny"] * case["nx"] > 9000 * 9000 and k != "d8_area":
        return None
    if k == "d8_area":  # codes and areas are whole numbers
        n = float(case["ny"] * case["nx"])
        return [None, None, torch.tensor([0.0, n, n], dtype=torch.float64)]
    s = prepare(case, seed)
    if k == "batch":
        out = []
        for z, r in zip(s["dems"], s["rains"]):
            if case["routing"] == "d8":
                out.append([None, _d8_water(_codes(z, "steepest", False), r)])
            else:
                f = _fractions(z, {"p": 1.1})
                out.append([None, _mfd_water(f, _levels(f, z.shape[1]), r)])
        return out
    z = s["z"].detach()
    rain = s["rain"].detach() if "rain" in s else torch.ones_like(z)
    if k in ("d8", "d8_step", "filled"):
        code = _codes(z, case.get("rule", "steepest"), bool(case.get("edge_route")))
        if k == "filled" and not case["water"]:
            return None  # areas are whole numbers
        w = _d8_water(code, rain)
        if k != "d8_step":
            return [w, None]
        mb = torch.stack([w[code == 255].sum(), rain.double().sum(),
                          torch.tensor(float(z.numel()), dtype=torch.float64, device=z.device)])
        return [None, w, None, mb]
    if k == "fill":
        return [_filled(z)]
    f = _fractions(z, case)
    levels = _levels(f, z.shape[1])
    w = _mfd_water(f, levels, rain)
    if k == "mfd":
        return [w]
    if k == "train":
        g, dz = _mfd_grads(z, f, levels, w, s["grad"].double(), case["p"])
        return [w, dz, g]
    gbar = torch.where(sum(f) > 0, torch.zeros_like(w), 2.0 * w)
    g, dz = _mfd_grads(z, f, levels, w, gbar, case["p"])
    return [g, dz]
