"""MFD and adjoint tile solve at the edges of its tiles (80x64 inner cells, an
8-cell halo, 64 levels listed at once) and both global phases behind it.

A cell's value is a fixed sequence of fp32 operations on its dependencies'
values (the compensated dot product in code order), whichever kernel computes
it, so the results are compared bit for bit with the same operations done by
numpy, level by level, on the library's own fractions (which the parity tests
check against the oracle)."""
import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

OFF = ((1, 0), (0, -1), (-1, 0), (0, 1), (1, -1), (-1, -1), (-1, 1), (1, 1))


def _rough(ny, nx):
    return inputs.fractal_dem(ny, nx, beta=2.2, tilt=0.0, seed=17)


def _ramp(ny, nx):
    """Falls along x and, ten times slower, along y: chains as long as the grid
    is wide, every cell with several receivers."""
    y, x = np.mgrid[0:ny, 0:nx].astype(np.float64)
    return (3.0 * (nx - x) + 0.3 * (ny - y)).astype(np.float32)


def _dot8(hi, lo, f, vh, vl):
    s, c = hi, lo
    for k in range(8):
        p = f[k] * vh[k]
        pe = (f[k].astype(np.float64) * vh[k] - p).astype(np.float32)
        pe = (f[k].astype(np.float64) * vl[k] + pe).astype(np.float32)
        t = s + p
        b = t - s
        e = (s - (t - b)) + (p - b)
        s, c = t, c + (e + pe)
    h = s + c
    return h, c - (h - s)


def _solve(mask, frac, init, adjoint):
    """Two-float values of the forward (donors) or transposed (receivers)
    system on the fractions frac[cell, code] of the receiver mask."""
    ny, nx = mask.shape
    n = ny * nx
    step = [dy * nx + dx for dx, dy in OFF]
    m, f = mask.reshape(-1), frac.reshape(n, 8)
    recv = [((m >> k) & 1).astype(bool) for k in range(8)]
    ids = np.arange(n)
    # dep[k]: cells that depend on their neighbour k, with that edge's fraction
    dep, wt = [], []
    for k in range(8):
        if adjoint:
            dep.append(recv[k])
            wt.append(f[:, k])
        else:
            d, w = np.zeros(n, bool), np.zeros(n, np.float32)
            src = ids[recv[k ^ 2]]  # gives in direction k ^ 2: its receiver's neighbour k
            d[src + step[k ^ 2]] = True
            w[src + step[k ^ 2]] = f[src, k ^ 2]
            dep.append(d)
            wt.append(w)
    wait = np.sum(dep, axis=0).astype(np.int32)
    hi, lo = init.reshape(-1).astype(np.float32).copy(), np.zeros(n, np.float32)
    level, zero = ids[wait == 0], np.float32(0)
    while level.size:
        fs, vh, vl = [], [], []
        for k in range(8):
            on = dep[k][level]
            j = np.where(on, level + step[k], 0)
            fs.append(np.where(on, wt[k][level], zero))
            vh.append(np.where(on, hi[j], zero))
            vl.append(np.where(on, lo[j], zero))
        hi[level], lo[level] = _dot8(hi[level], lo[level], fs, vh, vl)
        nxt = []
        for k in range(8):  # cells whose neighbour k ^ 2 ... this level's cells were waited for
            t = level + step[k]
            t = t[(t >= 0) & (t < n)]
            t = t[dep[k ^ 2][t] & np.isin(t + step[k ^ 2], level, assume_unique=True)]
            wait[t] -= 1
            nxt.append(t[wait[t] == 0])
        level = np.unique(np.concatenate(nxt))
    return hi.reshape(ny, nx), lo.reshape(ny, nx)


def _check(ny, nx, make, flags, with_rain):
    from paper_2606_12800_gb300 import api
    z = torch.from_numpy(make(ny, nx)).cuda()
    rain = inputs.rain_field(ny, nx, 3) if with_rain else np.ones((ny, nx), np.float32)
    out = api.route_mfd(z, 30.0, 1.1, torch.from_numpy(rain).cuda() if with_rain else None, flags,
                        want_lo=True, want_mask=True)
    assert api.get_status() == 0
    mask, frac = api.receivers_mfd(z, 30.0, 1.1, flags, frac=True)
    mask, frac = mask.cpu().numpy(), frac.cpu().numpy()
    np.testing.assert_array_equal(out["mask"].cpu().numpy(), mask)
    hi, lo = _solve(mask, frac, rain, adjoint=False)
    np.testing.assert_array_equal(out["w"].cpu().numpy(), hi)
    np.testing.assert_array_equal(out["w_lo"].cpu().numpy(), lo)
    # adjoint of a given gradient, through the same tiles the other way round
    gbar = inputs.rain_field(ny, nx, 9)
    R = api.routing_mfd(out["mask"], z, 30.0, 1.1, flags)
    g, _ = api.adjoint(R, out["w"], out["w_lo"], dLdw=torch.from_numpy(gbar).cuda())
    assert api.get_status() == 0
    np.testing.assert_array_equal(g.cpu().numpy(), _solve(mask, frac, gbar, adjoint=True)[0])


@pytest.mark.parametrize("shape", [(15, 63), (16, 64), (17, 65), (18, 66), (33, 129), (1, 70), (70, 1), (2, 2),
                                   (31, 64), (32, 65), (34, 63)])
@pytest.mark.parametrize("flags", [0, oracle.EDGE_ROUTE])
@pytest.mark.parametrize("p", [0.5, 1.0, 1.1, 4.5])
def test_mfd_weights_tile_edges(shape, flags, p):
    """Masks (with and without fractions) bit for bit, fractions against FP64 at
    the edges of the tiles.  A fraction's error: the powers' 1e-7 (p 4.5:
    the slope's rounding times p) twice, and its own rounding."""
    from paper_2606_12800_gb300 import api
    z = inputs.fractal_dem(*shape, beta=2.0, tilt=0.0, seed=6)
    zt = torch.from_numpy(z).cuda()
    m_ref, f_ref = oracle.receivers_mfd(z, 30.0, p, flags)
    m, f = api.receivers_mfd(zt, 30.0, p, flags, frac=True)
    np.testing.assert_array_equal(m.cpu().numpy(), m_ref)
    np.testing.assert_array_equal(api.receivers_mfd(zt, 30.0, p, flags).cpu().numpy(), m_ref)
    f = f.cpu().numpy().astype(np.float64).reshape(-1, 8)
    f_ref = f_ref.reshape(-1, 8)
    assert np.all(np.abs(f - f_ref) <= 1e-6 * f_ref)


@pytest.mark.parametrize("shape", [(15, 63), (16, 64), (17, 65), (33, 129), (3, 70), (70, 3), (2, 2)])
@pytest.mark.parametrize("flags", [0, oracle.EDGE_ROUTE])
def test_mfd_grad_z_tile_edges(shape, flags):
    """dL/dz against its formula in FP64 on the library's fractions and adjoint,
    at the edges of the 64x16 tiles.  Per edge: the adjoint's leading words are
    rounded (2^-24 each), six fp32 operations follow."""
    from paper_2606_12800_gb300 import api
    ny, nx = shape
    z = inputs.fractal_dem(ny, nx, beta=2.0, tilt=0.0, seed=8)
    zt = torch.from_numpy(z).cuda()
    out = api.route_mfd(zt, 30.0, 1.1, None, flags, want_lo=True, want_mask=True)
    gbar = torch.from_numpy(inputs.rain_field(ny, nx, 4)).cuda()
    R = api.routing_mfd(out["mask"], zt, 30.0, 1.1, flags)
    g, dz = api.adjoint(R, out["w"], out["w_lo"], dLdw=gbar, want_dz=True)
    _, f = api.receivers_mfd(zt, 30.0, 1.1, flags, frac=True)
    f = f.cpu().numpy().astype(np.float64)
    g, w = g.double().cpu().numpy(), out["w"].double().cpu().numpy()
    z = z.astype(np.float64)
    ref, tol = np.zeros((ny, nx)), np.full((ny, nx), 1e-30)
    for y in range(ny):
        for x in range(nx):
            on = [k for k in range(8) if f[y, x, k] > 0]
            G = sum(f[y, x, k] * g[y + OFF[k][1], x + OFF[k][0]] for k in on)
            for k in on:
                yn, xn = y + OFF[k][1], x + OFF[k][0]
                c = 1.1 * w[y, x] * f[y, x, k] / (z[y, x] - z[yn, xn])
                a, e = c * (g[yn, xn] - G), c * (g[yn, xn] + G) * 8 * 2.0 ** -24
                ref[y, x] += a
                ref[yn, xn] -= a
                tol[y, x] += e
                tol[yn, xn] += e
    assert np.all(np.abs(dz.double().cpu().numpy() - ref) <= tol)


@pytest.mark.parametrize("shape", [(64, 80), (63, 79), (65, 81), (128, 160), (129, 161), (3, 250), (250, 3), (1, 96)])
@pytest.mark.parametrize("make", [_rough, _ramp])
@pytest.mark.parametrize("flags", [0, oracle.EDGE_ROUTE])
def test_mfd_tile_edges(shape, make, flags):
    _check(*shape, make, flags, with_rain=flags != 0)


@pytest.mark.parametrize("shape", [(420, 700), (1100, 1300)])
def test_mfd_global_phases(shape):
    """Almost every cell global: few enough to poll, and too many."""
    _check(*shape, _ramp, oracle.EDGE_ROUTE, with_rain=True)
