"""D8 global phases at the edges of the skeleton's tiles (32x32 with water,
64x64 for areas alone) and on both sides of the polling kernel's limit."""
import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import _lib, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SKEL, WALK = _lib.FR_GLOBAL_SKELETON, _lib.FR_GLOBAL_WALKERS


@pytest.mark.parametrize("shape", [(96, 96), (95, 97), (97, 127), (128, 129), (129, 160), (257, 191)])
@pytest.mark.parametrize("gflags", [0, SKEL, WALK])
def test_filled_dem_tile_edges(shape, gflags):
    """Rivers through a filled DEM: water (one rounding of the leading word and
    the two-float sum, the bar of every D8 water test) and exact areas."""
    from paper_2606_12800_gb300 import api
    z = oracle.fill(inputs.fractal_dem(*shape, beta=2.1, tilt=0.0, seed=21))
    rain = inputs.rain_field(*shape, 5)
    d, w, _, order = oracle.route_d8(z, 30.0, rain, oracle.EDGE_ROUTE)
    _, a = oracle.accumulate_d8(d, order, None)
    R = api.routing_d8(torch.from_numpy(d).cuda(), gflags)
    rt = torch.from_numpy(rain).cuda()
    for want_w in (True, False):
        for want_area in (True, False):
            if not (want_w or want_area):
                continue
            o = api.accumulate(R, rt, want_w=want_w, want_lo=want_w, want_area=want_area)
            assert api.get_status() == 0
            if want_w:
                got = o["w"].double().cpu().numpy()
                assert np.max(np.abs(got - w) / np.maximum(w, 1e-30)) <= 1e-6
            if want_area:
                np.testing.assert_array_equal(o["area"].cpu().numpy().astype(np.uint64), a)


@pytest.mark.parametrize("shape", [(420, 700), (1100, 1300)])
def test_plane_walked(shape):
    """A plane without the skeleton: few enough global cells to poll, and too
    many.  Every row is one river."""
    from paper_2606_12800_gb300 import api
    ny, nx = shape
    z = torch.from_numpy(np.ascontiguousarray(inputs.planar_dem(ny, nx, 0.01, 30.0))).cuda()
    d = api.receivers_d8(z, 30.0, _lib.FR_EDGE_ROUTE)
    o = api.accumulate(api.routing_d8(d, WALK), None, want_w=True, want_area=True, device=d.device)
    assert api.get_status() == 0
    ref = np.broadcast_to(np.arange(1, nx + 1), (ny, nx))
    np.testing.assert_array_equal(o["area"].cpu().numpy(), ref)
    np.testing.assert_array_equal(o["w"].cpu().numpy(), ref.astype(np.float32))


def test_d8_polling_has_no_wait_limit():
    """The wait limit is for the MFD and adjoint phases: a D8 accumulation whose
    global cells are polled finishes under a limit of zero, as the walkers do."""
    from paper_2606_12800_gb300 import api
    z = inputs.fractal_dem(300, 700, beta=2.1, tilt=0.0, seed=22)
    d, _, _, order = oracle.route_d8(z, 30.0)
    _, a = oracle.accumulate_d8(d, order, None)
    R = api.routing_d8(torch.from_numpy(d).cuda(), WALK)
    prev = api.set_wait_limit(0)
    try:
        o = api.accumulate(R, None, want_w=False, want_area=True, device="cuda")
        assert api.get_status() == 0
    finally:
        api.set_wait_limit(prev)
    np.testing.assert_array_equal(o["area"].cpu().numpy().astype(np.uint64), a)


@pytest.mark.parametrize("shape", [(300, 517), (4100, 4163)])
def test_skeleton_looks_ahead(shape):
    """The skeleton forced on rough terrain, where most tiles hold no global cell
    and a block goes through several flags' worth of tiles (rows that share
    words of the bitmap): the walkers' areas, and their water to two roundings."""
    from paper_2606_12800_gb300 import api
    z = torch.from_numpy(inputs.fractal_dem(*shape, beta=2.1, tilt=0.0, seed=23)).cuda()
    d = api.receivers_d8(z, 30.0, 0)
    out = {}
    for f in (SKEL, WALK):
        for want_w in (True, False):
            out[f, want_w] = api.accumulate(api.routing_d8(d, f), None, want_w=want_w, want_area=True,
                                            device=d.device)
            assert api.get_status() == 0
    ref = out[WALK, False]["area"]
    for k, o in out.items():
        assert torch.equal(o["area"], ref)
        if k[1]:
            torch.testing.assert_close(o["w"], ref.float(), rtol=2 * 2.0 ** -23, atol=0)
