"""The skeleton with water on both sides of the rule that gives long, narrow grids
64x64 tiles and others 32x32: planes, where every row is one river of known water,
and filled terrain against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import _lib, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 3000), (63, 2048), (65, 2047), (320, 2048), (321, 2049), (1536, 2048),
                                   (1537, 2050), (70, 4099)])
@pytest.mark.parametrize("across", [False, True])
def test_planes(shape, across):
    from paper_2606_12800_gb300 import api
    ny, nx = shape
    z = np.ascontiguousarray(inputs.planar_dem(ny, nx, 0.01, 30.0))
    ref = np.broadcast_to(np.arange(1, nx + 1), (ny, nx))
    if across:  # the same rivers down the columns
        z, ref = np.ascontiguousarray(z.T), ref.T
    zt = torch.from_numpy(z).cuda()
    for want_area in (True, False):
        for flags in (0, _lib.FR_GLOBAL_SKELETON):
            o = api.route_d8(zt, 30.0, None, _lib.FR_EDGE_ROUTE | flags, want_lo=True, want_area=want_area)
            assert api.get_status() == 0
            np.testing.assert_array_equal(o["w"].cpu().numpy(), ref.astype(np.float32))
            assert not o["w_lo"].any()
            if want_area:
                np.testing.assert_array_equal(o["area"].cpu().numpy(), ref)


@pytest.mark.parametrize("shape", [(100, 2100), (2500, 64), (319, 2048), (330, 2051)])
def test_filled_terrain(shape):
    """Water to one rounding of its leading word, as in every water test."""
    from paper_2606_12800_gb300 import api
    z = oracle.fill(inputs.fractal_dem(*shape, beta=2.1, tilt=0.0, seed=31))
    rain = inputs.rain_field(*shape, 8)
    d, w, _, order = oracle.route_d8(z, 30.0, rain)
    _, a = oracle.accumulate_d8(d, order, None)
    zt, rt = torch.from_numpy(z).cuda(), torch.from_numpy(rain).cuda()
    for want_area in (True, False):
        o = api.route_d8(zt, 30.0, rt, _lib.FR_GLOBAL_SKELETON, want_area=want_area)
        assert api.get_status() == 0
        got = o["w"].double().cpu().numpy()
        assert np.max(np.abs(got - w) / np.maximum(w, 1e-30)) <= 1e-6
        if want_area:
            np.testing.assert_array_equal(o["area"].cpu().numpy().astype(np.uint64), a)
