"""D8 tile solve: aligned and unaligned tiles, tile edges (96x48 with water,
128x64 for areas alone, 64x32 on small grids and in batches) and routing bytes that are no codes."""
import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(48, 96), (64, 128), (47, 95), (65, 129), (145, 290), (144, 296), (200, 400), (1000, 1200)])
@pytest.mark.parametrize("shift", [0, 1])
def test_invalid_bytes_have_no_receiver(shape, shift):
    """Any byte above 7 is a cell without a receiver, on every loading path
    (shift: a base address off its alignment).  Areas are exact; water has one
    rounding of the leading word over the two-float sum."""
    from paper_2606_12800_gb300 import api
    ny, nx = shape
    z = inputs.fractal_dem(ny, nx, beta=2.0, tilt=0.01, seed=12)
    rain = inputs.rain_field(ny, nx, 2)
    d = oracle.receivers_d8(z, 30.0, oracle.EDGE_ROUTE)
    rng = np.random.default_rng(ny * nx)
    hit = rng.random(shape) < 0.05
    d[hit] = rng.integers(8, 256, size=int(hit.sum())).astype(np.uint8)
    ref = np.where(d < 8, d, oracle.SINK).astype(np.uint8)
    order = oracle.high_to_low_order(z)
    w_ref, _ = oracle.accumulate_d8(ref, order, rain)
    _, a_ref = oracle.accumulate_d8(ref, order, None)

    def place(a):
        buf = torch.empty(a.size + shift, dtype=torch.from_numpy(a).dtype, device="cuda")
        t = buf[shift:].view(ny, nx)
        t.copy_(torch.from_numpy(a))
        return t

    R = api.routing_d8(place(d))
    rt = place(rain)
    for want_w, want_area in ((True, True), (True, False), (False, True)):
        o = api.accumulate(R, rt, want_w=want_w, want_area=want_area)
        assert api.get_status() == 0
        if want_w:
            assert np.max(np.abs(o["w"].double().cpu().numpy() - w_ref) / np.maximum(w_ref, 1e-30)) <= 1e-6
        if want_area:
            np.testing.assert_array_equal(o["area"].cpu().numpy().astype(np.uint64), a_ref)
