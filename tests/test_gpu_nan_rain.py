"""Rain that is no number: water is NaN wherever such rain gets to, whatever the
NaN's bits (the polling phase marks unfinished cells by one pattern of them)."""
import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(40, 70), (300, 517), (304, 520), (1000, 1304)])
@pytest.mark.parametrize("bits", [0x7FC00000, 0x7FFFFFFF, 0xFFC0DEAD])
@pytest.mark.parametrize("share", [0.01, 1.0])
def test_nan_rain(shape, bits, share):
    from paper_2606_12800_gb300 import api
    ny, nx = shape
    z = inputs.fractal_dem(ny, nx, beta=2.1, tilt=0.0, seed=4)
    hit = np.random.default_rng(nx).random(shape) < share
    rain = np.ones(shape, np.float32)
    rain.view(np.uint32)[hit] = bits
    mark = hit.astype(np.float32)  # where water of a marked cell gets to
    zt, rt = torch.from_numpy(z).cuda(), torch.from_numpy(rain).cuda()
    for full in (False, True):
        o = api.route_d8(zt, 30.0, rt, want_lo=full)
        assert api.get_status() == 0
        _, ref, _, _ = oracle.route_d8(z, 30.0, mark)
        np.testing.assert_array_equal(np.isnan(o["w"].cpu().numpy()), ref > 0)
        o = api.route_mfd(zt, 30.0, 1.1, rt, want_lo=full)
        assert api.get_status() == 0
        # a share may round to nothing in 64 bits, but a receiver's weight is never 0 here
        _, _, ref, _ = oracle.route_mfd(z, 30.0, 1.1, mark)
        np.testing.assert_array_equal(np.isnan(o["w"].cpu().numpy()), ref > 0)
        if bits == 0xFFC0DEAD:
            b = api.route_batch([zt, zt], [rt, rt], kind="mfd")
            assert api.batch_status(b) == 0
            np.testing.assert_array_equal(np.isnan(b[1]["w"].cpu().numpy()), ref > 0)
