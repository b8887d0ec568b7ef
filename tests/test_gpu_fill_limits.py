"""fr_fill's limit on sweeps: what one limit allows a larger one allows too, the
count reported never exceeds it, and a surface that is still moving is refused."""
import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import _lib

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _channel(ny, nx):
    """A one-cell channel to and fro between high walls: thousands of tile
    crossings from its far end to the way out."""
    z = np.full((ny, nx), 50.0, np.float32)
    z[1:ny - 1:2, 1:nx - 1] = 1.0
    for i, k in enumerate(range(2, ny - 2, 2)):
        z[k, nx - 2 if i % 2 == 0 else 1] = 1.0
    z[0, 1] = 0.5
    return z


def test_fill_limit_is_monotone():
    from paper_2606_12800_gb300 import api
    z = _channel(1025, 1025)
    ref, zt = oracle.fill(z), torch.from_numpy(z).cuda()
    for limit in (4095, 4096, 100000):
        F, sweeps = api.fill(zt, max_sweeps=limit)
        np.testing.assert_array_equal(F.cpu().numpy(), ref)
        assert 1 < sweeps <= limit


@pytest.mark.parametrize("shape", [(5, 5), (64, 64), (66, 66)])
def test_fill_small_limits(shape):
    """One sweep that changes something is one too few; a grid of one tile is
    done after the first, however its channel winds."""
    from paper_2606_12800_gb300 import api
    z = _channel(*shape)
    zt = torch.from_numpy(z).cuda()
    with pytest.raises(_lib.FrError) as e:
        api.fill(zt, max_sweeps=1)
    assert e.value.status == _lib.FR_ERR_NO_PROGRESS
    if max(shape) <= 64:
        F, sweeps = api.fill(zt, max_sweeps=2)
        assert sweeps == 2
        np.testing.assert_array_equal(F.cpu().numpy(), oracle.fill(z))
    F, sweeps = api.fill(zt, max_sweeps=4000)
    np.testing.assert_array_equal(F.cpu().numpy(), oracle.fill(z))
