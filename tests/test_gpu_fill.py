"""Depression filling at the edges of its 64x64 tiles, against the
priority-flood oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _spiral(ny, nx):
    """A one-cell channel that winds through the grid between high walls: the
    path out of its end turns at every wall."""
    z = np.full((ny, nx), 50.0, np.float32)
    for k in range(1, ny - 1, 2):
        z[k, 1:nx - 1] = 1.0
    for i, k in enumerate(range(2, ny - 2, 2)):
        z[k, nx - 2 if i % 2 == 0 else 1] = 1.0
    z[0, 1] = 0.5
    return z


@pytest.mark.parametrize("shape", [(2, 2), (3, 64), (63, 66), (64, 64), (65, 65), (66, 130), (127, 67),
                                   (130, 193), (129, 256)])
@pytest.mark.parametrize("limit", [100000, 4000])
@pytest.mark.parametrize("shift", [0, 1])
def test_fill_tile_edges(shape, limit, shift):
    """limit: both lengths of a sweep; shift: a base address off 16 bytes."""
    from paper_2606_12800_gb300 import api
    ny, nx = shape
    rng = np.random.default_rng(ny * 1000 + nx)
    for z in (inputs.fractal_dem(ny, nx, beta=2.2, tilt=0.0, seed=3) - 500.0, _spiral(ny, nx),
              rng.integers(-3, 3, size=shape).astype(np.float32)):
        z = z.astype(np.float32)
        buf = torch.empty(ny * nx + shift, dtype=torch.float32, device="cuda")
        zt = buf[shift:].view(ny, nx)
        zt.copy_(torch.from_numpy(z))
        F, _ = api.fill(zt, max_sweeps=limit)
        np.testing.assert_array_equal(F.cpu().numpy(), oracle.fill(z))
