"""Donor counts of D8 codes at the edges of the count kernel's tiles (128x64, eight
rows a warp, four columns a lane), on rows and base addresses off their alignment."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import _lib, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1), (1, 300), (300, 1), (2, 2), (7, 4), (8, 128), (9, 132), (63, 127), (64, 128),
                                   (65, 129), (64, 256), (72, 131), (129, 260), (1100, 1028)])
@pytest.mark.parametrize("flags", [0, oracle.EDGE_ROUTE, oracle.D8_LOWEST, oracle.D4 | oracle.EDGE_ROUTE])
@pytest.mark.parametrize("shift", [0, 1])
def test_donor_counts(shape, flags, shift):
    from paper_2606_12800_gb300 import api
    ny, nx = shape
    z = inputs.fractal_dem(ny, nx, beta=2.0, tilt=0.0, seed=ny + nx)
    ref = oracle.receivers_d8(z, 30.0, flags)
    want = np.zeros((ny + 2, nx + 2), np.uint8)
    for k in range(8):
        y, x = np.nonzero(ref == k)
        np.add.at(want, (y + 1 + oracle.OFFY[k], x + 1 + oracle.OFFX[k]), 1)
    zt = torch.from_numpy(z).cuda()
    d, n = (torch.full((ny * nx + shift + 8,), 77, dtype=torch.uint8, device="cuda") for _ in range(2))
    P = ctypes.c_void_p
    _lib.check(_lib.load().fr_receivers_d8(P(zt.data_ptr()), nx, ny, 30.0, flags, P(d.data_ptr() + shift),
                                           P(n.data_ptr() + shift), api._stream()), "fr_receivers_d8")
    for t, r in ((d, ref), (n, want[1:-1, 1:-1])):
        t = t.cpu().numpy()
        np.testing.assert_array_equal(t[shift:shift + ny * nx].reshape(ny, nx), r)
        assert (t[:shift] == 77).all() and (t[shift + ny * nx:] == 77).all()
