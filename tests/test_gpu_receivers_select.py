"""D8 codes where the largest slope does not decide alone: ties, level ground
and slopes that underflow to zero, on both receiver kernels and in a batch, bit
for bit against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _surfaces(ny, nx):
    rng = np.random.default_rng(ny * 31 + nx)
    yield rng.integers(0, 3, size=(ny, nx)).astype(np.float32), 30.0      # ties and level ground
    yield (rng.integers(0, 3, size=(ny, nx)) * np.float32(1e-8)).astype(np.float32), 1e38  # every slope underflows
    yield (rng.integers(0, 9, size=(ny, nx)) * np.float32(1e-7)).astype(np.float32), 2e37  # some do
    yield np.zeros((ny, nx), np.float32), 30.0
    yield inputs.fractal_dem(ny, nx, beta=2.0, tilt=0.0, seed=5) - np.float32(500.0), 30.0


@pytest.mark.parametrize("shape", [(3, 5), (4, 127), (5, 129), (9, 257), (64, 128), (66, 260), (131, 132), (1024, 1028)])
@pytest.mark.parametrize("flags", [0, oracle.EDGE_ROUTE, oracle.D8_LOWEST, oracle.D4 | oracle.EDGE_ROUTE])
def test_ties_flats_and_underflow(shape, flags):
    from paper_2606_12800_gb300 import api
    for z, dx in _surfaces(*shape):
        zt = torch.from_numpy(np.ascontiguousarray(z)).cuda()
        ref = oracle.receivers_d8(z, dx, flags)
        np.testing.assert_array_equal(api.receivers_d8(zt, dx, flags).cpu().numpy(), ref)
        out = api.route_batch([zt, zt[:2].contiguous()], kind="d8", dx=dx, flags=flags)
        np.testing.assert_array_equal(out[0]["route"].cpu().numpy(), ref)
        np.testing.assert_array_equal(out[1]["route"].cpu().numpy(),
                                      oracle.receivers_d8(np.ascontiguousarray(z[:2]), dx, flags))
