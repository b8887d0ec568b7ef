"""What takes over when more cells are global than the polling phase takes: the
walkers (D8) and the rounds (slope split and both adjoints), alone and over a
batch, their answer to a cycle, and the rounds' barrier when its wait runs out.
Every case checks that the local phase did leave that many cells.  No test waits
without a limit: walkers end by count, the barrier after the wait limit."""
import numpy as np
import pytest

from paper_2606_12800_gb300 import _lib, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NY, NX = 1100, 1300
WALK, EDGE = _lib.FR_GLOBAL_WALKERS, _lib.FR_EDGE_ROUTE
NO_PROGRESS = _lib.FR_ERR_NO_PROGRESS


def _poll_limit():
    """At most four cells a lane, four blocks of 256 lanes an SM."""
    return torch.cuda.get_device_properties(0).multi_processor_count * 4 * 256 * 4


def _left(ws):
    """Cells the local phase left (the list's length, word 4 of the workspace)."""
    return int(ws[:64].view(torch.int64)[4])


def _ws(mfd):
    from paper_2606_12800_gb300 import api
    return api.workspace(NX, NY, torch.device("cuda", torch.cuda.current_device()), mfd=mfd)


@pytest.fixture
def plane():
    return torch.from_numpy(np.ascontiguousarray(inputs.planar_dem(NY, NX, 0.01, 30.0))).cuda()


@pytest.fixture
def ramp():
    """Falls along x and, ten times slower, along y."""
    y, x = np.mgrid[0:NY, 0:NX].astype(np.float64)
    return torch.from_numpy((3.0 * (NX - x) + 0.3 * (NY - y)).astype(np.float32)).cuda()


def test_rounds_give_up_at_the_barrier(ramp):
    from paper_2606_12800_gb300 import api
    good = api.route_mfd(ramp, 30.0, 1.1, None, EDGE, want_lo=True, want_mask=True)
    assert api.get_status() == 0 and _left(_ws(True)) > _poll_limit()
    R = api.routing_mfd(good["mask"], ramp, 30.0, 1.1, EDGE)
    g, _ = api.adjoint(R, good["w"], good["w_lo"])
    assert api.get_status() == 0 and _left(_ws(True)) > _poll_limit()
    prev = api.set_wait_limit(0)
    try:
        api.route_mfd(ramp, 30.0, 1.1, None, EDGE)
        assert api.get_status() == NO_PROGRESS
        api.adjoint(R, good["w"], good["w_lo"])
        assert api.get_status() == NO_PROGRESS
        b = api.route_batch([ramp], kind="mfd", flags=EDGE)
        assert api.batch_status(b) == NO_PROGRESS
    finally:
        api.set_wait_limit(prev)
    again = api.route_mfd(ramp, 30.0, 1.1, None, EDGE)
    assert api.get_status() == 0 and torch.equal(again["w"], good["w"])
    assert torch.equal(api.adjoint(R, good["w"], good["w_lo"])[0], g)


def test_rounds_end_at_a_cycle(ramp):
    from paper_2606_12800_gb300 import api
    o = api.route_mfd(ramp, 30.0, 1.1, None, EDGE, want_lo=True, want_mask=True)
    mask = o["mask"].clone()
    mask[500, 650], mask[500, 651] = 1, 4  # east and back
    R = api.routing_mfd(mask, ramp, 30.0, 1.1, EDGE)
    api.accumulate(R, None, want_w=True, device=mask.device)
    assert api.get_status() == NO_PROGRESS and _left(_ws(True)) > _poll_limit()
    api.adjoint(R, o["w"], o["w_lo"])
    assert api.get_status() == NO_PROGRESS and _left(_ws(True)) > _poll_limit()


def test_d8_ends_at_a_cycle(plane):
    """The walkers forward, the rounds of the adjoint."""
    from paper_2606_12800_gb300 import api
    d = api.receivers_d8(plane, 30.0, EDGE)
    o = api.accumulate(api.routing_d8(d, WALK), None, want_w=True, want_area=True, device=d.device)
    assert api.get_status() == 0
    d[500, 650], d[500, 651] = 0, 2
    R = api.routing_d8(d, WALK)
    for want_w, want_area in ((True, True), (True, False), (False, True)):
        api.accumulate(R, None, want_w=want_w, want_area=want_area, device=d.device)
        assert api.get_status() == NO_PROGRESS and _left(_ws(False)) > _poll_limit()
    api.adjoint(R, o["w"])
    assert api.get_status() == NO_PROGRESS and _left(_ws(False)) > _poll_limit()


def test_batch_of_planes_walks(plane):
    """Every row is one river, in each of the batch's grids."""
    from paper_2606_12800_gb300 import api
    small = plane[:300, -700:].contiguous()
    outs = api.route_batch([plane, small, plane], kind="d8", flags=EDGE, want_area=True)
    assert api.batch_status(outs) == 0 and _left(outs[0]["_ws"]) > _poll_limit()
    for o in outs:
        ny, nx = o["area"].shape
        ref = np.broadcast_to(np.arange(1, nx + 1), (ny, nx))
        np.testing.assert_array_equal(o["area"].cpu().numpy(), ref)
        np.testing.assert_array_equal(o["w"].cpu().numpy(), ref.astype(np.float32))


def test_batch_of_ramps_goes_by_rounds(ramp):
    """The sums are the same sequence of operations as a single call's."""
    from paper_2606_12800_gb300 import api
    small = ramp[:300, -700:].contiguous()
    outs = api.route_batch([small, ramp], kind="mfd", flags=EDGE, want_lo=True)
    assert api.batch_status(outs) == 0 and _left(outs[0]["_ws"]) > _poll_limit()
    for z, o in zip((small, ramp), outs):
        ref = api.route_mfd(z, 30.0, 1.1, None, EDGE, want_lo=True)
        assert api.get_status() == 0
        assert torch.equal(o["w"], ref["w"]) and torch.equal(o["w_lo"], ref["w_lo"])
