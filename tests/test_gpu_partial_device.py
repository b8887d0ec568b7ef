"""D8 routing where the whole GPU is not to be had: on a stream of some of its SMs
(a green context) the cooperative polling kernel does not fit and the walkers do
the same work; a captured graph, which may be launched on such a stream, holds no
cooperative kernel at all (that is read from the graph, none is launched there)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    """A stream of a green context of at least eight SMs."""
    cu = ctypes.CDLL("libcuda.so.1")
    torch.zeros(1, device="cuda")
    # resource descriptions are 144 bytes or a little more by driver version
    sm, part, rest = (ctypes.create_string_buffer(4096) for _ in range(3))
    desc, ctx, s = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    n = ctypes.c_uint(1)
    calls = (lambda: cu.cuDeviceGetDevResource(torch.cuda.current_device(), sm, 1),
             lambda: cu.cuDevSmResourceSplitByCount(part, ctypes.byref(n), sm, rest, 0, 8),
             lambda: cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1),
             lambda: cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, torch.cuda.current_device(), 1),
             lambda: cu.cuGreenCtxStreamCreate(ctypes.byref(s), ctx, 1, 0))
    for c in calls:
        if c() != 0:
            pytest.skip("no green context on this driver")
    yield torch.cuda.ExternalStream(s.value)
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(s)
    cu.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("shape", [(160, 192), (1000, 1100)])
def test_d8_on_some_of_the_sms(stream, shape):
    from paper_2606_12800_gb300 import api
    z = inputs.fractal_dem(*shape, beta=2.1, tilt=0.0, seed=4)
    zt = torch.from_numpy(z).cuda()
    rain = torch.from_numpy(inputs.rain_field(*shape, 3)).cuda()
    ref = api.route_d8(zt, 30.0, rain, want_lo=True)
    assert api.get_status() == 0
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        out = api.route_d8(zt, 30.0, rain, want_lo=True)
        assert api.get_status() == 0
        batch = api.route_batch([zt, zt], [rain, rain], want_area=True)
        assert api.batch_status(batch) == 0
    torch.cuda.synchronize()
    for o in (out, batch[0], batch[1]):
        assert torch.equal(o["w"], ref["w"]) and torch.equal(o["area"], ref["area"])
    assert torch.equal(out["w_lo"], ref["w_lo"])
    _, _, area, _ = oracle.route_d8(z, 30.0)
    np.testing.assert_array_equal(ref["area"].cpu().numpy().astype(np.uint64), area)


def _cooperative_nodes(call):
    """Kernels that `call` enqueues, and how many of them are cooperative: from
    the nodes of a captured graph."""
    cu = ctypes.CDLL("libcuda.so.1")
    call()  # allocations and kernel attributes before the capture
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    graph = ctypes.c_void_p()
    with torch.cuda.stream(side):
        call()
        side.synchronize()
        s = ctypes.c_void_p(side.cuda_stream)
        assert cu.cuStreamBeginCapture_v2(s, 2) == 0
        try:
            keep = call()
        finally:
            assert cu.cuStreamEndCapture(s, ctypes.byref(graph)) == 0
    n = ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kernels = coop = 0
    for i in range(n.value):
        kind, value = ctypes.c_int(-1), (ctypes.c_int * 16)()
        node = ctypes.c_void_p(nodes[i])
        assert cu.cuGraphNodeGetType(node, ctypes.byref(kind)) == 0
        if kind.value != 0:
            continue
        kernels += 1
        assert cu.cuGraphKernelNodeGetAttribute(node, 2, ctypes.byref(value)) == 0
        coop += value[0] != 0
    cu.cuGraphDestroy(graph)
    del keep
    return kernels, coop


@pytest.mark.parametrize("shape", [(160, 192), (1000, 1100)])
def test_captured_d8_is_not_cooperative(shape):
    from paper_2606_12800_gb300 import api
    z = torch.from_numpy(inputs.fractal_dem(*shape, beta=2.1, tilt=0.0, seed=4)).cuda()
    kernels, coop = _cooperative_nodes(lambda: api.route_d8(z, 30.0, z, want_lo=True))
    assert kernels >= 4 and coop == 0
    # the attribute is read right: the slope split's polling is cooperative
    kernels, coop = _cooperative_nodes(lambda: api.route_mfd(z, 30.0, 1.1))
    assert kernels >= 3 and coop >= 1
