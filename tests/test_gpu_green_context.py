"""Plans on a stream of a green context, which has a part of the device's SMs: the resident
2D launches, whose CTAs must all be on an SM at once, keep to that part (or give way to
the per-step kernels where a shot needs more), and every result is the one of the whole
device: traces bit for bit, gradients to 1e-6 (relative L2; another kernel family may
run, which sums the density terms and the images in another order)."""
import ctypes

import numpy as np
import pytest

from paper_2110_03345_gb300 import binding, inputs
from _helpers import gpu_forward, gpu_gradient, rel_l2

pytestmark = pytest.mark.gpu

SM, RES = 1, 96 + 48   # resource type, bytes of a resource (type, padding, union) at least


@pytest.fixture(params=[16, 64])
def green_stream(request):
    """A stream of a green context of about `param` SMs."""
    import torch
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("the driver has no green contexts")
    buf = lambda: ctypes.create_string_buffer(4 * RES)  # noqa: E731
    res, part, rest = buf(), buf(), buf()
    n = ctypes.c_uint(1)
    desc, ctx, st = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    ok = lambda e: e == 0  # noqa: E731
    assert ok(cu.cuDeviceGetDevResource(0, res, SM))
    assert ok(cu.cuDevSmResourceSplitByCount(part, ctypes.byref(n), res, rest, 0, request.param))
    sms = ctypes.c_uint.from_buffer(part, 96).value
    assert request.param <= sms < ctypes.c_uint.from_buffer(res, 96).value
    assert ok(cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1))
    assert ok(cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, 0, 1))
    assert ok(cu.cuGreenCtxStreamCreate(ctypes.byref(st), ctx, 1, 0))
    yield torch.cuda.ExternalStream(st.value)
    torch.cuda.synchronize()
    assert ok(cu.cuStreamDestroy_v2(st)) and ok(cu.cuGreenCtxDestroy(ctx))


@pytest.mark.parametrize("shape,shots", [((100, 120), 1), ((100, 120), 3), ((256, 256), 2), ((700, 748), 1)])
def test_plans_keep_to_the_streams_sms(green_stream, shape, shots):
    import torch
    nt = 90
    p = inputs.breast_problem(shape, 0.3e-3, nt, nelem=24, shots=[8 * i for i in range(shots)], order=8, nb=10,
                              radius=0.3 * min(shape) * 0.3e-3)
    ref, _ = gpu_forward(p)
    J0, g0, _, _ = gpu_gradient(p, 0.5 * ref)
    torch.cuda.synchronize()
    with torch.cuda.stream(green_stream):
        got, plan = gpu_forward(p)
        J1, g1, d1, _ = gpu_gradient(p, 0.5 * ref)
    if max(shape) < 128:   # one tile per shot at most: still resident
        assert plan.stats()["launches"] < nt
    assert np.array_equal(got, ref) and np.array_equal(d1, ref)
    assert abs(J1 - J0) <= 1e-12 * J0 and rel_l2(g1, g0) < 1e-6
