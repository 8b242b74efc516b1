"""Contexts whose stream belongs to a green context, a part of the device's SMs: a march planned for all of them
may not be placed there, so the steps are launched one by one, with the same result."""
import ctypes as C

import pytest

from test_gpu_resident import _same, _solver, _start
from test_gpu_resident_timeout import _solver2, _state2, _status

pytestmark = pytest.mark.gpu


@pytest.fixture
def green_stream():
    """A stream on 16 SMs or the least the device partitions into."""
    import torch
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("driver without green contexts")
    whole, part = C.create_string_buffer(1024), C.create_string_buffer(1024)
    n, dev, desc, ctx, st = C.c_uint(1), C.c_int(), C.c_void_p(), C.c_void_p(), C.c_void_p()
    assert cu.cuDeviceGet(C.byref(dev), 0) == 0
    assert cu.cuDeviceGetDevResource(dev, whole, 1) == 0                                      # 1: SMs
    assert cu.cuDevSmResourceSplitByCount(part, C.byref(n), whole, None, 0, 16) == 0
    assert cu.cuDevResourceGenerateDesc(C.byref(desc), part, 1) == 0
    assert cu.cuGreenCtxCreate(C.byref(ctx), desc, dev, 1) == 0                               # 1: default stream
    assert cu.cuGreenCtxStreamCreate(C.byref(st), ctx, 1, 0) == 0                             # 1: non-blocking
    yield torch.cuda.ExternalStream(st.value)
    torch.cuda.synchronize()
    assert cu.cuStreamDestroy_v2(st) == 0
    assert cu.cuGreenCtxDestroy(ctx) == 0


@pytest.mark.parametrize("shape", [(4, 32, 4), (48, 48, 48)])
def test_marches_are_launched_on_a_part_of_the_device(green_stream, shape):
    import torch
    from paper_0809_4730_gb300.glbe import GLBE_ERR_STATE
    B = _solver(shape, "y", "f32", False)
    _start(B)
    B.step(30)
    B.sync()
    torch.cuda.synchronize()
    A = _solver(shape, "y", "f32", False, stream=green_stream)
    assert _status(lambda: A.set_barrier_test(1 << 24, -1)) == GLBE_ERR_STATE
    with torch.cuda.stream(green_stream):
        _start(A)
        A.step(30)
        got = A.get_state()
    A.sync()
    _same(got, B.get_state())
    with torch.cuda.stream(green_stream):
        _start(A)
    _start(B)
    assert A.solve(1e-30, 47)[:2] == B.solve(1e-30, 47)[:2] == (4, 47)
    A.close()
    B.close()


def test_2d_marches_are_launched_on_a_part_of_the_device(green_stream):
    import torch
    from paper_0809_4730_gb300.glbe import GLBE_ERR_STATE
    B = _solver2()
    _state2(B)
    B.step(30)
    B.sync()
    torch.cuda.synchronize()
    A = _solver2(stream=green_stream)
    assert _status(lambda: A.set_barrier_test(1 << 24, -1)) == GLBE_ERR_STATE
    with torch.cuda.stream(green_stream):
        _state2(A)
        A.step(30)
        got = A.get_state()
    A.sync()
    _same(got, B.get_state())
    A.close()
    B.close()
