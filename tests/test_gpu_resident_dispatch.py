"""Which calls the resident march takes: the sizes on both sides of each line (the lines are those of 152 SMs),
the shortest march, and that both routes give the same state."""
import pytest

from test_gpu_resident import _same, _solver, _start
from test_gpu_resident_timeout import LIMIT, _solver2, _state2, _status

pytestmark = pytest.mark.gpu

# (shape, walls, storage, coupled, whether the steps meet at the counting barrier)
SIZES = [((86, 86, 84), "yz", "f32", False, True), ((88, 86, 84), "yz", "f32", False, False),      # pairs
         ((88, 88, 90), "yz", "bf16", False, True), ((90, 88, 90), "yz", "bf16", False, False),
         ((88, 88, 90), "", "f16", False, True), ((90, 88, 90), "", "f16", False, False),
         ((57, 58, 58), "yz", "bf16", False, True), ((59, 58, 58), "yz", "bf16", False, False),    # one node a thread
         ((69, 70, 72), "yz", "f32", False, True), ((71, 70, 72), "yz", "f32", False, False),
         ((70, 69, 72), "y", "f32c", False, True), ((70, 71, 72), "y", "f32c", False, False),
         ((68, 67, 68), "y", "f32", True, True), ((68, 68, 68), "y", "f32", True, False),          # coupled
         ((68, 67, 68), "y", "f32c", True, True), ((68, 68, 68), "y", "f32c", True, False),
         ((62, 61, 61), "y", "bf16", True, True), ((62, 62, 62), "y", "bf16", True, False)]
SIZES2 = [((90, 91), dict(), False), ((91, 91), dict(), True), ((278, 279), dict(), True), ((279, 279), dict(), False),
          ((91, 91), dict(induction=0), True), ((279, 279), dict(induction=0), False),
          ((91, 91), dict(storage="bf16"), True), ((279, 279), dict(storage="bf16"), False),
          ((112, 111), dict(storage="f32"), False), ((112, 112), dict(storage="f32"), True),
          ((278, 279), dict(storage="f32"), True), ((279, 279), dict(storage="f32"), False),
          ((181, 181), dict(storage="bf16", induction=0), False), ((182, 181), dict(storage="bf16", induction=0), True),
          ((278, 279), dict(storage="f32", induction=0), True), ((279, 279), dict(storage="f32", induction=0), False),
          ((700, 700), dict(storage="bf16", induction=0), False)]


def _meets(S):
    from paper_0809_4730_gb300.glbe import GLBE_ERR_STATE, GlbeError
    try:
        S.set_barrier_test(1 << 24, -1)
    except GlbeError as e:
        assert e.status == GLBE_ERR_STATE
        return False
    return True


def _compare(A, B, start):
    start(A)
    start(B)
    for n in (4, 5, 13, 39, 40):
        A.step(n)
    for _ in range(101):
        B.step(1)
    A.sync()
    _same(A.get_state(), B.get_state())
    A.close()
    B.close()


@pytest.mark.parametrize("shape,walls,storage,mhd,meets", SIZES)
def test_lines(shape, walls, storage, mhd, meets):
    import torch
    A, B = _solver(shape, walls, storage, mhd), _solver(shape, walls, storage, mhd)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert _meets(A) == meets
    _compare(A, B, _start)


@pytest.mark.parametrize("shape,kw,meets", SIZES2)
def test_2d_lines(shape, kw, meets):
    import torch
    A, B = _solver2(shape, **kw), _solver2(shape, **kw)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert _meets(A) == meets
    _compare(A, B, _state2)


@pytest.mark.parametrize("make,start,least", [(lambda: _solver((48, 48, 48), "y", "f32", False), _start, 5),
                                             (lambda: _solver2(), _state2, 5),
                                             (lambda: _solver2((200, 200), storage="f32", induction=0), _state2, 40)])
def test_the_shortest_march(make, start, least):
    """Where the blocks meet at the counting barrier: with one of them absent, only a march runs out."""
    from paper_0809_4730_gb300.glbe import GLBE_ERR_TIMEOUT
    S = make()
    start(S)
    S.set_barrier_test(LIMIT, 0)
    for n in (0, 1, 2, 3, least - 1):
        S.step(n)
        S.sync()
    if least == 40:
        assert S.solve(1e-30, 100)[0] == GLBE_ERR_TIMEOUT      # its step limit: a solve of these replays launches
    S.step(least)
    assert _status(S.sync) == GLBE_ERR_TIMEOUT
    S.close()
