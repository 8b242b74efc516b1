"""A barrier wait of a resident march that runs out: one block leaves the launch at once, so the others' first
wait ends at a short poll limit.  The march must not hang, the host must learn of it, nothing may march from
the incomplete state, and a new state must march as in a context that never failed."""
import pytest

from test_gpu_resident import _same, _solver, _start

pytestmark = pytest.mark.gpu

LIMIT = 1 << 14          # polls: some ten milliseconds
# one tile a block and several tiles a block, in pairs and one node a thread
CASES = [((32, 32, 9), "f32", True), ((48, 48, 48), "f32", False), ((48, 48, 48), "f32c", True),
         ((51, 48, 48), "bf16", False)]


def _status(call):
    from paper_0809_4730_gb300.glbe import GlbeError
    with pytest.raises(GlbeError) as e:
        call()
    return e.value.status


def _timed_out(S, absent=0):
    S.set_barrier_test(LIMIT, absent)
    S.step(13)
    S.set_barrier_test(1 << 24, -1)


def _solver2(shape=(128, 300), **kw):
    from paper_0809_4730_gb300.glbe import Solver2D
    return Solver2D(*shape, wall_lo=(0, 1), wall_hi=(0, 1), gamma=0.2, nu=0.05, F=(2e-6, 1e-6),
                    **dict(dict(storage="f32c", induction=1, gamma_m=0.2, eta=0.05, chi=0.05, mu=1.0, B0=(0.002, 0.004)),
                           **kw))


def _state2(S):
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    r = lambda q, s: s * (2 * torch.rand(q, S.N, device="cuda", generator=g) - 1)  # noqa: E731
    S.set_state(r(9, 1e-4), r(10, 1e-5) if S.induction else None, r(2, 1e-7) if S.induction else None, 0)


@pytest.mark.parametrize("reported", [True, False])
@pytest.mark.parametrize("shape,storage,mhd", CASES)
def test_a_new_state_marches_as_before(shape, storage, mhd, reported):
    from paper_0809_4730_gb300.glbe import GLBE_ERR_TIMEOUT
    A, B = _solver(shape, "y", storage, mhd), _solver(shape, "y", storage, mhd)
    _start(B)
    data = B.checkpoint()
    for _ in range(23):
        B.step(1)
    for restore in (lambda: _start(A), lambda: A.restore(data)):
        _start(A)
        A.step(4)
        _timed_out(A)
        A.step(20)                            # does not march: the barrier's count is stale
        if reported:
            assert _status(A.sync) == GLBE_ERR_TIMEOUT
        restore()
        A.step(23)
        A.sync()
        _same(A.get_state(), B.get_state())
        assert [h["t"] for h in A.history()] == [10, 20]
    A.close()
    B.close()


def test_2d_a_new_state_marches_as_before():
    from paper_0809_4730_gb300.glbe import GLBE_ERR_TIMEOUT
    A, B = _solver2(), _solver2()
    _state2(B)
    for _ in range(23):
        B.step(1)
    _state2(A)
    A.step(4)
    _timed_out(A, absent=1)
    A.step(20)
    assert _status(A.sync) == GLBE_ERR_TIMEOUT
    _state2(A)
    A.step(23)
    A.sync()
    _same(A.get_state(), B.get_state())
    A.close()
    B.close()


def test_contexts_without_a_counting_barrier_refuse_the_hook():
    from paper_0809_4730_gb300.glbe import GLBE_ERR_ARG, GLBE_ERR_STATE
    for S in (_solver((4, 32, 4), "y", "f32", False), _solver((48, 48, 48), "y", "f32", False, variant=1)):
        assert _status(lambda: S.set_barrier_test(LIMIT, 0)) == GLBE_ERR_STATE
        S.close()
    S = _solver((48, 48, 48), "y", "f32", False)
    assert _status(lambda: S.set_barrier_test(0, 0)) == GLBE_ERR_ARG
    S.close()


def test_every_synchronising_call_reports_until_a_state_is_set():
    import torch
    from paper_0809_4730_gb300.glbe import GLBE_ERR_STATE, GLBE_ERR_TIMEOUT
    calls = {"sync": lambda S: S.sync(), "residual": lambda S: S.residual(), "history": lambda S: S.history(),
             "checkpoint": lambda S: S.checkpoint()}
    S = _solver((48, 48, 48), "y", "f32c", True)
    w = torch.ones(3, S.N, device="cuda")
    for first in calls:
        _start(S)
        S.step(12)
        _timed_out(S)
        for name in (first, *calls):
            assert _status(lambda: calls[name](S)) == GLBE_ERR_TIMEOUT, (first, name)
        S.step(1)                             # also over a step launched by itself
        assert _status(S.sync) == GLBE_ERR_TIMEOUT
        for adjoint in (lambda: S.adjoint_steady(w, max_iters=20), lambda: S.adjoint_unrolled(4, 2, w)):
            assert _status(adjoint) == GLBE_ERR_STATE
    # not known to the host before the adjoint waits for the stream
    _start(S)
    _timed_out(S)
    assert _status(lambda: S.adjoint_steady(w, max_iters=20)) == GLBE_ERR_STATE
    _start(S)
    for call in calls.values():
        call(S)
    S.close()


def test_2d_every_synchronising_call_reports_until_a_state_is_set():
    from paper_0809_4730_gb300.glbe import GLBE_ERR_TIMEOUT
    calls = {"sync": lambda S: S.sync(), "residual": lambda S: S.residual(), "history": lambda S: S.history()}
    S = _solver2()
    for first in calls:
        _state2(S)
        S.step(12)
        _timed_out(S)
        for name in (first, *calls):
            assert _status(lambda: calls[name](S)) == GLBE_ERR_TIMEOUT, (first, name)
    _state2(S)
    for call in calls.values():
        call(S)
    S.close()


@pytest.mark.parametrize("two_d", [False, True])
def test_replays_of_a_captured_march_are_checked(two_d):
    """The wait runs out in replays alone: a synchronising call after the capture has found nothing."""
    import torch
    from paper_0809_4730_gb300.glbe import GLBE_ERR_TIMEOUT
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        S = _solver2() if two_d else _solver((48, 48, 48), "y", "f32", True)
        start = _state2 if two_d else _start
        start(S)
        S.step(20)
        S.sync()
        g = torch.cuda.CUDAGraph()
        S.set_barrier_test(LIMIT, 0)
        with torch.cuda.graph(g, stream=side):
            S.step(20)
        S.set_barrier_test(1 << 24, -1)
        S.sync()
        S.sync()
        g.replay()
        assert _status(S.sync) == GLBE_ERR_TIMEOUT
        start(S)
        S.sync()
        g.replay()
        assert _status(S.residual) == GLBE_ERR_TIMEOUT
        start(S)
        S.step(20)
        S.sync()
    S.close()


@pytest.mark.parametrize("two_d", [False, True])
def test_solve_does_not_pass_a_timed_out_wait_off_as_its_step_limit(two_d):
    from paper_0809_4730_gb300.glbe import GLBE_ERR_STATE, GLBE_ERR_TIMEOUT
    S = _solver2() if two_d else _solver((48, 48, 48), "y", "f32", False)
    start = _state2 if two_d else _start
    # the wait runs out in the steps up to a residual level, in the solve's own march, and before the call
    for before, cap in ((0, 400), (20, 400), (20, 7), (20, 0)):
        start(S)
        S.step(before)
        S.set_barrier_test(LIMIT, 0)
        if cap == 0:
            S.step(5)
        for _ in range(2):
            assert _status(lambda: S.solve(1e-30, cap)) == GLBE_ERR_STATE
        S.set_barrier_test(1 << 24, -1)
        assert _status(lambda: S.solve(1e-30, cap)) == GLBE_ERR_STATE
    start(S)
    status, t, r = S.solve(1e-30, 40)
    assert status == GLBE_ERR_TIMEOUT and t == 40 and r > 0
    S.close()


@pytest.mark.parametrize("two_d", [False, True])
def test_a_part_of_a_state_does_not_make_up_for_a_timed_out_wait(two_d):
    """Without dg or F_L those parts stay as the march left them, at different levels."""
    from paper_0809_4730_gb300.glbe import GLBE_ERR_TIMEOUT
    S = _solver2() if two_d else _solver((48, 48, 48), "y", "f32", True)
    (_state2 if two_d else _start)(S)
    df, dg, FL = S.get_state()
    for part in ((df,), (df, dg), (df, None, FL)):
        for reported in (True, False):
            S.set_state(df, dg, FL)
            S.sync()
            _timed_out(S)
            if reported:
                assert _status(S.sync) == GLBE_ERR_TIMEOUT
            S.set_state(*part)
            S.step(12)
            assert _status(S.sync) == GLBE_ERR_TIMEOUT
    S.set_state(df, dg, FL)
    S.set_state(df)                           # over a whole state a part is as good as ever
    S.step(12)
    S.sync()
    S.close()
