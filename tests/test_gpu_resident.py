"""The resident march of small grids (many steps in one launch) against the same steps launched one by
one: states bit for bit, residual records to the rounding of their block sums, at the sizes where the
march changes form (one cluster, one tile a block, several tiles a block, single launches)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# one node and up; one cluster (up to 4096 nodes) and past it; one tile of 256 nodes on each of 152 SMs and past
# it; several tiles a block; the largest of the dense forms and past them; odd nx; seams and walls on every axis
SHAPES = [((1, 3, 1), "y"), ((4, 32, 4), "y"), ((27, 19, 1), "y"), ((16, 16, 16), "yz"), ((17, 16, 16), "xyz"),
          ((64, 32, 19), "y"), ((64, 32, 20), "yz"), ((63, 41, 37), "xy"), ((62, 60, 64), ""), ((70, 70, 70), "yz"),
          ((72, 72, 72), "yz")]


def _solver(shape, walls, storage, mhd, **kw):
    from paper_0809_4730_gb300.glbe import Solver
    w = tuple(int(c in walls) for c in "xyz")
    kw = dict(wall_lo=w, wall_hi=w, gamma=0.2, nu=0.05, F=(2e-6, 1e-6, -1e-6), storage=storage, **kw)
    if mhd:
        kw.update(induction=1, gamma_m=0.2, eta=0.05, chi=0.05, mu=1.0, B0=(0.002, 0.004, -0.001))
    return Solver(*shape, **kw)


def _start(S, seed=3):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda q, s: s * (2 * torch.rand(q, S.N, device="cuda", generator=g) - 1)  # noqa: E731
    S.set_state(r(19, 1e-4), r(21, 1e-5) if S.induction else None, r(3, 1e-7) if S.induction else None, 0)


def _same(a, b):
    for x, y in zip(a, b):
        assert (x is None) == (y is None)
        if x is not None:
            assert bool((x == y).all())


@pytest.mark.parametrize("mhd", [False, True])
@pytest.mark.parametrize("storage", ["f32", "f32c", "bf16", "f16"])
def test_march_equals_single_steps(storage, mhd):
    for shape, walls in SHAPES:
        A, B = _solver(shape, walls, storage, mhd), _solver(shape, walls, storage, mhd)
        _start(A)
        _start(B)
        A.step(2)
        A.step(21)                   # from level 2 over two residual levels
        for _ in range(23):
            B.step(1)
        _same(A.get_state(), B.get_state())
        ha, hb = A.history(), B.history()
        assert [h["t"] for h in ha] == [h["t"] for h in hb] == [10, 20]
        for x, y in zip(ha, hb):
            # FP32 sums of at most 512 terms a tile, in another order
            assert abs(x["den"] - y["den"]) <= 512 * 2.0 ** -23 * y["den"]
            assert abs(x["num"] - y["num"]) <= 512 * 2.0 ** -23 * y["num"]
            assert x["nonfinite"] == y["nonfinite"] == 0
        # the snapshot and the counters carry on
        A.step(12)
        for _ in range(12):
            B.step(1)
        _same(A.get_state(), B.get_state())
        assert [h["t"] for h in A.history()] == [10, 20, 30]
        A.close()
        B.close()


@pytest.mark.parametrize("shape,storage,mhd", [((4, 32, 4), "f32", False), ((16, 32, 16), "f32c", True),
                                              ((48, 48, 48), "f32c", False)])
def test_solve_stops_where_single_steps_would(shape, storage, mhd):
    A, B = _solver(shape, "y", storage, mhd), _solver(shape, "y", storage, mhd)
    _start(A)
    _start(B)
    for _ in range(10 * 60):
        B.step(1)
    levels = {h["t"]: h["r"] for h in B.history()}
    tol = levels[300]
    want = min(t for t, r in levels.items() if r <= tol)
    st, t, r = A.solve(tol * (1 + 1e-4), 590)
    assert st == 0 and t == want and A.t == want + 1 and abs(r - levels[want]) <= 1e-3 * r
    C = _solver(shape, "y", storage, mhd)
    _start(C)
    for _ in range(want + 1):
        C.step(1)
    _same(A.get_state(), C.get_state())
    # a capped solve takes every step, also the ones after the last whole chunk
    st, t, _ = A.solve(1e-30, 37)
    assert st == 4 and t == want + 38 and A.t == want + 38
    for _ in range(37):
        C.step(1)
    _same(A.get_state(), C.get_state())
    for S in (A, B, C):
        S.close()


@pytest.mark.parametrize("shape", [(4, 32, 4), (32, 32, 24)])
def test_divergence_ends_a_solve_and_is_reported(shape):
    import torch
    from paper_0809_4730_gb300.glbe import GLBE_ERR_DIVERGED, GlbeError
    S = _solver(shape, "y", "f32", False)
    df = torch.zeros(19, S.N, device="cuda")
    df.reshape(19, shape[2], shape[1], shape[0])[0, 0, shape[1] // 2, 0] = float("nan")   # off the walls
    S.set_state(df)
    with pytest.raises(GlbeError) as e:
        S.solve(1e-9, 400)
    assert e.value.status == GLBE_ERR_DIVERGED
    assert S.t == 11                     # ended at the first residual level that saw it
    _start(S)                            # a new state is marched as usual
    S.step(20)
    assert np.isfinite(S.residual().r)
    S.close()


# 2D: one cluster and past it, one tile on each of 152 SMs and past it, several tiles a block, the largest of
# the dense forms and past them
SHAPES2 = [((1, 5), "y"), ((64, 64), "y"), ((65, 64), "xy"), ((128, 304), "y"), ((129, 304), ""), ((333, 501), "x"),
           ((700, 700), "y"), ((1100, 1000), "y")]


@pytest.mark.parametrize("mhd", [False, True])
@pytest.mark.parametrize("storage", ["f32", "f32c", "bf16"])
def test_2d_march_equals_single_steps(storage, mhd):
    import torch
    from paper_0809_4730_gb300.glbe import Solver2D
    for shape, walls in SHAPES2:
        w = tuple(int(c in walls) for c in "xy")
        kw = dict(wall_lo=w, wall_hi=w, gamma=0.2, nu=0.05, F=(2e-6, 1e-6), storage=storage)
        if mhd:
            kw.update(induction=1, gamma_m=0.2, eta=0.05, chi=0.05, mu=1.0, B0=(0.002, 0.004))
        A, B = Solver2D(*shape, **kw), Solver2D(*shape, **kw)
        g = torch.Generator(device="cuda").manual_seed(3)
        r = lambda q, s: s * (2 * torch.rand(q, A.N, device="cuda", generator=g) - 1)  # noqa: E731
        st = (r(9, 1e-4), r(10, 1e-5) if mhd else None, r(2, 1e-7) if mhd else None, 0)
        A.set_state(*st)
        B.set_state(*st)
        A.step(2)
        A.step(21)
        for _ in range(23):
            B.step(1)
        _same(A.get_state(), B.get_state())
        # the same FP32 partials; their FP64 sum in another order past one cluster
        ha, hb = A.history(), B.history()
        assert [h.t for h in ha] == [h.t for h in hb] == [10, 20]
        for x, y in zip(ha, hb):
            rel = 0.0 if A.N <= 4096 else 1e-13
            assert abs(x.num - y.num) <= rel * y.num and abs(x.den - y.den) <= rel * y.den
            assert abs(x.r - y.r) <= rel * y.r and abs(x.mass - y.mass) <= rel * y.mass
        # a capped solve takes every step
        status, t, _ = A.solve(1e-30, 18)
        assert status == 4 and t == 41
        for _ in range(18):
            B.step(1)
        _same(A.get_state(), B.get_state())
        A.close()
        B.close()


def test_two_streams_march_apart():
    import torch
    out = []
    solvers = []
    for k in range(2):
        with torch.cuda.stream(torch.cuda.Stream()):
            S = _solver((40, 40, 40), "yz", "f32", True)
            _start(S, seed=k)
            solvers.append(S)
    for _ in range(5):
        for S in solvers:
            S.step(40)
    for k, S in enumerate(solvers):
        S.sync()
        with torch.cuda.stream(S.stream):
            out.append([x.clone() for x in S.get_state()])
        S.sync()
    for k, S in enumerate(solvers):
        T = _solver((40, 40, 40), "yz", "f32", True)
        _start(T, seed=k)
        T.step(200)
        _same(T.get_state(), out[k])
        T.close()
        S.close()


@pytest.mark.parametrize("shape", [(4, 32, 4), (40, 40, 40), (80, 80, 72)])
def test_captured_march_replays(shape):
    """A march captured in the caller's graph (cluster, cooperative and overlapped launches) replays as the
    same steps taken directly, its residual levels counted on the device."""
    import torch
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        A = _solver(shape, "yz" if shape[2] > 4 else "y", "f32c", True)
        _start(A)
        A.step(20)
        A.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            A.step(20)
        for _ in range(3):
            g.replay()
        side.synchronize()
        got = [x.clone() for x in A.get_state()]
        levels = [h["t"] for h in A.history()]
        A.sync()
    B = _solver(shape, "yz" if shape[2] > 4 else "y", "f32c", True)
    _start(B)
    B.step(80)
    _same(got, B.get_state())
    assert levels == [h["t"] for h in B.history()] == [10, 20, 30, 40, 50, 60, 70]
    A.close()
    B.close()
