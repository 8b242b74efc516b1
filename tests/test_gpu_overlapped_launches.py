"""Chains of overlapped launches on grids so small that whole successors of a kernel sit waiting while it
runs: replayed from a graph, and then enqueued without a pause, against the same steps each waited for.
The kernels are the same, so the fields and the residual records have the same bits."""
import pytest

pytestmark = pytest.mark.gpu

FLOW = dict(wall_lo=(0, 1, 1), wall_hi=(0, 1, 1), gamma=0.3, nu=0.05, F=(2e-5, 1e-5, -1e-5))
MHD = dict(induction=1, gamma_m=0.3, eta=0.05, chi=0.3, mu=1.0, B0=(0.01, 0.02, -0.01))
CAVITY = dict(wall_lo=(1, 1, 1), wall_hi=(1, 1, 1), gamma=0.3, nu=0.05, U_lid=(0.02, 0.0, 0.0))
BOX = dict(box=((4, 4, 4), (15, 13, 12)))

# explicit one-node and paired forms, the SRT collision, stochastic rounding, the cavity with and without its
# extended domain: everything that is launched step by step whatever the grid's size
CASES = [("one_f32", dict(FLOW, storage="f32", variant=1)), ("one_f32c", dict(FLOW, storage="f32c", variant=1, **MHD)),
         ("one_bf16", dict(FLOW, storage="bf16", variant=1, **MHD)), ("one_f16", dict(FLOW, storage="f16", variant=1)),
         ("pair_f32", dict(FLOW, storage="f32", variant=2)), ("pair_bf16", dict(FLOW, storage="bf16", variant=2, **MHD)),
         ("pair_f16", dict(FLOW, storage="f16", variant=2)),
         ("srt_f32", dict(FLOW, storage="f32", collision=1, **MHD)), ("srt_bf16", dict(FLOW, storage="bf16", collision=1)),
         ("sr_bf16", dict(FLOW, storage="bf16sr", **MHD)), ("sr_f16", dict(FLOW, storage="f16sr")),
         ("lid_f32", dict(CAVITY, storage="f32")), ("lid_bf16", dict(CAVITY, storage="bf16")),
         ("box_f32c", dict(CAVITY, storage="f32c", **MHD, **BOX)), ("box_bf16", dict(CAVITY, storage="bf16", **MHD, **BOX))]
FLOW2 = dict(wall_lo=(0, 1), wall_hi=(0, 1), gamma=0.3, nu=0.05, F=(2e-5, 1e-5))
MHD2 = dict(induction=1, gamma_m=0.3, eta=0.05, chi=0.3, mu=1.0, B0=(0.01, 0.02))
CASES2 = [("one_f32", dict(FLOW2, storage="f32", variant=1, **MHD2)), ("one_f32c", dict(FLOW2, storage="f32c", variant=1)),
          ("one_f32c_mhd", dict(FLOW2, storage="f32c", variant=1, **MHD2)),
          ("pair_f32", dict(FLOW2, storage="f32", variant=2)), ("pair_bf16", dict(FLOW2, storage="bf16", variant=2, **MHD2))]


def _run(make):
    import torch
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        A = make()
        A.step(20)                            # an even level, a residual snapshot: the graph can be replayed
        A.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            A.step(20)
        for _ in range(3):
            g.replay()
        A.step(20)
        got = [x for x in A.fields() if x is not None]
        A.sync()
        ha = A.history()
    B = make()
    for _ in range(100):
        B.step(1)
        B.sync()
    want = [x for x in B.fields() if x is not None]
    B.sync()
    assert len(got) == len(want)
    for x, y in zip(got, want):
        assert bool(torch.isfinite(x).all()) and bool((x == y).all())
    key = (lambda h: (h["num"], h["den"], h["mass"])) if isinstance(ha[0], dict) else (lambda h: (h.num, h.den, h.mass))
    assert [key(h) for h in ha] == [key(h) for h in B.history()] and len(ha) >= 8
    A.close()
    B.close()


@pytest.mark.parametrize("shape", [(20, 18, 17), (34, 30, 29)])
@pytest.mark.parametrize("name,kw", CASES, ids=[n for n, _ in CASES])
def test_chain_equals_synchronised_steps(name, kw, shape):
    from paper_0809_4730_gb300.glbe import Solver
    _run(lambda: Solver(*shape, **kw))


@pytest.mark.parametrize("shape", [(64, 48), (194, 101)])
@pytest.mark.parametrize("name,kw", CASES2, ids=[n for n, _ in CASES2])
def test_2d_chain_equals_synchronised_steps(name, kw, shape):
    from paper_0809_4730_gb300.glbe import Solver2D
    _run(lambda: Solver2D(*shape, **kw))
