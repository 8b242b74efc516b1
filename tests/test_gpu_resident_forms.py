"""The resident march against single steps over the options that reach it beside the plain ones: force fields,
ghost planes of a slab (never updated, gathered from as fluid), rates of their own, and levels that start off a
multiple of ten."""
import pytest

from test_gpu_resident import _same, _solver, _start
from test_gpu_resident_timeout import _solver2, _state2

pytestmark = pytest.mark.gpu

# one cluster, one tile a block, several tiles a block; even and odd nx
SHAPES = [(6, 24, 8), (7, 24, 8), (32, 30, 20), (33, 30, 20), (50, 48, 40), (51, 48, 40)]
OPTIONS = {"force1": dict(force_field=1), "force3": dict(force_field=3), "ghost_lo": dict(ghost_lo=1),
           "ghost_hi": dict(ghost_hi=1), "ghosts": dict(ghost_lo=1, ghost_hi=1, force_field=3),
           "rates": dict(s=[1.0 + 0.02 * k for k in range(19)], rho0=1.1)}


def _compare(A, B, start):
    import torch
    for S in (A, B):
        if S.params.force_field:
            g = torch.Generator(device="cuda").manual_seed(11)
            S.set_force(2e-6 * (2 * torch.rand(S.params.force_field, S.N, device="cuda", generator=g) - 1))
        start(S)
    for n in (7, 16, 9):
        A.step(n)
    for _ in range(32):
        B.step(1)
    A.sync()
    _same(A.get_state(), B.get_state())
    _same(A.fields(), B.fields())
    status, t, _ = A.solve(1e-30, 27)
    assert (status, t) == (4, 59)
    for _ in range(27):
        B.step(1)
    _same(A.get_state(), B.get_state())
    A.close()
    B.close()


@pytest.mark.parametrize("option", list(OPTIONS))
@pytest.mark.parametrize("storage,mhd", [("f32", False), ("bf16", False), ("f16", True), ("f32c", False), ("f32c", True)])
def test_options(storage, mhd, option):
    for shape in SHAPES:
        _compare(_solver(shape, "y", storage, mhd, **OPTIONS[option]), _solver(shape, "y", storage, mhd, **OPTIONS[option]),
                 _start)


@pytest.mark.parametrize("shape", [(33, 60), (64, 64), (100, 90), (197, 190)])
@pytest.mark.parametrize("storage,mhd", [("f32", 0), ("bf16", 1), ("f32c", 0), ("f32c", 1)])
def test_2d_force_field(shape, storage, mhd):
    kw = dict(storage=storage, induction=mhd, force_field=2)
    _compare(_solver2(shape, **kw), _solver2(shape, **kw), _state2)
