"""Residual sums of the resident march's forms of several tiles a block: no FP32 sum spans more nodes than a
launched block's 256, so they differ from the launched steps' in the order of FP64 additions alone."""
import pytest

from test_gpu_resident import _same, _solver, _start

pytestmark = pytest.mark.gpu


# past one tile on each SM: pairs (even nx, x periodic), one node a thread, coupled
@pytest.mark.parametrize("storage,mhd", [("f32", False), ("bf16", False), ("f16", False), ("f32c", False), ("f32", True)])
@pytest.mark.parametrize("shape,walls", [((62, 60, 64), ""), ((70, 70, 70), "yz"), ((63, 60, 50), "y")])
def test_partials_are_the_launched_ones(shape, walls, storage, mhd):
    A, B = _solver(shape, walls, storage, mhd), _solver(shape, walls, storage, mhd)
    _start(A)
    _start(B)
    A.step(31)
    for _ in range(31):
        B.step(1)
    _same(A.get_state(), B.get_state())
    # P positive terms added in FP64 in any order: each sum is within P 2^-53 of the exact one
    tol = 2 * ((A.N + 255) // 256) * 2.0 ** -53
    ha, hb = A.history(), B.history()
    assert [h["t"] for h in ha] == [h["t"] for h in hb] == [10, 20, 30]
    for x, y in zip(ha, hb):
        assert abs(x["num"] - y["num"]) <= tol * y["num"] and abs(x["den"] - y["den"]) <= tol * y["den"]
    A.close()
    B.close()
