"""The residual record against sums formed from the fields, at grid sizes where the reduction of the
per-block partials changes shape: one block, one chunk of partials, one more than a chunk, a remainder
chunk, and more chunks than one pass of a warp adds."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 8, 4), (64, 64, 16), (64, 65, 16), (61, 59, 53), (256, 128, 96)])
def test_record_matches_field_sums(shape):
    import torch
    from paper_0809_4730_gb300.glbe import Solver
    nx, ny, nz = shape
    S = Solver(nx, ny, nz, wall_lo=(0, 1, 0), wall_hi=(0, 1, 0), gamma=0.5, nu=0.05, F=(1e-5, 2e-6, -3e-6),
               storage="f32", variant=1)
    gen = torch.Generator(device="cuda").manual_seed(5)
    S.set_state(1e-3 * (torch.rand(19, S.N, device="cuda", generator=gen) - 0.5))
    S.step(10)
    _, u0, _ = S.fields()
    S_prev = u0.double()
    S.step(10)
    rho, u, _ = S.fields()      # level 20: the state that the next step's residual is taken on
    S.step(1)
    info = S.residual()
    assert info.t == 20
    u, rho = u.double(), rho.double()
    num, den = (u - S_prev).square().sum(), u.square().sum()
    # per block 256 FP32 terms summed in FP32 (relative 256 eps at most), FP64 from there on
    tol = 256 * 2.0 ** -24
    assert abs(info.den - float(den)) <= tol * float(den)
    assert abs(info.num - float(num)) <= 4 * tol * float(num)
    assert abs(info.r - (info.num / info.den) ** 0.5) <= 1e-14 * info.r
    fluid = nx * (ny - 2) * nz
    assert abs(info.mass - float(rho.sum())) <= fluid * 2.0 ** -24
    j = (rho * u).sum(1)
    scale = float((rho * u).abs().sum())
    for k in range(3):
        assert abs(info.momentum[k] - float(j[k])) <= tol * scale
    assert info.nonfinite == 0
    S.close()
