"""One-launch mixed solves on 8^3 and 16^3 with controls near and beyond what FP32 dot products hold.

The solves sum r.z and p.q as FP32 pairs, up to 2^120; beyond that in FP64, like the solver
of the larger grids.  At 1e19 times the target's control the vectors' products are finite in
FP32 and their sums are not: the solve converges, to the scaled solution (tolerance 1e-6, the
parity bar).  At 1e21 the products themselves overflow: no sample ends as solved, and the solve
and the step that reads such a record give MLSGD_ENONFINITE, with one inner iteration per step
as well as with the default.  (A sample whose r.z is finite while p.q is not takes steps of
length 0 and ends at the iteration cap, status 1; with an infinite r.z the step length is NaN
and the status 2.)
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2606_09291_gb300 import inputs  # noqa: E402

CFG = dict(n_levels=4, n0=4, n_modes=64, corr_len=0.3, sigma=1.0, theta=1.0, alpha=1e-4, seed=2, precision="mixed", rtol=1e-8,
           max_iter=400)


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09291_gb300 import mlsgd
    return mlsgd


def _solve(lib, grid, scale, **cfg):
    ctx = lib.Context(**dict(CFG, **cfg))
    N, S = 4 << grid, 3
    f64 = dict(dtype=torch.float64, device="cuda")
    la = torch.zeros(S, N ** 3, **f64)
    ctx.mlsgd_sample_field(0, grid, grid, 0, S, log_a=la)
    y, q, phi = torch.zeros(S, (N + 1) ** 3, **f64), torch.zeros(S, (N + 1) ** 3, **f64), torch.zeros(S, **f64)
    it, st = (torch.zeros(S, dtype=torch.int32, device="cuda") for _ in range(2))
    code = ctx.mlsgd_solve_state_adjoint(grid, S, la, torch.tensor(scale * inputs.z_test(32), **f64), y, q, phi, it, st)
    ctx.close()
    return code, y.cpu().numpy(), st.cpu().numpy()


@pytest.mark.parametrize("inner", [1, 6])
@pytest.mark.parametrize("grid", [1, 2])  # 8^3, 16^3
def test_sums_beyond_fp32(lib, grid, inner):
    code, ref, st = _solve(lib, grid, 1.0, inner_iters=inner)
    assert code == 0
    code, y, st = _solve(lib, grid, 1e19, inner_iters=inner)
    assert code == 0 and not st.any()
    assert np.abs(y / 1e19 - ref).max() <= 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("inner", [1, 6])
@pytest.mark.parametrize("grid", [1, 2])
def test_products_beyond_fp32(lib, grid, inner):
    code, y, st = _solve(lib, grid, 1e21, inner_iters=inner)
    assert code == 4 and (st & 2).any() and st.all()
    ctx = lib.Context(**dict(CFG, inner_iters=inner, ctrl_level=3))
    z = torch.tensor(1e21 * inputs.z_test(32), dtype=torch.float64, device="cuda")
    stats = [ctx.new_stats(0), ctx.new_stats(1), ctx.new_stats(2)]
    for level in (0, 1, 2):
        ctx.mlsgd_level_gradient(0, level, 0, 3, z if level == grid else z * 1e-21, stats[level])
    with pytest.raises(lib.MlsgdError) as e:
        ctx.mlsgd_step(stats, 0.0, z.clone())
    assert e.value.status == 4
    ctx.close()
