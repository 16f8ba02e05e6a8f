"""FP64 field synthesis (k_field): planes alone and in mirrored pairs, both field models.

Few samples take one plane per block, many take pairs; grids from 2^3 (one point per half
axis) up.  Against the oracle's direct sum; tolerance 1e-13 of the field's largest value
(n_modes products of four factors, a few roundings each).  The two forms add the same
terms in the same order, so a sample's field is the same bits in both.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mlmc, philox  # noqa: E402

MODELS = {"exponential": dict(n_modes=96, corr_len=0.15, field_model=0), "cosines": dict(n_modes=64, corr_len=0.15, field_model=1)}


@pytest.mark.parametrize("model", sorted(MODELS))
@pytest.mark.parametrize("grid", [0, 1, 2, 4])  # 2^3, 4^3, 8^3, 32^3
def test_planes_and_pairs(model, grid):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09291_gb300 import mlsgd
    c = dict(n_levels=5, n0=2, sigma=1.0, theta=1.0, alpha=1e-4, seed=9, **MODELS[model])
    ctx = mlsgd.Context(**c)
    N = 2 << grid
    S = 2 * 152 // (N // 2) + 1  # the first count that takes pairs
    many = torch.zeros(S, N ** 3, dtype=torch.float64, device="cuda")
    xi = torch.zeros(S, c["n_modes"], dtype=torch.float64, device="cuda")
    one = torch.zeros(1, N ** 3, dtype=torch.float64, device="cuda")
    ctx.mlsgd_sample_field(2, grid, grid, 0, S, xi=xi, log_a=many)
    ctx.mlsgd_sample_field(2, grid, grid, S - 1, 1, log_a=one)
    assert torch.equal(many[S - 1], one[0])
    W = mlmc.Workload(**c)
    x = xi.cpu().numpy()
    pick = sorted({0, S // 2, S - 1})
    ref = W.log_a(x[pick], grid).reshape(len(pick), -1)
    got = many.cpu().numpy()[pick]
    assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()
    ctx.close()
