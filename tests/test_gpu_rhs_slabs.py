"""The right-hand side of a control grid at least eight times finer than the grid, by slabs of control planes.

The slabs follow the scratch, which follows the sample count; the sums do not.  So a sample's
solve has the same bits alone, in a larger batch (one slab or a few) and in the allocation-free
call, and the record of a chunked batch does not see the chunks.  Against the oracle's B z at
1e-12 of its largest value (2 r (2 r + 2) products in a sum, r up to 64).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fem  # noqa: E402
from paper_2606_09291_gb300 import inputs  # noqa: E402

CFG = dict(n_levels=7, n0=4, n_modes=16, corr_len=0.3, sigma=1.0, theta=1.0, alpha=1e-4, seed=2, max_iter=400)
BAR = {"fp64": dict(rtol=1e-13), "mixed": dict(rtol=1e-8)}


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09291_gb300 import mlsgd
    return mlsgd


def _solve(lib, precision, grid, S, z, noalloc=False):
    ctx = lib.Context(**dict(CFG, precision=precision, **BAR[precision]))
    N = CFG["n0"] << grid
    f64 = dict(dtype=torch.float64, device="cuda")
    la = torch.zeros(S, N ** 3, **f64)
    ctx.mlsgd_sample_field(0, grid, grid, 0, S, log_a=la)
    y, q, phi = torch.zeros(S, (N + 1) ** 3, **f64), torch.zeros(S, (N + 1) ** 3, **f64), torch.zeros(S, **f64)
    it, st = (torch.zeros(S, dtype=torch.int32, device="cuda") for _ in range(2))
    f = ctx.mlsgd_solve_state_adjoint_noalloc if noalloc else ctx.mlsgd_solve_state_adjoint
    assert f(grid, S, la, z, y, q, phi, it, st) == 0
    ctx.close()
    return [t.cpu().numpy() for t in (y, q, phi, it)] + [la.cpu().numpy()]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("grid", [0, 1, 2, 3, 4])  # 4^3 (r = 64) to 32^3 (r = 8) under a 256^3 control, 64^3 by node rows
def test_bits_do_not_follow_the_batch(lib, precision, grid):
    Nc = 256
    z = torch.tensor(inputs.z_test(Nc) + inputs.z_random(Nc, 2), dtype=torch.float64, device="cuda")
    ref = _solve(lib, precision, grid, 1, z)
    for S in ((2, 6, 20) if grid < 4 else (2, 3)):
        for a, b in zip(ref, _solve(lib, precision, grid, S, z)):
            assert np.array_equal(a[0], b[0])
    if grid < 3:
        for a, b in zip(ref, _solve(lib, precision, grid, 1, z, noalloc=True)):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("grid", [0, 1, 2])
def test_against_oracle(lib, grid):
    Nc, N = 256, CFG["n0"] << grid
    z = inputs.z_test(Nc) + inputs.z_random(Nc, 2)
    y, _, _, _, la = _solve(lib, "fp64", grid, 1, torch.tensor(z, dtype=torch.float64, device="cuda"))
    lev = fem.Level(N)
    inner, b = lev.interior, lev.interpolation(Nc).T @ z / Nc ** 3
    A = lev.restrict(lev.stiffness(np.exp(la[0])))
    # the solve's own residual, at its rtol, beside the right-hand side's rounding
    assert np.abs(b[inner] - A @ y[0][inner]).max() <= 1e-12 * np.abs(b).max() + 1e-13 * np.linalg.norm(b[inner])
