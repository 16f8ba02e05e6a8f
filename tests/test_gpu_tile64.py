"""FP64 solves on grids whose passes march tiles (32^3 and up): true residual and chunking.

The residual is formed by the oracle's sparse matrix, so a wrong operator or right-hand
side shows whatever the solver reports; a wrong smoother shows in the iteration count.
The stop test is on the recursive residual, which the true one follows to about
eps |A| |y| / |b| (1e-13 at 64^3), so 2 rtol bounds it.  Tiles are 32 x 16 nodes and
segments 4 planes: 31 and 63 interior nodes leave a ragged end in each direction.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import fem  # noqa: E402
from paper_2606_09291_gb300 import inputs  # noqa: E402

CFG = dict(n_levels=5, n0=8, ctrl_level=2, n_modes=28, corr_len=0.3, sigma=1.0, theta=1.0, alpha=1e-4, seed=4)
RTOL = 1e-10


def _solve(lib, grid, S, z, **cfg):
    ctx = lib.Context(**dict(dict(CFG, precision="fp64", rtol=RTOL, max_iter=100), **cfg))
    N = 8 << grid
    f64 = dict(dtype=torch.float64, device="cuda")
    la = torch.zeros(S, N ** 3, **f64)
    ctx.mlsgd_sample_field(0, grid, grid, 0, S, log_a=la)
    y, q, phi = torch.full((S, (N + 1) ** 3), 7.0, **f64), torch.full((S, (N + 1) ** 3), 7.0, **f64), torch.zeros(S, **f64)
    it, st = (torch.zeros(S, dtype=torch.int32, device="cuda") for _ in range(2))
    code = ctx.mlsgd_solve_state_adjoint(grid, S, la, torch.tensor(z, **f64), y, q, phi, it, st)
    ctx.close()
    return code, la.cpu().numpy(), y.cpu().numpy(), q.cpu().numpy(), phi.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09291_gb300 import mlsgd
    return mlsgd


@pytest.mark.parametrize("grid,S", [(2, 1), (2, 9), (3, 3)])
def test_true_residual(lib, grid, S):
    N = 8 << grid
    z = inputs.z_test(32) + inputs.z_random(32, 3)
    code, la, y, q, phi, it, st = _solve(lib, grid, S, z)
    assert code == 0 and not st.any() and (it > 0).all() and it.max() <= 40
    lev = fem.Level(N)
    inner, rhs = lev.interior, lev.interpolation(32).T @ z / 32 ** 3
    for s in {0, S - 1}:
        A = lev.restrict(lev.stiffness(np.exp(la[s])))
        for v, b in ((y[s], rhs), (q[s], lev.mass() @ (y[s] - lev.nodal_target()))):
            assert np.linalg.norm(b[inner] - A @ v[inner]) <= 2 * RTOL * np.linalg.norm(b[inner])
            assert not np.delete(v, inner).any()


@pytest.mark.parametrize("grid", [2, 3])
def test_chunks_and_batches_leave_the_bits(lib, grid):
    z = inputs.z_test(32) + inputs.z_random(32, 3)
    ref = _solve(lib, grid, 2, z)
    for other in [_solve(lib, grid, 2, z, z_chunks=c) for c in (1, 3, 64)] + [_solve(lib, grid, 40, z)]:
        for a, b in zip(ref[1:], other[1:]):
            assert np.array_equal(a, b[:2])


@pytest.mark.parametrize("grid", [0, 1])  # 8^3, 16^3
def test_cluster_solves_do_not_depend_on_the_wave(lib, grid):
    """The blocks per SM follow the sample count (one block on an SM, several, more than a wave): the same bits."""
    z = inputs.z_test(32) + inputs.z_random(32, 3)
    ref = _solve(lib, grid, 1, z)
    for S in (15, 20, 40, 150, 250):
        for a, b in zip(ref[1:], _solve(lib, grid, S, z)[1:]):
            assert np.array_equal(a, b[:1])
