"""One-launch solves on 8^3 and 16^3 grids against the CPU oracle, at the edges of their dispatch.

4^3 (level by level) and 32^3 (fused passes) are the neighbouring grids of the rule; sample
counts run from one to more than one wave of blocks.  Tolerances are the parity bars of
the two paths: 1e-6 for the mixed path at rtol 1e-8, 1e-10 for FP64 at rtol 1e-13.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mlmc  # noqa: E402
from paper_2606_09291_gb300 import inputs  # noqa: E402

CFG = dict(n_levels=4, n0=4, n_modes=64, corr_len=0.3, sigma=1.0, theta=1.0, alpha=1e-4, seed=2)


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09291_gb300 import mlsgd
    return mlsgd


def _solve(lib, grid, S, z, **cfg):
    ctx = lib.Context(**dict(dict(CFG, max_iter=400), **cfg))
    N = 4 << grid
    f64 = dict(dtype=torch.float64, device="cuda")
    la = torch.zeros(S, N ** 3, **f64)
    ctx.mlsgd_sample_field(0, grid, grid, 0, S, log_a=la)
    y, q, phi = torch.full((S, (N + 1) ** 3), 7.0, **f64), torch.full((S, (N + 1) ** 3), 7.0, **f64), torch.zeros(S, **f64)
    it, st = (torch.zeros(S, dtype=torch.int32, device="cuda") for _ in range(2))
    code = ctx.mlsgd_solve_state_adjoint(grid, S, la, torch.tensor(z, **f64), y, q, phi, it, st)
    ctx.close()
    return code, la.cpu().numpy(), y.cpu().numpy(), q.cpu().numpy(), phi.cpu().numpy(), it.cpu().numpy(), st.cpu().numpy()


def _check(grid, la, y, q, phi, z, tol, picks):
    W = mlmc.Workload(n0=4, n_levels=4, n_modes=64, corr_len=0.3, sigma=1.0, theta=1.0, alpha=1e-4, seed=2)
    for s in picks:
        ref = W.solve_state_adjoint(la[s], z, grid)
        for a, b in ((y[s], ref["y"]), (q[s], ref["q"])):
            assert np.abs(a - np.asarray(b).ravel()).max() <= tol * np.abs(b).max()
        assert abs(phi[s] - ref["phi"]) <= tol * abs(ref["phi"])


@pytest.mark.parametrize("grid", [0, 1, 2, 3])  # 4^3, 8^3, 16^3, 32^3
@pytest.mark.parametrize("S", [1, 5])
@pytest.mark.parametrize("knobs", [dict(), dict(inner_iters=1), dict(inner_iters=9, inner_iters_next=2), dict(ir_steps=3)])
def test_mixed_against_oracle(lib, grid, S, knobs):
    z = inputs.z_test(32) + inputs.z_random(32, 3)
    code, la, y, q, phi, it, st = _solve(lib, grid, S, z, precision="mixed", rtol=1e-8, **knobs)
    assert code == 0 and not st.any() and (it > 0).all()
    _check(grid, la, y, q, phi, z, 1e-6, range(S))


@pytest.mark.parametrize("grid", [0, 1, 2, 3])
@pytest.mark.parametrize("S", [1, 47])
def test_fp64_against_oracle(lib, grid, S):
    z = inputs.z_test(32) + inputs.z_random(32, 3)
    code, la, y, q, phi, it, st = _solve(lib, grid, S, z, precision="fp64", rtol=1e-13)
    assert code == 0 and not st.any() and (it > 0).all()
    _check(grid, la, y, q, phi, z, 1e-10, sorted({0, S // 2, S - 1}))


@pytest.mark.parametrize("grid,S", [(1, 700), (2, 310)])
def test_mixed_more_than_one_wave(lib, grid, S):
    z = inputs.z_test(32)
    code, la, y, q, phi, it, st = _solve(lib, grid, S, z, precision="mixed", rtol=1e-8)
    assert code == 0 and not st.any()
    _check(grid, la, y, q, phi, z, 1e-6, (0, S // 2, S - 1))
    one = _solve(lib, grid, 2, z, precision="mixed", rtol=1e-8)
    assert np.array_equal(y[:2], one[2]) and np.array_equal(q[:2], one[3]) and np.array_equal(it[:2], one[5])


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("grid", [1, 2])
def test_zero_nonfinite_and_capped(lib, grid, precision):
    z = np.zeros(32 ** 3)
    code, la, y, q, phi, it, st = _solve(lib, grid, 3, z, precision=precision, rtol=1e-8)
    assert code == 0 and not y.any() and not st.any()
    z[100] = np.inf
    code, la, y, q, phi, it, st = _solve(lib, grid, 3, z, precision=precision, rtol=1e-8)
    assert code == 4 and (st & 2).all()
    ctx = lib.Context(**dict(CFG, max_iter=1, precision=precision, rtol=1e-14))
    N = 4 << grid
    f64 = dict(dtype=torch.float64, device="cuda")
    la = torch.zeros(2, N ** 3, **f64)
    buf = [torch.zeros(2, (N + 1) ** 3, **f64), torch.zeros(2, (N + 1) ** 3, **f64), torch.zeros(2, **f64),
           torch.zeros(2, dtype=torch.int32, device="cuda"), torch.zeros(2, dtype=torch.int32, device="cuda")]
    assert ctx.mlsgd_solve_state_adjoint(grid, 2, la, torch.tensor(inputs.z_test(32), **f64), *buf) == 3
    assert (buf[4].cpu().numpy() == 1).all()
    ctx.close()


@pytest.mark.parametrize("grid", [3, 4, 5])  # 32^3: the whole solve; 64^3 and 128^3: the V-cycle from 32^3 down
@pytest.mark.parametrize("knobs", [dict(), dict(inner_iters=1), dict(ir_steps=2, inner_iters=4, inner_iters_next=7)])
def test_clusters_and_passes_agree(lib, grid, knobs):
    """Up to 32 samples the 32^3 level runs in clusters, above in passes: the same bits."""
    z = inputs.z_test(32) + inputs.z_random(32, 3)
    big = _solve(lib, grid, 33, z, precision="mixed", rtol=1e-8, n_levels=6, ctrl_level=3, **knobs)
    few = _solve(lib, grid, 3, z, precision="mixed", rtol=1e-8, n_levels=6, ctrl_level=3, **knobs)
    for a, b in zip(big[1:], few[1:]):
        assert np.array_equal(a[:3], b)


def test_cluster_zero_and_nonfinite(lib):
    z = np.zeros(32 ** 3)
    code, la, y, q, phi, it, st = _solve(lib, 3, 3, z, precision="mixed", rtol=1e-8)
    assert code == 0 and not y.any() and not st.any()
    z[100] = np.inf
    code, la, y, q, phi, it, st = _solve(lib, 3, 3, z, precision="mixed", rtol=1e-8)
    assert code == 4 and (st & 2).all()
