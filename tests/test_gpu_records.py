"""Record merges and the multilevel combine (k_merge_field, k_combine_step) against numpy.

The cases are the merge's forms (empty destination, empty source, either side with the
larger shift, equal shifts), cell counts from less than one block to several cells per
thread, and every number of levels the combine is instantiated for at its edges.
Tolerance: a merged cell takes four rounded FP64 operations, a sum of n cells in pairs
of trees and strided chains at most n / (8 152 256) + 64 roundings: 1e-13 relative to
the largest value covers both with room.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-13


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09291_gb300 import mlsgd
    return mlsgd


def _ctx(lib, n_levels, ctrl_level, theta=10.0):
    return lib.Context(n_levels=n_levels, n0=2, ctrl_level=ctrl_level, n_modes=8, corr_len=0.3, sigma=1.0, theta=theta,
                       alpha=1e-2, rtol=1e-8, max_iter=10, precision="fp64")


def _record(lib, rng, level, cells, count, shift):
    st = lib.Stats(level, cells)
    f = rng.standard_normal(cells) if count else np.zeros(cells)
    sc = np.array([count, shift, rng.random(), rng.random(), rng.random(), shift, 5.0, 0.0]) if count else \
        np.array([0.0, -np.inf, 0, 0, 0, -np.inf, 0, 0])
    st.field.copy_(torch.tensor(f))
    st.scalars.copy_(torch.tensor(sc))
    return st, f, sc


@pytest.mark.parametrize("na,sa,nb,sb", [(0, 0.0, 7, 0.3), (5, 0.2, 0, 0.0), (5, 0.2, 7, 0.3), (5, 0.3, 7, 0.2), (5, 0.3, 7, 0.3),
                                         (0, 0.0, 0, 0.0)])
@pytest.mark.parametrize("ctrl_level", [0, 2, 6])  # 8, 512 and 2097152 cells
def test_merge_forms(lib, na, sa, nb, sb, ctrl_level):
    ctx = _ctx(lib, ctrl_level + 1, ctrl_level)
    cells, theta = ctx.n_ctrl, 10.0
    rng = np.random.default_rng(3)
    a, fa, xa = _record(lib, rng, 0, cells, na, sa)
    b, fb, xb = _record(lib, rng, 0, cells, nb, sb)
    ctx.mlsgd_stats_merge(a, b)
    f, s = a.field.cpu().numpy(), a.scalars.cpu().numpy()
    n = na + nb
    if n == 0:
        assert np.array_equal(f, fa) and np.array_equal(s, xa)
        return
    sh = max(xa[1], xb[1])
    wa = np.exp(theta * (xa[1] - sh)) if na else 0.0
    wb = np.exp(theta * (xb[1] - sh)) if nb else 0.0
    d, dy = fa * wa - fb * wb, xa[2] * wa - xb[2] * wb
    ref = fb * wb + (na / n) * d
    assert np.abs(f - ref).max() <= TOL * np.abs(ref).max()
    assert s[0] == n and s[1] == sh
    ry = xb[2] * wb + (na / n) * dy
    r3 = xa[3] * wa ** 2 + xb[3] * wb ** 2 + dy * dy * na * nb / n
    r4 = xa[4] * wa ** 2 + xb[4] * wb ** 2 + (d * d).sum() / cells * na * nb / n
    assert abs(s[2] - ry) <= TOL * abs(ry) and abs(s[3] - r3) <= TOL * r3 and abs(s[4] - r4) <= TOL * r4
    ctx.close()


@pytest.mark.parametrize("L,ctrl_level", [(1, 0), (2, 1), (3, 2), (6, 6), (9, 3), (9, 6)])
@pytest.mark.parametrize("adaptive", [False, True])
def test_combine_levels(lib, L, ctrl_level, adaptive):
    ctx = _ctx(lib, L if L > ctrl_level else ctrl_level + 1, ctrl_level)
    cells, theta, alpha, tau = ctx.n_ctrl, 10.0, 1e-2, 0.25
    rng = np.random.default_rng(5)
    recs = [_record(lib, rng, l, cells, 4 + l, 0.1 + 0.01 * l) for l in range(L)]
    z, prev = rng.standard_normal(cells), rng.standard_normal(cells)
    zt, gt = torch.tensor(z, device="cuda"), torch.tensor(prev, device="cuda")
    if adaptive:
        rep = ctx.mlsgd_step_adaptive([r[0] for r in recs], 1.0, tau, zt, gt)
    else:
        rep = ctx.mlsgd_step([r[0] for r in recs], tau, zt, grad=gt)
    cs = max(r[2][1] for r in recs)
    fac = [np.exp(theta * (r[2][1] - cs)) for r in recs]
    ey = sum(f * r[2][2] for f, r in zip(fac, recs))
    ex = sum(f * r[1] for f, r in zip(fac, recs))
    g = ex / max(np.exp(-theta * cs), ey) + alpha * z
    gn = np.sqrt((g * g).sum() / cells)
    assert np.abs(gt.cpu().numpy() - g).max() <= TOL * np.abs(g).max()
    assert abs(rep["grad_norm"] - gn) <= TOL * gn
    zn = z - rep["tau"] * g
    assert np.abs(zt.cpu().numpy() - zn).max() <= TOL * np.abs(zn).max()
    for l in range(L):
        m2 = (recs[l][1] ** 2).sum() / cells
        assert abs(rep["mean_dx_norm2"][l] - m2) <= TOL * m2
    if adaptive:
        lh = np.sqrt(((g - prev) ** 2).sum()) / (tau * np.sqrt((prev ** 2).sum()))
        assert abs(rep["l_hat"] - lh) <= TOL * lh
    ctx.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n0,level,ctrl_level", [(4, 0, 0), (4, 0, 2), (4, 1, 3), (4, 2, 4), (4, 3, 5), (4, 3, 2), (8, 2, 2), (8, 2, 1),
                                                 (2, 1, 6)])
def test_level_record_against_oracle(lib, precision, n0, level, ctrl_level):
    """Level grids coarser than, equal to and finer than the control grid (every right-hand
    side and statistics kernel), two calls merged, against the oracle at the parity bars."""
    from oracle import mlmc
    from paper_2606_09291_gb300 import inputs
    L = max(level, ctrl_level) + 1
    c = dict(n_levels=L, n0=n0, n_modes=16, corr_len=0.3, sigma=1.0, theta=5.0, alpha=1e-4, seed=6, ctrl_level=ctrl_level)
    rtol, tol = (1e-13, 1e-10) if precision == "fp64" else (1e-8, 1e-6)
    Nc = n0 << ctrl_level
    z = inputs.z_test(Nc) + inputs.z_random(Nc, 2)
    ctx = lib.Context(**dict(c, rtol=rtol, max_iter=400, precision=precision))
    zt = torch.tensor(z, dtype=torch.float64, device="cuda")
    st = ctx.new_stats(level)
    ctx.mlsgd_level_gradient(3, level, 0, 2, zt, st)
    ctx.mlsgd_level_gradient(3, level, 2, 3, zt, st)
    W = mlmc.Workload(**c)
    ref = mlmc.level_batch(W, 3, level, range(5), z)
    h = st.host()
    fac = np.exp(5.0 * (h["shift"] - ref["shift"]))
    f, o = st.field.cpu().numpy() * fac, ref["stats"].mean_x
    assert h["count"] == 5
    assert np.abs(f - o).max() <= tol * np.abs(o).max()
    assert abs(h["s2_dx"] * fac ** 2 - ref["stats"].s2_x) <= tol * ref["stats"].s2_x
    ctx.close()
