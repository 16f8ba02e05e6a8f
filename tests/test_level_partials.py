"""The statistics kernels' block partial sums stay inside their buffer (level_partial_cap entries).

On the CPU: the blocks of every launch that writes them, over the control and level grids,
precisions and sample counts at the edges of the dispatch.  On the GPU: records at those
counts against the oracle, at the parity bars of the two paths.
"""
import numpy as np
import pytest

CASES = [(n0, level, ctrl) for n0, level, ctrl in [(8, 0, 0), (8, 0, 2), (8, 1, 1), (8, 1, 2), (8, 2, 2), (8, 2, 1), (16, 1, 1), (16, 2, 2),
                                                   (4, 3, 3), (4, 2, 0)]]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n0,level,ctrl", CASES)
def test_blocks_within_the_buffer(precision, n0, level, ctrl):
    from launch_host import Host
    for S in (1, 15, 16, 17, 70, 300)[:4 if n0 << level > 32 else 6]:
        h = Host(precision, n0=n0, n_levels=max(level, ctrl) + 1, ctrl_level=ctrl, max_batch=300)
        assert h.level_gradient(level, S) == 0
        blocks = sum(g[0] * g[1] * g[2] for name, g, *_ in h.launches()
                     if any(k in name for k in ("k_level_field", "k_level_pairs", "k_lvl_field", "k_lvl_s2")))
        assert 0 < blocks <= h.L.fake_level_partial_cap(n0 << ctrl, n0 << level), (S, blocks)
        h.close()


@pytest.mark.gpu
@pytest.mark.parametrize("precision,n0,level,ctrl,S", [
    ("mixed", 8, 2, 2, 16), ("mixed", 8, 2, 2, 17),                # samples of a cell split over threads
    ("mixed", 8, 0, 1, 9), ("mixed", 8, 0, 1, 70), ("fp64", 8, 0, 1, 70),  # more samples than blocks or warps
    ("mixed", 8, 1, 2, 17)])
def test_record_against_oracle(precision, n0, level, ctrl, S):
    torch = pytest.importorskip("torch")
    import __graft_entry__
    __graft_entry__.build()
    from oracle import mlmc
    from paper_2606_09291_gb300 import inputs, mlsgd
    c = dict(n_levels=max(level, ctrl) + 1, n0=n0, n_modes=16, corr_len=0.3, sigma=1.0, theta=5.0, alpha=1e-4, seed=6, ctrl_level=ctrl)
    rtol, tol = (1e-13, 1e-10) if precision == "fp64" else (1e-8, 1e-6)
    Nc = n0 << ctrl
    z = inputs.z_test(Nc) + inputs.z_random(Nc, 2)
    ctx = mlsgd.Context(**dict(c, rtol=rtol, max_iter=400, precision=precision))
    st = ctx.new_stats(level)
    ctx.mlsgd_level_gradient(3, level, 0, S, torch.tensor(z, dtype=torch.float64, device="cuda"), st)
    ref = mlmc.level_batch(mlmc.Workload(**c), 3, level, range(S), z)
    h = st.host()
    fac = np.exp(5.0 * (h["shift"] - ref["shift"]))
    f, o = st.field.cpu().numpy() * fac, ref["stats"].mean_x
    assert h["count"] == S
    assert np.abs(f - o).max() <= tol * np.abs(o).max()
    assert abs(h["s2_dx"] * fac ** 2 - ref["stats"].s2_x) <= tol * ref["stats"].s2_x
    ctx.close()
