"""The step's division by E[Y] is correctly rounded: with one level and alpha = 0 the gradient is the mean
field over max(exp(-theta c), E[Y]), bit for bit what an IEEE division gives, from subnormal to large fields."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ey,shift", [(0.7, 2.0), (1.0 + 2.0 ** -52, 2.0), (3.1e-5, 4.0), (0.01, 0.0), (1e90, 1.0), (7e-70, 30.0)])
def test_bits(ey, shift):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09291_gb300 import mlsgd
    theta = 10.0
    ctx = mlsgd.Context(n_levels=1, n0=64, n_modes=8, corr_len=0.3, sigma=1.0, theta=theta, alpha=0.0, rtol=1e-8, max_iter=10)
    n = ctx.n_ctrl
    rng = np.random.default_rng(11)
    f = rng.standard_normal(n) * 2e-4
    f[: n // 4] = np.ldexp(rng.uniform(1, 2, n // 4), rng.integers(-1074, 130, n // 4))
    f[-8:] = 0.0
    st = mlsgd.Stats(0, n)
    st.field.copy_(torch.tensor(f))
    st.scalars.copy_(torch.tensor([8.0, shift, ey, 0.1, 0.1, shift, 0.0, 0.0], dtype=torch.float64))
    z, g = torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    ctx.mlsgd_step([st], 0.0, z, grad=g)
    assert np.array_equal(g.cpu().numpy(), f / max(np.exp(-theta * shift), ey))
    ctx.close()
