"""Statistics of a level whose nodal values are FP32 pairs down to subnormal words: the batch mean on a control
grid twice as fine against FP64 (the pairs' sums are exact there), at 1e-13 of its largest value."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def stats():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_09291_gb300 import build
    out = os.path.join(build.BUILD, "liblevel_stats.so")
    objs = [os.path.join(build.BUILD, os.path.basename(s) + ".o") for s in build.sources()]
    subprocess.run([os.environ.get("NVCC", "nvcc")] + build.ARCH + build.FLAGS +
                   ["-shared", os.path.join(HERE, "native", "level_stats.cpp")] + objs + ["-o", out, "-lcudart"], check=True)
    f = ctypes.CDLL(out).level_stats
    f.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int] + [ctypes.c_void_p] * 2 + [ctypes.c_int] * 2 + [ctypes.c_double] + \
        [ctypes.c_void_p] * 2 + [ctypes.c_int] * 2
    return f


def _cells(x, n1, Nc):  # nodal [S, n1^3] at the control cells, trilinear
    r = Nc // (n1 - 1)
    m = np.arange(Nc)
    P = np.zeros((Nc, n1))
    P[m, m // r], P[m, m // r + 1] = 1 - (m % r + 0.5) / r, (m % r + 0.5) / r
    return np.einsum("ai,bj,ck,sijk->sabc", P, P, P, x.reshape(-1, n1, n1, n1)).reshape(len(x), -1)


@pytest.mark.parametrize("exponent", [-10, -105, -126, -140])  # of the high words
@pytest.mark.parametrize("coarse", [False, True])
def test_mean(stats, exponent, coarse):
    Nf, Nc, S = 16, 32, 5
    rng = np.random.default_rng(7)

    def pairs(N):
        v = np.zeros((S, N + 1, N + 1, N + 1, 2), dtype=np.float32)
        shape = (S, N - 1, N - 1, N - 1)
        h = np.ldexp(rng.uniform(1, 2, shape), exponent).astype(np.float32) * rng.choice([-1, 1], shape).astype(np.float32)
        v[:, 1:-1, 1:-1, 1:-1, 0] = h
        v[:, 1:-1, 1:-1, 1:-1, 1] = (np.ldexp(rng.uniform(-0.5, 0.5, shape), exponent - 23)).astype(np.float32)
        return v.reshape(S, -1, 2)

    f, k = pairs(Nf), pairs(Nf // 2)
    x = f.astype(np.float64).sum(2)
    ref = _cells(x, Nf + 1, Nc)
    if coarse:
        ref = ref - _cells(k.astype(np.float64).sum(2), Nf // 2 + 1, Nc)
    ref = ref.mean(0)
    dev = dict(device="cuda")
    q, c = torch.tensor(f, **dev), torch.tensor(k, **dev)
    phi = torch.zeros(S, dtype=torch.float64, **dev)
    field = torch.zeros(Nc ** 3, dtype=torch.float64, **dev)
    sc = torch.tensor([0.0, -np.inf, 0, 0, 0, -np.inf, 0, 0], dtype=torch.float64, **dev)
    torch.cuda.synchronize()
    assert stats(q.data_ptr(), phi.data_ptr(), Nf, c.data_ptr() if coarse else None, phi.data_ptr() if coarse else None, S, Nc, 1.0,
                 field.data_ptr(), sc.data_ptr(), 1, int(coarse)) == 0
    assert np.abs(field.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
