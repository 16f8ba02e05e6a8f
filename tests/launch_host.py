"""The library's host code on a fake CUDA runtime (native/fake_cuda_runtime.cpp): no GPU, no kernel runs,
launches are checked and recorded.  Device pointers are host memory."""
import ctypes
import functools
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(maxsize=None)
def load():
    from paper_2606_09291_gb300 import build, mlsgd
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if nvcc is None or shutil.which("g++") is None:
        pytest.skip("needs nvcc and g++")
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s) + ".o") for s in build.sources()]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    out = os.path.join(build.BUILD, "libmlsgd_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I" + build.CSRC, "-I" + build.INCLUDE,
                    "-I" + inc, os.path.join(HERE, "native", "fake_cuda_runtime.cpp")] + objs + ["-o", out], check=True)
    L = ctypes.CDLL(out)
    vp, i32 = ctypes.c_void_p, ctypes.c_int
    L.mlsgd_create.argtypes = [ctypes.POINTER(mlsgd.Config), ctypes.POINTER(vp)]
    L.mlsgd_destroy.argtypes = [vp]
    L.mlsgd_last_error.argtypes = [vp]
    L.mlsgd_last_error.restype = ctypes.c_char_p
    L.mlsgd_n_ctrl_cells.argtypes = [vp]
    L.mlsgd_n_ctrl_cells.restype = ctypes.c_int64
    L.mlsgd_level_gradient.argtypes = [vp, i32, i32, ctypes.c_int64, i32, vp, ctypes.POINTER(mlsgd.LevelStats), vp]
    L.mlsgd_solve_state_adjoint.argtypes = L.mlsgd_solve_state_adjoint_noalloc.argtypes = [vp, i32, i32] + [vp] * 8
    L.fake_launch.argtypes = [i32, ctypes.POINTER(ctypes.c_uint)]
    L.fake_launch.restype = ctypes.c_char_p
    L.fake_refuse_opt_in.argtypes = [ctypes.c_char_p]
    L.fake_level_partial_cap.restype = ctypes.c_longlong
    return L


class Host:
    """A context on the fake runtime."""

    def __init__(self, precision, **cfg):
        from paper_2606_09291_gb300 import mlsgd
        self.m, self.L = mlsgd, load()
        c = mlsgd.Config()
        d = dict(n_levels=3, n0=8, ctrl_level=-1, n_modes=16, corr_len=0.3, sigma=1.0, theta=1.0, alpha=1e-4, rtol=1e-8, max_iter=4,
                 precision=dict(fp64=0, mixed=1)[precision])
        d.update(cfg)
        if d["ctrl_level"] < 0:
            d["ctrl_level"] = d["n_levels"] - 1
        for k, v in d.items():
            setattr(c, k, v)
        self.cfg, self.h = d, ctypes.c_void_p()
        assert self.L.mlsgd_create(ctypes.byref(c), ctypes.byref(self.h)) == 0
        self.z = np.zeros(self.L.mlsgd_n_ctrl_cells(self.h))
        self.reset()

    def reset(self):
        self.L.fake_reset()
        self.L.fake_refuse_opt_in(b"")
        self.L.fake_refuse_occupancy(0)
        self.L.cudaGetLastError()

    def close(self):
        self.L.mlsgd_destroy(self.h)

    def level_gradient(self, level, samples):
        field, sc = np.zeros(len(self.z)), np.zeros(8)
        st = self.m.LevelStats(level, field.ctypes.data, sc.ctypes.data)
        return self.L.mlsgd_level_gradient(self.h, 0, level, 0, samples, self.z.ctypes.data, ctypes.byref(st), None)

    def solve(self, grid, samples, noalloc=False):
        N = self.cfg["n0"] << grid
        y, q = np.zeros((samples, (N + 1) ** 3)), np.zeros((samples, (N + 1) ** 3))
        la, phi = np.zeros((samples, N ** 3)), np.zeros(samples)
        it, st = np.zeros(samples, np.int32), np.zeros(samples, np.int32)
        f = self.L.mlsgd_solve_state_adjoint_noalloc if noalloc else self.L.mlsgd_solve_state_adjoint
        return f(self.h, grid, samples, *(a.ctypes.data for a in (la, self.z, y, q, phi, it, st)), None)

    def launches(self, kernel=""):
        """[(name, grid, block, shared memory, device)] of the kernels whose name contains `kernel`."""
        v, out = (ctypes.c_uint * 8)(), []
        for i in range(self.L.fake_launches()):
            name = self.L.fake_launch(i, v).decode()
            if kernel in name:
                out.append((name, tuple(v[:3]), tuple(v[3:6]), v[6], v[7]))
        return out
