"""Every kernel's shared-memory opt-in is made on each device that a process uses (two devices of the fake runtime)."""
import subprocess
import sys

import pytest


def _calls(precision, **cfg):
    from launch_host import Host
    out = []
    for dev in (0, 1):
        h = Host(precision, n_levels=5, max_batch=40, **cfg)
        h.L.cudaSetDevice(dev)
        out += [h.level_gradient(level, samples) for level in range(5) for samples in ((2, 33) if level < 4 else (2,))]
        out.append(h.solve(0, 2, noalloc=True))
        h.close()
    print(*out)


@pytest.mark.parametrize("precision,cfg", [("fp64", {}), ("mixed", {}), ("mixed", {"stencil": 1}), ("mixed", {"ctrl_level": 1, "n_modes": 512})])
def test_second_device(precision, cfg):
    from launch_host import load
    load()
    code = "import sys; sys.path[:0] = %r; import test_launch_devices as t; t._calls(%r, **%r)" % (sys.path, precision, cfg)
    out = subprocess.run([sys.executable, "-c", code], stdout=subprocess.PIPE, check=True, timeout=600).stdout.split()
    assert [int(v) for v in out] == [0] * 20
