"""A kernel whose shared-memory opt-in is refused (a fake of the failing call): every call that needs it
reports the error, not only the first, and no solve goes on with a V-cycle step left out."""
import subprocess
import sys

import pytest

ECUDA = 5
# (kernel, precision, level, samples): a level gradient that launches it
CASES = [("k_vcycle64", "fp64", 2, 2), ("k_tile64", "fp64", 2, 2), ("k_small64ILi8", "fp64", 0, 2), ("k_small64ILi16", "fp64", 1, 2),
         ("k_small16", "mixed", 1, 2), ("k_solve32", "mixed", 2, 2), ("k_vcycle32", "mixed", 3, 2), ("k_slab", "mixed", 3, 2),
         ("k_coarse_vcycle", "mixed", 2, 33)]


def _calls(kernel, precision, level, samples):
    from launch_host import Host
    h = Host(precision, n_levels=4)
    h.L.fake_refuse_opt_in(kernel.encode())
    print(*[h.level_gradient(level, samples) for _ in range(3)])


@pytest.mark.parametrize("kernel,precision,level,samples", CASES)
def test_reported_by_every_call(kernel, precision, level, samples):
    # in a process of its own: what is set up is set up once
    code = "import sys; sys.path[:0] = %r; import test_launch_errors as t; t._calls(%r, %r, %d, %d)" % (
        sys.path, kernel, precision, level, samples)
    from launch_host import load
    load()
    out = subprocess.run([sys.executable, "-c", code], stdout=subprocess.PIPE, check=True, timeout=300).stdout.split()
    assert [int(v) for v in out] == [ECUDA] * 3


def test_pending_error_stays():
    """An error that was pending before a refused occupancy query is still reported."""
    code = ("import sys; sys.path[:0] = %r\nfrom launch_host import Host\nh = Host('fp64', n_levels=3)\n"
            "h.L.fake_refuse_occupancy(1)\nh.L.fake_set_last_error(700)\nprint(h.solve(0, 2))\n"
            "h.L.cudaGetLastError()\nprint(h.solve(0, 2))" % (sys.path,))
    from launch_host import load
    load()
    out = subprocess.run([sys.executable, "-c", code], stdout=subprocess.PIPE, check=True, timeout=300).stdout.split()
    assert [int(v) for v in out] == [ECUDA, 0]
