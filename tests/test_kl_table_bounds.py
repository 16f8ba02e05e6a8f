"""The host's mode table stays inside its candidate list for any number of modes (checked vector accesses), and
takes the same modes as the oracle."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import kl

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_09291_gb300", "csrc")
MAIN = """
#include <cstdio>
#include <cstdlib>
#include "kl_table.h"
int main(int, char** v) {
  const mlsgd::KLTable t = mlsgd::build_kl_table(std::atof(v[1]), std::atoi(v[2]));
  for (size_t k = 0; k < t.lam3.size(); ++k) std::printf("%d %d %d %.17g\\n", t.ix[k], t.iy[k], t.iz[k], t.lam3[k]);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("kl")
    (d / "main.cpp").write_text(MAIN)
    out = str(d / "kl")
    subprocess.run(["g++", "-std=c++17", "-O1", "-D_GLIBCXX_ASSERTIONS", "-I" + CSRC, str(d / "main.cpp"),
                    os.path.join(CSRC, "kl_table.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("modes", [2, 64, 66, 124, 126, 128, 512, 4096])  # 4^3 and 5^3 candidates and their neighbours
def test_modes(program, modes):
    r = subprocess.run([program, "0.2", str(modes)], stdout=subprocess.PIPE, stderr=subprocess.PIPE, check=True)
    got = np.array([line.split() for line in r.stdout.decode().splitlines()], dtype=float)
    assert got.shape == (modes, 4)
    idx, lam3 = kl.select_3d(kl.modes_1d(0.2, int(got[:, :3].max()) + 3)[1], modes)  # two 1D modes more than were taken
    assert np.array_equal(got[:, :3].astype(int), idx)
    assert np.abs(got[:, 3] - lam3).max() <= 1e-13 * lam3[0]
