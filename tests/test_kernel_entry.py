"""Every kernel waits for the kernels before it in its stream before it does anything else: its body begins
with pdl_entry or pdl_wait, so that its result does not rest on how it is launched."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_09291_gb300", "csrc")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__\s+void(?:\s+__launch_bounds__\([^{;]*?\))?\s+(\w+)\s*\(", src):
            i, depth = m.end(), 1
            while depth:  # to the end of the parameter list
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            yield os.path.basename(path), m.group(1), src[i:].lstrip()


def test_every_kernel_waits_first():
    found = list(_kernels())
    assert len(found) >= 50
    late = [(f, k) for f, k, body in found if not re.match(r"\{\s*pdl_(entry|wait)\(\);", body)]
    assert not late, late
