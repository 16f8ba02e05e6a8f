"""Any accepted number of z chunks launches every pass with a valid grid (more chunks than segments mean one each)."""
import pytest


@pytest.mark.parametrize("z_chunks", [1, 3, 64, 2 ** 31 - 1])
@pytest.mark.parametrize("precision,stencil,level", [("fp64", 0, 2), ("fp64", 0, 3), ("mixed", 0, 3), ("mixed", 1, 2), ("mixed", 1, 3)])
def test_grids(precision, stencil, level, z_chunks):
    from launch_host import Host
    h = Host(precision, n_levels=4, z_chunks=z_chunks, stencil=stencil, ir_steps=0)
    assert h.level_gradient(level, 2) == 0
    kernel = "k_tile64" if precision == "fp64" else ("k_tile32" if stencil else "k_slab")
    segments = {"k_tile64": (8 << level) // 4, "k_tile32": (8 << level) // 8, "k_slab": (8 << level) // 8}[kernel]
    fine = max(g[2] for name, g, *_ in h.launches(kernel))
    assert fine <= 2 * min(z_chunks, segments)
    h.close()
