"""The vectors of a solve lie side by side in its scratch on every grid that a context accepts (2^3 to 1024^3)."""
import pytest


@pytest.mark.parametrize("elem", [4, 8])
@pytest.mark.parametrize("N", [2 << j for j in range(10)])
def test_vectors_do_not_overlap(N, elem):
    from launch_host import load
    for S in (1, 3):
        assert load().fake_check_carve(N, S, elem) == 0
