"""The Gaussian draws' radius, which every kernel that draws G forms without a
branch: bit for bit sqrtf's, for all 2^24 values that it is taken of."""
import pytest

pytestmark = pytest.mark.gpu


def test_radius_is_the_correctly_rounded_root():
    import paper_2203_02798_gb300 as lsk
    assert lsk.debug_radius() == 0
