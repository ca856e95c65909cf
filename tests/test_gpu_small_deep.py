"""Default steps of small spaces with the deepest trees, where the persistent kernel's
CTAs outnumber or nearly outnumber the configurations, against the four kernels."""
import pytest

from test_gpu_small_step import both, kt  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radices,depth", [([2], 14), ([3, 5], 14), ([7, 9, 16], 14), ([16, 16, 16], 14),
                                           ([3, 11, 16], 13), ([16, 16, 8], 13), ([3, 11, 16, 4], 13)])
def test_deep_trees(kt, radices, depth):  # noqa: F811
    both(kt, radices, 32, depth, 5, 4)
