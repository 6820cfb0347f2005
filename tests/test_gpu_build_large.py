"""The line between treelets restructured by a warp and by a thread: the four-wide
tree of the scenes on both sides of it, and of a much larger one, reaches every
triangle once."""
import pytest

from tests import test_gpu_build_edges as edges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, shape", [(400000, "even"), (400001, "even"), (400001, "cluster"), (1000003, "chain")])
def test_both_sides_of_the_line(n, shape):
    edges.test_four_wide_tree_reaches_every_triangle_once(n, shape)
