"""The upward scan's choice of tile for a leaf, at the line (2^19 groups)."""
import pytest

from tests import test_gpu_up_tiles as tiles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf", [(1 << 19) - 1, 1 << 19, (1 << 19) + 2047])
def test_groups_at_the_line(leaf):
    tiles.test_groups(leaf, 3001)
