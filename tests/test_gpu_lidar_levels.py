"""The warp-per-ray LiDAR traversal at the tree sizes where its expansions change: a node is expanded by
four levels, the root by the levels left over, so trees of 4, 8 and 12 levels, whose root takes a
whole expansion, and those of one level more, whose root takes one.  Against the FP64 oracle with the
tolerance of test_gpu_lidar."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import scenes as S
from tests.test_gpu_lidar_warp import _compare, _node, _one_env

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# leaves of 8: 16 (levels 4) 64..128 Gaussians, 17 (5) 129; 256 (8) to 2048, 257 (9) 2049; 4096 (12) to 32,768, 4097 (13)
@pytest.mark.parametrize("n", [65, 127, 128, 129, 1025, 2047, 2048, 2049, 20_000, 32_768, 32_769])
def test_levels_by_four(n):
    rng = np.random.default_rng(n)
    _compare(_one_env([_node(rng, n, 0.5, -3.0, 0.0)]), S.lidar_pattern(7, 45, -25, 25, -30, 60, tile=None), f"n={n}")
