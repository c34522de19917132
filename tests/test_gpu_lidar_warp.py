"""The warp-per-ray LiDAR traversal at the sizes where it can go wrong: trees whose level counts
do and do not divide by five (one leaf up to four expansions), more slots than one batch of
roots, and rays with more hits in one place than the pending buffer holds (so that it is cut and
further rounds resume), among them hits at exactly the same distance.  Against the FP64 oracle
with the tolerance of test_gpu_lidar."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import scenes as S
from tests.test_gpu_lidar import _check, _oracle, _trace

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _node(rng, n, half, log_scale, logit, centre=(1.0, 0.0, 0.0)):
    nd = S.uniform_cube_node(rng, n, half, log_scale, 0.3, logit, 0.3, 0, None)
    nd.mean[:] += np.asarray(centre, np.float32)
    return nd


def _one_env(nodes, poses=None):
    cam = (50.0, 50.0, 16.0, 16.0, 32, 32, np.eye(3, 4))
    return S.scene_from_lists("warp", nodes, [list(range(len(nodes)))], [poses or [np.eye(3, 4)] * len(nodes)], [[cam]])


def _compare(sc, dirs, what, zorder=True):
    from paper_2507_21981_gb300.render import DeviceScene
    ds = DeviceScene(sc, device="cuda:0", spatial_order=zorder)
    se, sp = np.zeros(1, np.int32), np.eye(3, 4, dtype=np.float32)[None]
    d, a = _trace(ds, se, sp, dirs)
    ref = _oracle(ds.scene, se, sp, dirs)
    assert (ref.a > 0.01).any()
    _check(d, a, ref, what)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 16, 17, 255, 256, 257, 512, 513, 4096, 8193, 40_000])
def test_tree_sizes(n):
    rng = np.random.default_rng(n)
    _compare(_one_env([_node(rng, n, 0.5, -3.0, 0.0)]), S.lidar_pattern(7, 45, -25, 25, -30, 60, tile=None), f"n={n}")


@pytest.mark.parametrize("K", [31, 32, 33, 70])
def test_many_slots(K):
    rng = np.random.default_rng(K)
    nodes = [_node(rng, int(rng.integers(1, 60)), 0.3, -2.5, 0.0) for _ in range(K)]
    poses = [S.random_pose(rng, 0.3) for _ in range(K)]
    for P in poses:
        P[0, 3] += 1.5
    _compare(_one_env(nodes, poses), S.lidar_pattern(6, 40, -30, 30, -40, 80, tile=None), f"K={K}")


@pytest.mark.parametrize("n,spread", [(90, 0.0), (97, 0.0), (300, 0.0), (1000, 0.0), (1000, 0.02), (3000, 0.3)])
def test_more_hits_than_the_pending_buffer(n, spread):
    """n faint Gaussians of one place (spread 0: the same mean, so the same t* on every ray up to
    their shapes; all rays hit all of them), stored in random order."""
    rng = np.random.default_rng(n)
    nd = _node(rng, n, max(spread, 1e-9), -1.5, -4.2)
    if spread == 0.0:
        nd.mean[:] = [1.0, 0.0, 0.0]
        nd.log_scale[:] = -1.5
    _compare(_one_env([nd]), S.lidar_pattern(5, 24, -12, 12, -12, 24, tile=None), f"n={n} spread={spread}", zorder=False)
