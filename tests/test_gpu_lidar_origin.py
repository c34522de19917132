"""A LiDAR whose origin lies exactly on a Gaussian's mean, with r_min = 0: the hit at distance 0 comes first.
Two round Gaussians on the beam, at 0 and 2 m, give D = (1 - a0) a1 2 and A = 1 - (1 - a0)(1 - a1) in
closed form; FP32 carries a few roundings of values below 2, within 1e-6.  Once by itself and once
in a dense pattern, whose packets are traced together."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import scenes as S
from tests.scene_utils import colour_sh, node, single_view
from tests.test_gpu_lidar import _trace

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dense", [False, True])
def test_hit_at_the_origin(dense):
    from paper_2507_21981_gb300.render import DeviceScene
    logits = np.array([0.3, -0.4])
    a0, a1 = 1.0 / (1.0 + np.exp(-logits))
    sc = single_view([node([[0.0, 0.0, 0.0], [2.0, 0.0, 0.0]], np.full((2, 3), np.log(0.05)), logits=logits,
                           sh=colour_sh(np.full((2, 3), 0.5)))])
    ds = DeviceScene(sc, device="cuda:0")
    dirs = np.array([[1.0, 0.0, 0.0]], np.float32)
    if dense:
        dirs = np.repeat(dirs, 256 * 256, axis=0)
    d, a = _trace(ds, np.zeros(1, np.int32), np.eye(3, 4, dtype=np.float32)[None], dirs, r_min=0.0)
    assert np.abs(d - (1 - a0) * a1 * 2.0).max() <= 1e-6
    assert np.abs(a - (1 - (1 - a0) * (1 - a1))).max() <= 1e-6
