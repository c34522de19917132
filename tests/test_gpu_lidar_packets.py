"""Dense beam patterns, whose packets of 32 neighbouring rays are traced together, against the same rays
traced one by one (a call of fewer than 65,536 rays takes no packets), bit for bit: patterns with packets
on both sides of the cone, ray counts that are no multiple of 32 and cross sensors within a
packet, sensors that see different nodes, rays with more hits than a packet's buffer, and trees of one
leaf.  The one-by-one form is held to the oracle in test_gpu_lidar.py."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import dgs as D
from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scene(rng, logit=0.0, ls=-3.0, n=(4000, 7, 900)):
    nodes = []
    for k, m in enumerate(n):
        nd = S.uniform_cube_node(rng, m, 0.6, ls, 0.4, logit, 0.5, 0, None)
        nd.mean[:] += np.asarray([1.5 + k, 0.0, 0.0], np.float32)
        nodes.append(nd)
    I = np.eye(3, 4)
    cam = (50.0, 50.0, 16.0, 16.0, 32, 32, I)
    return S.scene_from_lists("packets", nodes, [[0, 1, 2], [0, 2]], [[I, I, I], [I, S.random_pose(rng, 0.3)]],
                              [[cam], [cam]])


def _trace(r, ds, env, pose, dirs):
    out = r.lidar_trace(ds, D.lidar_sensors(np.asarray(env, np.int32), np.asarray(pose, np.float32)), None, dirs)
    return [t.cpu() for t in out]


@pytest.mark.parametrize("channels,azimuths,span,envs,logit,ls", [
    (256, 256, 20.0, [0], 0.0, -3.0),            # every packet inside the cone
    (256, 256, 21.46, [0], 0.0, -3.0),           # two thirds of them
    (256, 256, 21.48, [0], 0.0, -3.0),           # fewer than half: none is taken
    (256, 256, 90.0, [0], 0.0, -3.0),            # none
    (200, 173, 6.0, [0, 1], 0.0, -3.0),          # 34,600 rays a sensor: packets across two, and a cut one
    (257, 256, 2.0, [1], 1.5, -2.0),
    (192, 256, 6.0, [0, 1, 0], -4.2, -1.0),      # far more than 32 hits a ray: packets given up
])
def test_packets_equal_single_rays(channels, azimuths, span, envs, logit, ls):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    rng = np.random.default_rng(channels)
    ds = DeviceScene(_scene(rng, logit, ls), device="cuda:0", spatial_order=True)
    r = Renderer()
    r.lidar_build(ds)
    d = S.lidar_pattern(channels, azimuths, -span / 4, span / 4, -span / 2, span)
    dirs = torch.as_tensor(d, device="cuda:0")
    pose = np.tile(np.eye(3, 4)[None], (len(envs), 1, 1))
    pose[:, 1, 3] = 0.05 * np.arange(len(envs))
    got = _trace(r, ds, envs, pose, dirs)
    assert r.launches() == 3                     # setup, packets, rays
    assert len(envs) * len(d) >= 65536 and float(got[1].max()) > 0.3
    for s in range(len(envs)):
        for a in range(0, len(d), 30000):
            ref = _trace(r, ds, envs[s:s + 1], pose[s:s + 1], dirs[a:a + 30000])
            assert r.launches() == 2
            for x, y in zip(got, ref):
                assert torch.equal(x[s, a:a + 30000], y[0]), (s, a)
    r.close()
