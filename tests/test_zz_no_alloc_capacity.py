"""Batches that fill dgs_render_noalloc's 64 MiB almost to the last: many (view, slot) entries, most of
them empty (132 bytes of tables each are allowed for), and few instances of very many tile pairs on
a grid of 16 tile bits (16 1/3 bytes a pair), where the two passes of the tile sort share one
look-back region.  Both must fit, and equal dgs_render bit for bit."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import dgs as D
from paper_2507_21981_gb300 import scenes as S
from tests.scene_utils import colour_sh, node

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _compare(sc, **opts):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    ds = DeviceScene(sc, device="cuda:0")
    r = Renderer(mode="batched", **opts)
    ref = r.render(ds)
    assert float(ref[2].max()) > 0.1
    out = tuple(torch.full_like(t, -1.0) for t in ref)
    rc = D.dgs_render_noalloc(r.options, ds.nodes, ds.n_nodes, ds.env_node_ids, ds.n_envs, ds.max_nodes, ds.node_poses,
                              ds.cams, ds.cams_per_env, ds.max_cams, *out, None, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert rc == D.DGS_OK, D.STATUS_NAMES.get(rc, rc)
    assert all(torch.equal(a, b) for a, b in zip(out, ref))
    st = r.stats()
    r.close()
    return st


def test_many_empty_slots():
    n_envs, slots = 1000, 503                       # 503,000 entries: 66.4 of 67.1 MB at 132 bytes
    nd = node([[0.0, 0.0, 2.0]], np.full((1, 3), np.log(0.3)), logits=[1.0], sh=colour_sh([[0.7, 0.3, 0.5]]))
    cam = (8.0, 8.0, 4.0, 2.0, 8, 4, np.eye(3, 4))
    sc = S.scene_from_lists("slots", [nd], [[0]] * n_envs, [[np.eye(3, 4)]] * n_envs, [[cam]] * n_envs)
    ids = np.full((n_envs, slots), -1, np.int32)
    ids[:, 0] = sc.env_node_ids[:, 0]
    poses = np.tile(np.eye(3, 4), (n_envs, slots, 1, 1))
    sc.env_node_ids, sc.node_poses = ids, poses
    _compare(sc)


def test_many_pairs_per_instance():
    # 66 splats wider than the image, 2048 x 1920 in tiles of 8x8: 66 x 61,440 pairs
    n = 66
    means = np.stack([np.linspace(-0.1, 0.1, n), np.zeros(n), 2.0 + 0.01 * np.arange(n)], axis=1)
    rgb = np.random.default_rng(0).uniform(0, 1, (n, 3))
    nd = node(means, np.full((n, 3), np.log(4.0)), logits=np.full(n, -4.0), sh=colour_sh(rgb))
    cam = (1800.0, 1800.0, 1024.0, 960.0, 2048, 1920, np.eye(3, 4))
    sc = S.scene_from_lists("pairs", [nd], [[0]], [[np.eye(3, 4)]], [[cam]])
    st = _compare(sc, tile_w=8, tile_h=8)
    assert st["n_pairs"] == n * 61_440 and st["key_bits"] == 16
