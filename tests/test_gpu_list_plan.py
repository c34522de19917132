"""Batches at the edges of the list building's plan render as their envs do one by one, bit for bit:
count tables of one scan partition (4096 entries) less, exactly and more, and 16 and 18 views, the
last whose view fits above the depth key in 32 bits and the first whose view is a key of its own.
(An env alone takes other sizes of every list: its count table is a 64th, its depth key holds two
views.)"""
import pytest

from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _env(sc, e):
    s = slice(e, e + 1)
    return S.Scene(sc.name, sc.nodes, sc.env_node_ids[s], sc.node_poses[s], sc.cams_per_env[s], sc.cam_intr[s],
                   sc.cam_res[s], sc.cam_pose[s], sc.meta)


@pytest.mark.parametrize("n_envs,n_bg", [(32, 62 * 32), (32, 63 * 32), (32, 64 * 32 - 5), (32, 64 * 32 + 1),
                                         (8, 3000), (9, 3000)])
@pytest.mark.parametrize("mode", ["batched", "graph"])
def test_batch_equals_its_envs(n_envs, n_bg, mode):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    # two cameras per env; one object of a single chunk: (chunks of the background + 1) x 2 n_envs entries
    sc = S.config2(seed=21, n_envs=n_envs, n_bg=n_bg, n_obj=32, n_objects=1, width=96, height=64, sh_degree=1)
    ds = DeviceScene(sc, device="cuda:0")
    r, one = Renderer(mode=mode), Renderer(mode="batched")
    r.render(ds)
    out = r.render(ds)
    assert float(out[2].max()) > 0
    at = 0
    for e in range(n_envs):
        de = DeviceScene(_env(sc, e), device="cuda:0")
        ref = one.render(de)
        for a, b in zip(out, ref):
            assert torch.equal(a[at:at + de.n_pixels], b), e
        at += de.n_pixels
    r.close()
    one.close()
