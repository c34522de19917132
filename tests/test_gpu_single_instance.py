"""A view group whose only visible instance lies in one of its views: the depth sort then has one value,
which in groups of more than 16 views carries its view in its high bits and must lose it like any
other.  Render (eager and replayed), backward and the no-allocation render equal, bit for bit, the env
that sees the Gaussian rendered alone; the other views are background.  One 8x4 sub-tile per view,
so gradients are sums in one order."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import dgs as D
from paper_2507_21981_gb300 import scenes as S
from tests.scene_utils import colour_sh, node

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scene(n_views, seen):
    """n_views envs of one camera and one Gaussian, in front of the camera in env `seen` only."""
    nd = node([[0.1, 0.0, 0.0]], np.full((1, 3), np.log(0.15)), logits=[1.0], sh=colour_sh([[0.7, 0.3, 0.5]]))
    poses = []
    for e in range(n_views):
        P = np.eye(3, 4)
        P[2, 3] = 2.0 if e == seen else -2.0
        poses.append([P])
    cam = (8.0, 8.0, 4.0, 2.0, 8, 4, np.eye(3, 4))
    return S.scene_from_lists("single", [nd], [[0]] * n_views, poses, [[cam]] * n_views)


def _upstream():
    g = torch.Generator().manual_seed(3)
    return torch.randn((32, 3), generator=g).cuda(), torch.randn((32,), generator=g).cuda()


@pytest.mark.parametrize("n_views,seen", [(1, 0), (2, 1), (16, 15), (17, 0), (17, 16), (18, 17), (40, 33)])
def test_one_instance_in_the_group(n_views, seen):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    one = DeviceScene(_scene(1, 0), device="cuda:0")
    r = Renderer()
    ref = [t.clone() for t in r.render(one)]
    assert r.stats()["n_visible"] == 1 and float(ref[2].max()) > 0.3
    up_rgb, up_depth = _upstream()
    ref_g, ref_p = r.backward(one, ref[0], ref[1], up_rgb, up_depth)
    ds = DeviceScene(_scene(n_views, seen), device="cuda:0")
    sl = ds.view_slice(seen)

    def check(out):
        for a, b in zip(out, ref):
            assert torch.equal(a[sl], b)
            rest = a.clone()
            rest[sl] = 0
            assert not rest.any()

    out = r.render(ds)
    assert r.stats()["n_visible"] == 1 and r.stats()["n_groups"] == 1
    check(out)
    grads = [torch.zeros_like(t) for t in out[:2]]
    grads[0][sl], grads[1][sl] = up_rgb, up_depth
    g, p = r.backward(ds, out[0], out[1], *grads)
    assert all(torch.equal(g[0][k], ref_g[0][k]) for k in g[0])
    assert torch.equal(p[seen], ref_p[0]) and float(p[seen].abs().max()) > 0
    gr = Renderer(mode="graph")
    gr.render(ds)
    check(gr.render(ds))
    assert gr.stats()["path"] == D.DGS_PATH_GRAPH
    flat = tuple(torch.full_like(t, -1.0) for t in out)
    rc = D.dgs_render_noalloc(r.options, ds.nodes, ds.n_nodes, ds.env_node_ids, ds.n_envs, ds.max_nodes, ds.node_poses,
                              ds.cams, ds.cams_per_env, ds.max_cams, *flat, None,
                              torch.cuda.current_stream().cuda_stream)
    assert rc == D.DGS_OK
    torch.cuda.synchronize()
    check(flat)
    r.close()
    gr.close()
