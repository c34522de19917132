"""The count scan's bounded look-back running out: dgs_options.test_fault = 1 mutes its second partition
of 4096 entries, so a table of three and more waits in vain.  The eager render, the backward and the
no-allocation render stop with DGS_ERR_TIMEOUT before anything is written through the offsets, and
with the fault cleared the same context renders what a fresh one does.  A replay whose depth sort
runs out (its captured capacity holds a third partition that the first call's count did not need)
reports it too.  No wait is longer than spin_limit_us a wave of blocks."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import dgs as D
from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunks", [4096 * 2 + 1, 4096 * 3])
def test_count_scan_wait_runs_out(chunks):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    # one view whose count table has chunks + 1 entries (the object's one): a last partition of two
    # entries, or of one
    sc = S.config1(seed=6, n_bg=chunks * 32, n_obj=20, res=64, f=55.0)
    sc.nodes[0].mean[:, 2] -= 8.0
    sc.nodes[0].mean[:500, 2] += 8.0                 # few in front of the camera
    ds = DeviceScene(sc, device="cuda:0")
    fresh = Renderer()
    ref = fresh.render(ds)
    assert 0 < fresh.stats()["n_visible"] < 3072     # one partition of the sort: its wait has none before it
    r = Renderer(spin_limit_us=2000, test_fault=1)
    with pytest.raises(D.DgsError) as ei:
        r.render(ds)
    assert ei.value.code == D.DGS_ERR_TIMEOUT and "count scan" in str(ei.value)
    with pytest.raises(D.DgsError) as ei:
        r.backward(ds, ref[0], ref[1], torch.ones_like(ref[0]))
    assert ei.value.code == D.DGS_ERR_TIMEOUT
    out = tuple(torch.zeros_like(t) for t in ref)

    def noalloc():
        return D.dgs_render_noalloc(r.options, ds.nodes, ds.n_nodes, ds.env_node_ids, ds.n_envs, ds.max_nodes,
                                    ds.node_poses, ds.cams, ds.cams_per_env, ds.max_cams, *out, None,
                                    torch.cuda.current_stream().cuda_stream)

    assert noalloc() == D.DGS_ERR_TIMEOUT
    r.set_options(test_fault=0)
    got = r.render(ds)
    assert noalloc() == D.DGS_OK
    torch.cuda.synchronize()
    for a, b, c in zip(got, ref, out):
        assert torch.equal(a, b) and torch.equal(c, b)
    r.close()
    fresh.close()


def test_replayed_sort_wait_runs_out():
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    # 6000 instances fill two partitions of the depth sort (nobody waits behind the muted one); 6500 need
    # three and still fit the captured 1.25 x 6000 + 1024
    sc = S.config1(seed=7, n_bg=6000, n_obj=500, res=64, f=40.0)
    for nd in sc.nodes:
        nd.mean *= np.float32(0.2)
    ds = DeviceScene(sc, device="cuda:0")
    poses = ds.node_poses.clone()
    away = poses.clone()
    away[0, 1, 11] = -50.0                            # the object behind the camera
    r = Renderer(mode="graph", spin_limit_us=2000, test_fault=1)
    ds.node_poses.copy_(away)
    r.render(ds)
    ref = [t.clone() for t in r.render(ds)]
    assert r.stats()["path"] == D.DGS_PATH_GRAPH and r.stats()["n_visible"] == 6000
    ds.node_poses.copy_(poses)
    with pytest.raises(D.DgsError) as ei:
        r.render(ds)
    assert ei.value.code == D.DGS_ERR_TIMEOUT and "scan or sort" in str(ei.value)
    ds.node_poses.copy_(away)
    again = r.render(ds)
    assert r.stats()["path"] == D.DGS_PATH_GRAPH
    assert all(torch.equal(a, b) for a, b in zip(again, ref))
    r.close()
