"""The three forms of the depth sort's view key -- above the depth key (up to 16 views), packed into the
instance numbers' high bits (more), and gathered from a view array (test_fault 4 on either) -- give
the same tile lists, which the host checks in the eager renders (check_binning), and the same images
bit for bit; one view of each batch is held to the oracle."""
import pytest

from paper_2507_21981_gb300 import dgs as D
from paper_2507_21981_gb300 import scenes as S
from tests.test_gpu_failure import _check_oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["batched", "graph"])
@pytest.mark.parametrize("n_envs", [1, 8, 9, 20])        # 2, 16 | 18, 40 views
def test_gathered_view_key_equals_the_other_forms(n_envs, mode):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    sc = S.config2(seed=5, n_envs=n_envs, n_bg=20_000, n_obj=1_000, width=96, height=72, f=75.0)
    ds = DeviceScene(sc, device="cuda:0", spatial_order=True)
    outs = []
    for tf in (0, 4):
        r = Renderer(mode=mode, test_fault=tf, views_per_group=2 * n_envs, **({"check_binning": 1} if mode == "batched" else {}))
        out = r.render(ds)
        if mode == "graph":
            out = r.render(ds)
            assert r.stats()["path"] == D.DGS_PATH_GRAPH
        assert r.stats()["n_groups"] == 1 and r.stats()["n_pairs"] > 0
        outs.append([t.clone() for t in out])
        r.close()
    assert all(torch.equal(a, b) for a, b in zip(*outs))
    _check_oracle(ds.scene, ds, outs[0], v=2 * n_envs - 1)
