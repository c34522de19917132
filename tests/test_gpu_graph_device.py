"""Graph mode keeps its output buffers, and so replays, for a scene made with device="cuda" (no
index) as for one made with "cuda:0"; the images equal the eager ones bit for bit."""
import pytest

from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device", ["cuda", "cuda:0"])
def test_second_render_replays(device):
    from paper_2507_21981_gb300 import dgs as D
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    ds = DeviceScene(S.config1(seed=4, n_bg=800, n_obj=200), device=device)
    e = Renderer(mode="batched")
    ref = [t.clone() for t in e.render(ds)]
    r = Renderer(mode="graph")
    r.render(ds)
    out = r.render(ds)
    assert r.stats()["path"] == D.DGS_PATH_GRAPH and r.stats()["graph_captures"] == 1
    assert all(torch.equal(a, b) for a, b in zip(out, ref))
    e.close()
    r.close()
