"""The compositor's forms (plain, randomising, checkpointing; 14 or 16 resident blocks by the group's number
of blocks) give the same images: batches on both sides of each line, 640x480 views of 4800 blocks,
equal the per-view renders, whose groups are below all of them, bit for bit."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 6 and 7 views: 28,800 | 33,600 blocks; 10 and 11: 48,000 | 52,800; 20 and 21: 96,000 | 100,800
@pytest.mark.parametrize("n_views,form", [(6, "plain"), (7, "plain"), (10, "augment"), (11, "augment"),
                                          (20, "keep"), (21, "keep")])
def test_batch_equals_views(n_views, form):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    sc = S.config2(seed=8, n_envs=(n_views + 1) // 2, n_bg=20_000, n_obj=500, sh_degree=0)
    if n_views % 2:
        sc.cams_per_env[-1] = 1
    ds = DeviceScene(sc, device="cuda:0", spatial_order=True)
    assert ds.n_views == n_views
    outs = []
    for mode in ("plain", "batched"):
        r = Renderer(mode=mode, views_per_group=n_views, keep_lists=int(form == "keep" and mode == "batched"))
        if form == "augment":
            clip = torch.as_tensor(S.overlay_frames(1, 2, 320, 240), device="cuda:0")
            r.set_augment(S.augment_params(1, n_views, 2, 320, 240), clip)
        outs.append([t.clone() for t in r.render(ds)])
        assert r.stats()["n_groups"] == (n_views if mode == "plain" else 1)
        r.close()
    assert float(outs[0][2].max()) > 0.5
    assert all(torch.equal(a, b) for a, b in zip(*outs))
