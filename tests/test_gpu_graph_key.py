"""Graph mode on batches of one structure whose captured values differ: equal totals (pixels, tiles,
count-table entries, buffers) but other tile bits of the keys, another first tile of the second view
group, or another first count-table entry of it.  Each is captured anew and renders what an eager
renderer does, bit for bit; a batch that differs in none of these replays."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import dgs as D
from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _scene(sizes, n_a=1500, n_b=300):
    """One env per view size, a camera each; nodes a and b, the former in even envs, the latter in odd."""
    rng = np.random.default_rng(5)
    nodes = [S.uniform_cube_node(rng, n, 1.0, -2.5, 0.3, 0.5, 0.5, 0, None) for n in (n_a, n_b)]
    I = np.eye(3, 4)
    P = np.eye(3, 4)
    P[2, 3] = 4.0
    cams = [[(0.9 * w, 0.9 * w, w / 2.0, h / 2.0, w, h, P)] for w, h in sizes]
    return S.scene_from_lists("key", nodes, [[e % 2] for e in range(len(sizes))], [[I]] * len(sizes), cams)


def _render(r, ds):
    out = [t.clone() for t in r.render(ds)]
    return out, r.stats()


def _set_sizes(ds, sizes):
    for cam, (w, h) in zip(ds.cams, sizes):
        cam.width, cam.height = w, h
        cam.fx = cam.fy = 0.9 * w
        cam.cx, cam.cy = w / 2.0, h / 2.0


def _check(first, change, views_per_group):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    ds = DeviceScene(first, device="cuda:0")
    opts = dict(views_per_group=views_per_group)
    g, e = Renderer(mode="graph", **opts), Renderer(mode="batched", **opts)
    _render(g, ds)
    out, st = _render(g, ds)
    assert st["path"] == D.DGS_PATH_GRAPH and st["n_groups"] == (2 if views_per_group else 1)
    assert all(torch.equal(a, b) for a, b in zip(out, _render(e, ds)[0]))
    change(ds)
    for path in (D.DGS_PATH_CAPTURED, D.DGS_PATH_GRAPH):
        out, st = _render(g, ds)
        ref, _ = _render(e, ds)
        assert all(torch.equal(a, b) for a, b in zip(out, ref)) and float(ref[2].max()) > 0
        assert st["path"] == path
    g.close()
    e.close()


@pytest.mark.parametrize("views_per_group", [0, 1])
def test_other_tile_bits(views_per_group):
    # 60 + 60 tiles of 16x16 (6 bits and the dead index), then 100 + 20 (7): 30720 pixels either way
    _check(_scene([(160, 96), (160, 96)]), lambda ds: _set_sizes(ds, [(160, 160), (80, 64)]), views_per_group)


def test_sizes_swapped_across_the_groups():
    _check(_scene([(160, 96), (80, 64)]), lambda ds: _set_sizes(ds, [(80, 64), (160, 96)]), 1)


def test_node_tables_swapped_across_the_groups():
    def swap(ds):
        ds.env_node_ids[:] = ds.env_node_ids[::-1].copy()
    _check(_scene([(160, 96), (160, 96)]), swap, 1)


def test_sizes_swapped_within_a_group_replay():
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    ds = DeviceScene(_scene([(160, 96), (80, 64)]), device="cuda:0")
    g, e = Renderer(mode="graph"), Renderer(mode="batched")
    _render(g, ds)
    _set_sizes(ds, [(80, 64), (160, 96)])
    ref = _render(e, ds)[0]
    for _ in range(2):                       # (the first may outgrow the captured sizes and capture again)
        out, st = _render(g, ds)
        assert all(torch.equal(a, b) for a, b in zip(out, ref))
    assert st["path"] == D.DGS_PATH_GRAPH
    g.close()
    e.close()
