"""Fusing views of very different sizes (dgs_tsdf_integrate), whose depths one pass normalises packed
1024 pixels to a block: views of one pixel up to more than a block, at offsets with gaps, 1, 3 and
130 of them (the last read from the view table).  One call equals, bit for bit, a call per view: the
field and the weight hold a voxel's whole state between views."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (3, 2), (160, 120), (7, 5), (33, 31), (32, 32), (1, 40), (64, 16), (250, 3)]


def _views(n_views):
    rng = np.random.default_rng(n_views)
    cams, offs, at = [], [], 5
    for v in range(n_views):
        w, h = SIZES[v % len(SIZES)] if n_views > 1 else (160, 120)
        az = 2 * np.pi * v / n_views
        P = S.look_at(np.array([np.cos(az), np.sin(az), 0.2]), np.zeros(3))
        cams.append((float(w), float(w), w / 2.0, h / 2.0, w, h, P.astype(np.float32)))
        offs.append(at)
        at += w * h + int(rng.integers(0, 9))
    depth = rng.uniform(0.8, 1.1, at).astype(np.float32)
    alpha = (rng.random(at) > 0.2).astype(np.float32)
    return cams, np.asarray(offs, np.int64), depth * alpha, alpha


@pytest.mark.parametrize("n_views", [1, 3, 9, 130])
def test_one_call_equals_a_call_per_view(n_views):
    from paper_2507_21981_gb300 import dgs as D
    from paper_2507_21981_gb300.render import Renderer
    cams, offs, depth, alpha = _views(n_views)
    d, a = torch.as_tensor(depth).cuda(), torch.as_tensor(alpha).cuda()
    r = Renderer()
    stream = torch.cuda.current_stream().cuda_stream
    fields = []
    for calls in ([slice(0, n_views)], [slice(v, v + 1) for v in range(n_views)]):
        F, W = torch.zeros((20, 18, 37), device="cuda"), torch.zeros((20, 18, 37), device="cuda")
        for s in calls:
            rc = D.dgs_tsdf_integrate(r.ctx, F, W, 37, 18, 20, [-0.25, -0.12, -0.13], 0.0135, 0.05, 100.0, 0.5,
                                      D.cameras(cams[s]), len(cams[s]), d, a, np.ascontiguousarray(offs[s]), stream)
            assert rc == D.DGS_OK, D.dgs_last_error(r.ctx)
        fields.append((F, W))
    assert float(fields[0][1].max()) >= 1
    assert all(torch.equal(x, y) for x, y in zip(*fields))
    r.close()
