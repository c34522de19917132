"""Upstream gradients that are NaN or infinite (a masked division's 0 times infinity, at pixels that no
Gaussian covers) reach the Gaussians that touch their pixel and no others: a sub-tile of covered and
uncovered pixels gives, with NaN or infinity at the uncovered ones, bit for bit the gradients that it
gives with zeros there.  The image is one 8x4 sub-tile, so every accumulator is added to once per
batch and the sums have one order.  List lengths lie around the adjoint's batches (16 and 32)."""
import numpy as np
import pytest

from tests.scene_utils import colour_sh, node, single_view

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _splats(us, z0=2.0):
    """One Gaussian per projected column us[i] of an 8x4 image (f = 8), 0.7 px wide, at growing depths."""
    us = np.asarray(us, np.float64)
    z = z0 + 0.01 * np.arange(len(us))
    means = np.stack([(us - 4.0) * z / 8.0, np.zeros(len(us)), z], axis=1)
    rgb = np.tile([0.8, 0.4, 0.6], (len(us), 1))
    return single_view([node(means, np.full((len(us), 3), np.log(0.1)), logits=np.full(len(us), -2.5),
                             sh=colour_sh(rgb))], f=8.0, W=8, H=4)


def _grads(sc, up_rgb, up_depth, keep):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer
    ds = DeviceScene(sc, device="cuda:0")
    r = Renderer(keep_lists=keep)
    rgb, depth, alpha = r.render(ds)
    g, poses = r.backward(ds, rgb, depth, up_rgb.cuda(), up_depth.cuda())
    out = [t.cpu() for n in g for t in n.values()] + [poses.cpu()]
    r.close()
    return alpha.cpu(), out


def _upstream(seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randn((32, 3), generator=g), torch.randn((32,), generator=g)


@pytest.mark.parametrize("keep", [0, 1])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("n", [1, 4, 17, 33])
def test_uncovered_pixels_do_not_matter(n, bad, keep):
    sc = _splats(np.linspace(1.0, 2.5, n))
    rgb, depth = _upstream(n)
    alpha, _ = _grads(sc, rgb, depth, keep)
    out = alpha == 0
    assert 4 <= int(out.sum()) < 28
    rgb[out], depth[out] = 0.0, 0.0
    _, ref = _grads(sc, rgb, depth, keep)
    assert all(bool(torch.isfinite(t).all()) for t in ref) and float(ref[0].abs().max()) > 0
    rgb[out], depth[out] = bad, bad
    _, got = _grads(sc, rgb, depth, keep)
    for a, b in zip(got, ref):
        assert torch.equal(a, b)


def test_a_covered_pixel_reaches_its_own_gaussian_only():
    sc = _splats([1.0, 7.0])                          # three sigmas (2.1 px) apart from each other's pixels
    rgb, depth = _upstream(5)
    _, ref = _grads(sc, rgb, depth, 0)
    rgb[8], depth[8] = float("nan"), float("nan")     # column 0 of the second row: the first Gaussian's
    _, got = _grads(sc, rgb, depth, 0)
    assert bool(torch.isnan(got[0][0]).any()) and bool(torch.isnan(got[4][0]).any())
    for a, b in zip(got[:5], ref[:5]):
        assert torch.equal(a[1], b[1])
