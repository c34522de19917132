"""The autograd function with a graph-mode renderer, whose render() hands out the same tensors every
call: two forwards of equal pixel count before one backward give each scene the gradients that a
batched renderer gives it, and the renderer's own tensors stay out of the autograd graph.  Gradients
are sums of floating-point additions in no fixed order: within 1e-3 of an entry plus 1e-5 of the
largest, the bound that test_gpu_backward.py puts beside its error model."""
import pytest

from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _grads(mode, device):
    from paper_2507_21981_gb300.render import DeviceScene, Renderer, render_differentiable
    r = Renderer(mode=mode)
    scenes, params, outs = [], [], []
    for seed in (11, 12):
        ds = DeviceScene(S.config1(seed=seed, n_bg=600, n_obj=200, res=48, f=41.0), device=device)
        ps = ds.param_list()
        for p in ps:
            p.requires_grad_(True)
        scenes.append(ds)
        params.append([*ps, ds.node_poses.clone().requires_grad_(True)])
    for _ in range(2):                        # the second round replays where the mode does
        outs = [render_differentiable(r, ds, ps[-1]) for ds, ps in zip(scenes, params)]
    loss = sum((rgb * rgb).sum() + depth.sum() for rgb, depth, _ in outs)
    grads = [torch.autograd.grad(loss, ps, retain_graph=True) for ps in params]
    plain = r.render(scenes[0])
    assert not any(t.requires_grad for t in plain)
    plain[0].cpu().numpy()
    images = [t.detach().clone() for o in outs for t in o]
    r.close()
    return grads, images


@pytest.mark.parametrize("device", ["cuda", "cuda:0"])
def test_two_forwards_before_the_backward(device):
    got, images = _grads("graph", device)
    ref, ref_images = _grads("batched", device)
    assert all(torch.equal(a, b) for a, b in zip(images, ref_images))
    assert not torch.equal(images[0], images[3])
    for gs, rs in zip(got, ref):
        for a, b in zip(gs, rs):
            assert torch.allclose(a, b, rtol=1e-3, atol=1e-5 * float(b.abs().max()))
