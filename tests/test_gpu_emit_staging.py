"""SH coefficients at a 16-byte aligned address (read in vectors where a vector holds coefficients of
one Gaussian) and one element further on (read one by one) give the same images bit for bit, and the
same gradients up to the order of the atomic additions, for every degree and storage type and a
Gaussian count that ends inside a 32-Gaussian chunk."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import scenes as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("degree", [0, 1, 2, 3])
def test_aligned_and_unaligned_coefficients_agree(degree, dtype):
    from paper_2507_21981_gb300.render import DeviceScene, GradBuffers, Renderer
    sc = S.config1(seed=13, n_bg=1003, n_obj=37)
    rng = np.random.default_rng(5)
    for nd in sc.nodes:
        nd.sh = (rng.standard_normal((nd.n, (degree + 1) ** 2, 3)) * 0.2).astype(np.float32)
        nd.sh_degree = degree
    ds = DeviceScene(sc, device="cuda:0", dtype=dtype)
    r = Renderer()
    up = torch.as_tensor(rng.standard_normal((ds.n_pixels, 3)).astype(np.float32)).cuda()
    out = r.render(ds)
    ga = GradBuffers(ds)
    r.backward(ds, out[0], out[1], up, out=ga)
    keep = []
    for k in range(ds.n_nodes):
        sh = ds.tensors[k]["sh"]
        moved = torch.empty(sh.numel() + 8, dtype=sh.dtype, device=sh.device)
        assert moved.data_ptr() % 16 == 0 and sh.data_ptr() % 16 == 0
        moved[1:1 + sh.numel()] = sh.reshape(-1)
        ds.nodes[k].sh = moved.data_ptr() + sh.element_size()
        keep.append(moved)
    out2 = r.render(ds)
    assert all(torch.equal(a, b) for a, b in zip(out, out2))
    # the SH gradients one element off a 16-byte boundary too
    gb = GradBuffers(ds)
    for k in range(ds.n_nodes):
        g = torch.zeros(ds.tensors[k]["sh"].numel() + 8, device="cuda:0")
        gb.arr[k].sh = g.data_ptr() + 4
        gb.node_grads[k]["sh"] = g[1:1 + ds.tensors[k]["sh"].numel()].view(ds.tensors[k]["sh"].shape)
        keep.append(g)
    r.backward(ds, out[0], out[1], up, out=gb)
    # both sum the same FP32 terms, at most some thousand per entry, in another order
    for a, b in zip(ga.node_grads, gb.node_grads):
        for name in GradBuffers.NAMES:
            scale = float(a[name].abs().max())
            assert float((a[name] - b[name]).abs().max()) <= 2e-5 * scale, name
    assert float(ga.node_grads[0]["sh"].abs().max()) > 0
    r.close()
