"""The adjoint compositor's batches against the FP64 oracle's adjoint: lists that end below, at and
above a step of 4, a replay of 16, a batch of 32 and a scan step of 128 records, translucent so
that no pixel ends, on an image whose second tile is cut.  Tolerances are those of
test_gpu_backward.py."""
import numpy as np
import pytest

from paper_2507_21981_gb300 import scenes as S
from tests.test_gpu_backward import _compare, _gradients

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4, 5, 15, 16, 17, 31, 32, 33, 63, 65, 127, 130])
def test_list_lengths(n):
    sc = S.config1(seed=40 + n, n_bg=n, n_obj=1)
    for nd in sc.nodes:
        nd.mean = (nd.mean * np.float32(0.15)).astype(np.float32)
        nd.log_scale = np.full_like(nd.log_scale, -1.2) + (nd.log_scale - nd.log_scale.mean()) * np.float32(0.2)
        nd.opacity_logit = np.full_like(nd.opacity_logit, -3.0)
    sc.cam_res[:] = (24, 16)
    sc.cam_intr[:] = (30.0, 30.0, 12.0, 8.0)
    node_grads, gposes, ref = _gradients(sc, seed=n)
    assert max(float(g["sh"].abs().max()) for g in node_grads) > 0
    _compare(sc, node_grads, gposes, ref)
