"""The fusion kernels' split over row lengths (dgs_tsdf_integrate) against the FP64 oracle: rows
below, at and above one round of 32 voxels, one, two and four rounds per warp with remainders, both
forms of the voxel centre (row length a multiple of four or not), and view tables passed with the
launch (up to 128 views) or read from memory.  Tolerances are those of test_gpu_tsdf.py: the weight
exactly and the field within 1e-4, away from the decisions the oracle flags."""
import numpy as np
import pytest

from oracle import tsdf as T
from paper_2507_21981_gb300 import scenes as S
from tests.test_gpu_tsdf import _check, _gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,n_views", [(7, 5), (28, 5), (31, 5), (32, 40), (33, 41), (61, 5), (64, 5), (100, 5),
                                        (130, 5), (200, 5), (257, 5), (40, 128), (45, 129), (20, 129)])
def test_rows(nx, n_views):
    c = np.array([0.05, -0.1, 0.1])
    cams, Dv, Av = S.sphere_depth_views(c, 0.2, n_views=n_views, width=72, height=56, f=64.0, dist=1.0, seed=nx)
    ny, nz, vox = 13, 11, 0.5 / max(nx, 13)
    origin = (c - 0.5 * vox * np.array([nx, ny, nz]) + np.array([0.0, 0.0, 0.2])).astype(np.float32)   # across the surface
    F0, W0 = np.zeros((nz, ny, nx)), np.zeros((nz, ny, nx))
    gF, gW = _gpu(F0, W0, origin, vox, 0.04, 100.0, 0.5, cams, Dv.reshape(-1), Av.reshape(-1))
    rF, rW, amb = T.integrate(F0, W0, origin.astype(np.float64), np.float32(vox), np.float32(0.04), 100.0, 0.5, cams,
                              Dv, Av)
    _check(gF, gW, rF, rW, amb, min_seen=100)
