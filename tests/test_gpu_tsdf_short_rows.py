"""The fusion's two forms (rows in segments of 128 voxels; voxels in storage order, whatever their rows)
at the edges between them, where a row's last segment leaves a sixteenth of its lanes idle, and
at rows of a few voxels, against the FP64 oracle.  Tolerances are those of test_gpu_tsdf.py."""
import numpy as np
import pytest

from oracle import tsdf as T
from paper_2507_21981_gb300 import scenes as S
from tests.test_gpu_tsdf import _check, _gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [1, 3, 4, 31, 32, 119, 120, 121, 127, 128, 129, 240, 241, 256])
def test_row_lengths(nx):
    c = np.array([0.05, -0.1, 0.1])
    cams, Dv, Av = S.sphere_depth_views(c, 0.2, n_views=5, width=72, height=56, f=64.0, dist=1.0, seed=nx)
    ny, nz, vox = 13, 11, 0.5 / max(nx, 13)
    origin = (c - 0.5 * vox * np.array([nx, ny, nz]) + np.array([0.0, 0.0, 0.2])).astype(np.float32)   # across the surface
    F0, W0 = np.zeros((nz, ny, nx)), np.zeros((nz, ny, nx))
    gF, gW = _gpu(F0, W0, origin, vox, 0.04, 100.0, 0.5, cams, Dv.reshape(-1), Av.reshape(-1))
    rF, rW, amb = T.integrate(F0, W0, origin.astype(np.float64), np.float32(vox), np.float32(0.04), 100.0, 0.5, cams,
                              Dv, Av)
    _check(gF, gW, rF, rW, amb, min_seen=20)
