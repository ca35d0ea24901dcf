"""The row generators and the truncation at the sizes where their tilings can
go wrong: lists shorter than a warp's share, remainders, windows and images
outside the usual ones."""
import numpy as np
import pytest
import torch

from paper_1607_06170_gb300 import inputs as I
from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_1607_06170_gb300 import build, psf

    build.build()
    return psf


@pytest.mark.parametrize("Wt,nx,ny,dx,k", [(3, 21, 13, 1.0, 59), (4, 7, 9, 3.0, 120), (2, 18, 19, 7.0, 250),
                                           (0, 5, 5, 2.0, 61)])
def test_voxel_driven_shapes(P, orc, Wt, nx, ny, dx, k):
    """Pixel counts that leave a remainder, few lines (threads share one), a
    window of either array length, pixels beyond the ring polygon (7 mm)."""
    w = I.workload("RING2D")
    s, t, ls = w["scanner"], w["table"], w["lors"]
    im = I.image(nx, ny, 1, dx, dx, 1.0)
    T, eta = P.response_build(s, t)
    To, _ = orc.table_build(s, t)
    A = P.voxel_homog(s, t, T, eta, im, ls, k, Wt).cpu().numpy()
    Ao, margin = orc.voxel_homog(s, t, To, im, I.workload_lors(w), k, Wt)
    assert margin.min() > 1e-5  # no response decision within reach of FP32 rounding
    scale = np.abs(Ao).max(0, keepdims=True)
    assert_close(A, Ao, 1e-5, 1e-6 * scale + 1e-30, "voxel-driven A")
