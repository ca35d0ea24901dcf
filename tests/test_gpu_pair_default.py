"""Which form an untuned plan with a declared grid projects with: pair-streamed
where a transaxial pair has enough rows and voxels, row by row otherwise; the same
values either way."""
import pytest
import torch

from paper_1607_06170_gb300 import inputs as I
from parity import assert_close

pytestmark = pytest.mark.gpu


def _case(name):
    """(scanner, LOR set, image, window, forward streamed?, back streamed?)"""
    w = I.workload("RING3D")
    ring2, ls = dict(w["scanner"], n_block_rings=2), dict(fan_half=12, max_ring_diff=15)
    ring1 = dict(w["scanner"], n_block_rings=1)
    return {
        # 1 row a pair
        "planar": (I.workload("RING2D")["scanner"], I.workload("RING2D")["lors"],
                   I.workload("RING2D")["image"], (3, 0), False, False),
        # 13 rows (direct planes only), 2,964 pairs
        "direct planes": (ring1, dict(fan_half=9, max_ring_diff=0), I.image(160, 160, 26, 0.8, 0.8, 1.1),
                          (1, 0), False, False),
        # 566 rows, 3,900 pairs: 566 (60 + 72) = 74,712 and 566 (160 + 160) = 181,120
        "coarse grid": (ring2, ls, I.image(60, 72, 26, 2.0, 2.0, 2.2), (1, 0), False, True),
        "fine grid": (ring2, ls, I.image(160, 160, 52, 0.8, 0.8, 1.1), (1, 0), True, True),
        # 504 pairs: at most four an SM
        "few pairs": (I.workload("RING3D_SMALL")["scanner"], I.workload("RING3D_SMALL")["lors"],
                      I.workload("RING3D_SMALL")["image"], (1, 0), True, True),
    }[name]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("name", ["planar", "direct planes", "coarse grid", "fine grid", "few pairs"])
def test_default_form(name, dtype):
    from paper_1607_06170_gb300 import build, psf as P

    build.build()
    s, ls, im, win, fwd, back = _case(name)
    tb = I.workload("RING2D" if name == "planar" else "RING3D_SMALL" if name == "few pairs" else
                    "RING3D")["table"]
    T, eta = P.response_build(s, tb)
    W = P.bin_spread_classes(s, tb, T, eta, ls, P.lor_set_classes(s, ls), *win)
    rows = P.sysmat_rows_set_typed(s, im, ls, dtype)
    nv = im["nx"] * im["ny"] * im["nz"]
    make = lambda: P.Matrix(*rows[:3], nv, row_scale=rows[3]).set_spread(s, ls, *win, W)
    M, R = make().set_image(im), make().set_launch(0)
    x, y = torch.rand(nv, device="cuda"), torch.rand(M.n_rows, device="cuda")
    P.timing_enable(True)
    got = (M.forward(x), M.back(y), M.sensitivity())
    ran = set(P.timing_read())
    P.timing_enable(False)
    assert ("csr_fwd_patch_kernel" in ran) == fwd and ("csr_fwd_kernel" in ran) == (not fwd)
    assert ("csr_back_single_kernel" in ran) == back and ("csr_back_kernel" in ran) == (not back)
    for g, o in zip(got, (R.forward(x), R.back(y), R.sensitivity())):
        # sums of the same positive products in another order: up to ~2e4 per voxel
        assert_close(g.cpu(), o.cpu(), 2e-5, 1e-6 * float(o.abs().max()), name)
