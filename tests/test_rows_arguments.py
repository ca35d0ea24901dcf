"""What the PSF-row calls refuse on the host, before any device work (no GPU
needed: every call here returns before it reads a pointer)."""
import ctypes as C

import pytest

from paper_1607_06170_gb300 import inputs as I

EINVAL = -1
DEV = C.c_void_p(16)  # stands for a device pointer; never read


@pytest.fixture(scope="module")
def L():
    from paper_1607_06170_gb300 import build, psf

    build.build()
    return psf


@pytest.mark.parametrize("half", [(-1, 0), (0, -1), (-1, -1), (-3, 0), (-4, -4), (40, 0)])
def test_psf_rows_refuse_windows(L, half):
    """Negative half windows (whose E * E is that of a small window) and one
    that is too large, in every call that takes them."""
    w = I.workload("RING2D")
    sc, im = L.scanner(w["scanner"]), L.image(w["image"])
    s, i, nnz, room = C.byref(sc), C.byref(im), C.c_int64(), C.c_int64()
    lib = L.lib()
    for col, val in ((None, None), (DEV, DEV)):  # size query, fill
        assert lib.psf_sysmat_rows(s, i, DEV, 5, DEV, *half, L.PSF_F32, DEV, col, val, None, 0,
                                   C.byref(nnz), None) == EINVAL
    assert lib.psf_psf_rows_workspace(s, i, 5, *half, C.byref(room)) == EINVAL
    assert lib.psf_psf_rows_merge(s, i, DEV, 5, DEV, *half, DEV, DEV, 1 << 30, C.byref(nnz),
                                  None) == EINVAL
