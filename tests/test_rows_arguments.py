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


@pytest.mark.parametrize("nx,rings,n", [(64, 1, 1 << 22), (256, 1, 5), (64, 80, 5)])
def test_psf_rows_emit_refuses_what_merge_refuses(L, nx, rings, n):
    """A list too long for a workspace, an image of too many voxels, a scanner of
    too many crystals."""
    w = I.workload("RING2D")
    sc = L.scanner(dict(w["scanner"], na_block=rings))
    im = L.image(I.image(nx, nx, 1, 1.0, 1.0, 1.0))
    s, i, nnz, room = C.byref(sc), C.byref(im), C.c_int64(), C.c_int64(-1)
    lib = L.lib()
    rc = lib.psf_psf_rows_workspace(s, i, n, 3, 0, C.byref(room))
    assert rc == EINVAL or (rc == 0 and room.value == 0)
    assert lib.psf_psf_rows_merge(s, i, DEV, n, DEV, 3, 0, DEV, DEV, 1 << 40, C.byref(nnz),
                                  None) == EINVAL
    assert lib.psf_psf_rows_emit(s, i, n, L.PSF_F32, DEV, DEV, DEV, DEV, None, None) == EINVAL
