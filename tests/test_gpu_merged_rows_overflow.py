"""PSF rows whose merge outgrew its workspace: what psf_psf_rows_emit then does."""
import ctypes as C

import pytest
import torch

from paper_1607_06170_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_emit_after_an_overflowed_merge(dtype):
    """Rows with a place in the workspace come out whole, the others stay as they
    were (a window of 25 x 25 equal weights over a planar ring: every row is a band
    far wider than the room for four times a ray's voxels)."""
    from paper_1607_06170_gb300 import build, psf as P

    build.build()
    w, Wt = I.workload("RING2D"), 12
    s, im = w["scanner"], w["image"]
    lors = P.lor_set_list(s, w["lors"])
    W = torch.ones((lors.shape[0], 2 * Wt + 1, 2 * Wt + 1), device="cuda")
    ptr, col, val, scale = P.sysmat_rows(s, im, lors, W, Wt, 0, dtype=dtype)  # falls back by itself
    n, L, sc, img = lors.shape[0], P.lib(), P.scanner(s), P.image(im)
    room, nnz = C.c_int64(), C.c_int64()
    assert L.psf_psf_rows_workspace(C.byref(sc), C.byref(img), n, Wt, 0, C.byref(room)) == 0
    ws = torch.empty(room.value, dtype=torch.uint8, device="cuda")
    p2 = torch.empty_like(ptr)
    rc = L.psf_psf_rows_merge(C.byref(sc), C.byref(img), P._ptr(lors), n, P._ptr(W), Wt, 0, P._ptr(p2),
                              P._ptr(ws), room.value, C.byref(nnz), P._stream())
    assert rc == P.PSF_ECAPACITY and nnz.value == len(col) and torch.equal(p2, ptr)
    c2 = torch.full_like(col, -7)
    v2 = torch.full_like(val, -7.0)
    s2 = None if scale is None else torch.empty_like(scale)
    assert L.psf_psf_rows_emit(C.byref(sc), C.byref(img), n, P._DT[dtype], P._ptr(p2), P._ptr(ws),
                               P._ptr(c2), P._ptr(v2), P._ptr(s2), P._stream()) == 0
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), ptr[1:] - ptr[:-1])
    blank = torch.zeros(n, dtype=torch.bool, device="cuda")
    blank[row[c2 == -7]] = True
    out = blank[row]
    assert bool(blank.any()) and not bool(blank[ptr[1:] > ptr[:-1]].all())
    assert bool((c2[out] == -7).all()) and bool((v2[out] == -7.0).all())
    assert torch.equal(c2[~out], col[~out]) and torch.equal(v2[~out], val[~out])
    if scale is not None:
        assert torch.equal(s2, scale)
