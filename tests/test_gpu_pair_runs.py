"""psf_back_sens on images too wide for the byte table over x and y: the pair's
cells found by their y rows, against the row launches on the same rows."""
import numpy as np
import pytest
import torch

from paper_1607_06170_gb300 import inputs as I
from parity import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ring():
    from paper_1607_06170_gb300 import build, psf as P

    build.build()
    w = I.workload("RING3D_SMALL")
    s, t, ls = w["scanner"], w["table"], w["lors"]
    T, eta = P.response_build(s, t)
    W = P.bin_spread_classes(s, t, T, eta, ls, P.lor_set_classes(s, ls), *w["window"])
    return P, s, ls, w["window"], W


# (nx + ny < 1024: the set generator)
SIZES = [(256, 256, 5), (257, 31, 9), (19, 300, 8), (480, 480, 3), (1000, 7, 2)]


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("nx,ny,nz", SIZES)
@pytest.mark.parametrize("case", ["set rows", "shuffled columns", "some pairs zero", "wrong grid"])
def test_wide_images(ring, case, nx, ny, nz, dtype):
    """Grids beyond 254 voxels a side, one beyond any byte table; rows of the set,
    rows whose voxels lie anywhere, values that are zero on whole pairs, a grid
    with x and y exchanged."""
    P, s, ls, win, W = ring
    im = I.image(nx, ny, nz, 36.0 / nx, 36.0 / ny, 17.6 / nz)
    nv = nx * ny * nz
    ptr, col, val, scale = P.sysmat_rows_set_typed(s, im, ls, dtype)
    if case == "shuffled columns":
        perm = torch.from_numpy(np.random.default_rng(3).permutation(nv)).cuda()
        col = perm[col.long()].int().contiguous()
    grid = I.image(ny, nx, nz, 1.0, 1.0, 1.0) if case == "wrong grid" else im
    make = lambda: P.Matrix(ptr, col, val, nv, row_scale=scale).set_spread(s, ls, *win, W)
    M, R = make().set_image(grid), make().set_launch(4, 128)
    y = torch.from_numpy(I.random_lor_values(M.n_rows, 42)).cuda()
    if case == "some pairs zero":
        nrp = P.len_ring_pairs(s, ls)
        y.view(-1, nrp)[::3] = 0.0
        y.view(-1, nrp)[1::3, ::2] = 0.0
    P.timing_enable(True)
    got = M.back_sens(y)
    ran = set(P.timing_read())
    P.timing_enable(False)
    assert "csr_back_pair_runs_kernel" in ran
    for g, o in zip(got, (R.back(y), R.sensitivity())):
        # sums of the same positive products in another order: up to ~2e4 per voxel
        assert_close(g.cpu(), o.cpu(), 2e-5, 1e-6 * float(o.abs().max()), case)
    M.autotune()  # whichever form it keeps
    for g, o in zip(M.back_sens(y), got):
        assert_close(g.cpu(), o.cpu(), 2e-5, 1e-6 * float(o.abs().max()), "tuned")
