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


@pytest.mark.parametrize("name", ["RING2D", "RING3D_SMALL"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 700, 1999])
def test_listed_rows_any_length(P, name, n):
    """Rows of a shuffled list, some ids out of range, are the set's rows bit
    for bit (out-of-range ids: empty rows), whatever the LORs per warp."""
    w = I.workload(name)
    s, im, ls = w["scanner"], w["image"], w["lors"]
    ptr, col, val = P.sysmat_rows_set(s, im, ls)
    L = P.lor_set_list(s, ls)
    pick = torch.from_numpy(np.random.default_rng(n).permutation(L.shape[0])[:n]).cuda()
    lors = L[pick].contiguous()
    bad = torch.arange(n, device="cuda") % 5 == 3
    lors[bad, 0] = I.n_crystals(s) + 7
    rp, rc, rv, _ = P.sysmat_rows(s, im, lors)
    cnt = torch.where(bad, 0, ptr[pick + 1] - ptr[pick])
    assert torch.equal(rp[1:] - rp[:-1], cnt)
    at = torch.repeat_interleave(ptr[pick] - rp[:-1], cnt) + torch.arange(int(cnt.sum()), device="cuda")
    assert torch.equal(rc, col[at]) and torch.equal(rv, val[at])


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


@pytest.mark.parametrize("Wt,Wa,N", [(0, 0, 1), (1, 0, 9), (0, 3, 49), (3, 3, 1)])
def test_truncation_whole_and_tiny_windows(P, orc, Wt, Wa, N):
    """Windows down to one entry, all entries kept, a count of windows that
    leaves warps without one; values whose FP32 total would overflow."""
    E = (2 * Wt + 1) * (2 * Wa + 1)
    rng = np.random.default_rng(7 + E)
    w = rng.uniform(0, 1, size=(131, E, E)).astype(np.float32)
    w[3] *= np.float32(1e38)
    idx, wk = P.spread_topn(torch.from_numpy(w).cuda(), Wt, Wa, N)
    out_o, idx_o = orc.spread_topn(w.astype(np.float64), Wt, Wa, N)
    np.testing.assert_array_equal(idx.cpu().numpy(), idx_o)
    keep = np.delete(np.arange(131), 3) if E > 1 else np.arange(131)  # row 3: beyond FP32
    wo = np.take_along_axis(out_o.reshape(131, -1), idx_o.astype(np.int64), 1)
    assert_close(wk.cpu().numpy()[keep], wo[keep], 2e-7, 1e-30, "kept weights")
    # its scaled weights are the double ones rounded (infinite beyond the range)
    with np.errstate(over="ignore"):
        want = wo[3].astype(np.float32)
    np.testing.assert_allclose(wk.cpu().numpy()[3], want, rtol=2e-7)


@pytest.mark.parametrize("case", ["wide window", "large list", "one row"])
def test_merged_rows_paths(P, case):
    """PSF rows whose merged entries outgrow the workspace (a wide window), whose
    workspace would be too large (a list over an image of many voxels) and of a
    single LOR: against S (G x) in 64 bits, and the 16-bit formats against FP32."""
    w = I.workload("RING2D")
    s, t, im, Wt = dict(w["scanner"]), w["table"], w["image"], 3
    if case == "wide window":
        Wt = 12
    elif case == "large list":
        s.update(n_blocks=32, radius=130.0)
        im = I.image(220, 200, 1, 0.8, 0.9, 1.0)
    nt = I.n_transaxial(s)
    lors = P.lor_set_list(s, dict(fan_half=nt // 2 - 1, max_ring_diff=0))
    lors = lors[32:33].contiguous() if case == "one row" else lors[:16000].contiguous()
    n, nv = lors.shape[0], im["nx"] * im["ny"]
    T, eta = P.response_build(s, t)
    W = P.bin_spread(s, t, T, eta, lors, Wt, 0)
    ptr, col, val, _ = P.sysmat_rows(s, im, lors, W, Wt, 0)
    d = col[1:].long() - col[:-1].long()
    inner = torch.ones(len(col) - 1, dtype=torch.bool, device="cuda") if len(col) else d.bool()
    ends = ptr[1:-1]
    inner[ends[(ends > 0) & (ends < len(col))] - 1] = False
    assert bool((d[inner] > 0).all()) and bool((val > 0).all())
    x = torch.rand(nv, device="cuda", dtype=torch.float64)

    def times(p, c, v):
        y = torch.zeros(n, device="cuda", dtype=torch.float64)
        row = torch.repeat_interleave(torch.arange(n, device="cuda"), p[1:] - p[:-1])
        return y.index_add_(0, row, v.double() * x[c.long()])

    gx = times(*P.sysmat_rows(s, im, lors)[:3])
    index = torch.full((nt, nt), -1, dtype=torch.int64, device="cuda")
    index[lors[:, 0].long(), lors[:, 1].long()] = torch.arange(n, device="cuda")
    want = torch.zeros(n, device="cuda", dtype=torch.float64)
    for d1 in range(-Wt, Wt + 1):
        for d2 in range(-Wt, Wt + 1):
            a, b = (lors[:, 0].long() + d1) % nt, (lors[:, 1].long() + d2) % nt
            to = torch.where(a != b, torch.maximum(index[a, b], index[b, a]), -1)
            on = (to >= 0) & (W[:, d1 + Wt, d2 + Wt] > 0)
            want.index_add_(0, to[on], W[on, d1 + Wt, d2 + Wt].double() * gx[on])
    # sums of positive FP32 products of at most 2 E^2 terms per voxel
    assert_close(times(ptr, col, val).cpu(), want.cpu(), 2 * (2 * Wt + 1) ** 2 * 6e-8,
                 1e-30, "merged rows")
    for dt, tol in (("bf16", 2.0 ** -8), ("f16", 2.0 ** -10)):
        p2, c2, v2, sc = P.sysmat_rows(s, im, lors, W, Wt, 0, dtype=dt)
        assert torch.equal(p2, ptr) and torch.equal(c2, col)
        per = torch.repeat_interleave(sc, ptr[1:] - ptr[:-1])
        assert float((v2.float() * per - val).abs().max()) <= tol * float(sc.max())


@pytest.mark.parametrize("n_sub", [2, 4, 8])
@pytest.mark.parametrize("norm", [0, 1, 2])
def test_planar_spreads(P, orc, n_sub, norm):
    """Planar spreads with 4, 16 and 64 sub-LORs (lanes idle, a half-warp, two
    chunks), a LOR count that leaves groups without one, every normalisation."""
    w = I.workload("RING2D")
    s, t = w["scanner"], dict(w["table"], n_sub_t=n_sub)
    T, eta = P.response_build(s, t)
    To, _ = orc.table_build(s, t)
    L = I.workload_lors(w)[:1999]
    got = P.bin_spread(s, t, T, eta, torch.from_numpy(L).cuda(), 3, 0, norm=norm).cpu().numpy()
    want = orc.spread(s, t, To, L, 3, 0, norm=norm)
    sure = orc.tie_margin(s, t, To, L) > 1e-5
    assert sure.mean() > 0.5
    scale = np.abs(want).reshape(len(L), -1).max(1)[:, None, None]
    assert_close(got[sure], want[sure], 1e-5, (1e-6 * scale + 1e-30)[sure], "planar spreads")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("start", ["nothing", "sens", "x0", "both"])
@pytest.mark.parametrize("iters", [0, 1, 3])
def test_mlem_forms(P, dtype, start, iters):
    """psf_mlem from every start against the single steps, on a plan at its
    default launches (fused) and at the work queue's."""
    from paper_1607_06170_gb300.torch_api import mlem

    w = I.workload("RING2D_NARROW")
    s, t, im, ls = w["scanner"], w["table"], w["image"], w["lors"]
    T, eta = P.response_build(s, t)
    lors = P.lor_set_list(s, ls)
    rows = P.sysmat_rows(s, im, lors, P.bin_spread(s, t, T, eta, lors, 3, 0), 3, 0, dtype=dtype)
    nv = im["nx"] * im["ny"]
    for chunk in (0, 2):
        M = P.Matrix(*rows[:3], nv, row_scale=rows[3]).set_launch(chunk, 128)
        y = M.forward(torch.from_numpy(I.phantom_discs(im, 3).reshape(-1)).cuda())
        sens = M.sensitivity()
        x0 = torch.rand(nv, device="cuda")
        got = mlem(M, y, iters, x0 if start in ("x0", "both") else None,
                   sens if start in ("sens", "both") else None)
        floor = 1e-12 * float(sens.max())
        x = torch.ones_like(sens)
        P.em_update(x, sens, sens, floor)
        x = x0.clone() if start in ("x0", "both") else x
        for _ in range(iters):
            P.em_update(x, M.back(P.em_ratio(y, M.forward(x))), sens, floor)
        # three iterations of FP32 sums of up to 2,000 terms in another order
        assert_close(got.cpu(), x.cpu(), 2e-5, 1e-6 * float(x.max()), "MLEM image")


@pytest.fixture(scope="module")
def ring3d(P):
    """Rows and spreads of the small 3D ring in each value format."""
    w = I.workload("RING3D_SMALL")
    s, t, im, ls = w["scanner"], w["table"], w["image"], w["lors"]
    T, eta = P.response_build(s, t)
    W = P.bin_spread_classes(s, t, T, eta, ls, P.lor_set_classes(s, ls), *w["window"])
    rows = {d: P.sysmat_rows_set_typed(s, im, ls, d) for d in ("f32", "bf16", "f16")}
    return w, W, rows


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("case", ["set rows", "shuffled columns", "some pairs zero", "cells past the table"])
def test_pair_streamed_projections(P, ring3d, dtype, case):
    """The pair-streamed forward, back and pair back-projection (the default with
    a declared image) against the work-queue kernels on the same rows: rows of
    the set; rows whose voxels lie anywhere; LOR values that are zero on whole
    transaxial pairs; a grid declared so that the cell lists are wrong and longer
    than the table."""
    w, W, rows = ring3d
    s, ls, im = w["scanner"], w["lors"], w["image"]
    ptr, col, val, scale = rows[dtype]
    nv = im["nx"] * im["ny"] * im["nz"]
    grid = im
    if case == "shuffled columns":
        perm = torch.from_numpy(np.random.default_rng(3).permutation(nv)).cuda()
        col = perm[col.long()].int().contiguous()
    elif case == "cells past the table":
        grid = I.image(96, 96, 1, 1.0, 1.0, 1.0)  # the same voxel count
    make = lambda: P.Matrix(ptr, col, val, nv, row_scale=scale).set_spread(s, ls, *w["window"], W)
    M, R = make().set_image(grid), make().set_launch(4, 128)
    x = torch.from_numpy(I.random_image(im, 41).reshape(-1)).cuda()
    y = torch.from_numpy(I.random_lor_values(M.n_rows, 42)).cuda()
    if case == "some pairs zero":
        nrp = P.len_ring_pairs(s, ls)
        y.view(-1, nrp)[::3] = 0.0
        y.view(-1, nrp)[1::3, ::2] = 0.0
    P.timing_enable(True)
    got = (M.forward(x), M.back(y), *M.back_sens(y))
    ran = set(P.timing_read())
    P.timing_enable(False)
    assert {"csr_fwd_patch_kernel", "csr_back_single_kernel", "csr_back_patch_kernel"} <= ran
    M.check()
    want = (R.forward(x), R.back(y), R.back(y), R.sensitivity())
    for g, o in zip(got, want):
        # sums of the same positive products in another order: up to ~2e4 per voxel
        assert_close(g.cpu(), o.cpu(), 2e-5, 1e-6 * float(o.abs().max()), case)


@pytest.mark.parametrize("plan", ["stored", "bf16 rows and weights", "traced"])
@pytest.mark.parametrize("n_ev,n_sub", [(4000, 4), (37, 1), (3, 5)])
def test_osem_by_events(P, ring3d, plan, n_ev, n_sub):
    """List-mode OSEM through psf_osem against the separate steps (a plan without
    the transpose of S): events outside the set, LORs hit several times, subsets
    without events, a given start image."""
    from paper_1607_06170_gb300.torch_api import listmode_osem

    w, W, rows = ring3d
    s, ls, im = w["scanner"], w["lors"], w["image"]
    nv = im["nx"] * im["ny"] * im["nz"]
    idx, wk = P.spread_topn(W, *w["window"], 5)
    wk, wsc = P.spread_topn_bf16(wk) if plan.startswith("bf16") else (wk, None)

    def make():
        if plan == "traced":
            M = P.Matrix.traced(s, im, ls)
        else:
            ptr, col, val, sc = rows["bf16" if plan.startswith("bf16") else "f32"]
            M = P.Matrix(ptr, col, val, nv, row_scale=sc)
        return M.set_spread_topn(s, ls, *w["window"], idx, wk, scale=wsc)

    M, R = make(), make()
    rng = np.random.default_rng(n_ev)
    ev = rng.choice(rng.integers(0, M.n_rows, max(n_ev // 2, 1)), n_ev)
    ev[::17] = -1
    ev = torch.from_numpy(ev.astype(np.int64)).cuda()
    x0 = torch.from_numpy(I.random_image(im, 7, 0.5, 1.5).reshape(-1)).cuda()
    for start in (None, x0):
        P.timing_enable(True)
        got = listmode_osem(M, ev, n_sub, 2, x0=start)
        ran = set(P.timing_read())
        P.timing_enable(False)
        assert "osem_ratio_kernel" in ran
        want = listmode_osem(R, ev, n_sub, 2, x0=start, sparse_adjoint=False)
        # products of up to eight sub-iterations of reordered FP32 sums
        assert_close(got.cpu(), want.cpu(), 5e-5, 1e-6 * float(want.max()) + 1e-30, "OSEM image")
