"""Branches that the usual scanners and images don't reach: rays nearly parallel
to an axis' planes in the listed-row kernel, a voxel index beyond the fast form
there, response tables of more nodes than a kernel argument holds, a ring of more
blocks than the voxel generator's tables hold."""
import math

import numpy as np
import pytest
import torch

from paper_1607_06170_gb300 import inputs as I
from parity import assert_close, compare_chord_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_1607_06170_gb300 import build, psf

    build.build()
    return psf


def _near(s, im, lors):
    """LORs with an axis crossed by less than 1/1024 voxel, but by more than the
    1e-9 that counts as parallel."""
    nt, nr = I.n_transaxial(s), I.n_rings(s)
    c = np.arange(nt)
    phi = 2 * math.pi * (c // s["nt_block"]) / s["n_blocks"]
    u = (c % s["nt_block"] - 0.5 * (s["nt_block"] - 1)) * (s["xtal_w_t"] + s["gap_t"])
    x = s["radius"] * np.cos(phi) - u * np.sin(phi)
    y = s["radius"] * np.sin(phi) + u * np.cos(phi)
    z = (np.arange(nr) - 0.5 * (nr - 1)) * (s["xtal_w_a"] + s["gap_a"])
    p = [np.stack([x[i % nt], y[i % nt], z[i // nt]], 1) for i in (lors[:, 0], lors[:, 1])]
    d = np.abs(p[1] - p[0]) / np.array([im["dx"], im["dy"], im["dz"]])
    return ((d > 1e-9) & (d < 1 / 1024)).any(1)


@pytest.mark.parametrize("n", [1, 2])
@pytest.mark.parametrize("axis", ["x", "y", "z"])
def test_listed_rows_of_nearly_parallel_rays(P, orc, axis, n):
    """One or two voxels of 3 m along an axis (two: the plane between them cuts
    the rays): count, CSR and padded rows equal the set's rows bit for bit, in
    lists of every group size, and the oracle's."""
    w = I.workload("RING3D_SMALL")
    s, ls = w["scanner"], w["lors"]
    a = {k: (n, 3000.0) if k == axis else v for k, v in
         dict(x=(24, 1.5), y=(23, 1.5), z=(16, 1.1)).items()}
    im = I.image(a["x"][0], a["y"][0], a["z"][0], a["x"][1], a["y"][1], a["z"][1])
    L = I.workload_lors(w)
    near = _near(s, im, L)
    assert near.sum() > 100
    ptr, col, val = P.sysmat_rows_set(s, im, ls)
    order = np.concatenate([np.flatnonzero(near), np.random.default_rng(1).permutation(len(L))])
    for m in (1, 33, 1500, len(order)):
        pick = torch.from_numpy(order[:m]).cuda()
        rp, rc, rv, _ = P.sysmat_rows(s, im, torch.from_numpy(L[order[:m]]).cuda())
        cnt = ptr[pick + 1] - ptr[pick]
        assert torch.equal(rp[1:] - rp[:-1], cnt)
        at = torch.repeat_interleave(ptr[pick] - rp[:-1], cnt) + torch.arange(int(cnt.sum()),
                                                                              device="cuda")
        assert torch.equal(rc, col[at]) and torch.equal(rv, val[at])
    some = np.flatnonzero(near)[::3]
    lors = torch.from_numpy(L[some]).cuda()
    got = P.sysmat_rows(s, im, lors)[:3]
    ref = orc.rows_geom(s, im, L[some])
    compare_chord_rows([g.cpu() for g in got], ref[:3], im["nx"] * im["ny"] * im["nz"])
    # the padded rows of the merge: a window of one entry of weight 1
    one = torch.ones((len(some), 1, 1), device="cuda")
    for g, o in zip(P.sysmat_rows(s, im, lors, one, 0, 0)[:3], got):
        assert torch.equal(g, o)


@pytest.mark.parametrize("axis", ["x", "y"])
def test_listed_rows_of_a_far_parallel_index(P, orc, axis):
    """Rays parallel to 200,001 planes half a micrometre apart, at indices on both
    sides of 2^17."""
    w = I.workload("RING2D")
    s, L = w["scanner"], I.workload_lors(w)
    fine, coarse = (200_001, 0.0005), (64, 1.0)
    (nx, dx), (ny, dy) = (fine, coarse) if axis == "x" else (coarse, fine)
    im = I.image(nx, ny, 1, dx, dy, 1.0)
    k = 0 if axis == "x" else 1
    p = np.stack([orc.face_point(s, int(i))[:2] for i in L.reshape(-1)]).reshape(-1, 2, 2)
    flat = np.abs(p[:, 0, k] - p[:, 1, k]) < 1e-12
    index = (p[:, 0, k] - (im["ox"] if k == 0 else im["oy"])) / fine[1]
    pick = flat & (index > 0) & (index < fine[0])
    assert (index[pick] > 1 << 17).any() and (index[pick] < 1 << 17).any()
    got = P.sysmat_rows(s, im, torch.from_numpy(L[pick]).cuda())[:3]
    compare_chord_rows([g.cpu() for g in got], orc.rows_geom(s, im, L[pick])[:3], im["nx"] * im["ny"])


@pytest.mark.parametrize("name,K,Ka", [("RING2D", 128, 1), ("RING2D", 127, 1), ("RING3D_SMALL", 120, 32)])
def test_spreads_of_many_nodes(P, orc, name, K, Ka):
    """2 K + Ka = 257 and 272 node tangents, found by the CTAs (and 255, the
    argument's)."""
    w = I.workload(name)
    s, (Wt, Wa) = w["scanner"], w["window"]
    t = dict(w["table"], n_ang_t=K, n_ang_a=Ka)
    # (the outermost node's reach stays within the table's offsets)
    t.update(dict(ang_max_t_deg=78.0) if name == "RING2D" else dict(max_off_t=18, max_off_a=10))
    T, eta = P.response_build(s, t)
    To, _ = orc.table_build(s, t)
    L = I.workload_lors(w)
    L = L[np.random.default_rng(0).permutation(len(L))[:70 if Wa else 700]]
    got = P.bin_spread(s, t, T, eta, torch.from_numpy(L).cuda(), Wt, Wa).cpu().numpy()
    want = orc.spread(s, t, To, L, Wt, Wa)
    sure = orc.tie_margin(s, t, To, L) > 1e-5
    assert sure.mean() > 0.5
    scale = np.abs(want).reshape(len(L), -1).max(1)[:, None, None]
    assert_close(got[sure], want[sure], 1e-5, (1e-6 * scale + 1e-30)[sure], "spreads")


@pytest.mark.parametrize("k", [17, 60])
def test_voxel_driven_without_tables(P, orc, k):
    """5,000 blocks of one crystal: their tables exceed the shared memory."""
    R = 5000
    s = I.scanner(R, 1, 1, 1, 2.0, 2.0, 10.0, 0.0, 0.0, 1.0005 / math.tan(math.pi / R), 0.0, 0.087)
    t, ls, im = I.workload("RING2D")["table"], dict(fan_half=1, max_ring_diff=0), I.image(5, 3, 1, 0.31, 0.37, 1.0)
    T, eta = P.response_build(s, t)
    To, _ = orc.table_build(s, t)
    A = P.voxel_homog(s, t, T, eta, im, ls, k, 3).cpu().numpy()
    Ao, margin = orc.voxel_homog(s, t, To, im, I.lor_list(s, 1, 0), k, 3)
    assert margin.min() > 1e-5 and Ao.max() > 0
    scale = np.abs(Ao).max(0, keepdims=True)
    assert_close(A, Ao, 1e-5, 1e-6 * scale + 1e-30, "voxel-driven A")
