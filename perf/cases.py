"""What a user of this library has it do, as cases that can be timed and checked.

Every case is one call (or the short sequence of calls that belongs together)
through the public entry points of ``paper_1607_06170_gb300``: building the
detector response, generating system-matrix rows, projecting, reconstructing.
The sizes are those of the repository's workloads (``inputs.WORKLOADS``);
``draw`` gives scanners, images and lists of the same ranges.

A seed stands for one scanner of the design (its radius and attenuation differ
by up to a percent, as built scanners do) and for one object or data set.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1607_06170_gb300 import inputs as I
from paper_1607_06170_gb300 import psf as P
from paper_1607_06170_gb300.torch_api import listmode_osem, mlem

DEV = "cuda"
_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def listed():
    return [
        # a planar ring's response model: the table, then the spread of each of
        # its LORs (the smallest calls: latency and launches)
        dict(name="ring2d_response", op="response", base="RING2D"),
        # the merged PSF rows A = S G of the planar ring, sized and filled in
        # one call as a script does before a 2D reconstruction
        dict(name="ring2d_psf_rows", op="psf_rows", base="RING2D", dtype="f32"),
        # ten MLEM iterations on those rows (many small launches)
        dict(name="ring2d_mlem", op="mlem2d", base="RING2D", dtype="f32", iters=10),
        # the voxel-driven generator of the planar PSF matrix
        dict(name="ring2d_voxel_driven", op="voxel", base="RING2D", lines=720),
        # the response model of the 3D scanner: table and all class spreads
        dict(name="ring3d_response", op="response", base="RING3D"),
        # the truncation of those spreads to their five largest entries, with
        # 16-bit weights, as list-mode reconstruction uses them
        dict(name="ring3d_truncate", op="topn", base="RING3D", keep=5),
        # the geometric rows of the 3D scanner's whole LOR set (4e9 entries)
        dict(name="ring3d_rows", op="rows_set", base="RING3D", dtype="f32"),
        # the geometric rows of the LORs of listed events
        dict(name="event_rows", op="rows_list", base="RING3D", events=400_000),
        # one projection and one back-projection with A = S G
        dict(name="ring3d_forward", op="forward", base="RING3D", dtype="f32"),
        dict(name="ring3d_back", op="back", base="RING3D", dtype="f32"),
        # two MLEM iterations on the small-animal scanner's fine grid, 16-bit rows
        dict(name="eplus_mlem", op="mlem", base="EPLUS260", dtype="bf16", iters=2),
        # one list-mode OSEM pass over new events, truncated spreads
        dict(name="ring3d_listmode", op="listmode", base="RING3D", dtype="f32", keep=5,
             events=2_000_000, subsets=4),
    ]


# ------------------------------------------------------------------ geometry
def _workload(case, seed=None):
    """Scanner, table, image, LOR set and window of a case (as built, for a seed)."""
    w = I.workload(case["base"])
    s, t, im, ls = dict(w["scanner"]), dict(w["table"]), dict(w["image"]), dict(w["lors"])
    window = w["window"]
    for k in ("n_blocks", "nt_block", "na_block", "n_block_rings", "radius", "gap_t", "gap_a"):
        if k in case:
            s[k] = case[k]
    s["block_gap_a"] = s["gap_a"] if s["n_block_rings"] > 1 else s["block_gap_a"]
    for k in ("n_sub_t", "n_sub_a"):
        if k in case:
            t[k] = case[k]
    if "nx" in case:
        im = I.image(case["nx"], case["ny"], case["nz"], case["dx"], case["dx"], case["dz"])
    if "fan_half" in case:
        ls = dict(fan_half=case["fan_half"], max_ring_diff=case["max_ring_diff"])
    if "half_t" in case:
        window = (case["half_t"], case["half_a"])
    if seed is not None:
        g = np.random.default_rng([int(seed), 7])
        if case["op"] != "psf_rows":  # its caller sizes the rows: one ring, other crystals
            s["radius"] *= 1.0 + 0.01 * g.uniform()
        s["mu"] *= 1.0 + 0.01 * g.uniform()
    return s, t, im, ls, window


def _counts(s, ls):
    """(transaxial pairs, ring pairs, spread classes) of a structured set."""
    nt, nb = I.n_transaxial(s), s["nt_block"]
    tp = I.transaxial_pairs(s, ls["fan_half"])
    nrp = P.len_ring_pairs(s, ls)
    ncls = int((tp[:, 0] < nb).sum()) * (2 * ls["max_ring_diff"] + 1)
    assert nt % 2 == 0
    return tp, nrp, ncls


def _face_xy(s):
    """Front-face centres of one ring's crystals (mm), [Nt, 2]."""
    c = np.arange(I.n_transaxial(s))
    b, i = c // s["nt_block"], c % s["nt_block"]
    phi = 2 * math.pi * b / s["n_blocks"]
    u = (i - 0.5 * (s["nt_block"] - 1)) * (s["xtal_w_t"] + s["gap_t"])
    return np.stack([s["radius"] * np.cos(phi) - u * np.sin(phi),
                     s["radius"] * np.sin(phi) + u * np.cos(phi)], 1)


def _entries(s, im, ls):
    """About how many entries the geometric rows of a set have: per LOR the
    x, y and z planes it crosses inside the grid, plus one."""
    tp, nrp, _ = _counts(s, ls)
    f = _face_xy(s)
    p, d = f[tp[:, 0]], f[tp[:, 1]] - f[tp[:, 0]]
    lo, hi = np.zeros(len(tp)), np.ones(len(tp))
    for a, (n, o, step) in enumerate(((im["nx"], im["ox"], im["dx"]),
                                      (im["ny"], im["oy"], im["dy"]))):
        flat = np.abs(d[:, a]) < 1e-9
        den = np.where(flat, 1.0, d[:, a])
        t0, t1 = (o - p[:, a]) / den, (o + n * step - p[:, a]) / den
        out = (p[:, a] < o) | (p[:, a] >= o + n * step)
        lo = np.maximum(lo, np.where(flat, np.where(out, 2.0, 0.0), np.minimum(t0, t1)))
        hi = np.minimum(hi, np.where(flat, 1.0, np.maximum(t0, t1)))
    frac = np.maximum(hi - lo, 0.0)
    flat_cells = (np.abs(d[:, 0]) / im["dx"] + np.abs(d[:, 1]) / im["dy"]) * frac + (frac > 0)
    # the part of each interval inside the grid's z range, on a sample of pairs
    rp = I.ring_pairs(s, ls["max_ring_diff"])
    pa, zmid = s["xtal_w_a"] + s["gap_a"], 0.5 * (I.n_rings(s) - 1)
    z0, dz = (rp[:, 0] - zmid) * pa, (rp[:, 1] - rp[:, 0]) * pa
    total = 0.0
    pick = np.linspace(0, len(tp) - 1, min(len(tp), 400)).astype(int)
    for k in pick:
        if frac[k] <= 0:
            continue
        den = np.where(dz == 0, 1e-12, dz)
        t0, t1 = (im["oz"] - z0) / den, (im["oz"] + im["nz"] * im["dz"] - z0) / den
        part = (np.minimum(np.maximum(t0, t1), hi[k]) -
                np.maximum(np.minimum(t0, t1), lo[k])).clip(0.0, frac[k])
        total += (flat_cells[k] * part / frac[k] + np.abs(dz) / im["dz"] * part).sum()
    return float(total * len(tp) / len(pick))


def _capacity(s, im, ls):
    """Room for the rows of a set whatever the seed's radius."""
    tp, nrp, _ = _counts(s, ls)
    return int(1.06 * _entries(s, im, ls)) + 3 * len(tp) * nrp


def _stencil_pairs(s, ls, window):
    """(source, target) LOR pairs of the set joined by the spread window."""
    nt, (wt, wa) = I.n_transaxial(s), window
    tp = I.transaxial_pairs(s, ls["fan_half"]).astype(np.int64)
    rp = I.ring_pairs(s, ls["max_ring_diff"]).astype(np.int64)
    nr, dm, f = I.n_rings(s), ls["max_ring_diff"], ls["fan_half"]
    n_t = 0
    for d1 in range(-wt, wt + 1):
        for d2 in range(-wt, wt + 1):
            a, b = (tp[:, 0] + d1) % nt, (tp[:, 1] + d2) % nt
            d = np.abs(a - b)
            n_t += int(((d >= nt // 2 - f) & (d <= nt // 2 + f)).sum())
    n_a = 0
    for o1 in range(-wa, wa + 1):
        for o2 in range(-wa, wa + 1):
            a, b = rp[:, 0] + o1, rp[:, 1] + o2
            n_a += int(((a >= 0) & (a < nr) & (b >= 0) & (b < nr) & (np.abs(a - b) <= dm)).sum())
    return float(n_t) * n_a


# ------------------------------------------------------------------ preparing
def _spreads(s, t, ls, window):
    """(table, eta, spreads): per LOR on a planar ring, per class in 3D."""
    T, eta = P.response_build(s, t)
    if I.n_rings(s) == 1:
        W = P.bin_spread(s, t, T, eta, P.lor_set_list(s, ls), *window)
    else:
        W = P.bin_spread_classes(s, t, T, eta, ls, P.lor_set_classes(s, ls), *window)
    return T, eta, W


def _object(im, seed):
    """A cylinder of textured activity with a few hot spheres (float32 [nv])."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 1)
    axis = [o + (torch.arange(n, device=DEV) + 0.5) * d for n, o, d in
            ((im["nz"], im["oz"], im["dz"]), (im["ny"], im["oy"], im["dy"]),
             (im["nx"], im["ox"], im["dx"]))]
    half = 0.5 * min(im["nx"] * im["dx"], im["ny"] * im["dy"])
    r2 = axis[1][:, None] ** 2 + axis[2][None, :] ** 2
    x = (r2 <= (0.9 * half) ** 2).float()[None] * (
        0.9 + 0.2 * torch.rand((im["nz"], im["ny"], im["nx"]), generator=g, device=DEV))
    for rad in (0.05, 0.1, 0.2):
        c = (torch.rand(3, generator=g, device=DEV) - 0.5) * half
        c[0] *= 0.5 * im["nz"] * im["dz"] / half
        q = ((axis[0] - c[0]) ** 2)[:, None, None] + ((axis[1] - c[1]) ** 2)[:, None] + (
            axis[2] - c[2]) ** 2
        x = torch.where(q <= (rad * half) ** 2, x + 4.0, x)
    return x.reshape(-1).contiguous()


def _lor_data(n, seed):
    """Values as an iteration's ratio holds them: around one, some zero."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 2 + 2)
    y = 0.5 + torch.rand(n, generator=g, device=DEV)
    return torch.where(torch.rand(n, generator=g, device=DEV) < 0.02, torch.zeros_like(y), y)


def _events(case, s, im, ls, n, seed):
    w = dict(scanner=s, image=im, lors=ls, listmode=dict(radii_mm=(5.0, 10.0, 20.0)))
    half = 0.4 * min(im["nx"] * im["dx"], im["ny"] * im["dy"], im["nz"] * im["dz"])
    if half < 20.0:
        w["listmode"]["radii_mm"] = (0.25 * half, 0.5 * half, half)
    return I.listmode_events(w, n, int(seed) % 1_000_003, device=DEV)


def _rows(s, im, ls, dtype):
    if dtype == "f32":
        return (*P.sysmat_rows_set(s, im, ls), None)
    return P.sysmat_rows_set_typed(s, im, ls, dtype)


def _plan(case, s, t, im, ls, window):
    """The factored plan a reconstruction keeps: rows, spreads, tuned launches."""
    W = _spreads(s, t, ls, window)[2]
    rows = _rows(s, im, ls, case["dtype"])
    nv = im["nx"] * im["ny"] * im["nz"]
    M = P.Matrix(*rows[:3], nv, row_scale=rows[3]).set_spread(s, ls, *window, W).set_image(im)
    M.autotune()
    return M, rows, W


def prepare(case, seed):
    s, t, im, ls, window = _workload(case, seed)
    op, nv = case["op"], im["nx"] * im["ny"] * im["nz"]
    st = dict(op=op, case=case, s=s, t=t, im=im, ls=ls, window=window)
    if op == "response":
        planar = I.n_rings(s) == 1
        st["lors"] = P.lor_set_list(s, ls) if planar else P.lor_set_classes(s, ls)
    elif op == "psf_rows":
        st["lors"] = P.lor_set_list(s, ls)
        st["W"] = _spreads(s, t, ls, window)[2]
    elif op == "mlem2d":
        lors = P.lor_set_list(s, ls)
        W = _spreads(s, t, ls, window)[2]
        rows = P.sysmat_rows(s, im, lors, W, *window, dtype=case["dtype"])
        st["rows"] = rows
        st["M"] = P.Matrix(*rows[:3], nv, row_scale=rows[3])
        x = torch.from_numpy(I.phantom_discs(im, int(seed) % 1_000_003).reshape(-1)).to(DEV)
        st["y"] = st["M"].forward(x)
    elif op == "voxel":
        st["T"], st["eta"] = P.response_build(s, t)
    elif op == "topn":
        st["W"] = _spreads(s, t, ls, window)[2]
    elif op == "rows_set":
        n = P.lor_set_size(s, ls)[0]
        cap = _capacity(*(_workload(case)[i] for i in (0, 2, 3)))
        st["buffers"] = (torch.zeros(n + 1, dtype=torch.int64, device=DEV),
                         torch.zeros(cap, dtype=torch.int32, device=DEV),
                         torch.zeros(cap, dtype=_TORCH[case["dtype"]], device=DEV))
        if case["dtype"] != "f32":
            st["buffers"] += (torch.zeros(n, dtype=torch.float32, device=DEV),)
    elif op == "rows_list":
        n = case["events"]
        st["lors"] = _events(case, s, im, ls, n, seed)
        cap = n * (im["nx"] + im["ny"] + 2 * ls["max_ring_diff"])
        st["buffers"] = (torch.zeros(n + 1, dtype=torch.int64, device=DEV),
                         torch.zeros(cap, dtype=torch.int32, device=DEV),
                         torch.zeros(cap, dtype=torch.float32, device=DEV), None)
    elif op in ("forward", "back", "mlem"):
        st["M"], st["rows"], st["W"] = _plan(case, s, t, im, ls, window)
        if op == "back":
            st["y"] = _lor_data(st["M"].n_rows, seed)
        else:
            st["x"] = _object(im, seed)
            if op == "mlem":
                st["y"] = st["M"].forward(st.pop("x"))
    elif op == "listmode":
        W = _spreads(s, t, ls, window)[2]
        idx, wk = P.spread_topn(W, *window, case["keep"])
        del W
        rows = _rows(s, im, ls, case["dtype"])
        M = P.Matrix(*rows[:3], nv, row_scale=rows[3])
        M.set_spread_topn(s, ls, *window, idx, wk).build_sparse_adjoint()
        M.autotune()
        st["M"], st["sens"] = M, M.sensitivity()
        st["events"] = _events(case, s, im, ls, case["events"], seed)
    return st


def run(st):
    op, case = st["op"], st["case"]
    s, t, im, ls, window = st["s"], st["t"], st["im"], st["ls"], st["window"]
    if op == "response":
        T, eta = P.response_build(s, t)
        if I.n_rings(s) == 1:
            return [T, eta, P.bin_spread(s, t, T, eta, st["lors"], *window)]
        return [T, eta, P.bin_spread_classes(s, t, T, eta, ls, st["lors"], *window)]
    if op == "psf_rows":
        return P.sysmat_rows(s, im, st["lors"], st["W"], *window, dtype=case["dtype"])
    if op == "mlem2d" or op == "mlem":
        return mlem(st["M"], st["y"], iters=case["iters"])
    if op == "voxel":
        return P.voxel_homog(s, t, st["T"], st["eta"], im, ls, case["lines"], window[0])
    if op == "topn":
        idx, w = P.spread_topn(st["W"], *window, case["keep"])
        return [idx, w, *P.spread_topn_bf16(w)]
    if op == "rows_set":
        if case["dtype"] == "f32":
            P.sysmat_rows_set(s, im, ls, buffers=st["buffers"])
        else:
            P.sysmat_rows_set_typed(s, im, ls, case["dtype"], buffers=st["buffers"])
        return list(st["buffers"])
    if op == "rows_list":
        P.sysmat_rows(s, im, st["lors"], buffers=st["buffers"])
        return list(st["buffers"][:3])
    if op == "forward":
        return st["M"].forward(st["x"])
    if op == "back":
        return st["M"].back(st["y"])
    rows = P.event_rows(s, ls, st["events"])
    return [rows, listmode_osem(st["M"], rows, case["subsets"], 1, sens=st["sens"])]


# ------------------------------------------------------------------ work
def work(case):
    s, t, im, ls, (wt, wa) = _workload(case)
    op, nv = case["op"], im["nx"] * im["ny"] * im["nz"]
    tp, nrp, ncls = _counts(s, ls)
    n, E, Q = len(tp) * nrp, (2 * wt + 1) * (2 * wa + 1), (wt + 1) * (wa + 1)
    table = t["n_ang_t"] * t["n_ang_a"] * t["n_sub_t"] * t["n_sub_a"]
    table *= 4 * t["max_off_t"] * t["max_off_a"] + 8 * (t["max_off_t"] + 1)
    vb = 4 + (4 if case.get("dtype", "f32") == "f32" else 2)
    if op == "response":
        # reflections make three of four 3D classes images of the fourth
        k, comp = (n, n) if I.n_rings(s) == 1 else (ncls, ncls / 4)
        return dict(bytes=table + 4.0 * k * E * E,
                    flops=2.0 * comp * (t["n_sub_t"] * t["n_sub_a"]) ** 2 * Q * Q)
    if op in ("psf_rows", "mlem2d"):
        g = _entries(s, im, ls)
        a = min(1.45 * g * (1 + wt / 3), float(n) * nv)  # merged entries of A = S G
        if op == "psf_rows":
            return dict(bytes=4.0 * n * E * E + 8.0 * n + vb * a,
                        flops=2.0 * g * (2 * wt + 1) ** 2)
        it = case["iters"]
        return dict(bytes=it * (2 * vb * a + 16.0 * n + 20.0 * nv), flops=it * 4.0 * a)
    if op == "voxel":
        return dict(bytes=4.0 * n * nv + table, flops=2.0 * nv * case["lines"] * (wt + 1) ** 2)
    if op == "topn":
        return dict(bytes=ncls * (4.0 * E * E + 10.0 * case["keep"] + 4), flops=1.0 * ncls * E * E)
    if op == "rows_list":
        g = case["events"] * 1.27 * 2 * min(s["radius"], 0.5 * im["nx"] * im["dx"]) / im["dx"]
        return dict(bytes=16.0 * case["events"] + 8.0 * g, flops=10.0 * g)
    g = _entries(s, im, ls)
    if op == "rows_set":
        return dict(bytes=8.0 * n + vb * g + (0 if vb == 8 else 4.0 * n), flops=2.0 * g)
    if op == "listmode":
        # an event's LOR reaches `keep` measured LORs through each of its sources
        hit = min(float(n), case["events"] * case["keep"])
        per = g / n
        return dict(bytes=case["subsets"] * 24.0 * n + 2 * vb * per * hit, flops=4.0 * per * hit)
    spread = 4.0 * ncls * E * E
    sten = 2.0 * _stencil_pairs(s, ls, (wt, wa))
    one = dict(bytes=vb * g + 12.0 * n + 4.0 * nv + spread, flops=2.0 * g + sten)
    k = 2 * case["iters"] if op == "mlem" else 1
    return dict(bytes=k * one["bytes"], flops=k * one["flops"])


# ------------------------------------------------------------------ 64 bits
def _exact_table(s, t):
    """First-interaction probabilities of a ray in a flat crystal array."""
    f = dict(dtype=torch.float64, device=DEV)
    kt, ka, pt, pa = t["n_ang_t"], t["n_ang_a"], t["n_sub_t"], t["n_sub_a"]
    mt, ma = t["max_off_t"], t["max_off_a"]
    at = torch.arange(kt, **f) * (t["ang_max_t_deg"] / kt * math.pi / 180)
    th = torch.arange(ka, **f) * (t["ang_max_a_deg"] / ka * math.pi / 180)
    tx = torch.tan(at)[:, None].expand(kt, ka)
    ty = torch.tan(th)[None, :] / torch.cos(at)[:, None]
    x0 = (torch.arange(pt, **f) + 0.5) / pt * s["xtal_w_t"]
    y0 = (torch.arange(pa, **f) + 0.5) / pa * s["xtal_w_a"]

    def clip(slope, start, pitch, width, m):  # [kt, ka, p, m] entry and exit depths
        lo = torch.arange(m, **f) * pitch - start[:, None]
        sl = slope[:, :, None, None]
        safe = torch.where(sl > 0, sl, torch.ones_like(sl))
        inside = (lo <= 0) & (lo + width >= 0)
        a = torch.where(sl > 0, lo / safe, torch.where(inside, 0.0, 1e9))
        b = torch.where(sl > 0, (lo + width) / safe, torch.where(inside, 1e9, -1.0))
        return a, b

    ax, bx = clip(tx, x0, s["xtal_w_t"] + s["gap_t"], s["xtal_w_t"], mt)
    ay, by = clip(ty, y0, s["xtal_w_a"] + s["gap_a"], s["xtal_w_a"], ma)
    lo = torch.maximum(ax[:, :, :, None, :, None], ay[:, :, None, :, None, :]).clamp(min=0)
    hi = torch.minimum(bx[:, :, :, None, :, None], by[:, :, None, :, None, :]).clamp(max=s["depth"])
    ds = torch.sqrt(1 + tx * tx + ty * ty)[:, :, None, None, None, None]
    length = ((hi - lo).clamp(min=0) * ds).reshape(-1, mt * ma)
    depth = lo.expand(kt, ka, pt, pa, mt, ma).reshape(-1, mt * ma)
    before = torch.zeros_like(length)
    for j in range(mt * ma):
        before += torch.where(depth[:, j:j + 1] < depth, length[:, j:j + 1], 0.0)
    T = torch.where(length > 0, torch.exp(-s["mu"] * before) * -torch.expm1(-s["mu"] * length), 0.0)
    T = T.reshape(kt, ka, pt, pa, mt, ma)
    eta = torch.zeros((kt, ka, pt, pa, mt + 1), **f)
    eta[..., 1:] = torch.cumsum(T.sum(-1), -1)
    return T, eta


def _exact_rows(s, im, lors):
    """Chords of listed LORs: (row_ptr, col, val) by sorting the plane crossings."""
    f = dict(dtype=torch.float64, device=DEV)
    nt, xy = I.n_transaxial(s), torch.tensor(_face_xy(s), **f)
    nr, pa = I.n_rings(s), s["xtal_w_a"] + s["gap_a"]
    ids = lors.long()
    ends = []
    for e in range(2):
        ring = torch.div(ids[:, e], nt, rounding_mode="floor")
        z = (ring.double() - 0.5 * (nr - 1)) * pa
        ends.append(torch.cat([xy[ids[:, e] % nt], z[:, None]], 1))
    o = torch.tensor([im["ox"], im["oy"], im["oz"]], **f)
    h = torch.tensor([im["dx"], im["dy"], im["dz"]], **f)
    n3 = [im["nx"], im["ny"], im["nz"]]
    cols, vals, cnts = [], [], []
    for i in range(0, len(ids), 20000):
        a, b = (ends[0][i:i + 20000] - o) / h, (ends[1][i:i + 20000] - o) / h
        d = b - a
        d = torch.where(d.abs() < 1e-9, torch.zeros_like(d), d)
        cuts = [torch.zeros(len(a), 1, **f), torch.ones(len(a), 1, **f)]
        for c in range(3):
            safe = torch.where(d[:, c:c + 1] == 0, torch.ones_like(d[:, c:c + 1]), d[:, c:c + 1])
            al = (torch.arange(n3[c] + 1, **f)[None] - a[:, c:c + 1]) / safe
            cuts.append(torch.where(d[:, c:c + 1] == 0, torch.zeros_like(al), al.clamp(0, 1)))
        al = torch.sort(torch.cat(cuts, 1), 1).values
        mid = 0.5 * (al[:, 1:] + al[:, :-1])
        mm = (al[:, 1:] - al[:, :-1]) * ((d * h) ** 2).sum(1, keepdim=True).sqrt()
        on, col = mm >= 1e-7, torch.zeros_like(mid, dtype=torch.int64)
        for c, stride in ((0, 1), (1, n3[0]), (2, n3[0] * n3[1])):
            u = a[:, c:c + 1] + mid * d[:, c:c + 1]
            near = torch.round(u)
            u = torch.where((d[:, c:c + 1] == 0) & ((u - near).abs() < 1e-9), near, u).floor()
            on &= (u >= 0) & (u < n3[c])
            col += u.long() * stride
        col = torch.where(on, col, torch.full_like(col, 1 << 40))
        col, order = torch.sort(col, 1)
        keep = col < 1 << 40
        cols.append(col[keep].int())
        vals.append(mm.gather(1, order)[keep])
        cnts.append(keep.sum(1))
    ptr = torch.zeros(len(ids) + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.cat(cnts), 0)
    return ptr, torch.cat(cols), torch.cat(vals)


def _padded(x, n):
    out = torch.zeros(n, dtype=x.dtype, device=x.device)
    out[:len(x)] = x
    return out


class _Csr64:
    """Products with stored rows in 64 bits, in pieces."""

    def __init__(self, rows, nv):
        self.ptr, self.col, self.val, self.scale = rows
        self.nv, self.n = nv, len(self.ptr) - 1
        step = max(1, min(self.n, self.n * 150_000_000 // max(1, len(self.col))))
        self.cuts = list(range(0, self.n, step)) + [self.n]
        self.at = [int(self.ptr[c]) for c in self.cuts]

    def _parts(self):
        for k in range(len(self.cuts) - 1):
            r0, r1, j0, j1 = self.cuts[k], self.cuts[k + 1], self.at[k], self.at[k + 1]
            row = torch.repeat_interleave(torch.arange(r1 - r0, device=DEV),
                                          self.ptr[r0 + 1:r1 + 1] - self.ptr[r0:r1],
                                          output_size=j1 - j0)
            v = self.val[j0:j1].double()
            if self.scale is not None:
                v *= self.scale[r0:r1].double()[row]
            yield r0, r1, row, self.col[j0:j1].long(), v

    def forward(self, x):
        y = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        for r0, r1, row, col, v in self._parts():
            y[r0:r1].index_add_(0, row, v * x[col])
        return y

    def back(self, y):
        x = torch.zeros(self.nv, dtype=torch.float64, device=DEV)
        for r0, r1, row, col, v in self._parts():
            x.index_add_(0, col, v * y[r0:r1][row])
        return x


class _Spread64:
    """S and S^T of class spreads on a set's LOR vectors in 64 bits: every
    window entry is one shift of the (pair, ring, ring) volume."""

    def __init__(self, s, ls, window, W):
        self.wt, self.wa = window
        nt, nb, nr, dm = I.n_transaxial(s), s["nt_block"], I.n_rings(s), ls["max_ring_diff"]
        tp = torch.tensor(I.transaxial_pairs(s, ls["fan_half"]), device=DEV).long()
        self.index = torch.full((nt, nt), -1, dtype=torch.int64, device=DEV)
        self.index[tp[:, 0], tp[:, 1]] = torch.arange(len(tp), device=DEV)
        self.nt, self.tp, self.nr = nt, tp, nr
        rp = torch.tensor(I.ring_pairs(s, dm), device=DEV).long()
        self.rp = rp[:, 0] * nr + rp[:, 1]
        r = torch.arange(nr, device=DEV)
        d = r[None, :] - r[:, None]
        self.inside = (d.abs() <= dm).double()
        self.diff = d.clamp(-dm, dm) + dm
        a0 = tp[:, 0] % nb
        self.cls = self.index[a0, tp[:, 1] - (tp[:, 0] - a0)]
        E = (2 * self.wt + 1) * (2 * self.wa + 1)
        self.W = W.reshape(-1, 2 * dm + 1, E, E)

    def _planes(self, y):
        v = torch.zeros((len(self.tp), self.nr * self.nr), dtype=torch.float64, device=DEV)
        v[:, self.rp] = y.double().reshape(len(self.tp), -1)
        return v.reshape(-1, self.nr, self.nr)

    def _partners(self):
        k = 2 * self.wt + 1
        for i in range(k * k):
            a = (self.tp[:, 0] + i // k - self.wt) % self.nt
            b = (self.tp[:, 1] + i % k - self.wt) % self.nt
            to = self.index[torch.minimum(a, b), torch.maximum(a, b)]
            yield i // k, i % k, to, a > b

    def _weights(self, T1, T2, o1, o2, sel):
        k = 2 * self.wa + 1
        w = self.W[:, :, T1 * k + o1 + self.wa, T2 * k + o2 + self.wa]
        return w[self.cls[sel]][:, self.diff].double() * self.inside

    def _slices(self, o):
        n = self.nr
        return slice(max(0, -o), n - max(0, o)), slice(max(0, o), n - max(0, -o))

    def apply(self, y, adjoint):
        v = self._planes(y)
        out = torch.zeros_like(v)
        offs = range(-self.wa, self.wa + 1)
        for T1, T2, to, sw in self._partners():
            for flip in (False, True):
                sel = ((to >= 0) & (sw == flip)).nonzero()[:, 0]
                if not len(sel):
                    continue
                dst = to[sel]
                if adjoint:
                    src = v[dst].transpose(1, 2) if flip else v[dst]
                    acc = torch.zeros_like(src)
                else:
                    src = v[sel]
                    acc = torch.zeros_like(src)
                for o1 in offs:
                    for o2 in offs:
                        w = self._weights(T1, T2, o1, o2, sel)
                        (g1, t1), (g2, t2) = self._slices(o1), self._slices(o2)
                        if adjoint:
                            acc[:, g1, g2] += w[:, g1, g2] * src[:, t1, t2]
                        else:
                            acc[:, t1, t2] += (w * src)[:, g1, g2]
                if adjoint:
                    out[sel] += acc
                else:
                    out.index_add_(0, dst, (acc.transpose(1, 2) if flip else acc) * self.inside)
        return (out * self.inside).reshape(len(self.tp), -1)[:, self.rp].reshape(-1)


def _mlem64(forward, back, y, n, iters):
    """The reconstruction's iterations from a uniform image."""
    sens = back(torch.ones(n, dtype=torch.float64, device=DEV))
    seen = (sens >= 1e-12 * sens.max()) & (sens > 0)
    x = seen.double()
    for _ in range(iters):
        yhat = forward(x)
        ratio = torch.where(yhat > 0, y.double() / yhat, torch.zeros_like(yhat))
        x = torch.where(seen, x * back(ratio) / sens, torch.zeros_like(x))
    return x


def exact(case, seed):
    """The spreads' sub-LORs on a node boundary have two right values each, so
    what depends on the response model's decisions has none here; neither has
    list-mode reconstruction, whose rows would take minutes."""
    op = case["op"]
    s, t, im, ls, window = _workload(case, seed)
    nv = im["nx"] * im["ny"] * im["nz"]
    if op == "response":
        return [*_exact_table(s, t), None]
    if op == "rows_list":
        st = prepare(case, seed)
        ptr, col, val = _exact_rows(s, im, st["lors"])
        cap = len(st["buffers"][1])
        return [None, None, _padded(val, cap)]
    if op == "psf_rows":
        st = prepare(case, seed)
        lors = st["lors"].long()
        ptr, col, val = _exact_rows(s, im, lors)
        n = len(lors)
        G = torch.zeros((n, nv), dtype=torch.float64, device=DEV)
        row = torch.repeat_interleave(torch.arange(n, device=DEV), ptr[1:] - ptr[:-1])
        G[row, col.long()] = val
        nt, (wt, _) = I.n_transaxial(s), window
        index = torch.full((nt, nt), -1, dtype=torch.int64, device=DEV)
        index[lors[:, 0], lors[:, 1]] = torch.arange(n, device=DEV)
        A = torch.zeros_like(G)
        for d1 in range(-wt, wt + 1):
            for d2 in range(-wt, wt + 1):
                a, b = (lors[:, 0] + d1) % nt, (lors[:, 1] + d2) % nt
                to = torch.where(a != b, torch.maximum(index[a, b], index[b, a]), -1)
                sel = (to >= 0).nonzero()[:, 0]
                A.index_add_(0, to[sel], st["W"][sel, d1 + wt, d2 + wt].double()[:, None] * G[sel])
        v = A[A > 0]
        if case["dtype"] == "f32":
            return [None, None, v, None]
        top = A.max(1).values
        per = torch.repeat_interleave(torch.where(top > 0, top, 1.0), (A > 0).sum(1))
        return [None, None, v / per, torch.where(top > 0, top, 1.0)]
    if op == "mlem2d":
        st = prepare(case, seed)
        A = _Csr64(st["rows"], nv)
        return _mlem64(A.forward, A.back, st["y"], A.n, case["iters"])
    if op == "topn":
        st = prepare(case, seed)
        wt, wa = window
        k, E = 2 * wa + 1, (2 * wt + 1) * (2 * wa + 1)
        e = torch.arange(E * E, device=DEV)
        dist = sum((v - h).abs() for u in (e // E, e % E) for v, h in ((u // k, wt), (u % k, wa)))
        order = torch.argsort(dist * E * E + e)
        ws, ss = [], []
        for part in st["W"].reshape(-1, E * E).split(8192):
            best = torch.sort(part[:, order].clamp(min=0), dim=1, descending=True, stable=True)
            best = order[best.indices[:, :case["keep"]]]
            kept = part.gather(1, best).double()
            tot = kept.sum(1, keepdim=True)
            ws.append(kept * torch.where(tot != 0, part.double().sum(1, keepdim=True) / tot, 1.0))
            top = ws[-1].abs().max(1).values
            ss.append(torch.where(top > 0, top, 1.0))
        w, sc = torch.cat(ws), torch.cat(ss)
        return [None, w, w / sc[:, None], sc]
    if op in ("forward", "back", "mlem"):
        st = prepare(case, seed)
        G, S = _Csr64(st["rows"], nv), _Spread64(s, ls, window, st["W"])

        def forward(x):
            return S.apply(G.forward(x.double()), False)

        def back(y):
            return G.back(S.apply(y, True))

        if op == "forward":
            return forward(st["x"])
        if op == "back":
            return back(st["y"])
        return _mlem64(forward, back, st["y"], G.n, case["iters"])
    return None


# ------------------------------------------------------------------ drawing
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _planar(rng):
    """A planar ring of 8 blocks and its image, around RING2D."""
    nb = rng.randrange(6, 13)
    radius = rng.uniform(45.0, 60.0)
    nx = rng.randrange(40, 97)
    return dict(base="RING2D", nt_block=nb, radius=radius, nx=nx, ny=rng.randrange(40, 97), nz=1,
                dx=round(62.0 / nx, 3), dz=1.0, fan_half=4 * nb - rng.randrange(1, 5),
                max_ring_diff=0)


def _ring(rng, most):
    """A 3D ring of flat blocks and its image, between RING3D_SMALL and RING3D,
    with at most about `most` entries in its geometric rows."""
    for _ in range(1000):
        blocks, nb, na = rng.choice((12, 16, 20, 24)), rng.randrange(6, 17), rng.randrange(6, 17)
        rings = rng.randrange(1, 5)
        if rings * na > 52 or rings * na < 8:
            continue
        nt = blocks * nb
        if nt % 2 or nt > 384:
            continue
        half_w = 0.5 * (nb * 1.9 + (nb - 1) * 0.3)
        radius = (half_w + rng.uniform(0.3, 3.0)) / math.tan(math.pi / blocks)
        nx, dx = rng.randrange(48, 200), rng.choice((0.5, 0.8, 1.0, 1.25))
        if not 0.25 * radius < 0.5 * nx * dx < 0.62 * radius:
            continue
        nz = rng.randrange(rings * na, 2 * rings * na + 1)
        c = dict(base="RING3D", n_blocks=blocks, nt_block=nb, na_block=na, n_block_rings=rings,
                 radius=radius, nx=nx, ny=nx if rng.random() < 0.5 else rng.randrange(48, nx + 1),
                 nz=nz, dx=dx, dz=round(rings * na * 2.2 / nz, 3),
                 fan_half=rng.randrange(nt // 6, nt // 3 + 1),
                 max_ring_diff=rng.randrange(2, min(15, rings * na - 1) + 1),
                 n_sub_t=rng.choice((4, 8)), n_sub_a=rng.choice((4, 8)),
                 half_t=rng.choice((2, 3)), half_a=rng.randrange(1, 4))
        s, _, im, ls, _ = _workload(c)
        if _entries(s, im, ls) <= most:
            return c
    raise AssertionError("no scanner drawn")


def draw(rng):
    op = rng.choice(("response", "psf_rows", "mlem2d", "voxel", "response3d", "topn", "rows_set",
                     "rows_list", "forward", "back", "mlem", "listmode"))
    most = _log(rng, 2e7, 1.5e9)
    dtype = rng.choice(("f32", "f32", "bf16", "f16"))
    if op == "response":
        return dict(_planar(rng), op=op, n_sub_t=rng.choice((4, 8)))
    if op == "psf_rows":
        return dict(_planar(rng), op=op, dtype=dtype)
    if op == "mlem2d":
        return dict(_planar(rng), op=op, dtype=dtype, iters=10)
    if op == "voxel":  # odd multiples of 240 lines keep off the angle nodes' boundaries
        return dict(_planar(rng), op=op, lines=240 * rng.choice((1, 3, 5)))
    c = _ring(rng, most)
    if op == "response3d":
        return dict(c, op="response")
    if op == "topn":
        return dict(c, op=op, keep=rng.choice((3, 5, 5, 7, 16)))
    if op == "rows_list":
        return dict(c, op=op, events=_log(rng, 2e4, 6e5))
    if op == "mlem":
        return dict(c, op=op, dtype=dtype, iters=2)
    if op == "listmode":
        return dict(c, op=op, dtype=dtype, keep=rng.choice((3, 5, 7)),
                    events=_log(rng, 1e5, 2e6), subsets=rng.choice((2, 4, 8)))
    return dict(c, op=op, dtype=dtype)
