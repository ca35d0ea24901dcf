// G x and G^T y of a structured set's stored rows, a transaxial pair at a time
// out of shared memory.
//
// The rows of a transaxial pair (all its ring pairs, consecutive in the CSR)
// meet the same 2D cells in every z slice, about 12 rows a voxel on the 3D
// ring.  One CTA per SM takes a pair and holds the pair's voxels -- its cells
// times the z slices -- in shared memory: the forward reads x there, the back-
// projection adds there and reduces each touched voxel into the image once
// (row by row the back-projection is bound by the L2's reductions, one an entry,
// and the forward by the latency of its image gathers).  Each streaming warp
// takes a contiguous part of the pair's entries in blocks of U chunks of 32, the
// next block already loading (the first of the next pair too, before the pair's
// voxels are exchanged), whatever the row boundaries: an entry's z slice comes
// from one multiply-high, its cell from a byte table over the x/y index, its row
// is the warp's running row.  One more warp prepares the next pair (row starts,
// row values, cell list) meanwhile, and passes over pairs whose row values are
// all 0 (a large plan with few values goes row by row: sample_sparse_kernel).
// An entry whose voxel is not in the table (cells past the ones held, or rows of
// any other structure) goes to the image directly, so any rows give the same
// result.  Bound by the warps' chains and the stream together: 3D ring,
// 3.97e9 entries (32 GB of columns and values, 4.7 ms at the copy rate): forward
// 9.14 -> 7.49 ms, back 13.4 -> 7.14 ms, pair 12.05 -> 10.6 ms (the pair had its
// voxels in shared memory already, found through a run table and two divisions,
// with per-lane row tracking); with BF16 values 7.5, 7.2 and 10.3 ms.
//
// Every wait is bounded; a warp that gives up still meets the others at the
// warps' barrier, where all leave together.
#pragma once

namespace psf {

// PS_FWD: out[row] = G_row . in (in: the image).  PS_BACK: out += G^T in (in: a
// value per row; out: the image).  PS_PAIR: out2 += (G^T in, G^T in2), the
// interleaved image pair.
enum { PS_FWD = 0, PS_BACK = 1, PS_PAIR = 2 };

// Streaming warps, and chunks of 32 entries a warp has in registers and again
// in flight.  The stream needs about 45 KB in flight on an SM, and every warp is
// a chain of shared-memory accesses (table, voxel; the additions' are compare-
// and-swap loops), so as many warps as leave the registers for the chunks.  3D
// ring, FP32, ms (warps x chunks): forward 24 x 8 7.49, 24 x 6 7.85, 31 x 4 7.66,
// 28 x 6 8.8 and 16 x 8 10.3; back 31 x 6 7.14, 31 x 4 7.21, 24 x 8 7.46, 16 x 8 8.6;
// pair 31 x 4 10.58, 31 x 6 10.72, 24 x 8 11.1.
template <int MODE>
struct PsShape {
    static constexpr int W = MODE == PS_FWD ? 24 : 31;
    static constexpr int U = MODE == PS_FWD ? 8 : MODE == PS_BACK ? 6 : 4;
    static constexpr int B = 32 * U, T = 32 * (W + 1);
};
constexpr int PS_NONE = 255;  // no cell in the byte table

struct PairGrid {
    int nx, ny, nz, nxy;
    unsigned zm;  // column -> z slice: umulhi(column, zm) >> zk
    int zk;
    int cap;      // cells of a pair held in shared memory
    int jm;       // ring-pair index of the row that lists the cells
    int nrp;
    size_t o_lut, o_rs, o_rq, o_bar, o_xy, o_patch, bytes;
};

// Shared-memory layout, cap from what is left (false: too little).
// vectors: LOR vectors projected together (2: the pair back-projection).
inline bool pair_layout(PairGrid &g, int vectors, size_t avail) {
    auto up = [](size_t b) { return (b + 15) & ~(size_t)15; };
    size_t at = 0;
    g.o_lut = at;
    at += up((size_t)g.nxy);
    g.o_rs = at;
    at += up(sizeof(int) * 2 * (g.nrp + 1));
    g.o_rq = at;
    at += up(sizeof(float) * 2 * vectors * g.nrp);
    g.o_bar = at;
    at += up(sizeof(uint64_t) * 4);
    g.o_xy = at;
    if (at >= avail) return false;
    int cap = (int)((avail - at) / (sizeof(float) * vectors * g.nz + 2 * sizeof(int)));
    cap = cap < PS_NONE - 1 ? cap : PS_NONE - 1;
    cap &= ~3;
    if (cap < 64) return false;
    g.cap = cap;
    at += up(sizeof(int) * 2 * cap);
    g.o_patch = at;
    g.bytes = at + sizeof(float) * vectors * (size_t)g.nz * cap;
    return true;
}

// A prepared pair: first row, first entry, entries, cells held (-1: no more).
struct PairHdr {
    long long row0, E0;
    int total, nc;
};

// Barrier of the streaming warps; true when any of them passed true.
template <int THREADS>
__device__ __forceinline__ bool pair_sync_or(bool bad) {
    int r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n"
        " barrier.cta.red.or.pred q, 1, %2, p;\n selp.s32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"((int)bad), "n"(THREADS)
        : "memory");
    return r != 0;
}

// A stored value as loaded (evict-first) and as a float: converting where it is
// used, not where it is loaded, keeps the loads in flight.
template <typename VT>
__device__ __forceinline__ VT ld_raw_cs(const VT *p) { return __ldcs(p); }
__device__ __forceinline__ float raw_f(float v) { return v; }
__device__ __forceinline__ float raw_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float raw_f(__half v) { return __half2float(v); }

// The sums over the warp of p[0 .. 3], sum k in the lanes with lane >> 3 == k:
// six shuffles, where four sums one after the other take twenty.
__device__ __forceinline__ float warp_sum4(const float p[4], int lane) {
    const unsigned F = 0xffffffffu;
    const bool h = lane & 16, q = lane & 8;
    const float a = (h ? p[2] : p[0]) + __shfl_xor_sync(F, h ? p[0] : p[2], 16);
    const float b = (h ? p[3] : p[1]) + __shfl_xor_sync(F, h ? p[1] : p[3], 16);
    float s = (q ? b : a) + __shfl_xor_sync(F, q ? a : b, 8);
    s += __shfl_xor_sync(F, s, 4);
    s += __shfl_xor_sync(F, s, 2);
    s += __shfl_xor_sync(F, s, 1);
    return s;
}

template <typename VT, int MODE>
__global__ void __launch_bounds__(PsShape<MODE>::T, 1) pair_stream_kernel(
    int64_t ntp, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
    const VT *__restrict__ val, const float *__restrict__ scale, const float *__restrict__ in,
    const float *__restrict__ in2, float *__restrict__ out, float2 *__restrict__ out2,
    unsigned long long *ctr, int *status, long long limit, PairGrid g,
    const unsigned long long *sparse) {
    if (MODE == PS_BACK && sparse && *sparse) return;  // the work queue has it
    extern __shared__ __align__(128) unsigned char rg_raw[];
    constexpr int NV = MODE == PS_PAIR ? 2 : 1;
    constexpr int PS_W = PsShape<MODE>::W, PS_U = PsShape<MODE>::U, PS_B = PsShape<MODE>::B,
                  PS_T = PsShape<MODE>::T;
    unsigned char *lut = rg_raw + g.o_lut;                       // [nxy] x/y index -> cell
    int *rs_all = reinterpret_cast<int *>(rg_raw + g.o_rs);      // [2][nrp + 1] row starts
    float *rq_all = reinterpret_cast<float *>(rg_raw + g.o_rq);  // [2][nrp][NV] row values / sums
    int *xy_all = reinterpret_cast<int *>(rg_raw + g.o_xy);      // [2][cap] cell -> x/y index
    float *patch = reinterpret_cast<float *>(rg_raw + g.o_patch);  // [NV][nz][cap]
    uint64_t *pfull = reinterpret_cast<uint64_t *>(rg_raw + g.o_bar), *pempty = pfull + 2;
    __shared__ PairHdr hdr[2];
    __shared__ int abort_flag;
    volatile int *abort_v = &abort_flag;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned F = 0xffffffffu;
    const int nrp = g.nrp, plane = g.nz * g.cap;
    if (t == 0) {
        for (int k = 0; k < 2; ++k) {
            mbar_init_n(pfull + k, 1);
            mbar_init_n(pempty + k, PS_W);
        }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = t; i < (g.nxy + 3) / 4; i += PS_T) reinterpret_cast<unsigned *>(lut)[i] = F;
    if (MODE != PS_FWD)
        for (int i = t; i < NV * plane; i += PS_T) patch[i] = 0.0f;
    else
        for (int i = t; i < 2 * nrp; i += PS_T) rq_all[i] = 0.0f;
    __syncthreads();
    auto wait = [&](uint64_t *bar, long long use, int hint) {  // the whole warp
        const bool ok = mbar_wait_sleep(bar, (uint32_t)(use & 1), limit, hint);
        if (__all_sync(F, ok) && !*abort_v) return true;
        if (!ok) {
            atomicExch(status, PSF_ETIMEOUT);
            *abort_v = 1;
        }
        return false;
    };
    if (warp == PS_W) {  // prepares pairs
        for (long long k = 0;; ++k) {
            const int b = (int)(k & 1);
            if (k >= 2 && !wait(pempty + b, (k >> 1) - 1, 2000)) return;
            int *rs = rs_all + b * (nrp + 1), *xy = xy_all + b * g.cap;
            float *rq = rq_all + b * nrp * NV;
            long long T = 0;
            int64_t E0 = 0;
            for (;;) {
                if (lane == 0) T = (long long)atomicAdd(ctr, 1ull);
                T = __shfl_sync(F, T, 0);
                if (T >= ntp) break;
                const int64_t row0 = T * nrp;
                bool any = MODE == PS_FWD;
                if (MODE != PS_FWD) {
#pragma unroll 8
                    for (int i = lane; i < nrp; i += 32) {
                        const float sc = scale ? __ldcs(scale + row0 + i) : 1.0f;
                        const float q = __ldcs(in + row0 + i) * sc;
                        rq[NV * i] = q;
                        any |= q != 0.0f;
                        if (NV == 2) {
                            const float q2 = __ldcs(in2 + row0 + i) * sc;
                            rq[2 * i + 1] = q2;
                            any |= q2 != 0.0f;
                        }
                    }
                }
                // a pair whose row values are all 0 adds nothing
                if (!__any_sync(F, any)) continue;
                E0 = ptr[row0];
#pragma unroll 8
                for (int i = lane; i <= nrp; i += 32) rs[i] = (int)(__ldcs(ptr + row0 + i) - E0);
                break;
            }
            if (T >= ntp) {
                if (lane == 0) {
                    hdr[b].nc = -1;
                    hdr[b].total = 0;
                    mbar_arrive(pfull + b);
                }
                return;
            }
            __syncwarp();
            const int m0 = rs[g.jm], nc_all = rs[g.jm + 1] - m0, nc = nc_all < g.cap ? nc_all : g.cap;
#pragma unroll 8
            for (int i = lane; i < nc; i += 32) {
                const int c = col[E0 + m0 + i];
                xy[i] = c - (int)(__umulhi((unsigned)c, g.zm) >> g.zk) * g.nxy;
            }
            if (lane == 0) {
                hdr[b].row0 = T * nrp;
                hdr[b].E0 = E0;
                hdr[b].total = rs[nrp];
                hdr[b].nc = nc;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(pfull + b);
        }
    }
    int c[PS_U], cn[PS_U];
    float v[PS_U];
    VT vn[PS_U];
    // the warp's part of a pair's entries: blocks [b0, b1)
    auto part = [&](int total, int &b0, int &b1) {
        const int nb = (total + PS_B - 1) / PS_B, per = (nb + PS_W - 1) / PS_W;
        b0 = warp * per;
        b1 = b0 + per < nb ? b0 + per : nb;
    };
    auto load = [&](long long E0, int total, int blk) {
        const int32_t *cp = col + E0;
        const VT *vp = val + E0;
        const int e0 = blk * PS_B + lane;
        if ((blk + 1) * PS_B <= total) {
#pragma unroll
            for (int u = 0; u < PS_U; ++u) {
                cn[u] = __ldcs(cp + e0 + 32 * u);
                vn[u] = ld_raw_cs(vp + e0 + 32 * u);
            }
        } else {
#pragma unroll
            for (int u = 0; u < PS_U; ++u) {
                const bool on = e0 + 32 * u < total;
                cn[u] = on ? __ldcs(cp + e0 + 32 * u) : -1;
                vn[u] = on ? ld_raw_cs(vp + e0 + 32 * u) : VT(0.0f);
            }
        }
    };
    bool bad = !wait(pfull, 0, 200);
    if (pair_sync_or<PS_W * 32>(bad)) return;
    PairHdr H = hdr[0];
    int b0, b1;
    part(H.total, b0, b1);
    if (b0 < b1) load(H.E0, H.total, b0);
    for (long long k = 0; H.nc >= 0; ++k) {
        const int b = (int)(k & 1);
        const int *rs = rs_all + b * (nrp + 1), *xy = xy_all + b * g.cap;
        float *rq = rq_all + b * nrp * NV;
        for (int i = t; i < H.nc; i += PS_W * 32) lut[xy[i]] = (unsigned char)i;
        if (MODE == PS_FWD) {  // two slices' cells in flight
            for (int iz = 2 * warp; iz < g.nz; iz += 2 * PS_W) {
                const float *s0 = in + (int64_t)iz * g.nxy;
                const int more = iz + 1 < g.nz ? g.nxy : 0;
                float *d0 = patch + iz * g.cap;
#pragma unroll 8
                for (int i = lane; i < H.nc; i += 32) {
                    const float *s = s0 + xy[i];
                    const float p = __ldg(s), q = __ldg(s + more);
                    d0[i] = p;
                    if (more) d0[g.cap + i] = q;
                }
            }
        }
        pair_sync_or<PS_W * 32>(false);
        int r = 0, rend = 0, rfirst = 0, nrow = 0;
        float qr = 0.0f, qr2 = 0.0f, acc = 0.0f, sums[4];
        if (b0 < b1) {  // the row of the part's first entry: largest r with rs[r] <= p
            const int p = b0 * PS_B;
            const int step = (nrp + 31) / 32, i = lane * step;
            r = step * (31 - __clz(__ballot_sync(F, i < nrp && rs[i] <= p)));
            for (int o = 1; o < step; o += 32) {
                const int j = r + lane + 1;
                const unsigned m = __ballot_sync(F, lane < step - o && j < nrp && rs[j] <= p);
                r += __popc(m);
                if (m != F) break;
            }
            rend = rs[r + 1];
            if (MODE != PS_FWD) qr = rq[NV * r];
            if (MODE == PS_PAIR) qr2 = rq[2 * r + 1];
            rfirst = r;
        }
        // the sums of the nrow rows before r, up to four at once; the part's
        // first row (and its last) may have entries in another warp's part
        auto put_rows = [&]() {
            const float sum = warp_sum4(sums, lane);
            const int j = lane >> 3, row = r - nrow + j;
            if ((lane & 7) == 0 && j < nrow) {
                if (row == rfirst)
                    atomicAdd(rq + row, sum);
                else
                    rq[row] = sum;
            }
            nrow = 0;
        };
#pragma unroll 1
        for (int blk = b0; blk < b1; ++blk) {
#pragma unroll
            for (int u = 0; u < PS_U; ++u) {
                c[u] = cn[u];
                v[u] = raw_f(vn[u]);
            }
            if (blk + 1 < b1) load(H.E0, H.total, blk + 1);
            int slot[PS_U];
#pragma unroll
            for (int u = 0; u < PS_U; ++u) {
                const int iz = (int)(__umulhi((unsigned)c[u], g.zm) >> g.zk);
                const int cell = c[u] >= 0 ? (int)lut[c[u] - iz * g.nxy] : PS_NONE;
                slot[u] = cell == PS_NONE ? -1 : iz * g.cap + cell;
            }
            if (MODE == PS_FWD) {
                float x[PS_U];
#pragma unroll
                for (int u = 0; u < PS_U; ++u) {
                    x[u] = 0.0f;
                    if (slot[u] >= 0)
                        x[u] = patch[slot[u]];
                    else if (c[u] >= 0)
                        x[u] = __ldg(in + c[u]);
                }
#pragma unroll
                for (int u = 0; u < PS_U; ++u) v[u] *= x[u];
            }
            const int pe = (blk + 1) * PS_B < H.total ? (blk + 1) * PS_B : H.total;
#pragma unroll
            for (int u = 0; u < PS_U; ++u) {
                const int eb = blk * PS_B + 32 * u, e = eb + lane;
                const int ce = eb + 32 < pe ? eb + 32 : pe;
                if (MODE != PS_FWD) {
                    float q = qr, q2 = qr2;
                    while (rend < ce) {  // row r ends in this chunk
                        ++r;
                        qr = rq[NV * r];
                        if (MODE == PS_PAIR) qr2 = rq[2 * r + 1];
                        if (e >= rend) {
                            q = qr;
                            q2 = qr2;
                        }
                        rend = rs[r + 1];
                    }
                    const float pv = v[u] * q;
                    if (slot[u] >= 0) {
                        atomicAdd(patch + slot[u], pv);
                        if (MODE == PS_PAIR) atomicAdd(patch + plane + slot[u], v[u] * q2);
                    } else if (c[u] >= 0) {
                        if (MODE == PS_PAIR)
                            atomicAdd(out2 + c[u], make_float2(pv, v[u] * q2));
                        else
                            atomicAdd(out + c[u], pv);
                    }
                } else {
                    while (rend < ce) {
                        const float mine = e < rend ? acc + v[u] : acc;
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (nrow == j) sums[j] = mine;
                        if (e < rend) v[u] = 0.0f;
                        acc = 0.0f;
                        ++r;
                        rend = rs[r + 1];
                        if (++nrow == 4) put_rows();
                    }
                    acc += v[u];
                }
            }
        }
        if (MODE == PS_FWD && b0 < b1) {
            if (nrow) put_rows();
            const float sum = warp_sum_f(acc);
            if (lane == 0) atomicAdd(rq + r, sum);
        }
        // the next pair's first block, before this one's voxels are exchanged
        bad = !wait(pfull + (b ^ 1), (k + 1) >> 1, 200);
        const PairHdr N = hdr[b ^ 1];
        part(N.total, b0, b1);
        if (!bad && N.nc >= 0 && b0 < b1) load(N.E0, N.total, b0);
        if (pair_sync_or<PS_W * 32>(bad)) return;
        if (MODE != PS_FWD) {  // each touched voxel into the image once
            for (int iz = warp; iz < g.nz; iz += PS_W) {
                const int64_t z0 = (int64_t)iz * g.nxy;
#pragma unroll 4
                for (int i = lane; i < H.nc; i += 32) {
                    const int at = iz * g.cap + i;
                    const float w = patch[at], w2 = MODE == PS_PAIR ? patch[plane + at] : 0.0f;
                    if (w != 0.0f || w2 != 0.0f) {
                        if (MODE == PS_PAIR) {
                            atomicAdd(out2 + z0 + xy[i], make_float2(w, w2));
                            patch[plane + at] = 0.0f;
                        } else {
                            atomicAdd(out + z0 + xy[i], w);
                        }
                        patch[at] = 0.0f;
                    }
                }
            }
        } else {
            for (int i = t; i < nrp; i += PS_W * 32) {
                const float y = rq[i];
                out[H.row0 + i] = scale ? y * scale[H.row0 + i] : y;
                rq[i] = 0.0f;
            }
        }
        for (int i = t; i < H.nc; i += PS_W * 32) lut[xy[i]] = (unsigned char)PS_NONE;
        pair_sync_or<PS_W * 32>(false);  // the table is clear before the next pair's cells
        if (lane == 0) mbar_arrive(pempty + b);
        H = N;
    }
}

}  // namespace psf
