// G^T of two LOR vectors a transaxial pair at a time, for wide images.
#pragma once

namespace psf {

// Division by a fixed divisor with a multiply and a shift (Granlund and
// Montgomery, 1994): for d >= 1 and every n < 2^N, n / d = (n m) >> k with
// k = N + ceil(log2 d) and m = ceil(2^k / d).
struct DivMagic {
    unsigned m;  // < 2^32 for N <= 30
    int k;
    __host__ __device__ unsigned div(unsigned n) const {
        return (unsigned)(((unsigned long long)n * m) >> k);
    }
};

static DivMagic div_magic(unsigned d, unsigned long long n_end) {
    int N = 1, l = 0;
    while (N < 32 && (1ull << N) < n_end) ++N;
    while ((1ull << l) < d) ++l;
    DivMagic q;
    q.k = N + l;
    q.m = (unsigned)(((1ull << q.k) + d - 1) / d);
    return q;
}

// Pair back-projection with each transaxial pair's voxels accumulated in shared
// memory, the voxels found by their y row (pair form -4: images whose byte table
// over x and y leaves pair_stream_kernel too little room for a pair's cells).  All
// ring pairs of a transaxial pair cut the same 2D cells, each voxel of the pair is
// hit by about 12 of its rows on a 3D ring, and the global 8-byte reductions of the
// row-by-row form are bound by the L2's reduction rate; here one CTA per SM takes
// pairs from a counter, adds every entry's two products into a [z slice][cell]
// array of float pairs in shared memory, and flushes each touched voxel with one
// global reduction.  The cells and their voxel-order positions are read from the
// pair's direct-plane row of the middle ring (one z slice holding every cell of a
// pair whose plane crosses the image): a per-y-row table gives a voxel's position
// from its x index for the y rows whose cells form one run of consecutive x, so it
// costs 24 bytes a y row where the byte table costs one a pixel; an entry outside
// the list (or past the array's capacity) is reduced into the image directly; a
// voxel's z slice and x/y index come from multiply-shift divisions.  The entries
// are read 128 per warp step, independently of row boundaries, and each lane keeps
// the start of its entries' next row in a register, so following the rows costs a
// shared-memory read only when a row ends.  Bound by the warps' chains.  ms, against
// (row by row; pair_stream_kernel where it takes the grid), 3D ring of 26 rings:
// 256 x 256 x 104, 3.1e9 entries 9.56 (13.96; 9.82), 400 x 400 x 63, 4.7e9 entries
// 13.22 (22.68; 13.99), 480 x 480 x 48, 5.6e9 entries 15.14 (30.04; no room).
constexpr int PR_T = 1024;

struct RunsGrid {
    int nx, ny, nz, nxy;
    DivMagic dxy, dx;  // column -> z slice, x/y index -> y row
    int cap;           // cells of a pair held in shared memory
    int jm;            // ring-pair index of the cell-list row
};

static size_t runs_smem_bytes(const RunsGrid &g, int nrp) {
    return sizeof(float) * 2 * (size_t)g.nz * g.cap + sizeof(int) * (size_t)g.cap +
           sizeof(int2) * (size_t)g.ny + sizeof(int) * 4 * (size_t)g.ny +
           sizeof(int) * ((size_t)nrp + 1) + sizeof(float2) * (size_t)nrp;
}

template <typename VT>
__global__ void __launch_bounds__(PR_T, 1) csr_back_pair_runs_kernel(
    int64_t ntp, int nrp, const int64_t *__restrict__ ptr, const int32_t *__restrict__ col,
    const VT *__restrict__ val, const float *__restrict__ scale, const float *__restrict__ ya,
    const float *__restrict__ yb, float2 *__restrict__ x2, unsigned long long *pair_ctr,
    RunsGrid g) {
    extern __shared__ __align__(16) unsigned char pr_raw[];
    float *px = reinterpret_cast<float *>(pr_raw);  // [nz][cap] sums of the first LOR vector
    float *ps = px + (size_t)g.nz * g.cap;          // [nz][cap] and of the second
    float2 *rq = reinterpret_cast<float2 *>(ps + (size_t)g.nz * g.cap);  // [nrp] row values
    int2 *run = reinterpret_cast<int2 *>(rq + nrp);  // [ny] y row -> x of its first cell,
                                                     //   first cell << 16 | cells (0: none)
    int *xyl = reinterpret_cast<int *>(run + g.ny);  // [cap] cell -> x/y index
    int *rs = xyl + g.cap;                           // [nrp + 1] row starts in the pair
    int *r_first = rs + nrp + 1, *r_x = r_first + g.ny, *r_end = r_x + g.ny,
        *r_gap = r_end + g.ny;  // [ny] each: run assembly
    __shared__ long long s_T;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    constexpr int NW = PR_T / 32;
    for (int i = t; i < 2 * g.nz * g.cap; i += PR_T) px[i] = 0.0f;
    for (;;) {
        __syncthreads();  // the previous pair's flush is complete
        if (t == 0) s_T = (long long)atomicAdd(pair_ctr, 1ull);
        __syncthreads();
        const long long T = s_T;
        if (T >= ntp) return;
        const int64_t row0 = T * nrp;
        const int64_t E0 = ptr[row0];
        for (int i = t; i <= nrp; i += PR_T) rs[i] = (int)(ptr[row0 + i] - E0);
        for (int i = t; i < nrp; i += PR_T) {
            const float sc = scale ? scale[row0 + i] : 1.0f;
            rq[i] = make_float2(ya[row0 + i] * sc, yb[row0 + i] * sc);
        }
        for (int i = t; i < g.ny; i += PR_T) {
            r_first[i] = -1;
            r_gap[i] = 0;  // runs started in this y row, or 2 when one has a gap
        }
        __syncthreads();
        const int m0 = rs[g.jm];
        const int nc_all = rs[g.jm + 1] - m0, nc = nc_all < g.cap ? nc_all : g.cap;
        for (int i = t; i < nc; i += PR_T) {  // the cell list and its y runs
            const int c = col[E0 + m0 + i];
            const int xy = c - (int)g.dxy.div((unsigned)c) * g.nxy;
            const int iy = (int)g.dx.div((unsigned)xy), ix = xy - iy * g.nx;
            xyl[i] = xy;
            int iyp = -1, ixp = 0, iyn = -1;
            if (i > 0) {
                const int cp = col[E0 + m0 + i - 1];
                const int xyp = cp - (int)g.dxy.div((unsigned)cp) * g.nxy;
                iyp = (int)g.dx.div((unsigned)xyp);
                ixp = xyp - iyp * g.nx;
            }
            if (i + 1 < nc) {
                const int cn = col[E0 + m0 + i + 1];
                const int xyn = cn - (int)g.dxy.div((unsigned)cn) * g.nxy;
                iyn = (int)g.dx.div((unsigned)xyn);
            }
            if (iyp != iy) {
                r_first[iy] = i;
                r_x[iy] = ix;
                atomicAdd(r_gap + iy, 1);
            } else if (ix != ixp + 1) {
                atomicAdd(r_gap + iy, 2);  // not consecutive in x
            }
            if (iyn != iy) r_end[iy] = i + 1;
        }
        __syncthreads();
        for (int i = t; i < g.ny; i += PR_T) {
            // a y row's cells are used only as one run of consecutive x (a
            // cell list out of voxel order could split a y row in two)
            const int f = r_first[i];
            run[i] = f >= 0 && r_gap[i] == 1 ? make_int2(r_x[i], (f << 16) | (r_end[i] - f))
                                             : make_int2(0, 0);
        }
        __syncthreads();
        // entries in blocks of 128, entry base + lane + 32 u of each block to
        // lane u-th (consecutive entries of a row are neighbouring cells of
        // one z slice: consecutive words of the arrays, so the lanes' shared
        // atomics fall on different banks); each warp takes a contiguous run
        // of blocks, every lane finds the row of its entries by stepping
        // forward, and the next block's entries are loaded while the current
        // one is added
        const int E = rs[nrp];
        const int nblk = (E + 127) >> 7;
        const int per = (nblk + NW - 1) / NW;
        const int b0 = warp * per, b1 = b0 + per < nblk ? b0 + per : nblk;
        if (b0 < b1) {
            int r[4];    // per u: largest r with rs[r] <= the lane's entry
            int nxt[4];  // and rs[r + 1], the start of the next row
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int key = (b0 << 7) + lane + 32 * u;
                int lo = 0, hi = nrp - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (rs[mid] <= key) lo = mid; else hi = mid - 1;
                }
                r[u] = lo;
                nxt[u] = rs[lo + 1];
            }
            int c4[4];
            float v4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int rel = (b0 << 7) + lane + 32 * u;
                c4[u] = rel < E ? __ldcs(col + E0 + rel) : 0;
                v4[u] = rel < E ? ld_val_cs(val, E0 + rel) : 0.0f;
            }
            const int32_t *cb = col + E0 + lane;
            const VT *vb = val + E0 + lane;
            for (int bk = b0; bk < b1; ++bk) {
                int cn[4];
                float vn[4];
                const int nx0 = ((bk + 1) << 7) + lane;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool ld = bk + 1 < b1 && nx0 + 32 * u < E;
                    cn[u] = ld ? __ldcs(cb + ((bk + 1) << 7) + 32 * u) : 0;
                    vn[u] = ld ? ld_val_cs(vb, ((bk + 1) << 7) + 32 * u) : 0.0f;
                }
                const int rel0 = (bk << 7) + lane;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int rel = rel0 + 32 * u;
                    if (rel < E) {
                        while (nxt[u] <= rel) {
                            ++r[u];
                            nxt[u] = rs[r[u] + 1];
                        }
                        const float2 q = rq[r[u]];
                        const float pa = v4[u] * q.x, pb = v4[u] * q.y;
                        const int c = c4[u];
                        const int iz = (int)g.dxy.div((unsigned)c), xy = c - iz * g.nxy;
                        const int iy = (int)g.dx.div((unsigned)xy);
                        const int2 ru = run[iy];
                        const int k = xy - iy * g.nx - ru.x;
                        const int pc = (ru.y >> 16) + k;
                        if (((unsigned)k < (unsigned)(ru.y & 0xffff)) & (iz < g.nz)) {
                            const int slot = iz * g.cap + pc;
                            atomicAdd(px + slot, pa);
                            atomicAdd(ps + slot, pb);
                        } else {
                            atomicAdd(x2 + c, make_float2(pa, pb));
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    c4[u] = cn[u];
                    v4[u] = vn[u];
                }
            }
        }
        __syncthreads();
        // flush each touched voxel with one reduction, and clear the array
        const float inv = 1.0f / (float)(nc > 0 ? nc : 1);
        for (int i = t; i < g.nz * nc; i += PR_T) {
            int iz = (int)((float)i * inv);
            iz -= iz * nc > i ? 1 : 0;
            iz += (iz + 1) * nc <= i ? 1 : 0;
            const int pc = i - iz * nc, slot = iz * g.cap + pc;
            const float2 v = make_float2(px[slot], ps[slot]);
            if (v.x != 0.0f || v.y != 0.0f) {
                atomicAdd(x2 + (int64_t)iz * g.nxy + xyl[pc], v);
                px[slot] = 0.0f;
                ps[slot] = 0.0f;
            }
        }
    }
}

}  // namespace psf
