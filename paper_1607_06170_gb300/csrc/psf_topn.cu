// Top-N truncation of LOR spreads (Sec. 4.3, Table 3): the window entries of
// each LOR ranked by weight, the first N kept and rescaled to the window's
// total.  Ranking rule (a reading; the paper only says "descending order"):
// a negative weight ranks as 0; equal weights rank the smaller offset
// |dt1|+|da1|+|dt2|+|da2| first, then the lower window index e1*E + e2.
#include <cuda_bf16.h>

#include "psf_common.cuh"

namespace psf {

constexpr int TN_W = 4;       // warps (LORs in flight) per CTA
constexpr int TN_MAX = 64;    // largest N
constexpr int TN_EE = 2432;   // largest window (a 7 x 7 x 7 x 7 window has 2401 entries)

// Entry a comes before entry b: larger weight, then smaller tie rank (unique).
__device__ __forceinline__ bool tn_before(float wa, unsigned ta, float wb, unsigned tb) {
    return wa > wb || (wa == wb && ta < tb);
}

// s + c += x, the rounding error of s + x kept in c (Knuth's two-sum): sums
// weights to about 2^-46 of their sum of magnitudes in FP32.
__device__ __forceinline__ void tn_add(float &s, float &c, float x) {
    const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z)));
    s = t;
}

// The same on two pairs at once (packed FP32 additions; a - b as b * -1 + a).
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(0xbf800000bf800000ull), "l"(a));
    return r;
}
__device__ __forceinline__ void tn_add2(uint64_t &s, uint64_t &c, float x, float y) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
    const uint64_t t = f2_add(s, v), z = f2_sub(t, s);
    c = f2_add(c, f2_add(f2_sub(s, f2_sub(t, z)), f2_sub(v, z)));
    s = t;
}

// The sum over the warp of s + c (every lane's pair ends up with it).
__device__ __forceinline__ void tn_warp(float &s, float &c) {
    for (int o = 16; o > 0; o >>= 1) {
        const float so = __shfl_xor_sync(0xffffffffu, s, o);
        const float co = __shfl_xor_sync(0xffffffffu, c, o);
        tn_add(s, c, so);
        c += co;
    }
}

// One warp per LOR.  The window is copied to shared memory (asynchronous
// copies, all in flight at once), and one pass over each lane's contiguous piece
// (an odd number of words, so the lanes' reads fall on different banks) gives
// its total and the piece's largest weight.  The N-th largest of the 32 pieces'
// largest weights bounds the N-th weight of the window from below, so only the
// pieces that reach it are read again, by the whole warp, for the entries that
// do; those (a handful) rank themselves against each other.  Windows with more
// than 32 such entries (ties, or no N positive pieces) and N above 32 take the
// entries one after the other, each from the piece that holds the next.  Totals
// and scale are pairs of FP32 numbers where no weight is negative (nothing
// cancels, so they keep 2^-46 of the total, and total / kept is 1 .. EE / N) and
// within FP32's range, else FP64 (whose pipe would cost more than all the rest).
// RING3D, N = 5, 84,227 windows, 809 MB: 0.26 ms (1.52 ms when every rank was
// another pass over the window in 64-bit keys with a CTA barrier, 0.40 ms when
// each was taken from its piece in turn, with FP64 totals; the pieces' largest
// weights as floats, not bits: 0.27 ms).
__global__ void __launch_bounds__(TN_W * 32) topn_kernel(const float *__restrict__ spread,
                                                         int64_t n, int Wt, int Wa, int N,
                                                         int piece, int32_t *__restrict__ idx,
                                                         float *__restrict__ wout) {
    extern __shared__ __align__(16) unsigned char tn_raw[];
    const int W2a = 2 * Wa + 1, E = (2 * Wt + 1) * W2a, EE = E * E, words = 32 * piece;
    unsigned *tie = reinterpret_cast<unsigned *>(tn_raw);  // [words] tie rank of an entry
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned F = 0xffffffffu, lt = (1u << lane) - 1u;
    float *win = reinterpret_cast<float *>(tie + words) + warp * (words + TN_MAX);  // [words]
    float *sel = win + words;                                                         // [N]
    for (int e = t; e < words; e += TN_W * 32) {
        const int e1 = e / E, e2 = e - e1 * E;
        const int dist = abs(e1 / W2a - Wt) + abs(e1 % W2a - Wa) + abs(e2 / W2a - Wt) +
                         abs(e2 % W2a - Wa);
        tie[e] = e < EE ? (unsigned)(dist * EE + e) : 0xffffffffu;
    }
    for (int e = EE + lane; e < words; e += 32) win[e] = 0.0f;  // padding: adds nothing
    __syncthreads();
    const uint32_t win32 = (uint32_t)__cvta_generic_to_shared(win);
    // entry e's weight as the rule ranks it (a negative one, or none, as 0;
    // padding after every entry)
    auto ranked = [&](int e) {
        const float w = win[e];
        return e < EE ? (w > 0.0f ? w : 0.0f) : -1.0f;
    };
    for (int64_t g = (int64_t)blockIdx.x * TN_W + warp; g < n; g += (int64_t)gridDim.x * TN_W) {
        const float *wg = spread + g * EE;
        {
            const float *src = wg + lane;
            uint32_t dst = win32 + 4 * lane;
#pragma unroll 8
            for (int e = lane; e < EE; e += 32, src += 32, dst += 128)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src)
                             : "memory");
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        // the lane's piece: its sum and its largest weight (0 for none positive), by
        // the weights' bits, which order as they do unless one is negative (or not
        // a number): then above infinity's, and that window's are compared again
        const float *mine = win + lane * piece;
        uint64_t s2 = 0, c2 = 0;
        unsigned top = __float_as_uint(mine[piece - 1]);
#pragma unroll 4
        for (int j = 0; j + 1 < piece; j += 2) {
            const float w = mine[j], v = mine[j + 1];
            tn_add2(s2, c2, w, v);
            top = max(top, max(__float_as_uint(w), __float_as_uint(v)));
        }
        const bool mixed = __any_sync(F, top > 0x7f800000u);
        float bw = __uint_as_float(top);
        if (mixed) {
            bw = 0.0f;
            for (int j = 0; j < piece; ++j) bw = fmaxf(bw, mine[j]);
        }
        float s, c, sb, cb;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(s), "=f"(sb) : "l"(s2));
        asm("mov.b64 {%0, %1}, %2;" : "=f"(c), "=f"(cb) : "l"(c2));
        tn_add(s, c, sb);
        tn_add(s, c, mine[piece - 1]);
        c += cb;
        tn_warp(s, c);
        // T: the N-th largest piece
        unsigned T = 0, left = N <= 32 ? F : 0u;
        for (int k = 0; k < N && left; ++k) {
            const bool in = (left >> lane) & 1u;
            T = __reduce_max_sync(F, in ? __float_as_uint(bw) : 0u);
            const unsigned who = __ballot_sync(F, in && __float_as_uint(bw) == T);
            left &= ~(who & (0u - who));
        }
        int cnt = 33;  // candidates (33: not this way)
        float cw = -1.0f;
        unsigned ct = 0xffffffffu;
        if (T > 0u && N <= 32) {
            const float tw = __uint_as_float(T);
            unsigned pieces = __ballot_sync(F, bw >= tw);
            cnt = 0;
            while (pieces && cnt <= 32) {
                const int l = __ffs(pieces) - 1;
                pieces &= pieces - 1;
                for (int j0 = 0; j0 < piece; j0 += 32) {
                    const int f = l * piece + j0 + lane;
                    const bool on = j0 + lane < piece && ranked(f) >= tw;
                    const unsigned m = __ballot_sync(F, on);
                    if (on && cnt + __popc(m & lt) < 32)
                        sel[32 + cnt + __popc(m & lt)] = __int_as_float(f);
                    cnt += __popc(m);
                }
            }
            __syncwarp();
            if (cnt <= 32 && lane < cnt) {
                const int f = __float_as_int(sel[32 + lane]);
                cw = win[f];
                ct = tie[f];
            }
        }
        float ks = 0.0f, kc = 0.0f;
        if (cnt <= 32) {  // (uniform) the candidates rank each other
            int rank = 0;
            for (int j = 0; j < cnt; ++j) {
                const float ow = __shfl_sync(F, cw, j);
                const unsigned ot = __shfl_sync(F, ct, j);
                rank += tn_before(ow, ot, cw, ct);
            }
            const bool keep = lane < cnt && rank < N;
            if (keep) idx[g * N + rank] = (int)(ct % (unsigned)EE);
            __syncwarp();
            if (keep) sel[rank] = cw;
            ks = keep ? cw : 0.0f;
            tn_warp(ks, kc);
        } else {
            // one after the other: (pw, pt) the last one taken; bw, bt: the first
            // entry after it in the lane's piece
            unsigned bt = 0xffffffffu;
            bw = -2.0f;
            for (int j = 0; j < piece; ++j) {
                const float r = ranked(lane * piece + j);
                const unsigned te = tie[lane * piece + j];
                if (tn_before(r, te, bw, bt)) {
                    bw = r;
                    bt = te;
                }
            }
            for (int k = 0; k < N; ++k) {
                // (the weight's bits order as the weight; a lane without entries
                // left takes no part)
                const unsigned top =
                    __reduce_max_sync(F, bw >= 0.0f ? __float_as_uint(bw) + 1u : 0u);
                const bool tops = bw >= 0.0f && __float_as_uint(bw) + 1u == top;
                const unsigned pt = __reduce_min_sync(F, tops ? bt : 0xffffffffu);
                const float pw = __uint_as_float(top - 1u);
                const int e = (int)(pt % (unsigned)EE), from = e / piece;
                const float w = win[e];
                tn_add(ks, kc, w);
                if (lane == 0) {
                    sel[k] = w;
                    idx[g * N + k] = e;
                }
                float nw = -2.0f;
                unsigned nt = 0xffffffffu;
                for (int j = lane; j < piece; j += 32) {
                    const int f = from * piece + j;
                    const float r = ranked(f);
                    const unsigned tf = tie[f];
                    if (tn_before(pw, pt, r, tf) && tn_before(r, tf, nw, nt)) {
                        nw = r;
                        nt = tf;
                    }
                }
                const unsigned nb =
                    __reduce_max_sync(F, nw >= 0.0f ? __float_as_uint(nw) + 1u : 0u);
                nt = __reduce_min_sync(
                    F, nw >= 0.0f && __float_as_uint(nw) + 1u == nb ? nt : 0xffffffffu);
                if (lane == from) {
                    bw = nb ? __uint_as_float(nb - 1u) : -2.0f;
                    bt = nt;
                }
            }
        }
        __syncwarp();  // sel is complete
        // scale = total / kept, 1 when nothing was kept
        if (!mixed && s > 1e-25f && s < 1e30f && ks > 1e-25f && ks < 1e30f) {
            const float q = __fdiv_rn(s, ks);
            const float rem = fmaf(-q, ks, s) + fmaf(-q, kc, c);
            const float ql = __fdiv_rn(rem, ks);
            for (int k = lane; k < N; k += 32) wout[g * N + k] = fmaf(sel[k], q, sel[k] * ql);
        } else {  // a negative weight, an end of FP32's range, or not a number
            double all = 0.0, kept = 0.0;
            for (int e = lane; e < EE; e += 32) all += (double)win[e];
            all = warp_sum_d(all);
            for (int k = 0; k < N; ++k) kept += (double)sel[k];
            const double scale = kept != 0.0 ? all / kept : 1.0;
            for (int k = lane; k < N; k += 32) wout[g * N + k] = (float)((double)sel[k] * scale);
        }
        __syncwarp();  // the window and sel are rewritten next
    }
}

}  // namespace psf

using namespace psf;

extern "C" int psf_spread_topn(const float *spread, int64_t n_lors, int32_t half_t,
                               int32_t half_a, int32_t n_keep, int32_t *idx, float *w,
                               void *stream) {
    PSF_RANGE("psf_spread_topn");
    if (n_lors < 0 || half_t < 0 || half_a < 0) return PSF_EINVAL;
    const int64_t E = (2 * (int64_t)half_t + 1) * (2 * (int64_t)half_a + 1);
    if (E * E > TN_EE) return PSF_EINVAL;
    if (n_keep < 1 || n_keep > TN_MAX || n_keep > E * E) return PSF_EINVAL;
    if (n_lors == 0) return PSF_OK;
    if (!spread || !idx || !w) return PSF_EINVAL;
    cudaStream_t st = as_stream(stream);
    int dev = 0, sms = 148;
    PSF_TRY(cudaGetDevice(&dev));
    PSF_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int piece = (int)((E * E + 31) / 32) | 1;  // entries of a lane, odd
    const size_t shm = sizeof(float) * (32 * piece * (1 + TN_W) + TN_MAX * TN_W);
    PSF_TRY(cudaFuncSetAttribute(topn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)shm));
    int per_sm = 0;
    PSF_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, topn_kernel, TN_W * 32, shm));
    const int64_t need = (n_lors + TN_W - 1) / TN_W, cap = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
    const int64_t grid = need < cap ? need : cap;
    {
        PSF_TIMED("topn_kernel", st);
        topn_kernel<<<(int)grid, TN_W * 32, shm, st>>>(spread, n_lors, half_t, half_a, n_keep,
                                                       piece, idx, w);
    }
    PSF_LAUNCHED();
    return PSF_OK;
}

namespace psf {

// Top-N weights -> BF16 codes with one FP32 scale per spread: scale = the
// largest |w| of the spread's kept weights (1 when they are all 0), code =
// w / scale rounded to the nearest BF16 (ties to even).  One warp per spread.
__global__ void topn_bf16_kernel(const float *__restrict__ w, int64_t n, int N,
                                 __nv_bfloat16 *__restrict__ w16, float *__restrict__ scale) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); g < n;
         g += warps) {
        float mx = 0.0f;
        for (int k = lane; k < N; k += 32) mx = fmaxf(mx, fabsf(w[g * N + k]));
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float sc = mx > 0.0f ? mx : 1.0f;
        for (int k = lane; k < N; k += 32) w16[g * N + k] = __float2bfloat16_rn(__fdiv_rn(w[g * N + k], sc));
        if (lane == 0) scale[g] = sc;
    }
}

}  // namespace psf

extern "C" int psf_spread_topn_bf16(const float *w, int64_t n_spreads, int32_t n_keep,
                                    void *w16, float *scale, void *stream) {
    PSF_RANGE("psf_spread_topn_bf16");
    if (n_spreads < 0 || n_keep < 1 || n_keep > TN_MAX) return PSF_EINVAL;
    if (n_spreads == 0) return PSF_OK;
    if (!w || !w16 || !scale) return PSF_EINVAL;
    cudaStream_t st = as_stream(stream);
    const int64_t blocks = (n_spreads + 7) / 8;
    const int grid = (int)(blocks < 65535 * 16 ? blocks : 65535 * 16);
    {
        PSF_TIMED("topn_bf16_kernel", st);
        topn_bf16_kernel<<<grid, 256, 0, st>>>(w, n_spreads, n_keep,
                                               static_cast<__nv_bfloat16 *>(w16), scale);
    }
    PSF_LAUNCHED();
    return PSF_OK;
}
