// K3: homogenization spread of each LOR (Sec. 2.2 Eq. 10, Sec. 2.3 Eq. 11-12)
// with the neighbouring-block path of Sec. 2.1.2 (Eq. 2, 4, 5).
//
// One CTA per LOR.  The sub-position centres of both crystal faces are staged
// in shared memory; each thread takes one sub-LOR (pair of sub-positions) at a
// time and evaluates the two single-photon responses restricted to the window
// quadrant the photon travels into (the response is one-sided).  Sub-LORs are
// grouped by their pair of travel directions, and each group's contribution is
// a small dense product sum_s r1_s (x) r2_s accumulated by the threads that own
// the outputs, chunk by chunk (FP32, deterministic order).  The per-LOR
// normalisation totals are FP64 block reductions.
#include "psf_common.cuh"
#include "psf_end.cuh"
#include "psf_lorset.cuh"

namespace psf {

constexpr int SP_THREADS = 256;
constexpr int SP_PATS = 16;  // travel-sign patterns of the two ends
struct SpreadSmem {
    float *R1, *R2;        // [SP_THREADS][Q]
    float *accp;           // [SP_PATS][Q*Q]
    float *wwin;           // [E*E]
    float *pts;            // end points: [2][Pt*Pa][4] = (x, y, z, s_entry)
    int *pat;              // [SP_THREADS]
    int *order;            // [SP_THREADS]
    int *cnt;              // [SP_PATS + 1] starts
    int *wcnt;             // [8 warps][SP_PATS]
    double *red;           // [2 * 8]
};

__global__ void __launch_bounds__(SP_THREADS) spread_kernel(
    Scan sc, Tab tb, const float *__restrict__ T, const double *__restrict__ eta,
    const int32_t *__restrict__ lors, int64_t n_lors, int Wt, int Wa, int norm,
    float *__restrict__ out, const int32_t *__restrict__ sym) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int Q = (Wt + 1) * (Wa + 1);
    const int E = (2 * Wt + 1) * (2 * Wa + 1);
    const int NP = tb.Pt * tb.Pa;
    const int nsub = NP * NP;
    SpreadSmem s;
    {
        unsigned char *p = smraw;
        s.red = (double *)p; p += sizeof(double) * 16;
        s.R1 = (float *)p; p += sizeof(float) * SP_THREADS * (Q + 1);
        s.R2 = (float *)p; p += sizeof(float) * SP_THREADS * (Q + 1);
        s.accp = (float *)p; p += sizeof(float) * SP_PATS * Q * Q;
        s.wwin = (float *)p; p += sizeof(float) * E * E;
        s.pts = (float *)p; p += sizeof(float) * 2 * NP * 4;
        s.pat = (int *)p; p += sizeof(int) * SP_THREADS;
        s.order = (int *)p; p += sizeof(int) * SP_THREADS;
        s.cnt = (int *)p; p += sizeof(int) * (SP_PATS + 1);
        s.wcnt = (int *)p;
    }
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int64_t lor = blockIdx.x; lor < n_lors; lor += gridDim.x) {
        const int id1 = lors[2 * lor], id2 = lors[2 * lor + 1];
        const int ring1 = id1 / sc.Nt, c1 = id1 - ring1 * sc.Nt;
        const int ring2 = id2 / sc.Nt, c2 = id2 - ring2 * sc.Nt;
        if (sym && sym[lor] >= 0) continue;  // an image of another class under the mirrors
        const int b1 = c1 / sc.Nb, i1 = c1 - b1 * sc.Nb;
        const int b2 = c2 / sc.Nb, i2 = c2 - b2 * sc.Nb;
        float *o = out + lor * (int64_t)E * E;
        const int nc = sc.Nt * sc.NR;
        // same block: the chord runs along a block face and enters neither
        // crystal; invalid crystal ids also get no spread
        if (b1 == b2 || id1 < 0 || id2 < 0 || id1 >= nc || id2 >= nc) {
            for (int k = t; k < E * E; k += SP_THREADS) o[k] = 0.0f;
            continue;
        }
        float sb1, cb1, sb2, cb2;
        sincospif(2.0f * b1 / sc.R, &sb1, &cb1);
        sincospif(2.0f * b2 / sc.R, &sb2, &cb2);
        // stage the sub-position centres of both faces
        for (int k = t; k < 2 * NP; k += SP_THREADS) {
            int end = k / NP, sp = k - end * NP;
            int p = sp / tb.Pa, q = sp - p * tb.Pa;
            int i = end ? i2 : i1, ring = end ? ring2 : ring1;
            float cb = end ? cb2 : cb1, sb = end ? sb2 : sb1;
            float se = (i - 0.5f * (sc.Nb - 1)) * sc.pt + ((p + 0.5f) / tb.Pt - 0.5f) * sc.wt;
            float ze = sc.z0 + ring * sc.pa + ((q + 0.5f) / tb.Pa - 0.5f) * sc.wa;
            float *P = s.pts + k * 4;
            P[0] = sc.radius * cb - se * sb;
            P[1] = sc.radius * sb + se * cb;
            P[2] = ze;
            P[3] = se;
        }
        for (int k = t; k < SP_PATS * Q * Q; k += SP_THREADS) s.accp[k] = 0.0f;
        double sfull = 0.0, swin = 0.0;
        __syncthreads();
        for (int base = 0; base < nsub; base += SP_THREADS) {
            int sidx = base + t;
            int pt_ = SP_PATS;  // empty slot
            if (sidx < nsub) {
                int s1 = sidx / NP, s2 = sidx - s1 * NP;
                const float *P1 = s.pts + s1 * 4;
                const float *P2 = s.pts + (NP + s2) * 4;
                float dx = P1[0] - P2[0], dy = P1[1] - P2[1], dz = P1[2] - P2[2];
                EndResp r1, r2;
                end_response(sc, tb, T, eta, i1, ring1, cb1, sb1, s1 / tb.Pa, s1 % tb.Pa, P1[3],
                             P1[2], dx, dy, dz, Wt, Wa, r1);
                end_response(sc, tb, T, eta, i2, ring2, cb2, sb2, s2 / tb.Pa, s2 % tb.Pa, P2[3],
                             P2[2], -dx, -dy, -dz, Wt, Wa, r2);
                if (r1.valid && r2.valid) {
                    float w1 = 0.0f, w2 = 0.0f;
                    for (int k = 0; k < Q; ++k) {
                        s.R1[t * (Q + 1) + k] = r1.q[k];  // odd stride: conflict-free
                        s.R2[t * (Q + 1) + k] = r2.q[k];
                        w1 += r1.q[k];
                        w2 += r2.q[k];
                    }
                    sfull += r1.eta * r2.eta;
                    swin += (double)w1 * (double)w2;
                    pt_ = ((r1.sgt > 0) << 3) | ((r1.sga > 0) << 2) | ((r2.sgt > 0) << 1) |
                          (r2.sga > 0);
                }
            }
            s.pat[t] = pt_;
            // stable counting sort of this chunk by pattern (warp ballots)
            for (int P = 0; P < SP_PATS; ++P) {
                unsigned m = __ballot_sync(0xffffffffu, pt_ == P);
                if (lane == 0) s.wcnt[warp * SP_PATS + P] = __popc(m);
            }
            __syncthreads();
            if (t == 0) {
                int acc = 0;
                for (int P = 0; P < SP_PATS; ++P) {
                    s.cnt[P] = acc;
                    for (int w = 0; w < SP_THREADS / 32; ++w) {
                        int c = s.wcnt[w * SP_PATS + P];
                        s.wcnt[w * SP_PATS + P] = acc;
                        acc += c;
                    }
                }
                s.cnt[SP_PATS] = acc;
            }
            __syncthreads();
            // rank within (warp, pattern)
            for (int P = 0; P < SP_PATS; ++P) {
                unsigned m = __ballot_sync(0xffffffffu, pt_ == P);
                if (pt_ == P) {
                    int r = __popc(m & ((1u << lane) - 1u));
                    s.order[s.wcnt[warp * SP_PATS + P] + r] = t;
                }
            }
            __syncthreads();
            if (t < Q * Q) {
                const int e1 = t / Q, e2 = t - e1 * Q;
                for (int P = 0; P < SP_PATS; ++P) {
                    int k0 = s.cnt[P], k1 = s.cnt[P + 1];
                    if (k1 == k0) continue;
                    float acc = 0.0f;
                    for (int k = k0; k < k1; ++k) {
                        int sl = s.order[k];
                        acc = fmaf(s.R1[sl * (Q + 1) + e1], s.R2[sl * (Q + 1) + e2], acc);
                    }
                    s.accp[P * Q * Q + t] += acc;
                }
            }
            __syncthreads();
        }
        // FP64 totals over the CTA
        sfull = warp_sum_d(sfull);
        swin = warp_sum_d(swin);
        if (lane == 0) {
            s.red[warp] = sfull;
            s.red[8 + warp] = swin;
        }
        for (int k = t; k < E * E; k += SP_THREADS) s.wwin[k] = 0.0f;
        __syncthreads();
        if (t == 0) {
            double a = 0.0, b = 0.0;
            for (int w = 0; w < SP_THREADS / 32; ++w) {
                a += s.red[w];
                b += s.red[8 + w];
            }
            s.red[0] = a;
            s.red[8] = b;
        }
        // fold the pattern-local blocks into the window
        const int W2a = 2 * Wa + 1;
        for (int P = 0; P < SP_PATS; ++P) {
            if (t < Q * Q) {
                float v = s.accp[P * Q * Q + t];
                if (v != 0.0f) {
                    int sgt1 = (P >> 3) & 1 ? 1 : -1, sga1 = (P >> 2) & 1 ? 1 : -1;
                    int sgt2 = (P >> 1) & 1 ? 1 : -1, sga2 = P & 1 ? 1 : -1;
                    int e1 = t / Q, e2 = t - e1 * Q;
                    int x1 = e1 / (Wa + 1), z1 = e1 - x1 * (Wa + 1);
                    int x2 = e2 / (Wa + 1), z2 = e2 - x2 * (Wa + 1);
                    int w1 = (sgt1 * x1 + Wt) * W2a + (sga1 * z1 + Wa);
                    int w2 = (sgt2 * x2 + Wt) * W2a + (sga2 * z2 + Wa);
                    s.wwin[w1 * E + w2] += v;
                }
            }
            __syncthreads();
        }
        // wwin holds sums over sub-LORs; sw is its total, sf the untruncated one
        double sf = s.red[0], sw = s.red[8];
        double scale = 1.0 / nsub;                                     // NONE: mean
        if (norm == PSF_NORM_EFF && sw > 0.0) scale = sf / (sw * nsub);  // total = mean eta1 eta2
        if (norm == PSF_NORM_UNIT && sw > 0.0) scale = 1.0 / sw;         // total = 1
        float fs = (float)scale;
        for (int k = t; k < E * E; k += SP_THREADS) o[k] = s.wwin[k] * fs;
        __syncthreads();
    }
}

static size_t spread_smem(const Tab &tb, int Wt, int Wa) {
    int Q = (Wt + 1) * (Wa + 1), E = (2 * Wt + 1) * (2 * Wa + 1);
    int NP = tb.Pt * tb.Pa;
    size_t b = sizeof(double) * 16;
    b += sizeof(float) * 2 * SP_THREADS * (Q + 1);
    b += sizeof(float) * SP_PATS * Q * Q;
    b += sizeof(float) * E * E;
    b += sizeof(float) * 2 * NP * 4;
    b += sizeof(int) * (2 * SP_THREADS + SP_PATS + 1 + 8 * SP_PATS);
    return b;
}


// K3 for the common windows (3 crystals to a side, axially 0, 2 or 3).  A LOR's sub-LORs are not
// evaluated one by one: the transaxial half of a response depends on the
// transaxial sub-positions (p1, p2) alone, and for one such pair the axial half
// (polar nodes, the cells that gap crossers meet) is a step function of the
// axial ones (q1, q2): seen from one q, two or three steps at most, as a rule,
// over the other end's.  So each q's few different rows ("variants") are
// evaluated once, and sum_{q1,q2} r1 (x) r2 is, over the runs of q2 in which
// r1(q1) stays, r1 (x) (sum_q2 r2): about 25 table rows and 12 outer products a
// pair for its Pa^2 sub-LORs (64).  A warp takes a 4 x 4 tile of pairs: first a
// lane the transaxial side of a pair's end, then, a few pairs at a time, a lane an
// end's q: the steps, its variants into shared memory, the runs' sums (two lanes to a
// q1), and the outer products with 16 lanes owning RB x CB blocks of the Q x Q
// quadrant product.  Pairs with different signs of travel land in different
// quadrants of the window: a pass for each pattern of signs.  Sums have a fixed
// order (FP32, deterministic); the totals that normalise them are FP64.  Bound
// by issue; warps are at different places of the code, which therefore has one
// copy of each part (with the sums of pairs without steps formed apart, 150 KB
// of code: 10 of 16 cycles of a warp went by without an instruction).  RING3D's
// 21,744 orbit classes x 4096 sub-LORs: 4.65 -> 3.2 ms (a sub-LOR per lane,
// 4096 outer products a LOR).
constexpr int SQ_T = 128;
constexpr int SQ_WARPS = SQ_T / 32;
constexpr int SQ_V = 3;  // most variants of a row that are staged (more: fewer q at a time)
constexpr int SQ_R = 16 * SQ_V;  // most sums of a batch: 16 lanes' runs
constexpr int SQ_S = 7;   // words of a staged side

template <int WT, int WA>
struct SqShape {
    static constexpr int Q = (WT + 1) * (WA + 1);
    static constexpr int E = (2 * WT + 1) * (2 * WA + 1);
    // each half-warp covers the Q x Q product with its 16 lanes, lane (rb, cb)
    // owning rows rb*RB.. and columns cb*CB.. of it; the two halves take
    // alternate staged sub-LORs and are summed at the end of a pass
    static constexpr int RB = (Q + 3) / 4;
    static constexpr int CB = (Q + 3) / 4;
    // floats from one staged row to the next: 16-byte parts, an odd number of
    // them, so that eight lanes storing a part each hit distinct banks
    static constexpr int QS = RB % 2 ? 4 * RB : 4 * RB + 4;
};

// A lane's operands of a staged row.
template <int N>
__device__ __forceinline__ void load_n(const float *p, float (&v)[N]) {
    if constexpr (N == 4) {
        const float4 w = *reinterpret_cast<const float4 *>(p);
        v[0] = w.x;
        v[1] = w.y;
        v[2] = w.z;
        v[3] = w.w;
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = p[i];
    }
}

// n rows of R2, with the rows of R1 that `at` names (in floats), into the
// accumulator: each half-warp takes every other one.
template <class S>
__device__ __forceinline__ void acc_rows(float (&acc)[S::RB][S::CB], const float *R1, const int *at,
                                         const float *R2, int n, int h, int rb, int cb) {
    R1 += rb * S::RB;
    R2 += h * S::QS + cb * S::CB;
#pragma unroll 2
    for (int row = h; row < n; row += 2) {
        float a[S::RB], b[S::CB];
        load_n<S::RB>(R1 + at[row], a);
        load_n<S::CB>(R2, b);
        R2 += 2 * S::QS;
#pragma unroll
        for (int i = 0; i < S::RB; ++i)
#pragma unroll
            for (int j = 0; j < S::CB; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
}

// A lane's half of a run's sum into its place.
template <class S, int PH>
__device__ __forceinline__ void put_sum(float *R, int half, const float4 (&sum)[PH]) {
#pragma unroll
    for (int k = 0; k < PH; ++k)
        if (half * PH + k < S::Q / 4) reinterpret_cast<float4 *>(R)[half * PH + k] = sum[k];
}

// Shared words of a warp, in order: variant rows [SQ_V][32][QS], sums
// [SQ_R][QS], variants' totals [SQ_V][32] (FP64), sides [SQ_S][32], steps [32],
// sums' r1 [SQ_R], pairs [16].
template <class S>
__host__ __device__ constexpr int spread_q_words() {
    return (SQ_V * 32 + SQ_R) * S::QS + 2 * SQ_V * 32 + SQ_S * 32 + 32 + SQ_R + 16;
}

template <int WT, int WA>
static size_t spread_q_smem(const Tab &tb) {
    using S = SqShape<WT, WA>;
    size_t b = sizeof(float) * SQ_WARPS * spread_q_words<S>();
    b += sizeof(double) * 2 * SQ_WARPS;            // FP64 partial totals
    b += sizeof(float) * 2 * (4 * tb.Pt + tb.Pa);  // sub-position centres
    b += sizeof(int) * 4;                          // sign masks, the LOR
    b += sizeof(float) * (2 * tb.Kt + tb.Ka);      // node tangents
    return b;
}

// queue: the next LOR to take (null: strided)
template <int WT, int WA>
__global__ void __launch_bounds__(SQ_T, 4) spread_q_kernel(
    Scan sc, Tab tb, const __grid_constant__ NodeTans tans, const float *__restrict__ T,
    const double *__restrict__ eta, const int32_t *__restrict__ lors, int64_t n_lors, int wt, int wa,
    int norm, float *__restrict__ out, const int32_t *__restrict__ sym, unsigned *queue) {
    using S = SqShape<WT, WA>;
    constexpr int Q = S::Q, RB = S::RB, CB = S::CB, QS = S::QS;
    const int W2a = 2 * wa + 1, E = (2 * wt + 1) * W2a;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int Pt = tb.Pt, Pa = tb.Pa;
    const int nsub = Pt * Pa * Pt * Pa;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    float *all = reinterpret_cast<float *>(smraw);
    constexpr int WORDS = spread_q_words<S>();
    static_assert(WORDS % 4 == 0 && QS % 4 == 0 && SQ_R % 4 == 0, "16-byte and 8-byte alignment");
    float *Rv = all + warp * WORDS, *Rs = Rv + SQ_V * 32 * QS;
    double *Es = reinterpret_cast<double *>(Rs + SQ_R * QS);
    float *side = reinterpret_cast<float *>(Es + SQ_V * 32);
    unsigned *steps = reinterpret_cast<unsigned *>(side + SQ_S * 32);
    int *row1 = reinterpret_cast<int *>(steps + 32), *pairs = row1 + SQ_R;
    // of all warps
    double *red = reinterpret_cast<double *>(all + SQ_WARPS * WORDS);  // [2][SQ_WARPS]
    float4 *pts = reinterpret_cast<float4 *>(red + 2 * SQ_WARPS);      // [2][Pt]: x, y, face
    float *zs = reinterpret_cast<float *>(pts + 2 * Pt);               // [2][Pa]
    // signs of travel: [0] transaxial, [1] axial; [2] the LOR
    int *masks = reinterpret_cast<int *>(zs + 2 * Pa);
    float *tabs = reinterpret_cast<float *>(masks + 4);
    const float *part = all;  // [Q*Q] of each warp, over its variant rows
    static_assert(Q * Q <= SQ_V * 32 * QS, "part fits the staged rows");
    const int hw = lane >> 4, rb = (lane >> 2) & 3, cb = lane & 3;
    const unsigned below = (1u << lane) - 1u;
    const bool need_eta = norm == PSF_NORM_EFF;
    // s = 2^lg: axial sub-positions of an end in a batch, nq batches to an end
    int lg = 0;
    while (lg < 4 && (1 << lg) < Pa) ++lg;
    const int s = 1 << lg, nq = (Pa + s - 1) >> lg;
    const GapConst gk = make_gapconst(sc, tb, tans, tabs);
    for (int64_t lor = blockIdx.x;; lor += gridDim.x) {
        __syncthreads();  // the LOR before: its readers of the shared arrays are done
        if (queue) {
            if (t == 0) masks[2] = (int)atomicAdd(queue, 1u);
            __syncthreads();
            lor = (unsigned)masks[2];
        }
        if (lor >= n_lors) break;
        if (sym && sym[lor] >= 0) continue;  // an image of another class under the mirrors
        const int id1 = lors[2 * lor], id2 = lors[2 * lor + 1];
        const int ring1 = id1 / sc.Nt, c1 = id1 - ring1 * sc.Nt;
        const int ring2 = id2 / sc.Nt, c2 = id2 - ring2 * sc.Nt;
        const int b1 = c1 / sc.Nb, i1 = c1 - b1 * sc.Nb;
        const int b2 = c2 / sc.Nb, i2 = c2 - b2 * sc.Nb;
        float *o = out + lor * (int64_t)E * E;
        const int nc = sc.Nt * sc.NR;
#pragma unroll 1
        for (int k = t; k < E * E; k += SQ_T) o[k] = 0.0f;
        if (b1 == b2 || id1 < 0 || id2 < 0 || id1 >= nc || id2 >= nc) continue;
        float sb1, cb1, sb2, cb2;
        sincospif(2.0f * b1 / sc.R, &sb1, &cb1);
        sincospif(2.0f * b2 / sc.R, &sb2, &cb2);
#pragma unroll 1
        for (int k = t; k < 2 * Pt; k += SQ_T) {
            const int end = k / Pt, p = k - end * Pt;
            const float cbk = end ? cb2 : cb1, sbk = end ? sb2 : sb1;
            const float u = (end ? i2 : i1) - 0.5f * (sc.Nb - 1);
            const float se = fmaf(u, sc.pt, ((p + 0.5f) / Pt - 0.5f) * sc.wt);
            pts[k] = make_float4(fmaf(sc.radius, cbk, -(se * sbk)), fmaf(sc.radius, sbk, se * cbk),
                                 se, 0.0f);
        }
#pragma unroll 1
        for (int k = t; k < 2 * Pa; k += SQ_T) {
            const int end = k / Pa, q = k - end * Pa;
            zs[k] = sc.z0 + (end ? ring2 : ring1) * sc.pa + ((q + 0.5f) / Pa - 0.5f) * sc.wa;
        }
        if (t < 2) masks[t] = 0;
        __syncthreads();
        // signs of travel of a transaxial pair: -1 (a photon leaves the ring
        // the wrong way), else end 1's times 2 plus end 2's (1: forwards)
        auto pair_dirs = [&](int p1, int p2, float &vn1, float &vt1, float &vn2, float &vt2) {
            const float4 P1 = pts[p1], P2 = pts[Pt + p2];
            const float dx = P1.x - P2.x, dy = P1.y - P2.y;
            end_dir(dx, dy, cb1, sb1, vn1, vt1);
            end_dir(-dx, -dy, cb2, sb2, vn2, vt2);
            if (!(vn1 > 0.0f && vn2 > 0.0f)) return -1;
            return ((vt1 >= 0.0f) << 1) | (vt2 >= 0.0f);
        };
        auto axial_signs = [](float dz) { return ((dz >= 0.0f) << 1) | (-dz >= 0.0f); };
        unsigned mt = 0, ma = 0;
#pragma unroll 1
        for (int k = t; k < Pt * Pt; k += SQ_T) {
            float vn1, vt1, vn2, vt2;
            const int s = pair_dirs(k / Pt, k % Pt, vn1, vt1, vn2, vt2);
            if (s >= 0) mt |= 1u << s;
        }
#pragma unroll 1
        for (int k = t; k < Pa * Pa; k += SQ_T) ma |= 1u << axial_signs(zs[k / Pa] - zs[Pa + k % Pa]);
        mt = __reduce_or_sync(0xffffffffu, mt);
        ma = __reduce_or_sync(0xffffffffu, ma);
        if (lane == 0 && mt) atomicOr(masks, (int)mt);
        if (lane == 0 && ma) atomicOr(masks + 1, (int)ma);
        __syncthreads();
        const unsigned tsigns = masks[0], asigns = masks[1];
        const bool one_sign = __popc(asigns) == 1;
        // a warp's pairs are a 4 x 4 tile: its table reads hit about 4 + 4 rows
        const int nt = (Pt + 3) >> 2;
        const int sub = nt * nt < SQ_WARPS ? SQ_WARPS : 1;  // warps that share a tile
        const int end = (lane >> lg) & 1, ring = end ? ring2 : ring1;
        int np = 0;
        const bool once = __popc(tsigns) * __popc(asigns) == 1;  // one pass
        // the pass's sums over the warps, with their places in the window: within
        // one pattern the quadrant-to-window map is one-to-one, so no two
        // threads meet
        auto each_sum = [&](int ts, int as, auto f) {
            const int g1 = ts >> 1 ? 1 : -1, g2 = ts & 1 ? 1 : -1;
            const int a1 = as >> 1 ? 1 : -1, a2 = as & 1 ? 1 : -1;
#pragma unroll 1
            for (int e = t; e < Q * Q; e += SQ_T) {
                const int e1 = e / Q, e2 = e - e1 * Q;
                const int x1 = e1 / (WA + 1), z1 = e1 - x1 * (WA + 1);
                const int x2 = e2 / (WA + 1), z2 = e2 - x2 * (WA + 1);
                if (x1 > wt || x2 > wt || z1 > wa || z2 > wa) continue;
                float sum = 0.0f;
#pragma unroll
                for (int w = 0; w < SQ_WARPS; ++w) sum += part[w * WORDS + e];
                f(((g1 * x1 + wt) * W2a + a1 * z1 + wa) * E + (g2 * x2 + wt) * W2a + a2 * z2 + wa,
                  sum);
            }
        };
        double sfull = 0.0, swin = 0.0;
#pragma unroll 1
        for (int pass = 0; pass < 16; ++pass) {
            const int ts = pass >> 2, as = pass & 3;  // (uniform over the CTA)
            if (!((tsigns >> ts) & 1) || !((asigns >> as) & 1)) continue;
            const int sga = (end ? as & 1 : as >> 1) ? 1 : -1;
            float acc[RB][CB];
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int j = 0; j < CB; ++j) acc[i][j] = 0.0f;
#pragma unroll 1
            for (int u = warp; u < nt * nt * sub; u += SQ_WARPS) {
                const int tile = u / sub;
                // a lane: the transaxial side of an end of a pair
                {
                    const int p1 = tile / nt * 4 + ((lane & 15) >> 2);
                    const int p2 = tile % nt * 4 + (lane & 3);
                    bool in = p1 < Pt && p2 < Pt;
                    float vn1, vt1, vn2, vt2;
                    if (in) in = pair_dirs(p1, p2, vn1, vt1, vn2, vt2) == ts;
                    const unsigned ins = __ballot_sync(0xffffffffu, in) & 0xffffu;
                    if (in) {
                        const QSide e = end_side(sc, tb, gk, hw ? i2 : i1, hw ? p2 : p1,
                                                 pts[hw ? Pt + p2 : p1].z, hw ? vn2 : vn1,
                                                 hw ? vt2 : vt1);
                        side[lane] = e.ih;
                        side[32 + lane] = e.h;
                        side[64 + lane] = e.run;
                        side[96 + lane] = __int_as_float(e.row0);
                        side[128 + lane] = __int_as_float(e.row1);
                        side[160 + lane] = __int_as_float(e.m);
                        side[192 + lane] = __int_as_float(2 * e.edge + e.gap);
                        if (lane < 16) pairs[__popc(ins & below)] = lane;
                    }
                    np = __popc(ins);
                }
                __syncwarp();
                // a lane: an end's q of a pair, against s of the other end's
#pragma unroll 1
                for (int b0 = u % sub * (16 >> lg); b0 < np; b0 += sub * (16 >> lg)) {
                    const int slot = b0 + (lane >> (lg + 1));
                    const bool in = slot < np;
                    QSide e = {};
                    if (in) {
                        const int l = pairs[slot] + 16 * end;
                        e.ih = side[l];
                        e.h = side[32 + l];
                        e.run = sga * side[64 + l];
                        e.row0 = __float_as_int(side[96 + l]);
                        e.row1 = __float_as_int(side[128 + l]);
                        e.m = __float_as_int(side[160 + l]);
                        e.edge = __float_as_int(side[192 + l]) >> 1;
                        e.gap = __float_as_int(side[192 + l]) & 1;
                    }
                    const bool gap = e.gap && (need_eta || e.edge < WT);
                    // the squares of s x s of (q1, q2)
#pragma unroll 1
                    for (int square = 0; square < nq * nq; ++square) {
                        const int o1 = square / nq * s, o2 = square % nq * s;  // its first q1, q2
                        const int q = (end ? o2 : o1) + (lane & (s - 1));
                        const float zq = q < Pa ? zs[end * Pa + q] : 0.0f;
                        const int ox = end ? o1 : o2;
                        const float *zx = zs + (1 - end) * Pa + ox;  // the other end's
                        // first members of the variants, members
                        unsigned starts = 0, members = 0;
                        int ka = 0;
                        if (in && q < Pa) {
                            int kl = 0, cl = 0;
                            ka = polar_seed(tb, e, fabsf(zq - zx[0]));
                            float lo = 1.0f, hi = 0.0f;  // adz of node ka: [lo, hi)
                            const int nx = min(s, Pa - ox);
#pragma unroll 1
                            for (int j = 0; j < nx; ++j) {
                                const float d = zq - zx[j], adz = fabsf(d);
                                if (!one_sign && axial_signs(end ? -d : d) != as) continue;
                                if (!(adz >= lo && adz < hi)) {
                                    ka = node_by_tan(gk.tanA, tb.Ka, adz, e.h, ka);
                                    lo = ka > 0 ? e.h * gk.tanA[ka - 1] : 0.0f;
                                    hi = ka < tb.Ka - 1 ? e.h * gk.tanA[ka] : CUDART_INF_F;
                                }
                                const int c = gap ? end_gap_cell(sc, tb, gk, e, zq, adz, sga, ring) : 0;
                                if (members == 0 || ka != kl || c != cl) starts |= 1u << j;
                                members |= 1u << j;
                                kl = ka;
                                cl = c;
                            }
                        }
                        // in pieces of step x step, in which no lane has more
                        // variants than are staged (two at most in 2 x 2)
                        int step = s;
                        while (step > 2) {
                            bool few = true;
                            for (int j = 0; j < s; j += step) {
                                const unsigned m = members & (((1u << step) - 1u) << j);
                                few = few && __popc((starts & m) | (m & -m)) <= SQ_V;
                            }
                            if (__all_sync(0xffffffffu, few)) break;
                            step >>= 1;
                        }
#pragma unroll 1
                        for (int piece = 0; piece < (s / step) * (s / step); ++piece) {
                            const int f1 = piece / (s / step) * step, f2 = piece % (s / step) * step;
                            const int fo = end ? f2 : f1, fx = end ? f1 : f2;
                            const bool act = (lane & (s - 1)) >= fo && (lane & (s - 1)) < fo + step;
                            const unsigned mem = act ? members & (((1u << step) - 1u) << fx) : 0;
                            const unsigned st = (starts & mem) | (mem & -mem);
                            const int nv = __popc(st);
                            const int nmax = __reduce_max_sync(0xffffffffu, nv);
                            __syncwarp();  // the rows before are read
                            steps[lane] = st;
                            unsigned rest = st;
#pragma unroll 1
                            for (int v = 0; v < nmax; ++v) {
                                if (v >= nv) continue;
                                const float adz = fabsf(zq - zx[__ffs(rest) - 1]);
                                rest &= rest - 1;
                                ka = node_by_tan(gk.tanA, tb.Ka, adz, e.h, ka);
                                float r[Q];
                                double es = 0.0;
#pragma unroll
                                for (int k = 0; k < Q; ++k) r[k] = 0.0f;
                                end_rows<WT, WA>(
                                    sc, tb, T, eta, e, ka, sga > 0 ? q : Pa - 1 - q,
                                    gap ? end_gap_cell(sc, tb, gk, e, zq, adz, sga, ring) : 0, sga, r,
                                    need_eta ? &es : nullptr);
                                float4 *dst = reinterpret_cast<float4 *>(Rv + (v * 32 + lane) * QS);
#pragma unroll
                                for (int k = 0; k < Q / 4; ++k)
                                    dst[k] = make_float4(r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3]);
                                Es[v * 32 + lane] = es;
                            }
                            __syncwarp();
                            // runs: lanes l1 (of end 1) and l1 + s share q1
                            const int l1 = lane & ~s, l2 = l1 + s - (lane & (s - 1));
                            const unsigned st1 = __shfl_sync(0xffffffffu, st, l1);
                            const unsigned mem1 = __shfl_sync(0xffffffffu, mem, l1);
                            const unsigned upto = (2u << (lane & (s - 1))) - 1u;
                            int at = 0;
                            float *pos[SQ_V];
#pragma unroll
                            for (int v = 0; v < SQ_V; ++v) {
                                const unsigned m = __ballot_sync(0xffffffffu, end == 0 && nv > v);
                                const int p = at + __popc(m & ((1u << l1) - 1u));
                                pos[v] = Rs + p * QS;
                                at += __popc(m);
                                if (end == 0 && nv > v) row1[p] = (v * 32 + lane) * QS;
                            }
                            if (need_eta)
#pragma unroll 1
                                for (int j = f2 + end; j < f2 + step; j += 2)
                                    if ((mem1 >> j) & 1) {
                                        const int v1 = __popc(st1 & ((2u << j) - 1u)) - 1;
                                        const int v2 = __popc(steps[l2 + j] & upto) - 1;
                                        sfull += Es[v1 * 32 + l1] * Es[v2 * 32 + l2 + j];
                                    }
                            constexpr int PARTS = Q / 4, PH = (PARTS + 1) / 2;
                            float4 sum[PH];
                            int v = -1;
#pragma unroll 1
                            for (int j = f2; j < f2 + step; ++j) {
                                if ((st1 >> j) & 1) {
                                    if (v >= 0) put_sum<S>(v == 0 ? pos[0] : pos[1], end, sum);
                                    ++v;
#pragma unroll
                                    for (int k = 0; k < PH; ++k) sum[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                                }
                                if ((mem1 >> j) & 1) {
                                    const float4 *src = reinterpret_cast<const float4 *>(
                                        Rv + ((__popc(steps[l2 + j] & upto) - 1) * 32 + l2 + j) * QS);
#pragma unroll
                                    for (int k = 0; k < PH; ++k) {
                                        if (end * PH + k >= PARTS) continue;
                                        const float4 x = src[end * PH + k];
                                        sum[k].x += x.x;
                                        sum[k].y += x.y;
                                        sum[k].z += x.z;
                                        sum[k].w += x.w;
                                    }
                                }
                            }
                            if (v >= 0)
                                put_sum<S>(v == 0 ? pos[0] : v == 1 ? pos[1] : pos[2], end, sum);
                            __syncwarp();
                            acc_rows<S>(acc, Rv, row1, Rs, at, hw, rb, cb);
                        }
                    }
                }
                __syncwarp();  // the sides and rows are read
            }
            // per-warp accumulators (the two halves summed) -> part
#pragma unroll
            for (int i = 0; i < RB; ++i)
#pragma unroll
                for (int j = 0; j < CB; ++j) {
                    acc[i][j] += __shfl_xor_sync(0xffffffffu, acc[i][j], 16);
                    const int e1 = rb * RB + i, e2 = cb * CB + j;
                    if (hw == 0 && e1 < Q && e2 < Q) Rv[e1 * Q + e2] = acc[i][j];
                }
            __syncthreads();
            each_sum(ts, as, [&](int at, float v) {
                swin += (double)v;
                if (!once) o[at] += v;
            });
            __syncthreads();  // the next pass may meet these entries; part aliases the staged rows
        }
        // FP64 totals: sfull over sub-LORs, sw over the window
        sfull = warp_sum_d(sfull);
        swin = warp_sum_d(swin);
        if (lane == 0) {
            red[warp] = sfull;
            red[SQ_WARPS + warp] = swin;
        }
        __syncthreads();
        double sf = 0.0, sw = 0.0;
#pragma unroll
        for (int w = 0; w < SQ_WARPS; ++w) {
            sf += red[w];
            sw += red[SQ_WARPS + w];
        }
        double scale = 1.0;
        if (norm == PSF_NORM_UNIT && sw > 0.0)
            scale = 1.0 / sw;  // total = 1
        else if (norm == PSF_NORM_EFF && sw > 0.0)
            scale = sf / (sw * nsub);  // total = mean eta1 eta2
        else
            scale = 1.0 / nsub;  // mean
        const float fs = (float)scale;
        if (once) {
            each_sum(__ffs(tsigns) - 1, __ffs(asigns) - 1, [&](int at, float v) { o[at] = v * fs; });
        } else {
#pragma unroll 1
            for (int k = t; k < E * E; k += SQ_T) o[k] *= fs;
        }
    }
}

// Spreads of a planar ring's LORs (one window row), whose crystals have only a
// few sub-positions: a CTA per LOR would keep 8 warps for 16 sub-LORs.  G lanes
// take a LOR (a half-warp for 16 sub-LORs), a lane a sub-LOR; the two responses
// go to shared memory over the whole window width, zero on the side the photon
// does not travel to, so the window is one small product sum_s r1_s (x) r2_s
// whatever the travel patterns, each lane owning a few of its entries (fixed
// order over s).  Responses and node decisions are spread_q_kernel's.  Bound by
// latency: RING2D, 2,016 LORs of 16 sub-LORs: 70 -> 15 us between events (about
// 5 us of which are the events'; 18 us with the node tangents found by the CTAs).
constexpr int SPL_T = 128;
constexpr int SPL_NSUB = 64;  // most sub-LORs: above, a warp's serial chunks lose to a CTA

template <int WT, int G>
__global__ void __launch_bounds__(SPL_T) spread_planar_kernel(
    Scan sc, Tab tb, const __grid_constant__ NodeTans tans, const float *__restrict__ T,
    const double *__restrict__ eta, const int32_t *__restrict__ lors, int64_t n_lors, int norm, float *__restrict__ out,
    const int32_t *__restrict__ sym) {
    constexpr int E = 2 * WT + 1, OWN = (E * E + G - 1) / G, NG = SPL_T / G;
    constexpr int RS = (2 * E) | 1;  // odd: the lanes' rows start in different banks
    extern __shared__ float spl_tabs[];          // node tangents
    __shared__ float R[NG][G][RS];                // a chunk's responses at both ends
    const GapConst gk = make_gapconst(sc, tb, tans, spl_tabs);
    __syncthreads();
    const int t = threadIdx.x, grp = t / G, l = t % G;
    const unsigned mask = G == 32 ? 0xffffffffu : ((1u << G) - 1u) << ((t & 31) / G * G);
    const int NP = tb.Pt * tb.Pa, nsub = NP * NP, nc = sc.Nt * sc.NR;
    for (int64_t lor = (int64_t)blockIdx.x * NG + grp; lor < n_lors;
         lor += (int64_t)gridDim.x * NG) {
        if (sym && sym[lor] >= 0) continue;  // an image of another class under the mirrors
        const int id1 = lors[2 * lor], id2 = lors[2 * lor + 1];
        const int ring1 = id1 / sc.Nt, c1 = id1 - ring1 * sc.Nt;
        const int ring2 = id2 / sc.Nt, c2 = id2 - ring2 * sc.Nt;
        const int b1 = c1 / sc.Nb, i1 = c1 - b1 * sc.Nb;
        const int b2 = c2 / sc.Nb, i2 = c2 - b2 * sc.Nb;
        float *o = out + lor * (int64_t)(E * E);
        if (b1 == b2 || id1 < 0 || id2 < 0 || id1 >= nc || id2 >= nc) {
            for (int e = l; e < E * E; e += G) o[e] = 0.0f;
            continue;
        }
        float sb1, cb1, sb2, cb2;
        sincospif(2.0f * b1 / sc.R, &sb1, &cb1);
        sincospif(2.0f * b2 / sc.R, &sb2, &cb2);
        float acc[OWN];
#pragma unroll
        for (int u = 0; u < OWN; ++u) acc[u] = 0.0f;
        double sfull = 0.0;
        for (int s0 = 0; s0 < nsub; s0 += G) {
            const int s = s0 + l, s1 = s / NP, s2 = s - s1 * NP;
            float *r1 = R[grp][l], *r2 = r1 + E;
#pragma unroll
            for (int e = 0; e < 2 * E; ++e) r1[e] = 0.0f;
            if (s < nsub) {
                const int p1 = s1 / tb.Pa, q1 = s1 - p1 * tb.Pa;
                const int p2 = s2 / tb.Pa, q2 = s2 - p2 * tb.Pa;
                const float se1 =
                    (i1 - 0.5f * (sc.Nb - 1)) * sc.pt + ((p1 + 0.5f) / tb.Pt - 0.5f) * sc.wt;
                const float ze1 = sc.z0 + ring1 * sc.pa + ((q1 + 0.5f) / tb.Pa - 0.5f) * sc.wa;
                const float se2 =
                    (i2 - 0.5f * (sc.Nb - 1)) * sc.pt + ((p2 + 0.5f) / tb.Pt - 0.5f) * sc.wt;
                const float ze2 = sc.z0 + ring2 * sc.pa + ((q2 + 0.5f) / tb.Pa - 0.5f) * sc.wa;
                const float x1 = sc.radius * cb1 - se1 * sb1, y1 = sc.radius * sb1 + se1 * cb1;
                const float x2 = sc.radius * cb2 - se2 * sb2, y2 = sc.radius * sb2 + se2 * cb2;
                const float dx = x1 - x2, dy = y1 - y2, dz = ze1 - ze2;
                float vn1, vt1, vn2, vt2;
                end_dir(dx, dy, cb1, sb1, vn1, vt1);
                end_dir(-dx, -dy, cb2, sb2, vn2, vt2);
                if (vn1 > 0.0f && vn2 > 0.0f) {
                    QResp<WT, 0> r;
                    end_resp_q<WT, 0>(sc, tb, gk, T, eta, i1, ring1, p1, q1, se1, ze1, vn1, vt1,
                                      dz, r);
                    const double e1 = r.eta;
                    const int g1 = vt1 >= 0.0f ? 1 : -1, g2 = vt2 >= 0.0f ? 1 : -1;
#pragma unroll
                    for (int x = 0; x <= WT; ++x) r1[WT + g1 * x] = r.q[x];
                    end_resp_q<WT, 0>(sc, tb, gk, T, eta, i2, ring2, p2, q2, se2, ze2, vn2, vt2,
                                      -dz, r);
#pragma unroll
                    for (int x = 0; x <= WT; ++x) r2[WT + g2 * x] = r.q[x];
                    sfull += e1 * r.eta;
                }
            }
            __syncwarp(mask);
            const int ns = nsub - s0 < G ? nsub - s0 : G;
#pragma unroll
            for (int u = 0; u < OWN; ++u) {
                const int e = l + u * G, e1 = e / E, e2 = e - e1 * E;
                if (e < E * E)
                    for (int k = 0; k < ns; ++k)
                        acc[u] = fmaf(R[grp][k][e1], R[grp][k][E + e2], acc[u]);
            }
            __syncwarp(mask);
        }
        // FP64 totals: sfull over sub-LORs, sw over the accumulated window
        double sw = 0.0;
#pragma unroll
        for (int u = 0; u < OWN; ++u) sw += (double)acc[u];
#pragma unroll
        for (int d = G / 2; d > 0; d >>= 1) {
            sfull += __shfl_xor_sync(mask, sfull, d);
            sw += __shfl_xor_sync(mask, sw, d);
        }
        double scale = 1.0 / nsub;                                          // NONE: mean
        if (norm == PSF_NORM_EFF && sw > 0.0) scale = sfull / (sw * nsub);  // total = mean eta1 eta2
        if (norm == PSF_NORM_UNIT && sw > 0.0) scale = 1.0 / sw;            // total = 1
        const float fs = (float)scale;
#pragma unroll
        for (int u = 0; u < OWN; ++u)
            if (l + u * G < E * E) o[l + u * G] = acc[u] * fs;
    }
}

template <int WT, int G>
static int launch_spread_planar(const Scan &sc, const Tab &tb, const float *T, const double *eta,
                                const int32_t *lors, int64_t n_lors, int norm, float *out,
                                const int32_t *sym, cudaStream_t st) {
    const size_t shm = sizeof(float) * (2 * tb.Kt + tb.Ka);
    int dev = 0, sms = 148;
    PSF_TRY(cudaGetDevice(&dev));
    PSF_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t need = (n_lors + SPL_T / G - 1) / (SPL_T / G), cap = (int64_t)sms * 8;
    {
        PSF_TIMED("spread_planar_kernel", st);
        spread_planar_kernel<WT, G><<<(int)(need < cap ? need : cap), SPL_T, shm, st>>>(
            sc, tb, make_nodetans(sc, tb), T, eta, lors, n_lors, norm, out, sym);
    }
    PSF_LAUNCHED();
    return PSF_OK;
}

template <int WT, int WA>
static int launch_spread_q(const Scan &sc, const Tab &tb, const float *T, const double *eta,
                           const int32_t *lors, int64_t n_lors, int wt, int wa, int norm, float *out,
                           const int32_t *sym, unsigned *queue, cudaStream_t st) {
    const size_t shm = spread_q_smem<WT, WA>(tb);
    if (shm > 200 * 1024) return PSF_EINVAL;
    PSF_TRY(cudaFuncSetAttribute(spread_q_kernel<WT, WA>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm));
    int dev = 0, sms = 148, per_sm = 0;
    PSF_TRY(cudaGetDevice(&dev));
    PSF_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PSF_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, spread_q_kernel<WT, WA>, SQ_T,
                                                          shm));
    if (per_sm < 1) per_sm = 1;
    const int64_t cap = (int64_t)sms * per_sm;
    {
        PSF_TIMED("spread_q_kernel", st);
        spread_q_kernel<WT, WA><<<(int)(n_lors < cap ? n_lors : cap), SQ_T, shm, st>>>(
            sc, tb, make_nodetans(sc, tb), T, eta, lors, n_lors, wt, wa, norm, out, sym, queue);
    }
    PSF_LAUNCHED();
    return PSF_OK;
}

}  // namespace psf

using namespace psf;


namespace psf {

// Symmetries of the spread classes of a structured set.  A: reflection
// through the axial centre plane (ring r -> NR-1-r for both crystals; the ring
// lattice has one pitch): ring difference d -> -d, every axial window offset
// negated.  T: reflection through block 0's centre plane (crystal x ->
// (Nb-1-x) mod Nt): every transaxial offset negated; when the reflected first
// crystal comes after the second the ends swap (the spread is transposed and
// d -> -d).  A and T are commuting involutions, so a class's orbit is
// {c, A c, T c, AT c}; the spread kernel computes the smallest class index of
// each orbit and the others are its images.  sym[c] = -1 for a computed class,
// else the computed class | SYM_A << 28 | SYM_T << 29 | SYM_SWAP << 30.
constexpr int SYM_A = 1, SYM_T = 2, SYM_SWAP = 4;

// T image of transaxial class tp: its class and whether the ends swap.
__device__ __forceinline__ void t_image(const LorSet &ls, const int32_t *tp_start, int64_t tp,
                                        int64_t *tp_t, bool *swap) {
    int a0, b0;
    ls.tp_decode(tp_start, tp, &a0, &b0);
    const int ma = (ls.Nb - 1 - a0 + ls.Nt) % ls.Nt, mb = (ls.Nb - 1 - b0 + ls.Nt) % ls.Nt;
    *swap = ma > mb;
    const int a1 = *swap ? mb : ma, b1 = *swap ? ma : mb;
    const int a10 = a1 % ls.Nb, b10 = b1 - (a1 - a10);
    *tp_t = tp_start[a10] + (b10 - ls.tp_lo(a10));
}

__global__ void spread_sym_kernel(LorSet ls, int32_t *__restrict__ sym) {
    extern __shared__ int32_t sy_pre[];  // tp_start [Nt + 1], rp_start [NR + 1]
    ls.stage_prefix(sy_pre, sy_pre + ls.Nt + 1);
    __syncthreads();
    const int D = 2 * ls.Dm + 1;
    const int64_t n_cls = ls.ntp_cls * D;
    if (blockIdx.x == 0 && threadIdx.x == 0) sym[n_cls] = 0;  // the spread kernel's queue
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_cls;
         c += (int64_t)gridDim.x * blockDim.x) {
        const int64_t tp = c / D;
        const int d = (int)(c - tp * D) - ls.Dm;
        int64_t tpt;
        bool sw;
        t_image(ls, sy_pre, tp, &tpt, &sw);
        const int dt = sw ? -d : d;
        const int64_t cA = tp * D + (-d + ls.Dm), cT = tpt * D + (dt + ls.Dm),
                      cAT = tpt * D + (-dt + ls.Dm);
        int64_t can = c < cA ? c : cA;
        can = can < cT ? can : cT;
        can = can < cAT ? can : cAT;
        if (can == c) {
            sym[c] = -1;
            continue;
        }
        // the map from the computed class to this one
        const int64_t ctp = can / D;
        const int cd = (int)(can - ctp * D) - ls.Dm;
        int64_t ctpt;
        bool csw;
        t_image(ls, sy_pre, ctp, &ctpt, &csw);
        const int cdt = csw ? -cd : cd;
        int flags;
        if (ctp * D + (-cd + ls.Dm) == c)
            flags = SYM_A;
        else if (ctpt * D + (cdt + ls.Dm) == c)
            flags = SYM_T | (csw ? SYM_SWAP : 0);
        else
            flags = SYM_A | SYM_T | (csw ? SYM_SWAP : 0);
        sym[c] = (int32_t)can | (flags << 28);
    }
}

// The classes that are images: W_c[e1][e2] = W_s[h(e1')][h(e2')] with
// (e1', e2') = (e2, e1) when the ends swap, h negating the axial offset
// (A) and/or the transaxial offset (T) of a window index.
__global__ void spread_mirror_kernel(int64_t n_cls, int Wt, int Wa,
                                     const int32_t *__restrict__ sym, float *__restrict__ out) {
    __shared__ int16_t hperm[4][256];  // window index maps per (A, T) flag pair
    const int W2a = 2 * Wa + 1, E = (2 * Wt + 1) * W2a, EE = E * E;
    for (int i = threadIdx.x; i < 4 * E; i += blockDim.x) {
        const int f = i / E, e = i - f * E;
        const int x = e / W2a, z = e - x * W2a;
        hperm[f][e] = (int16_t)(((f & SYM_T) ? 2 * Wt - x : x) * W2a + ((f & SYM_A) ? 2 * Wa - z : z));
    }
    __syncthreads();
    for (int64_t c = blockIdx.x; c < n_cls; c += gridDim.x) {
        const int32_t sv = sym[c];
        if (sv < 0) continue;
        const int64_t src = sv & 0x0fffffff;
        const int flags = sv >> 28;
        const int16_t *h = hperm[flags & 3];
        const bool swap = flags & SYM_SWAP;
        float *o = out + c * EE;
        const float *sp = out + src * EE;
        for (int e = threadIdx.x; e < EE; e += blockDim.x) {
            const int e1 = e / E, e2 = e - e1 * E;
            const int s1 = swap ? e2 : e1, s2 = swap ? e1 : e2;
            o[e] = sp[h[s1] * E + h[s2]];
        }
    }
}

static int bin_spread(const psf_scanner *scanner, const psf_table_desc *desc, const float *table,
                      const double *eta, const int32_t *lors, int64_t n_lors, int32_t half_t,
                      int32_t half_a, int32_t norm, float *spread, const int32_t *sym,
                      unsigned *queue, cudaStream_t st) {
    Scan sc;
    Tab tb;
    int rc = make_scan(scanner, &sc);
    if (rc) return rc;
    rc = make_tab(desc, sc, &tb, true);
    if (rc) return rc;
    if (half_t < 0 || half_a < 0 || (half_t + 1) * (half_a + 1) > SP_QMAX) return PSF_EINVAL;
    if (norm < PSF_NORM_NONE || norm > PSF_NORM_UNIT) return PSF_EINVAL;
    if (n_lors < 0) return PSF_EINVAL;
    if (n_lors == 0) return PSF_OK;
    if (!table || !eta || !lors || !spread) return PSF_EINVAL;
    if (tb.Pt * tb.Pa > 1024) return PSF_EINVAL;
    const int nsub = tb.Pt * tb.Pa * tb.Pt * tb.Pa;
    if (half_t == 3 && half_a == 0 && nsub <= SPL_NSUB && 2 * tb.Kt + tb.Ka <= 4096)
        return nsub <= 16
                   ? launch_spread_planar<3, 16>(sc, tb, table, eta, lors, n_lors, norm, spread,
                                                 sym, st)
                   : launch_spread_planar<3, 32>(sc, tb, table, eta, lors, n_lors, norm, spread,
                                                 sym, st);
    if (half_t == 3 && half_a == 0)
        return launch_spread_q<3, 0>(sc, tb, table, eta, lors, n_lors, half_t, half_a, norm, spread,
                                     sym, queue, st);
    if (half_t == 3 && (half_a == 2 || half_a == 3))
        return launch_spread_q<3, 3>(sc, tb, table, eta, lors, n_lors, half_t, half_a, norm, spread,
                                     sym, queue, st);
    size_t shm = spread_smem(tb, half_t, half_a);
    if (shm > 200 * 1024) return PSF_EINVAL;
    PSF_TRY(cudaFuncSetAttribute(spread_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)shm));
    int dev = 0, sms = 148;
    PSF_TRY(cudaGetDevice(&dev));
    PSF_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    int64_t grid = n_lors < (int64_t)sms * 8 ? n_lors : (int64_t)sms * 8;
    {
        PSF_TIMED("spread_kernel", st);
        spread_kernel<<<(int)grid, SP_THREADS, shm, st>>>(sc, tb, table, eta, lors, n_lors, half_t,
                                                          half_a, norm, spread, sym);
    }
    PSF_LAUNCHED();
    return PSF_OK;
}

}  // namespace psf

extern "C" int psf_bin_spread(const psf_scanner *scanner, const psf_table_desc *desc,
                              const float *table, const double *eta, const int32_t *lors,
                              int64_t n_lors, int32_t half_t, int32_t half_a, int32_t norm,
                              float *spread, void *stream) {
    PSF_RANGE("psf_bin_spread");
    return bin_spread(scanner, desc, table, eta, lors, n_lors, half_t, half_a, norm, spread,
                      nullptr, nullptr, as_stream(stream));
}

extern "C" int psf_bin_spread_classes(const psf_scanner *scanner, const psf_table_desc *desc,
                                      const float *table, const double *eta,
                                      const psf_lor_set *set, const int32_t *class_lors,
                                      int32_t half_t, int32_t half_a, int32_t norm,
                                      float *spread, void *stream) {
    PSF_RANGE("psf_bin_spread_classes");
    LorSet ls;
    int rc = make_lorset(scanner, set, &ls);
    if (rc) return rc;
    const int64_t n_cls = ls.ntp_cls * (2 * (int64_t)ls.Dm + 1);
    if (n_cls == 0) return PSF_OK;
    if (n_cls >= (1 << 28) || (2 * half_t + 1) * (2 * half_a + 1) > 256) return PSF_EINVAL;
    if (!class_lors || !spread) return PSF_EINVAL;
    cudaStream_t st = as_stream(stream);
    int32_t *sym = nullptr;
    // and the next class to compute: of a CTA's share, uneven parts are images
    PSF_TRY(cudaMallocAsync(&sym, sizeof(int32_t) * (n_cls + 1), st));
    int dev = 0, sms = 148;
    rc = cudaGetDevice(&dev) != cudaSuccess ||
                 cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess
             ? PSF_ECUDA
             : PSF_OK;
    if (!rc) {
        PSF_TIMED("spread_sym_kernel", st);
        spread_sym_kernel<<<grid_for(n_cls, 256), 256, sizeof(int32_t) * (ls.Nt + ls.NR + 2),
                            st>>>(ls, sym);
        if (cudaGetLastError() != cudaSuccess) rc = PSF_ECUDA;
    }
    // the smallest class of each orbit through the spread kernel ...
    if (!rc)
        rc = bin_spread(scanner, desc, table, eta, class_lors, n_cls, half_t, half_a, norm,
                        spread, sym, reinterpret_cast<unsigned *>(sym + n_cls), st);
    // ... the others as its images
    if (!rc) {
        PSF_TIMED("spread_mirror_kernel", st);
        spread_mirror_kernel<<<(int)(n_cls < (int64_t)sms * 8 ? n_cls : (int64_t)sms * 8), 256, 0,
                               st>>>(n_cls, half_t, half_a, sym, spread);
        if (cudaGetLastError() != cudaSuccess) rc = PSF_ECUDA;
    }
    cudaFreeAsync(sym, st);
    return rc;
}
