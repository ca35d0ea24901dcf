// Voxel-driven homogenization (Sec. 2.3, Eq. 11-12, Figs. 7-8), the paper's
// own matrix generator, for a planar (single crystal ring) scanner: a point
// source at each pixel centre emits k lines at theta_i = pi i / k with equal
// proportion 1/k; each line enters a crystal face at both ends and the
// detected pair (c1 + d1, c2 + d2) receives rho1[d1] rho2[d2] / k (Eq. 10,
// summed as Eq. 12) over the +-half_t window.  The hit geometry is FP64 (the
// sub-position decision of a hit on a cell boundary must not depend on
// rounding: such a hit is shared half and half by the two cells); the
// responses are the spread's (end_response: block0 and the gap path).
#include "psf_common.cuh"
#include "psf_end.cuh"
#include "psf_lorset.cuh"

namespace psf {

constexpr int VH_T = 256;
constexpr int VH_P = 12;             // most pixels of a CTA
constexpr int VH_MAX_ROWS = 16384;   // one pixel's column in shared memory

struct VhGeom {
    int R, Nb, Pt;
    double radius, wt, pt, width;  // width: transaxial block width
    double u_lo, u_hi;             // the side of the ring polygon in cells, off its ends
    double to_u, u0;               // face coordinate -> cell lattice: st * to_u + u0
    double Pp, iPp;                // cells per crystal pitch and its inverse
    bool whole;                    // no gaps: crystal i spans whole cells [i Pt, i Pt + Pt)
};

// What one end of a line needs of the block whose face plane it crosses: the
// same for every pixel, so it is computed when a pixel's line leaves through
// another block than the pixel before it, not per pixel.
struct VhBlock {
    int b;           // -1: none yet
    double idn, du;  // 1 / (direction . normal), cells per unit of path along the face
    int ent, ent1;   // table entries of sub-position 0: this block, the next one
    int sgt;         // travel direction along the face
    float cratio;    // cos(alpha) / cos(beta)
    bool valid, gap; // faces the photon, reaches the next block
};

// A pixel in the blocks' frames: the blocks' trigonometry and the pixel's
// normal and tangential coordinates from the CTA's tables, or (rings of so
// many blocks that the tables do not fit) computed when asked for.
template <bool STAGED>
struct VhFrame {
    int R;
    const double *cs, *pn, *pu;
    double cx, cy;
    __device__ __forceinline__ void trig(int b, double &c, double &s) const {
        if (STAGED) {
            c = cs[2 * b];
            s = cs[2 * b + 1];
        } else {
            sincospi(2.0 * b / R, &s, &c);
        }
    }
    __device__ __forceinline__ double normal(int b) const {
        if (STAGED) return pn[b];
        double c, s;
        trig(b, c, s);
        return cx * c + cy * s;
    }
    // tangential coordinate in cells of the face lattice
    __device__ __forceinline__ double cells(const VhGeom &g, int b) const {
        if (STAGED) return pu[b];
        double c, s;
        trig(b, c, s);
        return (cy * c - cx * s) * g.to_u + g.u0;
    }
};

template <bool STAGED>
__device__ __forceinline__ void vh_block(const VhGeom &g, const Scan &sc, const Tab &tb,
                                         const VhFrame<STAGED> &f, int b, double dx, double dy, VhBlock &k) {
    double cb, sb;
    f.trig(b, cb, sb);
    k.b = b;
    k.idn = 1.0 / (dx * cb + dy * sb);
    k.du = (dy * cb - dx * sb) * g.to_u;
    // the response's angles, as end_response forms them (no axial component)
    const float fx = (float)dx, fy = (float)dy;
    float fs, fc;
    sincospif(2.0f * b / sc.R, &fs, &fc);
    const float vn = fx * fc + fy * fs, vt = fy * fc - fx * fs;
    k.sgt = vt >= 0.0f ? 1 : -1;
    k.valid = vn > 0.0f;
    const float alpha = atan2f(fabsf(vt), vn);
    k.ent = (int)table_entry(tb, angle_node(alpha, tb.inv_dt, tb.Kt), 0, 0, 0);
    const float beta = alpha - sc.two_pi_R;
    k.gap = beta > 0.0f;
    k.cratio = 0.0f;
    k.ent1 = 0;
    if (k.gap) {
        k.cratio = cosf(alpha) / cosf(beta);
        k.ent1 = (int)table_entry(tb, angle_node(beta, tb.inv_dt, tb.Kt), 0, 0, 0);
    }
}

// The block whose face plane the ray leaves the ring polygon through: the
// plane crossed first.  (FP64, every block.)
template <bool STAGED>
__device__ __noinline__ int vh_exit(const VhGeom &g, const VhFrame<STAGED> &f, double dx,
                                    double dy) {
    int best = -1;
    double tmin = 1e300;
    for (int b = 0; b < g.R; ++b) {
        double cb, sb;
        f.trig(b, cb, sb);
        const double dn = dx * cb + dy * sb;
        if (!(dn > 1e-15)) continue;
        const double t = (g.radius - f.normal(b)) / dn;
        if (t > 0.0 && t < tmin) {
            tmin = t;
            best = b;
        }
    }
    return best;
}

// FP32 guess of the same block.
__device__ __forceinline__ int vh_guess(const VhGeom &g, const float2 *csf, const double *pn,
                                        float dx, float dy) {
    int best = -1;
    float tmin = 3e38f;
    for (int b = 0; b < g.R; ++b) {
        const float2 c = csf[b];
        const float dn = dx * c.x + dy * c.y;
        if (!(dn > 1e-5f)) continue;
        const float t = __fdividef((float)(g.radius - pn[b]), dn);
        if (t > 0.0f && t < tmin) {
            tmin = t;
            best = b;
        }
    }
    return best;
}

// Entries of the ray from a pixel along (dx, dy) into the crystal faces: the
// crystal and sub-position cell under the hit point (weight 1; a hit within
// 1e-9 cell of a cell boundary is shared by the two cells, weight 1/2 each,
// nothing past a block edge or into a gap).  k: the block of the pixel before,
// replaced when this ray leaves through another one.  Inside the
// polygon the block is the exit exactly when the hit lies within its side, so
// the kept block, then the FP32 guess, is tried with that test and every plane
// is only compared when both fail (or the pixel lies outside the polygon).
struct VhHit {
    int n, x0, p0, x1, p1;
    float w;
};

template <bool STAGED>
__device__ __forceinline__ VhHit vh_entry(const VhGeom &g, const Scan &sc, const Tab &tb,
                                          const VhFrame<STAGED> &f, const float2 *csf, bool inside,
                                          double dx, double dy, VhBlock &k) {
    VhHit h;
    h.n = 0;
    h.x0 = h.p0 = h.x1 = h.p1 = 0;
    h.w = 1.0f;
    double u = 0.0;
    auto hits = [&]() {  // within the side of block k.b, off its ends
        const double t = (g.radius - f.normal(k.b)) * k.idn;
        u = f.cells(g, k.b) + t * k.du;
        return k.idn > 0.0 && u > g.u_lo && u < g.u_hi;
    };
    if (!(inside && k.b >= 0 && hits())) {
        int b = STAGED && inside ? vh_guess(g, csf, f.pn, (float)dx, (float)dy) : -1;
        if (b >= 0 && b != k.b) vh_block(g, sc, tb, f, b, dx, dy, k);
        if (b < 0 || !hits()) {
            b = vh_exit(g, f, dx, dy);
            if (b < 0) return h;
            if (b != k.b) vh_block(g, sc, tb, f, b, dx, dy, k);
            hits();
        }
    }
    // cells of the face lattice: crystal i spans cells [i Pp, i Pp + Pt)
    const double ur = rint(u), off = u - ur;
    const bool on = fabs(off) < 1e-9;
    h.w = on ? 0.5f : 1.0f;
#pragma unroll 1
    for (int side = 0; side < (on ? 2 : 1); ++side) {
        int i, p;
        if (g.whole) {  // the lattice cell below (or beside) the hit, in integers
            const int cell = (int)ur - (on ? 1 - side : off < 0.0 ? 1 : 0);
            if (cell < 0 || cell >= g.Nb * g.Pt) continue;
            i = cell / g.Pt;
            p = cell - i * g.Pt;
        } else {
            const double uu = on ? ur - 0.5 + side : u;
            i = (int)floor(uu * g.iPp);
            if (i < 0 || i >= g.Nb) continue;
            const double cell = uu - i * g.Pp;
            if (cell >= g.Pt) continue;  // in the gap after crystal i
            p = (int)floor(cell);
        }
        if (h.n == 0) {
            h.x0 = i;
            h.p0 = p;
        } else {
            h.x1 = i;
            h.p1 = p;
        }
        ++h.n;
    }
    return h;
}

// Response of the crystals from entry crystal i on (q[0 .. WT], along the
// travel direction) of a photon entering at sub-position p: end_response's
// without an axial component, from the line's block quantities.
template <int WT>
__device__ __forceinline__ void vh_response(const Scan &sc, const Tab &tb,
                                            const float *__restrict__ T, const VhBlock &k, int i,
                                            int p, int iv1, int z, int Wt, float q[WT + 1]) {
    const int MM = tb.Mt * tb.Ma;
    const int iu = k.sgt > 0 ? p : tb.Pt - 1 - p;
    const float *Tb = T + (int64_t)(k.ent + iu * tb.Pa) * MM;
    const int edge = k.sgt > 0 ? sc.Nb - 1 - i : i;  // crystals of the block past the entry one
    const int nx0 = min(min(edge, Wt), tb.Mt - 1);
#pragma unroll
    for (int x = 0; x <= WT; ++x) q[x] = x <= nx0 ? ldg(Tb + x * tb.Ma) : 0.0f;
    if (!k.gap || edge >= Wt) return;  // the next block's crystals lie past the window
    const float s_entry = (i - 0.5f * (sc.Nb - 1)) * sc.pt + ((p + 0.5f) / tb.Pt - 0.5f) * sc.wt;
    const float nu = sc.half_w - k.sgt * s_entry;
    const float AP1 = sc.sigma + k.cratio * (sc.sigma + nu);
    const float qq = fmaxf(AP1 - sc.gt, 0.0f);
    const int m = f2i_rd(qq / sc.pt);
    const float f = qq - m * sc.pt;
    const float u1 = f < sc.wt ? (sc.wt - f) / sc.wt : 0.0f;
    const int iu1 = max(min(f2i_rd(u1 * tb.Pt), tb.Pt - 1), 0);
    const float *T1 = T + (int64_t)(k.ent1 + iu1 * tb.Pa + iv1) * MM + z;
#pragma unroll
    for (int X = 1; X <= WT; ++X) {
        const int j = X - edge - 1, x = m + 1 + j;
        if (X <= Wt && j >= 0 && j < sc.Nb && x < tb.Mt) q[X] += ldg(T1 + x * tb.Ma);
    }
}

// One CTA per P consecutive pixels; its threads take the lines, walk the
// pixels of each and add the pair products to the pixels' columns in shared
// memory, written out together (P neighbouring pixels of a row: whole
// sectors).  The FP64 work bounds it (2 lanes a clock on an SM): a line's
// direction is one FP64 sine and cosine for its P pixels, its block's normal
// component and angles are found once per block, the blocks' trigonometry and
// the pixels' block coordinates (in cells of the face lattice) once per CTA,
// which leaves 6 FP64 operations per line end and pixel.  RING2D, 720 lines:
// 7.03 -> 0.37 ms (a CTA per pixel that found all of this per line: 16 FP64
// sines a line end).  Neighbouring lines stay in a warp: they cross the same
// blocks (lines k / 32 apart in a warp: 0.57 ms, 9 of 32 lanes at work).
// split > 1 (few lines): split threads share a line, each with P / split pixels.
template <int WT, bool STAGED>
__global__ void __launch_bounds__(VH_T, WT <= 3 ? 3 : 2) voxel_homog_kernel(VhGeom g, Scan sc, Tab tb,
                                                           const float *__restrict__ T,
                                                           Img im, LorSet ls, int k, int Wt,
                                                           int P, int stride, int split,
                                                           float *__restrict__ A) {
    extern __shared__ __align__(16) unsigned char vh_raw[];
    const int SR = STAGED ? g.R : 0;                     // blocks with tables
    double *cs = reinterpret_cast<double *>(vh_raw);     // [SR][2] block cosine, sine
    double *pn = cs + 2 * SR;                            // [P][SR] pixel . normal
    double *pu = pn + P * SR;                            // [P][SR] its cells along the face
    float2 *csf = reinterpret_cast<float2 *>(pu + P * SR);  // [SR]
    float *vh_col = reinterpret_cast<float *>(csf + SR);      // [P][stride]
    int32_t *tp_start = reinterpret_cast<int32_t *>(vh_col + P * stride);
    int32_t *rp_start = tp_start + ls.Nt + 1;
    int *inside = rp_start + ls.NR + 1;  // [P]
    const int t = threadIdx.x;
    ls.stage_prefix(tp_start, rp_start);
    for (int b = t; b < SR; b += VH_T) {
        double sb, cb;
        sincospi(2.0 * b / g.R, &sb, &cb);
        cs[2 * b] = cb;
        cs[2 * b + 1] = sb;
        csf[b] = make_float2((float)cb, (float)sb);
    }
    const int64_t nvox = (int64_t)im.nx * im.ny;
    const int nrows = (int)ls.ntp;  // one crystal ring: rows are transaxial pairs
    const float inv_k = 1.0f / (float)k;
    // the axial entry of the gap path at z = z0 (end_response with dz = 0)
    const float zl = sc.z0 - (sc.z0 - 0.5f * sc.wa);
    const int k1 = f2i_rd(zl / sc.pa);
    const float fa = zl - k1 * sc.pa;
    const int k1s = fa <= sc.wa ? k1 : k1 + 1;
    const int iv1 = max(min(f2i_rd((fa <= sc.wa ? fa / sc.wa : 0.0f) * tb.Pa), tb.Pa - 1), 0);
    const int z = -k1s;  // its column that lands on the ring
    const bool gap_ok = z >= 0 && z < tb.Ma;
    auto pixel = [&](int64_t v, double &cx, double &cy) {
        const int iy = (int)(v / im.nx), ix = (int)(v - (int64_t)iy * im.nx);
        cx = im.ox + (ix + 0.5) * im.dx;
        cy = im.oy + (iy + 0.5) * im.dy;
    };
    for (int64_t v0 = (int64_t)blockIdx.x * P; v0 < nvox; v0 += (int64_t)gridDim.x * P) {
        const int np = nvox - v0 < P ? (int)(nvox - v0) : P;
        __syncthreads();  // the previous pixels' columns are written out
        for (int m = t; m < P * stride; m += VH_T) vh_col[m] = 0.0f;
        if (t < np) inside[t] = STAGED;
        __syncthreads();
        for (int j = t; j < np * SR; j += VH_T) {
            const int p = j / g.R, b = j - p * g.R;
            double cx, cy;
            pixel(v0 + p, cx, cy);
            pn[j] = cx * cs[2 * b] + cy * cs[2 * b + 1];
            pu[j] = (cy * cs[2 * b] - cx * cs[2 * b + 1]) * g.to_u + g.u0;
            if (!(pn[j] < g.radius)) inside[p] = 0;
        }
        __syncthreads();
        const int per = (np + split - 1) / split;
        for (int it = t; it < k * split; it += VH_T) {
            const int i = split == 1 ? it : it / split, part = it - i * split;
            double sth, cth;
            sincospi((double)i / k, &sth, &cth);
            VhBlock k1b, k2b;
            k1b.b = k2b.b = -1;
            const int pe = (part + 1) * per < np ? (part + 1) * per : np;
#pragma unroll 1
            for (int p = part * per; p < pe; ++p) {
                VhFrame<STAGED> f{g.R, cs, pn + p * SR, pu + p * SR, 0.0, 0.0};
                if (!STAGED) pixel(v0 + p, f.cx, f.cy);
                const bool in = inside[p];
                const VhHit h1 = vh_entry(g, sc, tb, f, csf, in, cth, sth, k1b);
                if (h1.n == 0) continue;
                const VhHit h2 = vh_entry(g, sc, tb, f, csf, in, -cth, -sth, k2b);
                if (h2.n == 0 || k1b.b == k2b.b || !k1b.valid || !k2b.valid) continue;
                float *column = vh_col + p * stride;
                const float wl = h1.w * h2.w * inv_k;
#pragma unroll 1
                for (int e = 0; e < h1.n * h2.n; ++e) {
                    const bool f1 = e < h2.n, f2 = e == 0 || e == h2.n;  // first cell of each end
                    const int x1 = f1 ? h1.x0 : h1.x1, p1 = f1 ? h1.p0 : h1.p1;
                    const int x2 = f2 ? h2.x0 : h2.x1, p2 = f2 ? h2.p0 : h2.p1;
                    VhBlock a1 = k1b, a2 = k2b;
                    a1.gap = k1b.gap && gap_ok;
                    a2.gap = k2b.gap && gap_ok;
                    float q1[WT + 1], q2[WT + 1];
                    vh_response<WT>(sc, tb, T, a1, x1, p1, iv1, z, Wt, q1);
                    vh_response<WT>(sc, tb, T, a2, x2, p2, iv1, z, Wt, q2);
                    const int ct1 = k1b.b * sc.Nb + x1, ct2 = k2b.b * sc.Nb + x2;
#pragma unroll
                    for (int a = 0; a <= WT; ++a) {
                        if (a > Wt || q1[a] == 0.0f) continue;
                        int X = ct1 + k1b.sgt * a;
                        X += X < 0 ? sc.Nt : (X >= sc.Nt ? -sc.Nt : 0);
#pragma unroll
                        for (int bb = 0; bb <= WT; ++bb) {
                            if (bb > Wt || q2[bb] == 0.0f) continue;
                            int Y = ct2 + k2b.sgt * bb;
                            Y += Y < 0 ? sc.Nt : (Y >= sc.Nt ? -sc.Nt : 0);
                            const int lo = X < Y ? X : Y, hi = X < Y ? Y : X;
                            if (X == Y || !ls.member(lo, hi, 0, 0)) continue;
                            atomicAdd(column + tp_start[lo] + (hi - ls.tp_lo(lo)),
                                      q1[a] * q2[bb] * wl);
                        }
                    }
                }
            }
        }
        __syncthreads();
        for (int j = t; j < nrows * P; j += VH_T) {
            const int m = j / P, p = j - m * P;
            if (p < np) A[(int64_t)m * nvox + v0 + p] = vh_col[p * stride + m];
        }
    }
}

}  // namespace psf

using namespace psf;

extern "C" int psf_voxel_homog(const psf_scanner *scanner, const psf_table_desc *desc,
                               const float *table, const double *eta, const psf_image *image,
                               const psf_lor_set *set, int32_t k, int32_t half_t, float *A,
                               void *stream) {
    PSF_RANGE("psf_voxel_homog");
    Scan sc;
    Tab tb;
    Img im;
    LorSet ls;
    int rc = make_scan(scanner, &sc);
    if (rc) return rc;
    rc = make_tab(desc, sc, &tb, true);
    if (rc) return rc;
    rc = make_img(image, &im);
    if (rc) return rc;
    rc = make_lorset(scanner, set, &ls);
    if (rc) return rc;
    if (ls.NR != 1 || im.nz != 1 || k < 1 || half_t < 0 || half_t + 1 > SP_QMAX) return PSF_EINVAL;
    if (ls.ntp > VH_MAX_ROWS || ls.ntp * (int64_t)im.nx * im.ny > ((int64_t)1 << 31)) return PSF_EINVAL;
    if (!table || !eta || !A) return PSF_EINVAL;
    VhGeom g;
    g.R = scanner->n_blocks;
    g.Nb = scanner->nt_block;
    g.Pt = desc->n_sub_t;
    g.radius = scanner->radius;
    g.wt = scanner->xtal_w_t;
    g.pt = scanner->xtal_w_t + scanner->gap_t;
    g.width = scanner->nt_block * scanner->xtal_w_t + (scanner->nt_block - 1) * scanner->gap_t;
    g.to_u = g.Pt / g.wt;
    g.u0 = 0.5 * g.width / g.wt * g.Pt;
    const double edge = g.radius * tan(M_PI / g.R) * (1.0 - 1e-9) * g.to_u;
    g.u_lo = g.u0 - edge;
    g.u_hi = g.u0 + edge;
    g.Pp = g.Pt * g.pt / g.wt;
    g.iPp = 1.0 / g.Pp;
    g.whole = g.pt == g.wt;
    cudaStream_t st = as_stream(stream);
    int dev = 0, sms = 148;
    PSF_TRY(cudaGetDevice(&dev));
    PSF_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int64_t nvox = (int64_t)im.nx * im.ny;
    const int stride = (int)((ls.ntp + 31) / 32 * 32 + 8);  // the pixels' columns 8 banks apart
    auto bytes = [&](int P, int SR) {
        return sizeof(double) * SR * (2 + 2 * P) + sizeof(float2) * SR + sizeof(float) * P * stride +
               sizeof(int32_t) * (ls.Nt + ls.NR + 2 + P);
    };
    // Pixels of a CTA: a line costs an SM's FP64 pipe about 3 units and each of
    // its pixels one, the SM's CTAs share the pipe, and whole waves of them run;
    // the fewest units (RING2D: 9 pixels, one wave, 0.37 ms; 4 pixels, three
    // waves, 0.47 ms).
    int P = 0;
    double best = 1e300;
    for (int p = 1; p <= VH_P; ++p) {
        const size_t b = bytes(p, g.R);
        if (b > 200 * 1024) break;
        const int per_sm = b <= 74 * 1024 ? 3 : b <= 112 * 1024 ? 2 : 1;
        const int64_t groups = (nvox + p - 1) / p, at_once = (int64_t)sms * per_sm;
        const double units = (double)((groups + at_once - 1) / at_once) * (3 + p) * per_sm;
        if (units < best) {
            best = units;
            P = p;
        }
    }
    const bool staged = P > 0;
    if (!staged) P = 1;  // thousands of blocks: no tables
    const size_t shm = bytes(P, staged ? g.R : 0);
    const int split = k <= VH_T / 4 && P >= 4 ? 4 : k <= VH_T / 2 && P >= 2 ? 2 : 1;
    const int64_t groups = (nvox + P - 1) / P;
    const int grid = (int)(groups < (int64_t)sms * 16 ? groups : (int64_t)sms * 16);
    auto launch = [&](auto kernel) -> int {
        PSF_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)shm));
        {
            PSF_TIMED("voxel_homog_kernel", st);
            kernel<<<grid, VH_T, shm, st>>>(g, sc, tb, table, im, ls, k, half_t, P, stride, split,
                                            A);
        }
        PSF_LAUNCHED();
        return PSF_OK;
    };
    // the response arrays' compile-time length: 4 covers the window in use
    if (!staged) return launch(voxel_homog_kernel<SP_QMAX - 1, false>);
    return half_t <= 3 ? launch(voxel_homog_kernel<3, true>)
                       : launch(voxel_homog_kernel<SP_QMAX - 1, true>);
}
