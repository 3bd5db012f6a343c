// PCM_FP64 Fock correction and gradient integrals (the interactions are those of
// f64.cuh; the potentials, which feed the linear solve, are in integrals.cu).
//
// Work is laid out for warps, because the FP64 pipe bounds every kernel here
// and a warp instruction that serves few lanes costs as much as a full one:
//   - the points in tiles of 32 that lie together (consecutive along a Hilbert
//     curve, ordered by exponent class within a tile);
//   - the primitive pairs of a class sorted by cell (the same curve) and, within
//     a cell, by exponent, so that a warp's pairs have the same reach.
// A tile's bounding sphere then tells, in a few FP32 instructions, whether a
// pair is beyond f64_far_T for all of the tile's points.  The gradient's point
// part runs a warp per point tile (a lane per point) over the pairs, the Fock
// accumulation a warp per 32 pairs (a lane per pair) over the point tiles.
// Against kernels with a seven-term Taylor step, the Hermite recurrence and FP64
// branches per interaction (25 / 41 FP64 instructions for ss / ps pairs; here 12 /
// 19 far and 16 / 27 near): Fock correction of a 150-atom s/sp cluster (6566 points)
// 72.1 -> 42.2 ms, gradient of a 100-atom s/p/d cluster 109.9 -> 68.3 ms.
#include <math.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "context.h"
#include "curve.cuh"
#include "f64.cuh"
#include "multipole64.cuh"

namespace pcm {

constexpr int F64_LSUM[6] = {0, 1, 2, 2, 3, 4};
constexpr int F64_SORT_POINTS = 1024;     // fewer points than this stay in library order
// side of a cell (bohr): expansions cost cells times points, direct interactions go by the
// cells' volume, so larger molecules take larger cells.  2.5 / 3.0 / 3.6, Fock correction and
// gradient: 200 s/sp atoms (8.4k points) 47.6 / 47.2 / 51.2 and 131 / 139 / 156 ms, 300 s/p/d
// (11.8k) 132 / 130 / 143 and 365 / 388 / 452, 550 s/p/d (23.5k) 388 / 347 / 350 and 1001 / 970 /
// 1071, 1000 s/p/d (43.5k) 1102 / 931 / 864 and 2696 / 2463 / 2552
constexpr double F64_CELL = 2.5, F64_CELL_LARGE = 3.0;
constexpr int F64_CELL_POINTS = 16000;    // from this many points on the larger one
constexpr int F64_PTBITS = 6;             // cells per side of the points' grid
constexpr int F64_RC_CLASSES = 16;        // up to this many exponent classes rho and cn are tabulated per (class, pair)
// From this many pairs and points on the cells' expansions are used: setting them up costs
// as much per pair as some hundred points one by one, and more with d shells, whose
// level is expanded for distant tiles only.  Measured without and with them, Fock
// correction / gradient: s and p shells 3.4k points 8.56 / 8.81 and 25.5 / 26.1 ms, 4.2k
// 12.5 / 11.8 and 37.2 / 35.2, 11.8k 158 / 92 (Fock); with d shells 4.6k 21.5 / 23.0 and
// 64.0 / 64.3, 5.1k 26.0 / 26.4 and 76.9 / 74.1, 7.8k (gradient) 224 / 170
constexpr int F64_MP_PAIRS = 40000;
constexpr int F64_MP_POINTS = 3500;
constexpr int F64_MP_POINTS_D = 5000;
// thread blocks that a launch aims at: many more than fit, so that blocks with few
// expanded cells and blocks with many even out (Fock correction of 300 s/sp atoms 100.8 ms
// with 16 per SM, 94.7 with 32, 91.6 with 64; gradient of 180 s/p/d atoms 180, 173, 169)
constexpr int F64_CTAS = 152 * 64;

// scratch that a context keeps: the partial sums of a Fock launch (more than this only
// where one row of them takes more; it takes rows from d classes, which have few pairs)
// and the table of rho and cn
constexpr size_t F64_S_BYTES = (size_t)128 << 20;
constexpr size_t F64_RC_BYTES = (size_t)1 << 30;

__device__ inline double f64_comp_factor(int l, int c)
{
    return l == 2 && (c == 1 || c == 2 || c == 4) ? 1.7320508075688772935 : 1.0;
}

// ---------------------------------------------------------------------------
// table of F_m / (2m-1)!! (f64.cuh): one warp per row, F_9 by quadrature (the
// lanes share the nodes), the others by downward recursion
// ---------------------------------------------------------------------------
constexpr int F64_GL = 24;
constexpr int F64_PANELS = 16;

__global__ void f64_table_kernel(const double *__restrict__ gx, const double *__restrict__ gw,
                                 double *__restrict__ tab)
{
    const int row = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (row >= F64_NROW) return;
    constexpr int TOP = F64_MTOP + 4;
    const double T = (double)row / F64_INV_DT;
    double s = 0.0;
    for (int k = lane; k < F64_GL * F64_PANELS; k += 32) {
        const double u = ((double)(k / F64_GL) + 0.5 * (gx[k % F64_GL] + 1.0)) / F64_PANELS;
        const double u2 = u * u;
        double w = 0.5 * gw[k % F64_GL] / F64_PANELS;
        for (int j = 0; j < TOP; ++j) w *= u2;
        s = fma(w, exp(-T * u2), s);
    }
    s = warp_sum(s);
    double F[TOP + 1];
    F[TOP] = s;
    const double eT = exp(-T);
#pragma unroll
    for (int m = TOP; m > 0; --m) F[m - 1] = fma(2.0 * T, F[m], eT) / (double)(2 * m - 1);
    if (lane != 0) return;
    double df = 1.0;
#pragma unroll
    for (int m = 0; m <= F64_MTOP; ++m) {
        if (m > 1) df *= (double)(2 * m - 1);
        double *c = tab + (size_t)row * F64_STRIDE + 6 * m;
        c[0] = F[m] / df;
        c[1] = -F[m + 1] / df;
        c[2] = F[m + 2] / (2.0 * df);
        c[3] = -F[m + 3] / (6.0 * df);
        c[4] = F[m + 4] / (24.0 * df);
        c[5] = 0.0;
    }
    // H_m upwards from H_0 = -sqrt(pi / T) erfc(sqrt T) / 2, all of one sign
    double *hrow = tab + F64_TABLE + (size_t)row * F64_STRIDE;
    const bool on = T >= F64_H_MIN - 0.1;
    double H[TOP + 1];
    H[0] = on ? -0.5 * sqrt(PCM_PI / T) * erfc(sqrt(T)) : 0.0;
#pragma unroll
    for (int m = 1; m <= TOP; ++m) H[m] = on ? fma((double)(2 * m - 1), H[m - 1], -eT) / (2.0 * T) : 0.0;
    df = 1.0;
#pragma unroll
    for (int m = 0; m <= F64_MTOP; ++m) {
        if (m > 1) df *= (double)(2 * m - 1);
        double *c = hrow + 6 * m;
        c[0] = H[m] / df;
        c[1] = -H[m + 1] / df;
        c[2] = H[m + 2] / (2.0 * df);
        c[3] = -H[m + 3] / (6.0 * df);
        c[4] = H[m + 4] / (24.0 * df);
        c[5] = 0.0;
    }
}

int f64_build_tables(pcm_ctx *c)
{
    std::vector<double> x, w;
    gauss_legendre(F64_GL, x, w);
    DBuf<double> g;
    PCM_TRY(g.alloc(2 * F64_GL));
    PCM_CUDA(cudaMemcpyAsync(g.p, x.data(), F64_GL * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    PCM_CUDA(cudaMemcpyAsync(g.p + F64_GL, w.data(), F64_GL * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    PCM_TRY(c->f64.tab.alloc(2 * (size_t)F64_TABLE));
    f64_table_kernel<<<(F64_NROW + 3) / 4, 128, 0, c->stream>>>(g.p, g.p + F64_GL, c->f64.tab.p);
    PCM_LAUNCHED(c);
    PCM_CUDA(cudaStreamSynchronize(c->stream));  // g is freed on return
    return PCM_OK;
}

// ---------------------------------------------------------------------------
// orders of points and pairs
// ---------------------------------------------------------------------------
__global__ void f64_point_key_kernel(int M, const double *__restrict__ px, const double *__restrict__ py,
                                     const double *__restrict__ pz, F64Box box, unsigned *__restrict__ key,
                                     int *__restrict__ val)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= M) return;
    key[k] = curve_key<F64_PTBITS>(px[k], py[k], pz[k], box);
    val[k] = k;
}

// one warp per tile of 32 points: order by class, gather, bounding sphere
__global__ void f64_point_tile_kernel(int M, const int *__restrict__ val, const double *__restrict__ px,
                                      const double *__restrict__ py, const double *__restrict__ pz,
                                      const int *__restrict__ pcls, int *__restrict__ idx, int *__restrict__ cls,
                                      const double *__restrict__ cls_zeta, F64Box box, F64Pt *__restrict__ xyz,
                                      float4 *__restrict__ x32, float4 *__restrict__ sph)
{
    const int tile = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (tile * 32 >= M) return;
    const int nt = min(32, M - tile * 32);
    const int at = tile * 32 + min(lane, nt - 1);
    const int k = val ? val[at] : at;
    const int e = pcls[k];
    int rank = 0;
    for (int o = 0; o < nt; ++o) {
        const int eo = __shfl_sync(0xffffffffu, e, o);
        rank += (eo < e || (eo == e && o < lane)) ? 1 : 0;
    }
    const double x = px[k], y = py[k], z = pz[k];
    const float fx = (float)(x - box.mid[0]), fy = (float)(y - box.mid[1]), fz = (float)(z - box.mid[2]);
    if (lane < nt) {
        idx[tile * 32 + rank] = k;
        cls[tile * 32 + rank] = e;
        xyz[tile * 32 + rank] = F64Pt{x, y, z, 0.0};
        x32[tile * 32 + rank] = make_float4(fx, fy, fz, (float)(1.0 / (cls_zeta[e] * cls_zeta[e])));
    }
    float lo[3] = {fx, fy, fz}, hi[3] = {fx, fy, fz};
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
    const float cx = 0.5f * (lo[0] + hi[0]), cy = 0.5f * (lo[1] + hi[1]), cz = 0.5f * (lo[2] + hi[2]);
    const float dx = fx - cx, dy = fy - cy, dz = fz - cz;
    float r2 = dx * dx + dy * dy + dz * dz;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
    if (lane == 0) sph[tile] = make_float4(cx, cy, cz, sqrtf(r2) * 1.0001f + box.slack);
}

__device__ __forceinline__ int f64_class_of(const F64Src &s, int g)
{
    int k = 0;
#pragma unroll
    for (int i = 1; i < 6; ++i) k += g >= s.off[i] ? 1 : 0;
    return k;
}

// rho and cn of f64.cuh for exponent z2 = zeta^2
__device__ __forceinline__ double2 f64_rho_cn(double p, double z2)
{
    const double rho = p * z2 / (p + z2);
    return make_double2(rho, 2.0 * sqrt(rho / PCM_PI));
}

// sorted pair data: kept index, centre and exponent, FP32 copies for the tests,
// and (for few exponent classes) rho and cn per class
__global__ void f64_pair_gather_kernel(int n, F64Src src, const int *__restrict__ val, int ncls,
                                       const double *__restrict__ cls_zeta, F64Box box, int *__restrict__ ord,
                                       double *__restrict__ P, float4 *__restrict__ info, double2 *__restrict__ rc)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    const int k = f64_class_of(src, g), r = (val ? val[g] : g) - src.off[k];
    const double x = src.Px[k][r], y = src.Py[k][r], z = src.Pz[k][r], p = src.p[k][r];
    ord[g] = r;
    P[g] = x;
    P[(size_t)n + g] = y;
    P[2 * (size_t)n + g] = z;
    P[3 * (size_t)n + g] = p;
    // an exponent beyond 1e30 acts as that one (rho is zeta^2 either way)
    info[g] = make_float4((float)(x - box.mid[0]), (float)(y - box.mid[1]), (float)(z - box.mid[2]),
                          (float)fmin(p, 1e30));
    if (rc)
        for (int e = 0; e < ncls; ++e) rc[(size_t)e * n + g] = f64_rho_cn(p, cls_zeta[e] * cls_zeta[e]);
}

// point tiles and sorted pairs of the current geometry and basis
int f64_prepare(pcm_ctx *c)
{
    F64Int &f = c->f64;
    const int M = c->M;
    const F64Box box = f.box = cavity_box(c, M < F64_CELL_POINTS ? F64_CELL : F64_CELL_LARGE);
    const F64Src src = kept_pairs(c, f.off);
    const int n = f.off[6];
    f.ntile = (M + 31) / 32;
    PCM_TRY(f.pt_idx.alloc(M));
    PCM_TRY(f.pt_cls.alloc(M));
    PCM_TRY(f.pt_xyz.alloc(M));
    PCM_TRY(f.pt_x32.alloc(M));
    PCM_TRY(f.pt_sph.alloc(f.ntile));
    const bool sort_pts = M >= F64_SORT_POINTS;
    if (sort_pts) {
        PCM_TRY(f.key.alloc(M));
        PCM_TRY(f.val.alloc(M));
        f64_point_key_kernel<<<(M + 127) / 128, 128, 0, c->stream>>>(M, c->px.p, c->py.p, c->pz.p, box, f.key.p,
                                                                    f.val.p);
        PCM_LAUNCHED(c);
        PCM_TRY(sort_pairs(c, M, 3 * F64_PTBITS, f.key, f.val));
    }
    f64_point_tile_kernel<<<(f.ntile + 3) / 4, 128, 0, c->stream>>>(M, sort_pts ? f.val.p : nullptr, c->px.p, c->py.p,
                                                                   c->pz.p, c->pcls.p, f.pt_idx.p, f.pt_cls.p,
                                                                   c->cls_zeta.p, box, f.pt_xyz.p, f.pt_x32.p,
                                                                   f.pt_sph.p);
    PCM_LAUNCHED(c);
    f.mp.on = false;
    if (n == 0) return PCM_OK;
    PCM_TRY(f.ord.alloc(n));
    PCM_TRY(f.P.alloc(4 * (size_t)n));
    PCM_TRY(f.info.alloc(n));
    f.use_rc = c->ncls <= F64_RC_CLASSES && (size_t)c->ncls * n * sizeof(double2) <= F64_RC_BYTES;
    if (f.use_rc) PCM_TRY(f.rc.alloc((size_t)c->ncls * n));
    // within a cell by exponent
    bool sorted;
    PCM_TRY(pair_order(c, src, box, false, &sorted));
    f64_pair_gather_kernel<<<(n + 127) / 128, 128, 0, c->stream>>>(n, src, sorted ? f.val.p : nullptr, c->ncls,
                                                                  c->cls_zeta.p, box, f.ord.p, f.P.p, f.info.p,
                                                                  f.use_rc ? f.rc.p : nullptr);
    PCM_LAUNCHED(c);
    const int points = f.off[6] > f.off[3] ? F64_MP_POINTS_D : F64_MP_POINTS;   // ds, dp or dd pairs
    if (n >= F64_MP_PAIRS && M >= points) PCM_TRY(mp_prepare(c, box, src, CURVE_HBITS, CURVE_PBITS));
    return PCM_OK;
}

// ---------------------------------------------------------------------------
// ESP preparation: density test of Eq. 18 over the sorted pairs of every class,
// one compaction, then the coefficients of f64_dot per kept pair
// ---------------------------------------------------------------------------
template <int LA, int LB>
__global__ void f64_flag_kernel(int off, int npair, const int *__restrict__ ord, const int *__restrict__ sp,
                                const int *__restrict__ ia, const int *__restrict__ ib, const int *__restrict__ spA,
                                const int *__restrict__ spB, const int *__restrict__ sh_bf,
                                const double *__restrict__ Q, const double *__restrict__ Pm, int nbf, double thresh,
                                unsigned char *__restrict__ flag)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= npair) return;
    const int r = ord[off + j];
    const int s = sp[r];
    const int A = spA[s], B = spB[s];
    const bool mirror = (A != B) || (ia[r] != ib[r]);
    const int fa = sh_bf[A], fb = sh_bf[B];
    double wmax = 0.0;
    for (int a = 0; a < ncart(LA); ++a)
        for (int b = 0; b < ncart(LB); ++b) {
            double w = Pm[(size_t)(fa + a) * nbf + fb + b];
            if (mirror) w += Pm[(size_t)(fb + b) * nbf + fa + a];
            wmax = fmax(wmax, fabs(w));
        }
    flag[off + j] = thresh <= 0.0 || wmax * Q[r] >= thresh ? 1 : 0;
}

// kept pairs before each class
__global__ void f64_class_counts_kernel(F64Src src, const int *__restrict__ pos, int *__restrict__ out)
{
    if (threadIdx.x < 7) out[threadIdx.x] = pos[src.off[threadIdx.x]];
}

// record of ESP pair j (list: sorted positions): centre and far-field terms of
// its Hermite density D_tuv = -(2 pi / p) K sum_ab W_ab c_a c_b E^ab_tuv
// (W_ab = P_ab + P_ba for a pair that stands for its mirror image too)
template <int LA, int LB>
__global__ void f64_coef_kernel(int nesp, int off, const int *__restrict__ list, const int *__restrict__ ord,
                                const int *__restrict__ sp, const int *__restrict__ ia, const int *__restrict__ ib,
                                const int *__restrict__ spA, const int *__restrict__ spB,
                                const int *__restrict__ sh_atom, const int *__restrict__ sh_off,
                                const int *__restrict__ sh_bf, const double *__restrict__ cnorm,
                                const double *__restrict__ xyz, const double *__restrict__ Px,
                                const double *__restrict__ Py, const double *__restrict__ Pz,
                                const double *__restrict__ pp, const double *__restrict__ pref,
                                const double *__restrict__ Pm, int nbf, int *__restrict__ elist,
                                double *__restrict__ rec, double *__restrict__ B_)
{
    constexpr int L = LA + LB;
    constexpr int NH = nherm(L);
    constexpr int NC = far_nterms(L);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nesp) return;
    const int r = ord[list[j]];
    elist[j] = r;
    const int s = sp[r];
    const int A = spA[s], B = spB[s];
    const int i1 = ia[r], i2 = ib[r];
    const bool mirror = (A != B) || (i1 != i2);
    const double p = pp[r];
    const double P[3] = {Px[r], Py[r], Pz[r]};
    const double *RA = xyz + 3 * sh_atom[A], *RB = xyz + 3 * sh_atom[B];
    E1T<LA, LB> Ex, Ey, Ez;
    const double inv2p = 0.5 / p;
    hermite_E1T<LA, LB>(P[0] - RA[0], P[0] - RB[0], inv2p, Ex);
    hermite_E1T<LA, LB>(P[1] - RA[1], P[1] - RB[1], inv2p, Ey);
    hermite_E1T<LA, LB>(P[2] - RA[2], P[2] - RB[2], inv2p, Ez);
    const double cc = cnorm[sh_off[A] + i1] * cnorm[sh_off[B] + i2];
    const int fa = sh_bf[A], fb = sh_bf[B];
    double D[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) D[h] = 0.0;
#pragma unroll
    for (int a = 0; a < ncart(LA); ++a) {
        const int ax = cart_e(LA, a, 0), ay = cart_e(LA, a, 1), az = cart_e(LA, a, 2);
#pragma unroll
        for (int b = 0; b < ncart(LB); ++b) {
            const int bx = cart_e(LB, b, 0), by = cart_e(LB, b, 1), bz = cart_e(LB, b, 2);
            double w = Pm[(size_t)(fa + a) * nbf + fb + b];
            if (mirror) w += Pm[(size_t)(fb + b) * nbf + fa + a];
            w *= cc * f64_comp_factor(LA, a) * f64_comp_factor(LB, b);
            // E_t vanishes for t > i + j
#pragma unroll
            for (int t = 0; t <= ax + bx; ++t)
#pragma unroll
                for (int u = 0; u <= ay + by; ++u) {
                    const double wxy = w * Ex.e[ax][bx][t] * Ey.e[ay][by][u];
#pragma unroll
                    for (int v = 0; v <= az + bz; ++v)
                        D[hidx(t, u, v)] = fma(wxy, Ez.e[az][bz][v], D[hidx(t, u, v)]);
                }
        }
    }
    constexpr FarContrib FC = far_contrib(L);
    const double g = -pref[r] * 0.88622692545275801365 / sqrt(p);   // sqrt(pi) / (2 sqrt(p))
    double G[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) G[k] = 0.0;
#pragma unroll
    for (int q = 0; q < FC.count; ++q) G[FC.term[q]] = fma(FC.w[q], D[FC.h[q]], G[FC.term[q]]);
    double *o = rec + (size_t)j * f64_rec(L);
    o[0] = P[0];
    o[1] = P[1];
    o[2] = P[2];
#pragma unroll
    for (int k = 0; k < NC; ++k) o[3 + k] = g * G[k];
    if (!B_) return;
    // the same density as shifts of solid harmonics, for the cells' moments
    constexpr MpMap MM = mp_map(L);
    double b[(L + 1) * (L + 1)];
#pragma unroll
    for (int q = 0; q < (L + 1) * (L + 1); ++q) b[q] = 0.0;
#pragma unroll
    for (int i = 0; i < MM.count; ++i) b[MM.s[i]] = fma(MM.B[i], D[MM.h[i]], b[MM.s[i]]);
#pragma unroll
    for (int q = 0; q < (L + 1) * (L + 1); ++q) B_[(size_t)q * nesp + j] = g * b[q];
}

template <int LA, int LB>
static int f64_flag_class(pcm_ctx *c, int k, const double *dP)
{
    PairClass &pc = c->cls[k];
    if (pc.npair == 0) return PCM_OK;
    f64_flag_kernel<LA, LB><<<(pc.npair + 127) / 128, 128, 0, c->stream>>>(
        c->f64.off[k], pc.npair, c->f64.ord.p, pc.sp.p, pc.ia.p, pc.ib.p, pc.spA.p, pc.spB.p, c->sh_bf.p, pc.Q.p, dP,
        c->nbf, c->opt.schwarz, c->f64.flag.p);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

template <int LA, int LB>
static int f64_coef_class(pcm_ctx *c, int k, const double *dP)
{
    PairClass &pc = c->cls[k];
    if (pc.nesp == 0) return PCM_OK;
    PCM_TRY(pc.elist.alloc(pc.npair));
    f64_coef_kernel<LA, LB><<<(pc.nesp + 127) / 128, 128, 0, c->stream>>>(
        pc.nesp, c->f64.off[k], c->f64.list.p + c->f64.eoff[k], c->f64.ord.p, pc.sp.p, pc.ia.p, pc.ib.p, pc.spA.p,
        pc.spB.p, c->sh_atom.p, c->sh_off.p, c->sh_bf.p, c->cnorm.p, c->xyz.p, pc.Px.p, pc.Py.p, pc.Pz.p, pc.p.p,
        pc.pref.p, dP, c->nbf, pc.elist.p, c->f64.rec.p + c->f64.roff[k],
        c->f64.mp.on ? c->f64.B.p + c->f64.boff[k] : nullptr);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

int f64_esp_prepare(pcm_ctx *c, const double *dP)
{
    F64Int &f = c->f64;
    const int n = f.off[6];
    for (int k = 0; k < 6; ++k) c->cls[k].nesp = c->cls[k].nesp_same = 0;
    for (int k = 0; k <= 6; ++k) f.eoff[k] = 0;
    if (n == 0) return PCM_OK;
    PCM_TRY(f.flag.alloc(n));
    PCM_TRY(f.list.alloc(n));
    PCM_TRY(f.pos.alloc((size_t)n + 1));
    PCM_TRY((f64_flag_class<0, 0>(c, 0, dP)));
    PCM_TRY((f64_flag_class<1, 0>(c, 1, dP)));
    PCM_TRY((f64_flag_class<1, 1>(c, 2, dP)));
    PCM_TRY((f64_flag_class<2, 0>(c, 3, dP)));
    PCM_TRY((f64_flag_class<2, 1>(c, 4, dP)));
    PCM_TRY((f64_flag_class<2, 2>(c, 5, dP)));
    PCM_TRY(compact_flags(c, f.flag.p, n, f.list.p, f.pos.p, c->iscal.p + 8));
    F64Src src{};
    for (int k = 0; k <= 6; ++k) src.off[k] = f.off[k];
    f64_class_counts_kernel<<<1, 32, 0, c->stream>>>(src, f.pos.p, c->iscal.p);
    PCM_LAUNCHED(c);
    PCM_CUDA(cudaMemcpyAsync(f.eoff, c->iscal.p, 7 * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    PCM_CUDA(cudaStreamSynchronize(c->stream));
    static constexpr int REC[6] = {f64_rec(0), f64_rec(1), f64_rec(2), f64_rec(2), f64_rec(3), f64_rec(4)};
    size_t total = 0, btotal = 0;
    for (int k = 0; k < 6; ++k) {
        c->cls[k].nesp = f.eoff[k + 1] - f.eoff[k];
        f.roff[k] = total;
        total += (size_t)REC[k] * c->cls[k].nesp;
        f.boff[k] = btotal;
        btotal += (size_t)((F64_LSUM[k] + 1) * (F64_LSUM[k] + 1)) * c->cls[k].nesp;
    }
    PCM_TRY(f.rec.alloc(std::max<size_t>(1, total)));
    if (f.mp.on) PCM_TRY(f.B.alloc(std::max<size_t>(1, btotal)));
    PCM_TRY((f64_coef_class<0, 0>(c, 0, dP)));
    PCM_TRY((f64_coef_class<1, 0>(c, 1, dP)));
    PCM_TRY((f64_coef_class<1, 1>(c, 2, dP)));
    PCM_TRY((f64_coef_class<2, 0>(c, 3, dP)));
    PCM_TRY((f64_coef_class<2, 1>(c, 4, dP)));
    PCM_TRY((f64_coef_class<2, 2>(c, 5, dP)));
    return PCM_OK;
}

// ---------------------------------------------------------------------------
// main kernels
// ---------------------------------------------------------------------------
// what the kernels read of the points and of one class's sorted pairs
struct F64Points {
    int M, ntile;
    const F64Pt *xyz;      // x, y, z, charge (Fock)
    const int *cls;
    const float4 *x32;       // x, y, z, zeta^-2 in FP32
    const float4 *sph;
    const double *cls_zeta;
    float zmin2;             // smallest zeta^2: the smallest rho, the longest reach
    float slack, pad;        // error bounds of the FP32 tests (f64_reaches, f64_is_near)
    const double *tab;
};

struct F64Pairs {
    int n;                   // pairs of the launch
    int stride;              // sorted pairs of all classes
    const int *list;         // sorted positions of the pairs (null: 0 .. n-1 from first)
    int first;
    const float4 *info;
    const double *P;         // 4 x stride
    const double2 *rc;       // ncls x stride, or null
    const double *rec;       // ESP records
    const int *cell;         // cell of every sorted pair, and the order of its expansion
    const unsigned char *order;   // for every (tile, cell); null: no expansions
    unsigned char omask;     // bits of an order that say it serves the class
    int ncell;
};

__device__ __forceinline__ bool f64_expanded(const F64Pairs &a, int tile, int cell)
{
    return (a.order[(size_t)tile * a.ncell + cell] & a.omask) != 0;
}

__device__ __forceinline__ double2 f64_load_rc(const F64Pairs &a, const F64Points &t, int e, int pos)
{
    if (a.rc) return __ldg(a.rc + (size_t)e * a.stride + pos);
    const double z = t.cls_zeta[e];
    return f64_rho_cn(a.P[3 * (size_t)a.stride + pos], z * z);
}

// resident blocks of 128 threads per SM the register allocation aims for: the
// FP64 pipe is full with two or three warps per scheduler
constexpr int f64_min_blocks(int terms) { return terms <= 11 ? 4 : (terms <= 24 ? 3 : 2); }

// Point part of the integral gradient (gc of Eq. 22): per point the sums over
// the ESP pairs of the derivatives with respect to P.  One point tile per block,
// a lane per point; the block's four warps and the grid's rows share the pairs
// in chunks of `ch` (at most 32: a lane per pair for the reach test).
// part[row][component][slot].
template <int L>
__global__ void __launch_bounds__(128, f64_min_blocks(far_nterms(L)))
    f64_grad_kernel(F64Pairs a, F64Points t, int ch, double *__restrict__ part)
{
    constexpr int NC = far_nterms(L);
    constexpr int REC = f64_rec(L);
    constexpr int LB = L + 1;      // highest b_n
    constexpr float FT = (float)f64_far_T(LB);
    __shared__ double red[4][3][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int tile = blockIdx.x;
    const int slot = min(tile * 32 + lane, t.M - 1);
    const F64Pt c = t.xyz[slot];
    const int e = t.cls[slot];
    const float4 c32 = t.x32[slot], sph = t.sph[tile];
    double acc[3] = {0.0, 0.0, 0.0};
    // one interaction per lane with pair j of the list.  FAR: every lane beyond
    // farT; NEAR: the near part of expanded pairs, lanes with `on`; else near or
    // far by T
    constexpr int FAR = 0, NEAR = 1, BOTH = 2;
    auto interact = [&](auto kind, int j, bool on) {
        const double2 *r = reinterpret_cast<const double2 *>(a.rec + (size_t)j * REC);
        double v[REC];
#pragma unroll
        for (int i = 0; i < REC / 2; ++i) {
            const double2 x = __ldg(r + i);
            v[2 * i] = x.x;
            v[2 * i + 1] = x.y;
        }
        double G[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) G[k] = v[3 + k];
        const double X = v[0] - c.x, Y = v[1] - c.y, Z = v[2] - c.z;
        const double R2 = fma(X, X, fma(Y, Y, Z * Z));
        double b[LB + 1];
        if constexpr (decltype(kind)::value == FAR)
            f64_far<LB>(R2, b);
        else if constexpr (decltype(kind)::value == NEAR)
            f64_near_minus_far<LB>(R2, f64_load_rc(a, t, e, a.list[j]), on, t.tab, b);
        else
            f64_terms<LB>(R2, f64_load_rc(a, t, e, a.list[j]), false, t.tab, b);
        f64_dot_grad<L>(X, Y, Z, b, G, acc);
    };
    for (int j0 = (blockIdx.y * 4 + w) * ch; j0 < a.n; j0 += gridDim.y * 4 * ch) {
        // a lane per pair: does it reach the tile, is its cell expanded for it
        const bool act = lane < ch && j0 + lane < a.n;
        bool nr = false, ex = false;
        float4 info = make_float4(0.f, 0.f, 0.f, 1.f);
        if (act) {
            const int pos = a.list[j0 + lane];
            info = a.info[pos];
            nr = f64_reaches(info, sph, t.zmin2, FT, t.slack);
            ex = a.order && f64_expanded(a, tile, a.cell[pos]);
        }
        const unsigned nm = __ballot_sync(0xffffffffu, nr), em = __ballot_sync(0xffffffffu, ex);
        const unsigned direct = __ballot_sync(0xffffffffu, act) & ~em;
        for (unsigned m = direct & ~nm; m; m &= m - 1)
            interact(std::integral_constant<int, FAR>{}, j0 + __ffs(m) - 1, true);
        for (unsigned m = direct & nm; m; m &= m - 1)
            interact(std::integral_constant<int, BOTH>{}, j0 + __ffs(m) - 1, true);
        // expanded pairs that reach the tile: each lane (point) takes the next
        // pair near it, so that the warp makes as many steps as its busiest lane
        // has near pairs
        unsigned near = 0;
        for (unsigned m = nm & em; m; m &= m - 1) {
            const int o = __ffs(m) - 1;
            const float4 b = make_float4(__shfl_sync(0xffffffffu, info.x, o), __shfl_sync(0xffffffffu, info.y, o),
                                         __shfl_sync(0xffffffffu, info.z, o), __shfl_sync(0xffffffffu, info.w, o));
            near |= f64_is_near(b.x - c32.x, b.y - c32.y, b.z - c32.z, 1.f / b.w + c32.w, FT, t.pad) ? 1u << o : 0u;
        }
        int o = 0;
        while (__any_sync(0xffffffffu, near != 0)) {
            const bool on = near != 0;
            if (on) o = __ffs(near) - 1;
            near &= near - 1;
            interact(std::integral_constant<int, NEAR>{}, j0 + o, on);
        }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) red[w][d][lane] = acc[d];
    __syncthreads();
    if (w == 0 && tile * 32 + lane < t.M) {
        const size_t S = (size_t)t.ntile * 32;
#pragma unroll
        for (int d = 0; d < 3; ++d)
            part[((size_t)blockIdx.y * 3 + d) * S + tile * 32 + lane] =
                (red[0][d][lane] + red[1][d][lane]) + (red[2][d][lane] + red[3][d][lane]);
    }
}

// g[d][point] -= q times the sum of the partial rows, in row order
__global__ void f64_grad_reduce_kernel(int M, int S, int rows, const double *__restrict__ part,
                                       const int *__restrict__ idx, const double *__restrict__ q,
                                       double *__restrict__ g)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= M) return;
    const int k = idx[s];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double v = 0.0;
        for (int r = 0; r < rows; ++r) v += part[((size_t)r * 3 + d) * S + s];
        g[(size_t)d * M + k] -= q[k] * v;
    }
}

// the points' charges beside their coordinates
__global__ void f64_point_charge_kernel(int M, const int *__restrict__ idx, const double *__restrict__ q,
                                        F64Pt *__restrict__ xyz)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < M) xyz[s].w = q[idx[s]];
}

// Fock accumulation: a warp per 32 sorted pairs (a lane per pair), over the
// point tiles blockIdx.y, + gridDim.y, ...; S[row][term][pair] = sum_k q_k b_n
// X^a Y^b Z^c per term of farfield.cuh (mapped to Hermite components by
// f64_fold_kernel; a term costs one FMA per interaction, the Hermite recurrence
// about two).
template <int L>
__global__ void __launch_bounds__(128, f64_min_blocks(far_nterms(L)))
    f64_fock_kernel(F64Pairs a, F64Points t, double *__restrict__ S)
{
    constexpr int NC = far_nterms(L);
    constexpr float FT = (float)f64_far_T(L);
    const int lane = threadIdx.x & 31;
    const int j = (blockIdx.x * 4 + (threadIdx.x >> 5)) * 32 + lane;
    if (j - lane >= a.n) return;
    const int jj = min(j, a.n - 1);
    const int pos = a.list ? a.list[jj] : a.first + jj;
    const double Px = a.P[pos], Py = a.P[(size_t)a.stride + pos], Pz = a.P[2 * (size_t)a.stride + pos];
    const float4 info = a.info[pos];
    const int cell = a.order ? a.cell[pos] : 0;
    double acc[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) acc[k] = 0.0;
    const float ip = 1.f / info.w;
    for (int tile = blockIdx.y; tile < t.ntile; tile += gridDim.y) {
        const bool reaches = f64_reaches(info, t.sph[tile], t.zmin2, FT, t.slack);
        const bool expanded = a.order && f64_expanded(a, tile, cell);
        const int s0 = tile * 32, nt = min(32, t.M - s0);
        if (!__all_sync(0xffffffffu, expanded)) {
            // one by one: every point, near or far by T where some pair reaches the tile
            if (!__any_sync(0xffffffffu, reaches && !expanded)) {
                for (int s = s0; s < s0 + nt; ++s) {
                    const F64Pt c = t.xyz[s];
                    const double X = Px - c.x, Y = Py - c.y, Z = Pz - c.z;
                    double b[L + 1];
                    f64_far<L>(fma(X, X, fma(Y, Y, Z * Z)), b);
                    const double q = expanded ? 0.0 : c.w;
#pragma unroll
                    for (int n = 0; n <= L; ++n) b[n] *= q;
                    f64_accumulate<L>(X, Y, Z, b, acc);
                }
            } else {
                int cur = -1;
                double2 rc = make_double2(1.0, 1.0);
                for (int s = s0; s < s0 + nt; ++s) {
                    const F64Pt c = t.xyz[s];
                    const int e = t.cls[s];
                    if (e != cur) {
                        cur = e;
                        rc = f64_load_rc(a, t, e, pos);
                    }
                    const double X = Px - c.x, Y = Py - c.y, Z = Pz - c.z;
                    double b[L + 1];
                    f64_terms<L>(fma(X, X, fma(Y, Y, Z * Z)), rc, expanded, t.tab, b);
#pragma unroll
                    for (int n = 0; n <= L; ++n) b[n] *= c.w;
                    f64_accumulate<L>(X, Y, Z, b, acc);
                }
            }
        }
        if (!__any_sync(0xffffffffu, reaches && expanded)) continue;
        // expanded pairs that reach the tile: each lane (pair) takes the next point
        // near it, so that the warp makes as many steps as its busiest lane has
        // near points
        unsigned near = 0;
        for (int i = 0; i < nt; ++i) {
            const float4 c = t.x32[s0 + i];
            near |= f64_is_near(info.x - c.x, info.y - c.y, info.z - c.z, ip + c.w, FT, t.pad) ? 1u << i : 0u;
        }
        if (!expanded) near = 0;
        int o = 0;
        while (__any_sync(0xffffffffu, near != 0)) {
            const bool on = near != 0;
            if (on) o = __ffs(near) - 1;
            near &= near - 1;
            const F64Pt c = t.xyz[s0 + o];
            const double X = Px - c.x, Y = Py - c.y, Z = Pz - c.z;
            double b[L + 1];
            f64_near_minus_far<L>(fma(X, X, fma(Y, Y, Z * Z)), f64_load_rc(a, t, t.cls[s0 + o], pos), on, t.tab, b);
#pragma unroll
            for (int n = 0; n <= L; ++n) b[n] *= c.w;
            f64_accumulate<L>(X, Y, Z, b, acc);
        }
    }
    if (j < a.n)
#pragma unroll
        for (int k = 0; k < NC; ++k) S[((size_t)blockIdx.y * NC + k) * a.n + j] = acc[k];
}

// sums of the rows into the first one, an accumulator per thread: classes with few
// pairs are split over up to a row per tile
__global__ void f64_rows_kernel(size_t n, int rows, double *__restrict__ S)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    int r = 0;
    for (; r + 4 <= rows; r += 4)
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] += S[(size_t)(r + k) * n + i];
    for (; r < rows; ++r) v[0] += S[(size_t)r * n + i];
    S[i] = (v[0] + v[1]) + (v[2] + v[3]);
}

// W_tuv = sqrt(pi) / (2 sqrt(p)) sum over the terms (the transpose of the
// mapping that made the ESP's coefficients) of the rows' sums, written at the
// kept pair's place (ord) or, without ord, at j
template <int L>
__global__ void f64_fold_kernel(F64Pairs a, int rows, const double *__restrict__ S, const double *__restrict__ V,
                                const int *__restrict__ ord, int ldw, double *__restrict__ W)
{
    constexpr int NC = far_nterms(L);
    constexpr int NH = nherm(L);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= a.n) return;
    double acc[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        double v = 0.0;
        for (int r = 0; r < rows; ++r) v += S[((size_t)r * NC + k) * a.n + j];
        acc[k] = v;
    }
    const int pos = a.list ? a.list[j] : a.first + j;
    const double g = 0.88622692545275801365 / sqrt(a.P[3 * (size_t)a.stride + pos]);
    constexpr FarContrib FC = far_contrib(L);
    double out[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) out[h] = 0.0;
#pragma unroll
    for (int q = 0; q < FC.count; ++q) out[FC.h[q]] = fma(FC.w[q], acc[FC.term[q]], out[FC.h[q]]);
    if (V) {
        // the cells' local expansions at the pair (multipole64.cu)
        constexpr MpMap MM = mp_map(L);
        double v[(L + 1) * (L + 1)];
#pragma unroll
        for (int q = 0; q < (L + 1) * (L + 1); ++q) v[q] = V[(size_t)q * a.n + j];
#pragma unroll
        for (int i = 0; i < MM.count; ++i) out[MM.h[i]] = fma(MM.V[i], v[MM.s[i]], out[MM.h[i]]);
    }
    const int at = ord ? ord[pos] : j;
#pragma unroll
    for (int h = 0; h < NH; ++h) W[(size_t)h * ldw + at] = g * out[h];
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static F64Points f64_points(pcm_ctx *c)
{
    F64Points t;
    t.M = c->M;
    t.ntile = c->f64.ntile;
    t.xyz = c->f64.pt_xyz.p;
    t.cls = c->f64.pt_cls.p;
    t.x32 = c->f64.pt_x32.p;
    t.sph = c->f64.pt_sph.p;
    t.cls_zeta = c->cls_zeta.p;
    t.zmin2 = (float)(c->h_cls_zeta[0] * c->h_cls_zeta[0]) * 0.99999f;
    t.slack = c->f64.box.slack;
    t.pad = 2001.f * t.slack * t.slack;
    t.tab = c->f64.tab.p;
    return t;
}

static F64Pairs f64_pairs(pcm_ctx *c, int k, bool esp)
{
    F64Int &f = c->f64;
    F64Pairs a;
    a.n = esp ? c->cls[k].nesp : c->cls[k].npair;
    a.stride = f.off[6];
    a.list = esp ? f.list.p + f.eoff[k] : nullptr;
    a.first = f.off[k];
    a.info = f.info.p;
    a.P = f.P.p;
    a.rc = f.use_rc ? f.rc.p : nullptr;
    a.rec = esp ? f.rec.p + f.roff[k] : nullptr;
    a.cell = f.mp.pcell.p;
    a.order = f.mp.on ? f.mp.order.p : nullptr;
    a.omask = mp_level(k) == 0 ? 0xff : MP_ALL;
    a.ncell = f.mp.ncell;
    return a;
}

// chunk length and grid rows of a point-part launch over n pairs
static void f64_grad_plan(int n, int ntile, int *ch, int *rows)
{
    *ch = (int)std::min<long long>(32, std::max<long long>(4, (long long)n * ntile / (4LL * F64_CTAS)));
    const int want = (F64_CTAS + ntile - 1) / ntile;
    *rows = std::max(1, std::min(want, (n + 4 * *ch - 1) / (4 * *ch)));
}

template <int L>
static int f64_grad_launch(pcm_ctx *c, int k, int ch, int rows, double *part)
{
    f64_grad_kernel<L><<<dim3(c->f64.ntile, rows), 128, 0, c->stream>>>(f64_pairs(c, k, true), f64_points(c), ch,
                                                                       part);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

// gk[3][M] += the point part of the gradient over the ESP pairs
int f64_grad_point(pcm_ctx *c, const double *dq, double *gk)
{
    const int nt = c->f64.ntile;
    const size_t S = (size_t)nt * 32;
    int ch[6], rows[6], total = 0;
    for (int k = 0; k < 6; ++k) {
        rows[k] = 0;
        if (c->cls[k].nesp == 0) continue;
        f64_grad_plan(c->cls[k].nesp, nt, &ch[k], &rows[k]);
        total += rows[k];
    }
    if (total == 0) return PCM_OK;
    const int far = c->f64.mp.on ? mp_rows(c) : 0;
    total += far;
    PCM_TRY(c->esp_part.alloc(total * 3 * S));
    double *part = c->esp_part.p;
    if (far) {
        PCM_TRY(mp_order(c, true));
        PCM_TRY(mp_grad_far(c, part));
        part += (size_t)far * 3 * S;
    }
    for (int k = 0; k < 6; ++k) {
        if (rows[k] == 0) continue;
        switch (F64_LSUM[k]) {
        case 0: PCM_TRY(f64_grad_launch<0>(c, k, ch[k], rows[k], part)); break;
        case 1: PCM_TRY(f64_grad_launch<1>(c, k, ch[k], rows[k], part)); break;
        case 2: PCM_TRY(f64_grad_launch<2>(c, k, ch[k], rows[k], part)); break;
        case 3: PCM_TRY(f64_grad_launch<3>(c, k, ch[k], rows[k], part)); break;
        case 4: PCM_TRY(f64_grad_launch<4>(c, k, ch[k], rows[k], part)); break;
        }
        part += (size_t)rows[k] * 3 * S;
    }
    f64_grad_reduce_kernel<<<(c->M + 127) / 128, 128, 0, c->stream>>>(c->M, (int)S, total, c->esp_part.p,
                                                                     c->f64.pt_idx.p, dq, gk);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

int f64_charges(pcm_ctx *c, const double *dq, bool gradient)
{
    f64_point_charge_kernel<<<(c->M + 127) / 128, 128, 0, c->stream>>>(c->M, c->f64.pt_idx.p, dq, c->f64.pt_xyz.p);
    PCM_LAUNCHED(c);
    if (c->f64.mp.on) {
        PCM_TRY(mp_order(c, gradient));
        PCM_TRY(mp_local(c));
    }
    return PCM_OK;
}

template <int L>
static int f64_w_launch(pcm_ctx *c, const F64Pairs &a, int level, const int *ord, double *W)
{
    const int nb = (a.n + 127) / 128;
    const int fit = (int)std::min<size_t>(1 << 20, F64_S_BYTES / (sizeof(double) * far_nterms(L) * a.n));
    const int rows = std::max(1, std::min({c->f64.ntile, (F64_CTAS + nb - 1) / nb, fit}));
    PCM_TRY(c->f64.S.alloc((size_t)rows * far_nterms(L) * a.n));
    f64_fock_kernel<L><<<dim3(nb, rows), 128, 0, c->stream>>>(a, f64_points(c), c->f64.S.p);
    PCM_LAUNCHED(c);
    if (rows > 2) {
        const size_t ns = (size_t)far_nterms(L) * a.n;
        f64_rows_kernel<<<(unsigned)((ns + 127) / 128), 128, 0, c->stream>>>(ns, rows, c->f64.S.p);
        PCM_LAUNCHED(c);
    }
    if (c->f64.mp.on) PCM_TRY(mp_l2p(c, level, L, a.n, a.list, a.first));
    f64_fold_kernel<L><<<(a.n + 31) / 32, 32, 0, c->stream>>>(a, rows > 2 ? 1 : rows, c->f64.S.p, c->f64.mp.on ? c->f64.mp.V.p : nullptr, ord,
                                                 a.n, W);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

// W[nherm(L)][pairs] of class k for the charges of f64_charges: over the kept
// pairs in kept order (the Fock correction, L = la + lb), or over the ESP pairs
// in ESP order (the gradient, L = la + lb + 1)
int f64_w(pcm_ctx *c, int k, bool esp, double *W)
{
    const F64Pairs a = f64_pairs(c, k, esp);
    if (a.n == 0) return PCM_OK;
    const int *ord = esp ? nullptr : c->f64.ord.p;
    const int level = mp_level(k);
    switch (F64_LSUM[k] + (esp ? 1 : 0)) {
    case 0: return f64_w_launch<0>(c, a, level, ord, W);
    case 1: return f64_w_launch<1>(c, a, level, ord, W);
    case 2: return f64_w_launch<2>(c, a, level, ord, W);
    case 3: return f64_w_launch<3>(c, a, level, ord, W);
    case 4: return f64_w_launch<4>(c, a, level, ord, W);
    case 5: return f64_w_launch<5>(c, a, level, ord, W);
    }
    return PCM_ERR_ARG;
}

}  // namespace pcm
