// Multipole far field of the PCM_FP64 integrals.
//
// Beyond f64_far_T every pair is a set of point multipoles at its centre
// (farfield.cuh), so the pairs of one cell act on distant points through the
// cell's moments, and distant charges act on them through a local expansion
// about the cell's centre.  With the solid harmonics
//   R_l^m = r^l P_l^m(cos t) e^{im phi} / (l+m)!,  I_l^m = (l-m)! P_l^m(cos t) e^{im phi} / r^{l+1}
// (no Condon-Shortley sign; negative m by conjugation and (-1)^m),
//   1/|r - s| = sum_{l, m} conj(R_l^m(s)) I_l^m(r),  |s| < |r|,
// and derivatives of R are other R with coefficients +-1:
//   dz R_l^m = R_{l-1}^m,  (dx - i dy) R_l^m = R_{l-1}^{m-1},  (dx + i dy) R_l^m = -R_{l-1}^{m+1},
// so a Hermite density D_tuv becomes (L+1)^2 real numbers B_s (mp_map), the
// moments are sums over pairs of B_s R_l^m shifted by (n, mu), and the
// Hermite components W_tuv at a pair are the transpose of that.  (Greengard and
// Rokhlin, J. Comput. Phys. 73, 325 (1987), for the expansions and their bounds.)
//
// Both harmonics factor into a real recurrence in l with the same coefficients,
//   b_m = 1, b_l = u b_{l-1} - gamma_lm v b_{l-2},
//   R_l^m = hn_lm b_l (x + iy)^m,          u = z,     v = r^2,
//   I_l^m = (2l-1)!! b_l ((x + iy)/r^2)^m / r,  u = z/r^2, v = 1/r^2,
// three FP64 instructions per (l, m), then two per real sum.
//
// A cell is expanded for a tile of points when some order up to MP_P leaves less
// than its rounding out of any interaction (mp_order_for, with the highest
// derivative that the classes of a level take), when all interactions have
// T >= F64_H_MIN (the near form of more diffuse pairs is far below their far
// form), and when the expansion costs less than its pairs do one by one.  Pairs of such a cell that still have T < f64_far_T
// somewhere in the tile add near minus far form for those points.
#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "context.h"
#include "f64.cuh"
#include "multipole64.cuh"

namespace pcm {

// ---------------------------------------------------------------------------
// constants: gamma_lm (negated), hn_lm, w_m (2l-1)!! in column order
// ---------------------------------------------------------------------------
struct MpTables {
    double ngam[MP_NLM], hn[MP_NLM], wd[MP_NLM], d[MP_NLM];
};

constexpr MpTables mp_tables()
{
    MpTables t{};
    for (int m = 0; m <= MP_P; ++m) {
        double h = 1.0;
        for (int k = 1; k <= m; ++k) h /= 2.0 * k;
        for (int l = m; l <= MP_P; ++l) {
            if (l > m) h *= (2.0 * l - 1.0) / (((double)l + m) * ((double)l - m));
            double df = 1.0;
            for (int k = 2 * l - 1; k > 1; k -= 2) df *= k;
            const int i = mp_at(l, m);
            t.ngam[i] = l >= m + 2 ? -((l - 1.0) * (l - 1.0) - (double)m * m) / ((2.0 * l - 1.0) * (2.0 * l - 3.0)) : 0.0;
            t.hn[i] = h;
            t.d[i] = df;
            t.wd[i] = (m == 0 ? 1.0 : 2.0) * df;
        }
    }
    return t;
}

__constant__ const MpTables c_mp = mp_tables();

// ---------------------------------------------------------------------------
// cells
// ---------------------------------------------------------------------------
__global__ void mp_mark_kernel(int n, const unsigned *__restrict__ key, int shift, unsigned mask,
                               unsigned char *__restrict__ flag)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < n) flag[(key[g] >> shift) & mask] = 1;
}

// cell of every sorted pair, the cells' ranges per class, centres, radii and smallest
// exponents
__global__ void mp_cells_kernel(int n, const unsigned *__restrict__ key, int shift, unsigned mask,
                                const int *__restrict__ id, F64Src src, F64Box box, int side,
                                const double *__restrict__ P, int maxcell, int *__restrict__ pcell,
                                int *__restrict__ cbeg, int *__restrict__ cend, double *__restrict__ cxyz,
                                int *__restrict__ crad, int *__restrict__ cpmin)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    const unsigned kg = key[g] >> shift;
    const int cell = id[kg & mask];
    pcell[g] = cell;
    int k = 0;
#pragma unroll
    for (int i = 1; i < 6; ++i) k += g >= src.off[i] ? 1 : 0;
    // the grid cell by the same arithmetic as the key's
    const double s = (double)side * box.inv;
    double c[3], r2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double x = P[(size_t)d * n + g];
        const int i = min(max((int)((x - box.lo[d]) * s), 0), side - 1);
        c[d] = box.lo[d] + (i + 0.5) / s;
        r2 += (x - c[d]) * (x - c[d]);
    }
    if (g == 0 || (key[g - 1] >> shift) != kg) {
        cbeg[k * maxcell + cell] = g;
#pragma unroll
        for (int d = 0; d < 3; ++d) cxyz[3 * cell + d] = c[d];
    }
    if (g == n - 1 || (key[g + 1] >> shift) != kg) cend[k * maxcell + cell] = g + 1;
    // largest distance (non-negative floats order as integers), rounded up
    atomicMax(&crad[cell], __float_as_int((float)sqrt(r2) * 1.000001f));
    atomicMin(&cpmin[cell], __float_as_int((float)fmin(P[3 * (size_t)n + g], 1e30) * 0.999999f));
}

// Order of the expansion of a cell for a tile of points, with MP_ALL if it serves all
// of the cell's classes, without if only those of level 0; 0: pair by pair.  extra:
// derivatives beyond the pairs' own (the gradient's one)
__global__ void mp_order_kernel(int ntile, int ncell, int maxcell, F64Box box, const float4 *__restrict__ sph,
                                const double *__restrict__ cxyz, const int *__restrict__ crad,
                                const int *__restrict__ cpmin, float zmin2, const int *__restrict__ cbeg,
                                const int *__restrict__ cend, int extra,
                                unsigned char *__restrict__ order)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ntile * ncell) return;
    const int t = i / ncell, c = i % ncell;
    const float4 s = sph[t];
    const float dx = s.x - (float)(cxyz[3 * c] - box.mid[0]), dy = s.y - (float)(cxyz[3 * c + 1] - box.mid[1]),
                dz = s.z - (float)(cxyz[3 * c + 2] - box.mid[2]);
    const float r = fmaxf(__int_as_float(crad[c]), 1e-3f);
    const float D = sqrtf(dx * dx + dy * dy + dz * dz) * 0.99999f - box.slack - s.w;
    unsigned char o = 0;
    // smallest T of an interaction: below F64_H_MIN the near form is the difference of
    // two larger numbers
    const float pm = __int_as_float(cpmin[c]), rho = pm / (pm + zmin2) * zmin2;
    if (D > r && rho * (D - r) * (D - r) >= 1.0001f * (float)F64_H_MIN) {
        // FP64 instructions per point: far forms of the cell's pairs
        // (12 ... 95 by class) against 5 per (l, m) and 8 per m
        const float cost[6] = {12.f, 19.f, 32.f, 32.f, 55.f, 95.f};
        const int deg[6] = {0, 1, 2, 2, 3, 4};
        float direct[MP_LEVELS] = {0.f, 0.f};   // pairs up to each level
        int n[MP_LEVELS] = {0, 0};
        for (int k = 0; k < 6; ++k) {
            const int pairs = cend[k * maxcell + c] - cbeg[k * maxcell + c];
            for (int v = mp_level(k); v < MP_LEVELS; ++v) {
                direct[v] += cost[k] * (float)pairs;
                if (pairs > 0) n[v] = deg[k];
            }
        }
        for (int v = 0; v < MP_LEVELS; ++v) {
            const int p = mp_order_for(r / D, n[v] + extra);
            if (p > 0 && direct[v] >= MP_GAIN * (2.5f * (p + 1) * (p + 2) + 8.f * (p + 1)))
                o = (unsigned char)p | (v == MP_LEVELS - 1 ? MP_ALL : 0);
        }
    }
    order[i] = o;
}

int mp_prepare(pcm_ctx *c, const F64Box &box, const F64Src &src, int bits, int shift)
{
    F64Mp &mp = c->f64.mp;
    const int n = src.off[6], side = 1 << bits, nc = side * side * side;
    mp.on = false;
    PCM_TRY(c->flags8.alloc(nc));
    PCM_TRY(mp.id.alloc((size_t)nc + 1));
    PCM_CUDA(cudaMemsetAsync(c->flags8.p, 0, nc, c->stream));
    mp_mark_kernel<<<(n + 255) / 256, 256, 0, c->stream>>>(n, c->f64.key.p, shift, nc - 1, c->flags8.p);
    PCM_LAUNCHED(c);
    PCM_TRY(compact_flags(c, c->flags8.p, nc, nullptr, mp.id.p, c->iscal.p));
    int cnt = 0;
    PCM_CUDA(cudaMemcpyAsync(&cnt, c->iscal.p, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    PCM_CUDA(cudaStreamSynchronize(c->stream));
    mp.ncell = cnt;
    PCM_TRY(mp.pcell.alloc(n));
    PCM_TRY(mp.range.alloc(12 * (size_t)cnt));
    PCM_TRY(mp.cxyz.alloc(3 * (size_t)cnt));
    PCM_TRY(mp.crad.alloc(cnt));
    PCM_TRY(mp.cpmin.alloc(cnt));
    PCM_TRY(mp.order.alloc((size_t)cnt * c->f64.ntile));
    PCM_CUDA(cudaMemsetAsync(mp.range.p, 0, 12 * (size_t)cnt * sizeof(int), c->stream));
    PCM_CUDA(cudaMemsetAsync(mp.crad.p, 0, (size_t)cnt * sizeof(int), c->stream));
    PCM_CUDA(cudaMemsetAsync(mp.cpmin.p, 0x7f, (size_t)cnt * sizeof(int), c->stream));   // above any exponent
    mp_cells_kernel<<<(n + 127) / 128, 128, 0, c->stream>>>(n, c->f64.key.p, shift, nc - 1, mp.id.p, src, box, side,
                                                           c->f64.P.p, cnt, mp.pcell.p, mp.range.p,
                                                           mp.range.p + 6 * (size_t)cnt, mp.cxyz.p, mp.crad.p,
                                                           mp.cpmin.p);
    PCM_LAUNCHED(c);
    mp.on = true;
    return PCM_OK;
}

// orders of the expansions for every (tile, cell)
int mp_order(pcm_ctx *c, bool gradient)
{
    F64Mp &mp = c->f64.mp;
    const int no = mp.ncell * c->f64.ntile;
    mp_order_kernel<<<(no + 127) / 128, 128, 0, c->stream>>>(
        c->f64.ntile, mp.ncell, mp.ncell, c->f64.box, c->f64.pt_sph.p, mp.cxyz.p, mp.crad.p,
        mp.cpmin.p, (float)(c->h_cls_zeta[0] * c->h_cls_zeta[0]) * 0.99999f, mp.range.p,
        mp.range.p + 6 * (size_t)mp.ncell, gradient ? 1 : 0, mp.order.p);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

// ---------------------------------------------------------------------------
// moments
// ---------------------------------------------------------------------------
// e_m = (x + iy)^m by the bits of m from the squares
__device__ __forceinline__ double2 mp_power(double x, double y, int m)
{
    double er = 1.0, ei = 0.0;
    while (m) {
        if (m & 1) {
            const double t = er * x - ei * y;
            ei = fma(er, y, ei * x);
            er = t;
        }
        m >>= 1;
        if (m) {
            const double t = (x - y) * (x + y);
            y = 2.0 * x * y;
            x = t;
        }
    }
    return make_double2(er, ei);
}

// scratch of the raw sums: the cells go in groups of this much
constexpr size_t P2M_RAW_BYTES = (size_t)128 << 20;
constexpr int P2M_NP = 32;                          // pairs per batch, a lane each
constexpr int P2M_NW = (MP_P + 2) / 2;              // warp w fills columns w and MP_P - w: MP_P + 2 rows each
constexpr int P2M_NT = 32 * P2M_NW;
static_assert(P2M_NT >= MP_NLM, "a thread per (l, m)");

__host__ __device__ constexpr size_t p2m_smem(int L)
{
    return ((size_t)MP_NLM * (P2M_NP + 1) + 2 * (size_t)(MP_P + 1) * P2M_NP + (size_t)(L + 1) * (L + 1) * P2M_NP) *
           sizeof(double);
}

// Raw sums of one class over a cell's ESP pairs: raw[cell][split][s][lm] (re, im)
// = sum B_s b_l (x + iy)^m.  A batch of 32 pairs: the warps fill b in shared
// memory (columns paired so that every warp has the same rows), then a thread
// per (l, m) adds the pairs' terms in pair order.  FP64-bound: about 60 warp
// instructions per pair for the columns and 16 (2 + 2 (L+1)^2) for the sums.
template <int L>
__global__ void __launch_bounds__(P2M_NT) mp_p2m_kernel(const int *__restrict__ beg,
                                                        const int *__restrict__ end, const int *__restrict__ pos,
                                                        int e0, const double *__restrict__ rec,
                                                        const double *__restrict__ B, int nesp,
                                                        const double *__restrict__ cxyz, double2 *__restrict__ raw)
{
    constexpr int NS = (L + 1) * (L + 1);
    constexpr int REC = f64_rec(L);
    extern __shared__ double sm[];
    double *sb = sm;                                            // [lm][33]
    double2 *se = reinterpret_cast<double2 *>(sm + (size_t)MP_NLM * (P2M_NP + 1) + (MP_NLM * (P2M_NP + 1)) % 2);
    double *sB = reinterpret_cast<double *>(se + (MP_P + 1) * P2M_NP);
    const int cell = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int j0 = pos[beg[cell]] - e0, j1 = pos[end[cell]] - e0;   // ESP pairs of the class in the cell
    const double cx = cxyz[3 * cell], cy = cxyz[3 * cell + 1], cz = cxyz[3 * cell + 2];
    double2 acc[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) acc[s] = make_double2(0.0, 0.0);
    int m = 0;
    if (threadIdx.x < MP_NLM)
        while (threadIdx.x >= mp_col(m + 1)) ++m;
    for (int jt = j0 + blockIdx.y * P2M_NP; jt < j1; jt += gridDim.y * P2M_NP) {
        const int nt = min(P2M_NP, j1 - jt);
        const int j = jt + min(lane, nt - 1);
        const double *r = rec + (size_t)j * REC;
        const double x = r[0] - cx, y = r[1] - cy, z = r[2] - cz;
        const double r2 = fma(x, x, fma(y, y, z * z));
        __syncthreads();
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            const int mc = side == 0 ? w : MP_P - w;
            if (side == 1 && mc == w) continue;
            se[mc * P2M_NP + lane] = mp_power(x, y, mc);
            const int o = mp_col(mc) - mc;
            double b1 = 1.0, b0 = 0.0;
            sb[(o + mc) * (P2M_NP + 1) + lane] = 1.0;
            for (int l = mc + 1; l <= MP_P; ++l) {
                const double b = fma(z, b1, c_mp.ngam[o + l] * (r2 * b0));
                sb[(o + l) * (P2M_NP + 1) + lane] = b;
                b0 = b1;
                b1 = b;
            }
        }
        for (int i = threadIdx.x; i < NS * P2M_NP; i += P2M_NT) {
            const int s = i / P2M_NP, q = i % P2M_NP;
            sB[q * NS + s] = q < nt ? B[(size_t)s * nesp + jt + q] : 0.0;
        }
        __syncthreads();
        if (threadIdx.x < MP_NLM)
            for (int q = 0; q < nt; ++q) {
                const double b = sb[threadIdx.x * (P2M_NP + 1) + q];
                const double2 e = se[m * P2M_NP + q];
                const double br = b * e.x, bi = b * e.y;
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    const double Bs = sB[q * NS + s];
                    acc[s].x = fma(Bs, br, acc[s].x);
                    acc[s].y = fma(Bs, bi, acc[s].y);
                }
            }
    }
    if (threadIdx.x < MP_NLM)
#pragma unroll
        for (int s = 0; s < NS; ++s)
            raw[(((size_t)cell * gridDim.y + blockIdx.y) * NS + s) * MP_NLM + threadIdx.x] = acc[s];
}

// entry (l, m) of a set of harmonics stored for m >= 0; zero outside |m| <= l <= MP_P
__device__ __forceinline__ double2 mp_get(const double2 *v, int l, int m)
{
    const int a = m < 0 ? -m : m;
    if (l < a || l > MP_P) return make_double2(0.0, 0.0);
    double2 x = v[mp_at(l, a)];
    if (m < 0) {
        const double s = (a & 1) ? -1.0 : 1.0;
        x = make_double2(s * x.x, -s * x.y);
    }
    return x;
}

// M_lm += sum over the sets of one class, shifted by (n, mu); one block per cell
template <int L>
__global__ void __launch_bounds__(P2M_NT) mp_combine_kernel(int nsplit, bool first, const double2 *__restrict__ raw,
                                                            double2 *__restrict__ M)
{
    constexpr int NS = (L + 1) * (L + 1);
    __shared__ double2 S[MP_NLM];
    const int cell = blockIdx.x, i = threadIdx.x;
    int m = 0, l = 0;
    if (i < MP_NLM) {
        while (i >= mp_col(m + 1)) ++m;
        l = i - mp_col(m) + m;
    }
    double2 v = make_double2(0.0, 0.0);
    if (i < MP_NLM && !first) v = M[(size_t)cell * MP_NLM + i];
    for (int s = 0; s < NS; ++s) {
        __syncthreads();
        if (i < MP_NLM) {
            double2 t = make_double2(0.0, 0.0);
            for (int g = 0; g < nsplit; ++g) {
                const double2 x = raw[(((size_t)cell * nsplit + g) * NS + s) * MP_NLM + i];
                t.x += x.x;
                t.y += x.y;
            }
            S[i] = make_double2(c_mp.hn[i] * t.x, c_mp.hn[i] * t.y);
        }
        __syncthreads();
        if (i >= MP_NLM) continue;
        int n = 0;
        while ((n + 1) * (n + 1) <= s) ++n;
        const int q = s - n * n;                    // 0: mu = 0; 2 mu - 1, 2 mu: real, imaginary part of mu
        const int mu = (q + 1) / 2;
        if (mu == 0) {
            const double2 a = mp_get(S, l - n, m);
            v.x += a.x;
            v.y += a.y;
        } else {
            const double2 a = mp_get(S, l - n, m + mu), b = mp_get(S, l - n, m - mu);
            const double sg = (mu & 1) ? -1.0 : 1.0;
            if (q & 1) {                            // Sr(m + mu) + (-1)^mu Sr(m - mu)
                v.x += a.x + sg * b.x;
                v.y += a.y + sg * b.y;
            } else {                                // i Si(m + mu) - i (-1)^mu Si(m - mu)
                v.x += -(a.y - sg * b.y);
                v.y += a.x - sg * b.x;
            }
        }
    }
    if (i < MP_NLM) M[(size_t)cell * MP_NLM + i] = v;
}

// the three sets of the moments' derivatives with respect to the pairs' centres,
// scaled for mp_m2p_kernel: w_m (2l-1)!!; of level 0 (blockIdx.y 0) and of both levels
__global__ void __launch_bounds__(P2M_NT) mp_scale_kernel(int ncell, const double2 *__restrict__ M,
                                                          double2 *__restrict__ out)
{
    __shared__ double2 v[MP_NLM];
    const int cell = blockIdx.x, i = threadIdx.x;
    if (i < MP_NLM) {
        v[i] = M[(size_t)cell * MP_NLM + i];
        if (blockIdx.y > 0) {
            const double2 x = M[((size_t)ncell + cell) * MP_NLM + i];
            v[i] = make_double2(v[i].x + x.x, v[i].y + x.y);
        }
    }
    __syncthreads();
    if (i >= MP_NLM) return;
    int m = 0;
    while (i >= mp_col(m + 1)) ++m;
    const int l = i - mp_col(m) + m;
    const double s = c_mp.wd[i];
    const double2 a = mp_get(v, l - 1, m + 1), b = mp_get(v, l - 1, m - 1), z = mp_get(v, l - 1, m);
    double2 *o = out + (((size_t)blockIdx.y * ncell + cell) * MP_NLM + i) * 3;
    o[0] = make_double2(0.5 * s * (b.x - a.x), 0.5 * s * (b.y - a.y));
    // (-a - b) / (2i) = i (a + b) / 2
    o[1] = make_double2(-0.5 * s * (a.y + b.y), 0.5 * s * (a.x + b.x));
    o[2] = make_double2(s * z.x, s * z.y);
}

// Point part of the gradient from the expanded cells: a warp per (tile, part of
// the cells), a lane per point; part[row][component][slot] as f64_grad_kernel's
// rows.  mom: the moments of level 0, then of all classes.  Nine FP64 instructions per
// (l, m): FP64-bound.
__global__ void __launch_bounds__(128) mp_m2p_kernel(int M, int ntile, int ncell, const F64Pt *__restrict__ xyz,
                                                     const unsigned char *__restrict__ order,
                                                     const double *__restrict__ cxyz, const double2 *__restrict__ mom,
                                                     double *__restrict__ part)
{
    constexpr int NV = 3;
    __shared__ double red[4][NV][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tile = blockIdx.x;
    const F64Pt c = xyz[min(tile * 32 + lane, M - 1)];
    double acc[NV];
#pragma unroll
    for (int d = 0; d < NV; ++d) acc[d] = 0.0;
    for (int cell = blockIdx.y * 4 + w; cell < ncell; cell += 4 * gridDim.y) {
        const int o8 = order[(size_t)tile * ncell + cell], p = o8 & ~MP_ALL;
        if (p == 0) continue;
        const double x = c.x - cxyz[3 * cell], y = c.y - cxyz[3 * cell + 1], z = c.z - cxyz[3 * cell + 2];
        double rs[1];
        f64_far<0>(fma(x, x, fma(y, y, z * z)), rs);
        const double v = rs[0] * rs[0], u = z * v, ex = x * v, ey = y * v;
        double er = rs[0], ei = 0.0;
        const double2 *mc = mom + ((size_t)(o8 & MP_ALL ? ncell : 0) + cell) * MP_NLM * NV;
        for (int m = 0; m <= p; ++m) {
            const int o = mp_col(m) - m;
            double b1 = 1.0, b0 = 0.0, sr[NV], si[NV];
#pragma unroll
            for (int d = 0; d < NV; ++d) {
                const double2 a = __ldg(mc + (size_t)(o + m) * NV + d);
                sr[d] = a.x;
                si[d] = a.y;
            }
            for (int l = m + 1; l <= p; ++l) {
                const double b = fma(u, b1, c_mp.ngam[o + l] * (v * b0));
#pragma unroll
                for (int d = 0; d < NV; ++d) {
                    const double2 a = __ldg(mc + (size_t)(o + l) * NV + d);
                    sr[d] = fma(b, a.x, sr[d]);
                    si[d] = fma(b, a.y, si[d]);
                }
                b0 = b1;
                b1 = b;
            }
#pragma unroll
            for (int d = 0; d < NV; ++d) acc[d] = fma(ei, si[d], fma(er, sr[d], acc[d]));
            const double t = er * ex - ei * ey;
            ei = fma(er, ey, ei * ex);
            er = t;
        }
    }
#pragma unroll
    for (int d = 0; d < NV; ++d) red[w][d][lane] = acc[d];
    __syncthreads();
    if (w == 0 && tile * 32 + lane < M) {
        const size_t S = (size_t)ntile * 32;
#pragma unroll
        for (int d = 0; d < NV; ++d)
            part[((size_t)blockIdx.y * NV + d) * S + tile * 32 + lane] =
                (red[0][d][lane] + red[1][d][lane]) + (red[2][d][lane] + red[3][d][lane]);
    }
}

// ---------------------------------------------------------------------------
// local expansions
// ---------------------------------------------------------------------------
constexpr int P2L_NW = 4;
constexpr size_t P2L_SMEM = (size_t)P2L_NW * (2 * (MP_P + 1) * 33 + 2 * MP_NLM) * sizeof(double);

// lam[level][split][cell][lm] = sum of q_k (2l-1)!!^-1 I_l^m(C_k - centre) over the
// cell's tiles (level 0: those expanded for it alone, level 1: those for all
// classes), a warp per share of the tiles: the lanes (points) write one column m
// at a time to shared memory, then a lane per (l, part) adds its 32 values to the
// warp's sums.
__global__ void __launch_bounds__(32 * P2L_NW) mp_p2l_kernel(int M, int ntile, int ncell,
                                                             const F64Pt *__restrict__ xyz,
                                                             const unsigned char *__restrict__ order,
                                                             const double *__restrict__ cxyz,
                                                             double2 *__restrict__ lam)
{
    extern __shared__ double sm[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cell = blockIdx.x;
    double *buf = sm + (size_t)w * (2 * (MP_P + 1) * 33 + 2 * MP_NLM), *acc = buf + 2 * (MP_P + 1) * 33;
    for (int i = lane; i < 2 * MP_NLM; i += 32) acc[i] = 0.0;
    __syncwarp();
    const double cx = cxyz[3 * cell], cy = cxyz[3 * cell + 1], cz = cxyz[3 * cell + 2];
    for (int tile = blockIdx.y * P2L_NW + w; tile < ntile; tile += gridDim.y * P2L_NW) {
        const int o8 = order[(size_t)tile * ncell + cell], p = o8 & ~MP_ALL;
        if (p == 0 || (o8 & MP_ALL ? 1 : 0) != (int)blockIdx.z) continue;
        const bool on = tile * 32 + lane < M;
        const F64Pt c = xyz[min(tile * 32 + lane, M - 1)];
        const double x = c.x - cx, y = c.y - cy, z = c.z - cz;
        double rs[1];
        f64_far<0>(fma(x, x, fma(y, y, z * z)), rs);
        const double v = rs[0] * rs[0], u = z * v, ex = x * v, ey = y * v;
        double er = on ? c.w * rs[0] : 0.0, ei = 0.0;
        for (int m = 0; m <= p; ++m) {
            const int o = mp_col(m) - m, rows = p - m + 1;
            double b1 = 1.0, b0 = 0.0;
            buf[lane] = er;
            buf[33 + lane] = ei;
            for (int l = m + 1; l <= p; ++l) {
                const double b = fma(u, b1, c_mp.ngam[o + l] * (v * b0));
                buf[2 * (l - m) * 33 + lane] = b * er;
                buf[(2 * (l - m) + 1) * 33 + lane] = b * ei;
                b0 = b1;
                b1 = b;
            }
            __syncwarp();
            for (int i = lane; i < 2 * rows; i += 32) {
                double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
#pragma unroll
                for (int k = 0; k < 32; k += 4) {
                    s0 += buf[i * 33 + k];
                    s1 += buf[i * 33 + k + 1];
                    s2 += buf[i * 33 + k + 2];
                    s3 += buf[i * 33 + k + 3];
                }
                acc[2 * (o + m) + i] += (s0 + s1) + (s2 + s3);
            }
            __syncwarp();
            const double t = er * ex - ei * ey;
            ei = fma(er, ey, ei * ex);
            er = t;
        }
    }
    __syncthreads();
    double *out = reinterpret_cast<double *>(lam + (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * ncell + cell) * MP_NLM);
    constexpr int ST = 2 * (MP_P + 1) * 33 + 2 * MP_NLM;
    for (int i = threadIdx.x; i < 2 * MP_NLM; i += 32 * P2L_NW) {
        double s = 0.0;
        for (int k = 0; k < P2L_NW; ++k) s += sm[(size_t)k * ST + 2 * (MP_P + 1) * 33 + i];
        out[i] = s;
    }
}

// lam: nsplit shares of the cell's tiles, those of a level and the ones above it.
// Coefficients of V_s = sum_{l, m >= 0} b_l (Re e_m A + Im e_m B) for ns sets s
// = (n, mu, part) of a class from s0 on: tab[cell][lm][s - s0] = (A, B); one block per
// cell
__global__ void __launch_bounds__(P2M_NT) mp_local_kernel(int s0, int ns, int nsplit, int ncell,
                                                          const double2 *__restrict__ lam, double2 *__restrict__ tab)
{
    __shared__ double2 L[MP_NLM];
    const int cell = blockIdx.x, i = threadIdx.x;
    int m = 0, l = 0;
    if (i < MP_NLM) {
        while (i >= mp_col(m + 1)) ++m;
        l = i - mp_col(m) + m;
        double2 t = make_double2(0.0, 0.0);
        for (int g = 0; g < nsplit; ++g) {
            const double2 x = lam[((size_t)g * ncell + cell) * MP_NLM + i];
            t.x += x.x;
            t.y += x.y;
        }
        L[i] = make_double2(c_mp.d[i] * t.x, c_mp.d[i] * t.y);
    }
    __syncthreads();
    if (i >= MP_NLM) return;
    const double h = c_mp.hn[i];
    double2 *o = tab + ((size_t)cell * MP_NLM + i) * ns;
    for (int s = s0; s < s0 + ns; ++s) {
        int n = 0;
        while ((n + 1) * (n + 1) <= s) ++n;
        const int q = s - n * n, mu = (q + 1) / 2;
        const double sg = (mu & 1) ? -1.0 : 1.0;
        double2 al, be = make_double2(0.0, 0.0);   // complex coefficients of Re R and Im R
        if (m == 0) {
            const double2 a = mp_get(L, l + n, mu);
            al = make_double2(sg * a.x, sg * a.y);
        } else {
            const double2 a = mp_get(L, l + n, m - mu), b = mp_get(L, l + n, m + mu);
            al = make_double2(a.x + sg * b.x, -a.y + sg * b.y);
            be = make_double2(a.y + sg * b.y, a.x - sg * b.x);   // i (conj(a) - sg b)
        }
        o[s - s0] = (q == 0 || (q & 1)) ? make_double2(h * al.x, h * be.x) : make_double2(h * al.y, h * be.y);
    }
}

// V[s][pair] for NS sets: a lane per sorted pair, reading its
// own cell's coefficients (the pairs of a cell follow one another, so a warp reads
// one cell or a few; taking the cells of a warp in turn instead cost the d classes,
// with few pairs per cell, five times as much).
template <int NS>
__global__ void __launch_bounds__(128) mp_l2p_kernel(int n, int stride, const int *__restrict__ list, int first,
                                                     const double *__restrict__ P, const int *__restrict__ pcell,
                                                     const double *__restrict__ cxyz,
                                                     const double2 *__restrict__ tab, double *__restrict__ V)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int jj = min(j, n - 1);
    const int pos = list ? list[jj] : first + jj;
    const int cell = pcell[pos];
    const double x = P[pos] - cxyz[3 * cell], y = P[(size_t)stride + pos] - cxyz[3 * cell + 1],
                 z = P[2 * (size_t)stride + pos] - cxyz[3 * cell + 2];
    const double r2 = fma(x, x, fma(y, y, z * z));
    const double2 *t = tab + (size_t)cell * MP_NLM * NS;
    double out[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) out[s] = 0.0;
    double er = 1.0, ei = 0.0;
    for (int m = 0; m <= MP_P; ++m) {
        const int o = mp_col(m) - m;
        double b1 = 1.0, b0 = 0.0, sa[NS], sb[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            const double2 a = __ldg(t + (size_t)(o + m) * NS + s);
            sa[s] = a.x;
            sb[s] = a.y;
        }
        for (int l = m + 1; l <= MP_P; ++l) {
            const double b = fma(z, b1, c_mp.ngam[o + l] * (r2 * b0));
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                const double2 a = __ldg(t + (size_t)(o + l) * NS + s);
                sa[s] = fma(b, a.x, sa[s]);
                sb[s] = fma(b, a.y, sb[s]);
            }
            b0 = b1;
            b1 = b;
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) out[s] = fma(ei, sb[s], fma(er, sa[s], out[s]));
        const double q = er * x - ei * y;
        ei = fma(er, y, ei * x);
        er = q;
    }
    if (j < n)
#pragma unroll
        for (int s = 0; s < NS; ++s) V[(size_t)s * n + j] = out[s];
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <int L>
static int mp_moments_class(pcm_ctx *c, int k, bool first, double2 *M)
{
    F64Int &f = c->f64;
    F64Mp &mp = f.mp;
    constexpr int NS = (L + 1) * (L + 1);
    // several blocks share a cell's pairs where a class has many; d classes have few
    const int split = L <= 1 ? 4 : (L == 2 ? 2 : 1);
    static_assert(p2m_smem(L) + 8 <= 227 * 1024, "shared memory");
    const size_t per = (size_t)split * NS * MP_NLM;   // raw sums per cell
    const int group = (int)std::min<size_t>(mp.ncell, P2M_RAW_BYTES / (per * sizeof(double2)));
    PCM_TRY(mp.raw.alloc(group * per));
    PCM_CUDA(cudaFuncSetAttribute(mp_p2m_kernel<L>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)p2m_smem(L) + 8));
    for (int c0 = 0; c0 < mp.ncell; c0 += group) {
        const int nc = std::min(group, mp.ncell - c0);
        const int *beg = mp.range.p + (size_t)k * mp.ncell + c0, *end = mp.range.p + (size_t)(6 + k) * mp.ncell + c0;
        mp_p2m_kernel<L><<<dim3(nc, split), P2M_NT, p2m_smem(L) + 8, c->stream>>>(
            beg, end, f.pos.p, f.eoff[k], f.rec.p + f.roff[k], f.B.p + f.boff[k], c->cls[k].nesp,
            mp.cxyz.p + 3 * (size_t)c0, mp.raw.p);
        PCM_LAUNCHED(c);
        mp_combine_kernel<L><<<nc, P2M_NT, 0, c->stream>>>(split, first, mp.raw.p, M + (size_t)c0 * MP_NLM);
        PCM_LAUNCHED(c);
    }
    return PCM_OK;
}

// point part of the gradient from the expanded cells: mp_rows rows of partial sums
int mp_rows(pcm_ctx *c)
{
    const int nt = c->f64.ntile;
    return std::max(1, std::min((c->f64.mp.ncell + 3) / 4, (152 * 16 + nt - 1) / nt));
}

int mp_grad_far(pcm_ctx *c, double *part)
{
    F64Int &f = c->f64;
    F64Mp &mp = f.mp;
    const size_t nm = (size_t)mp.ncell * MP_NLM;
    PCM_TRY(mp.M.alloc(MP_LEVELS * nm));
    PCM_CUDA(cudaMemsetAsync(mp.M.p, 0, MP_LEVELS * nm * sizeof(double2), c->stream));   // levels without pairs
    bool first[MP_LEVELS] = {true, true};
    for (int k = 0; k < 6; ++k) {
        if (c->cls[k].nesp == 0) continue;
        const int v = mp_level(k);
        double2 *M = mp.M.p + v * nm;
        switch (k) {
        case 0: PCM_TRY(mp_moments_class<0>(c, k, first[v], M)); break;
        case 1: PCM_TRY(mp_moments_class<1>(c, k, first[v], M)); break;
        case 2:
        case 3: PCM_TRY(mp_moments_class<2>(c, k, first[v], M)); break;
        case 4: PCM_TRY(mp_moments_class<3>(c, k, first[v], M)); break;
        case 5: PCM_TRY(mp_moments_class<4>(c, k, first[v], M)); break;
        }
        first[v] = false;
    }
    PCM_TRY(mp.mom.alloc(MP_LEVELS * nm * 3));
    mp_scale_kernel<<<dim3(mp.ncell, MP_LEVELS), P2M_NT, 0, c->stream>>>(mp.ncell, mp.M.p, mp.mom.p);
    PCM_LAUNCHED(c);
    mp_m2p_kernel<<<dim3(f.ntile, mp_rows(c)), 128, 0, c->stream>>>(c->M, f.ntile, mp.ncell, f.pt_xyz.p, mp.order.p,
                                                                   mp.cxyz.p, mp.mom.p, part);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

// local expansions of every cell from the points' charges
int mp_local(pcm_ctx *c)
{
    F64Int &f = c->f64;
    F64Mp &mp = f.mp;
    mp.lsplit = std::max(1, std::min((f.ntile + P2L_NW - 1) / P2L_NW, (152 * 16 + mp.ncell - 1) / mp.ncell));
    PCM_TRY(mp.lam.alloc(MP_LEVELS * (size_t)mp.lsplit * mp.ncell * MP_NLM));
    PCM_CUDA(cudaFuncSetAttribute(mp_p2l_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P2L_SMEM));
    mp_p2l_kernel<<<dim3(mp.ncell, mp.lsplit, MP_LEVELS), 32 * P2L_NW, P2L_SMEM, c->stream>>>(
        c->M, f.ntile, mp.ncell, f.pt_xyz.p, mp.order.p, mp.cxyz.p, mp.lam.p);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

// V[(L+1)^2][n] at the pairs (list, or the sorted positions from first) of a level
int mp_l2p(pcm_ctx *c, int level, int L, int n, const int *list, int first)
{
    F64Int &f = c->f64;
    F64Mp &mp = f.mp;
    const int ns = (L + 1) * (L + 1);
    PCM_TRY(mp.V.alloc((size_t)ns * n));
    PCM_TRY(mp.tab.alloc((size_t)mp.ncell * MP_NLM * std::min(ns, 9)));
    const int nb = (n + 127) / 128;
    const int *pc = mp.pcell.p;
#define PCM_L2P(N, S0)                                                                                            \
    do {                                                                                                          \
        mp_local_kernel<<<mp.ncell, P2M_NT, 0, c->stream>>>(                                                      \
            S0, N, (MP_LEVELS - level) * mp.lsplit, mp.ncell,                                                     \
            mp.lam.p + (size_t)level * mp.lsplit * mp.ncell * MP_NLM, mp.tab.p);                                  \
        PCM_LAUNCHED(c);                                                                                          \
        mp_l2p_kernel<N><<<nb, 128, 0, c->stream>>>(n, f.off[6], list, first, f.P.p, pc, mp.cxyz.p, mp.tab.p,     \
                                                    mp.V.p + (size_t)(S0) * n);                                   \
        PCM_LAUNCHED(c);                                                                                          \
    } while (0)
    // at most nine sets per launch, so that their sums stay in registers and their
    // coefficients take 71 KB per cell
    switch (L) {
    case 0: PCM_L2P(1, 0); break;
    case 1: PCM_L2P(4, 0); break;
    case 2: PCM_L2P(9, 0); break;
    case 3: PCM_L2P(8, 0); PCM_L2P(8, 8); break;
    case 4: PCM_L2P(9, 0); PCM_L2P(8, 9); PCM_L2P(8, 17); break;
    case 5: PCM_L2P(9, 0); PCM_L2P(9, 9); PCM_L2P(9, 18); PCM_L2P(9, 27); break;
    default: return PCM_ERR_ARG;
    }
#undef PCM_L2P
    return PCM_OK;
}

}  // namespace pcm
