// Orders of primitive pairs along a curve through their centres and by exponent,
// so that the pairs of a warp lie together and reach equally far.
#include <math.h>

#include <algorithm>

#include "context.h"
#include "curve.cuh"

namespace pcm {

// fewer pairs than this stay in their order: sorting costs ten launches
constexpr int ORDER_MIN = 4096;

// class, then cell along the curve and exponent bin (half octaves from 0.2,
// ascending), or exponent bin and cell
__global__ void pair_key_kernel(int n, F64Src src, F64Box box, bool exponent_first, unsigned *__restrict__ key,
                                int *__restrict__ val)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    int k = 0;
#pragma unroll
    for (int i = 1; i < 6; ++i) k += g >= src.off[i] ? 1 : 0;
    const int r = g - src.off[k];
    const unsigned h = curve_key<CURVE_HBITS>(src.Px[k][r], src.Py[k][r], src.Pz[k][r], box);
    const unsigned pb = min(max((int)floorf(2.f * log2f(5.f * (float)src.p[k][r])), 0), (1 << CURVE_PBITS) - 1);
    key[g] = ((unsigned)k << (3 * CURVE_HBITS + CURVE_PBITS)) |
             (exponent_first ? (pb << (3 * CURVE_HBITS)) | h : (h << CURVE_PBITS) | pb);
    val[g] = g;
}

// cube around the cavity with 2^CURVE_HBITS cells a side, of `cell` or larger
F64Box cavity_box(pcm_ctx *c, double cell)
{
    F64Box box;
    double ext = 1e-3;
    for (int d = 0; d < 3; ++d) {
        double lo = 1e300, hi = -1e300;
        for (int I = 0; I < c->natom; ++I) {
            lo = std::min(lo, c->h_xyz[3 * I + d] - c->h_radius[I]);
            hi = std::max(hi, c->h_xyz[3 * I + d] + c->h_radius[I]);
        }
        box.lo[d] = lo;
        box.mid[d] = lo + 0.5 * (hi - lo);
        ext = std::max(ext, hi - lo);
    }
    // an FP32 coordinate of up to ext / 2 is off by 2^-25 of ext, the difference of two by
    // 2^-23, so a distance by less than 2^-22; beyond 1e18 bohr, where squares leave
    // FP32, there is no bound and every test errs on the FP64 side
    box.slack = ext < 2e18 ? (float)(ext * 0x1p-21) : INFINITY;
    box.inv = 1.0 / (std::max(cell, ext * (1.0 + 1e-9) / (1 << CURVE_HBITS)) * (1 << CURVE_HBITS));
    return box;
}

// the kept pairs of every class
F64Src kept_pairs(pcm_ctx *c, int off[7])
{
    F64Src src;
    int n = 0;
    for (int k = 0; k < 6; ++k) {
        src.off[k] = off[k] = n;
        src.Px[k] = c->cls[k].Px.p;
        src.Py[k] = c->cls[k].Py.p;
        src.Pz[k] = c->cls[k].Pz.p;
        src.p[k] = c->cls[k].p.p;
        n += c->cls[k].npair;
    }
    src.off[6] = off[6] = n;
    return src;
}

// Sorts the pairs of src: *sorted false if they are too few (the order is the
// identity), else c->f64.val holds their indices over all classes in order and
// c->f64.key the keys.
int pair_order(pcm_ctx *c, const F64Src &src, const F64Box &box, bool exponent_first, bool *sorted)
{
    const int n = src.off[6];
    *sorted = n >= ORDER_MIN;
    if (!*sorted) return PCM_OK;
    PCM_TRY(c->f64.key.alloc(n));   // a sort may have exchanged these with its scratch
    PCM_TRY(c->f64.val.alloc(n));
    pair_key_kernel<<<(n + 127) / 128, 128, 0, c->stream>>>(n, src, box, exponent_first, c->f64.key.p, c->f64.val.p);
    PCM_LAUNCHED(c);
    return sort_pairs(c, n, 3 + 3 * CURVE_HBITS + CURVE_PBITS, c->f64.key, c->f64.val);
}

// ---------------------------------------------------------------------------
// PCM_MIXED Fock: the pairs by exponent and then cell.  The packed Fock kernel
// takes the near form for a warp's 32 or 64 pairs and two points when any of these
// interactions is near (22% of them on 300 atoms in shell-pair order, 7.5% in this
// one; cell before exponent: 9%); every pair's own sums are the same in any order.
// Fock correction of 300 s/sp atoms 6.35 -> 5.1 ms, of 1000 s/p/d atoms 74.1 -> 70.4.
// ---------------------------------------------------------------------------
struct FockOrderSrc {
    const float *x32[6];     // 6 x pairs: split centres
};

__global__ void fock_order_kernel(int n, F64Src src, FockOrderSrc x, const int *__restrict__ val,
                                  int *__restrict__ ord, double *__restrict__ p, float *__restrict__ x32)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n) return;
    int k = 0;
#pragma unroll
    for (int i = 1; i < 6; ++i) k += g >= src.off[i] ? 1 : 0;
    const int o = src.off[k], np = src.off[k + 1] - o, j = g - o, r = val[g] - o;
    ord[g] = r;
    p[g] = src.p[k][r];
#pragma unroll
    for (int d = 0; d < 6; ++d) x32[6 * (size_t)o + (size_t)d * np + j] = x.x32[k][(size_t)d * np + r];
}

// sorted exponent sums and split centres of src's pairs in `out` (x32: per class
// the FP32 split centres)
int fock_order(pcm_ctx *c, const F64Src &src, const float *const x32[6], FockOrder &out)
{
    PCM_TRY(pair_order(c, src, cavity_box(c, 3.0), true, &out.on));
    if (!out.on) return PCM_OK;
    const int n = src.off[6];
    for (int k = 0; k < 7; ++k) out.off[k] = src.off[k];
    PCM_TRY(out.ord.alloc(n));
    PCM_TRY(out.p.alloc(n));
    PCM_TRY(out.x32.alloc(6 * (size_t)n));
    FockOrderSrc x;
    for (int k = 0; k < 6; ++k) x.x32[k] = x32[k];
    fock_order_kernel<<<(n + 127) / 128, 128, 0, c->stream>>>(n, src, x, c->f64.val.p, out.ord.p, out.p.p, out.x32.p);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

}  // namespace pcm
