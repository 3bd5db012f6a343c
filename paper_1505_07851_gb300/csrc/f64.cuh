// FP64 pair-point interactions in few FP64 instructions.
//
// The FP64 pipe of this GPU issues 1.67 lanes per clock and SM (measured; 77
// cycles per warp instruction and scheduler), so an FP64 integral kernel costs
// its FP64 instructions and nothing else: loads, integer work and FP32 tests
// hide behind them, and FP64 comparisons and conversions cost as much as an
// FMA.  An interaction of a pair (exponent p, centre P) with a point (zeta, C)
// is written in the form of farfield.cuh,
//   sum_n b_n Q_n(X, Y, Z),  (X, Y, Z) = P - C,
// with per-pair polynomials Q_n and
//   far  (T = rho R^2 >= f64_far_T): b_n = R^-(2n+1),
//   near:                            b_n = cn (2 rho)^n F_n(T) / (2n-1)!!,  cn = 2 sqrt(rho / pi)
// (U / (sqrt(pi) / (2 sqrt(p))) = 2 sqrt(rho / pi)), so both forms share the
// polynomials.  Beyond f64_far_T the two agree to below 1e-16 relative.
#pragma once
#include <string.h>

#include "common.cuh"
#include "farfield.cuh"

namespace pcm {

// smallest T at which F_0..F_m equal their asymptotic forms to 1e-16 relative
// (the neglected part of F_m is about e^-T 2^m T^(m-1/2) / ((2m-1)!! sqrt(pi)) of it)
__host__ __device__ constexpr double f64_far_T(int m)
{
    return m == 0 ? 35.0 : (m == 1 ? 39.5 : (m == 2 ? 43.0 : (m == 3 ? 46.5 : (m == 4 ? 49.5 : 52.5))));
}

// Table of F_m(T) / (2m-1)!!, m = 0..5, at T_i = i / 256 as Taylor coefficients
// in d = T - T_i (five terms: |d| <= 1/512, the next one is below 2^-55 of F_m):
// per row and m six doubles, c0..c4 and a pad, so that a row is read in 16-byte
// words.  1/256 instead of 1/32 costs 4 MB (resident in L2) and saves two FMAs
// and the d / k scalings per F_m.
constexpr int F64_MTOP = 5;
constexpr int F64_INV_DT = 256;
constexpr int F64_NROW = 54 * F64_INV_DT + 2;
constexpr int F64_STRIDE = 6 * (F64_MTOP + 1);
// A second table of the same layout follows: H_m(T) = F_m(T) - F_m's asymptotic
// form = -int_1^inf u^2m e^(-T u^2) du, for T >= F64_H_MIN: its Taylor step is as
// exact there, and F_5 is still 0.64 of its asymptotic form (0.13 at T = 3, 0.0015 at
// T = 1, where the sum of the two would lose three digits).
constexpr int F64_TABLE = F64_NROW * F64_STRIDE;
constexpr double F64_H_MIN = 6.0;
// adding 1.5 * 2^44 leaves round(256 T) in the low word of the sum
constexpr double F64_MAGIC = 26388279066624.0;

// ESP pair record: P, then the coefficients of the terms, padded to 16 bytes
__host__ __device__ constexpr int f64_rec(int L) { return (3 + far_nterms(L) + 1) / 2 * 2; }

// b_n of the far form; 1/R from the hardware estimate (2^-20) and one
// third-order step: r0 (1 + e/2 + 3 e^2/8), e = 1 - R^2 r0^2, error 5 e^3 / 16 < 2^-58
template <int L>
__device__ __forceinline__ void f64_far(double R2, double (&b)[L + 1])
{
    double r0;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(R2));
    const double e = fma(-R2 * r0, r0, 1.0);
    const double rs = fma(r0 * e, fma(e, 0.375, 0.5), r0);
    b[0] = rs;
    if constexpr (L > 0) {
        const double rs2 = rs * rs;
#pragma unroll
        for (int n = 1; n <= L; ++n) b[n] = b[n - 1] * rs2;
    }
}

// words of a double
__host__ __device__ __forceinline__ int hi_word(double v)
{
#ifdef __CUDA_ARCH__
    return __double2hiint(v);
#else
    long long b;
    memcpy(&b, &v, sizeof(b));
    return (int)(b >> 32);
#endif
}

__host__ __device__ __forceinline__ unsigned lo_word(double v)
{
#ifdef __CUDA_ARCH__
    return (unsigned)__double2loint(v);
#else
    long long b;
    memcpy(&b, &v, sizeof(b));
    return (unsigned)b;
#endif
}

// FP32 value of a non-negative double from its high word (20 mantissa bits,
// towards zero; values outside FP32's normal range become its smallest or largest),
// without the conversion's FP64-pipe slot
__host__ __device__ __forceinline__ float f64_trunc32(double v)
{
    int h = hi_word(v);
    h = h < 0x38100000 ? 0x38100000 : (h > 0x47efffff ? 0x47efffff : h);
    const int f = (h - 0x38000000) << 3;
#ifdef __CUDA_ARCH__
    return __int_as_float(f);
#else
    float x;
    memcpy(&x, &f, sizeof(x));
    return x;
#endif
}

// T = rho R^2 below `top`?  In FP32 from the truncated factors: T itself may be
// larger by up to 2^-19 of it.  Every read of the table is behind this test.
__host__ __device__ __forceinline__ bool f64_below(double R2, double rho, float top)
{
    return f64_trunc32(R2) * f64_trunc32(rho) < top;
}

// FP32 tests on coordinates from the middle of the cavity.  `slack` bounds the error
// of a distance between two of them (context.h), so that both tests only err on the
// side of the FP64 evaluation.
//
// may a pair (b: centre, exponent) have T < farT at a point of the tile (s: sphere)?
__host__ __device__ __forceinline__ bool f64_reaches(const float4 &b, const float4 &s, float zmin2, float farT,
                                                     float slack)
{
    const float dx = b.x - s.x, dy = b.y - s.y, dz = b.z - s.z;
    const float d = fmaxf(sqrtf(dx * dx + dy * dy + dz * dz) * 0.99999f - slack - s.w, 0.f);
    return b.w * zmin2 * d * d < 1.00001f * farT * (b.w + zmin2);
}

// T < farT for one interaction, s = 1/p + 1/zeta^2 = 1/rho?  A distance that is off by
// slack leaves R^2 within 0.05% and `pad` = 2001 slack^2 of it.
__host__ __device__ __forceinline__ bool f64_is_near(float x, float y, float z, float s, float farT, float pad)
{
    return fmaf(x, x, fmaf(y, y, z * z)) < fmaf(1.001f * farT + 0.05f, s, pad);
}

// row of the table from t = T + F64_MAGIC; the bound is for arguments that are no T
__host__ __device__ __forceinline__ int f64_row(double t)
{
    const unsigned i = lo_word(t);
    return (int)(i < (unsigned)F64_NROW ? i : (unsigned)F64_NROW - 1u);
}

// b_n of the near form; lanes without `use` read row 0 and return garbage
template <int L>
__device__ __forceinline__ void f64_near(double R2, double rho, double cn, bool use, const double *__restrict__ tab,
                                         double (&b)[L + 1])
{
    const double t = fma(rho, R2, F64_MAGIC);
    const int i = use ? f64_row(t) : 0;
    const double d = fma(rho, R2, F64_MAGIC - t);
    const double2 *row = reinterpret_cast<const double2 *>(tab + (size_t)i * F64_STRIDE);
    double f = cn;
#pragma unroll
    for (int n = 0; n <= L; ++n) {
        const double2 c01 = __ldg(row + 3 * n), c23 = __ldg(row + 3 * n + 1);
        const double c4 = __ldg(reinterpret_cast<const double *>(row + 3 * n + 2));
        const double F = fma(fma(fma(fma(c4, d, c23.y), d, c23.x), d, c01.y), d, c01.x);
        if (n > 0) f *= rho + rho;
        b[n] = f * F;
    }
}

// monomials X^a Y^b Z^c of degree 1..L in Hermite index order (mono[0] unused)
template <int L>
__device__ __forceinline__ void f64_monomials(double X, double Y, double Z, double (&mono)[nherm(L)])
{
    constexpr MonoTab MT = mono_tab(L);
    if constexpr (L > 0) {
        mono[1] = X;
        mono[2] = Y;
        mono[3] = Z;
#pragma unroll
        for (int i = 4; i < nherm(L); ++i) {
            const int a = MT.a[i], b = MT.b[i], c = MT.c[i];
            if (a > 0)
                mono[i] = mono[hidx(a - 1, b, c)] * X;
            else if (b > 0)
                mono[i] = mono[hidx(a, b - 1, c)] * Y;
            else
                mono[i] = mono[hidx(a, b, c - 1)] * Z;
        }
    }
}

// acc[d] += d/dP_d of sum_n b_n Q_n (coefficients G: the terms of farfield.cuh),
// with b_0..b_{L+1}: both forms have d b_n / dX = -(2n + 1) X b_{n+1}
template <int L>
__device__ __forceinline__ void f64_dot_grad(double X, double Y, double Z, const double (&b)[L + 2],
                                             const double (&G)[far_nterms(L)], double (&acc)[3])
{
    constexpr FarTerms FT = far_terms(L);
    double S = b[1] * G[0];
    if constexpr (L > 0) {
        double mono[nherm(L)];
        f64_monomials<L>(X, Y, Z, mono);
        mono[0] = 1.0;
#pragma unroll
        for (int n = 1; n <= L; ++n) {
            double Q = 0.0, D[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int k = 1; k < far_nterms(L); ++k) {
                if (FT.n[k] != n) continue;
                const int e[3] = {FT.a[k], FT.b[k], FT.c[k]};
                if (e[0] + e[1] + e[2] == 0) {
                    Q += G[k];
                    continue;
                }
                Q = fma(G[k], mono[hidx(e[0], e[1], e[2])], Q);
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    if (e[d] > 0) {
                        const double g = e[d] > 1 ? (double)e[d] * G[k] : G[k];
                        const int h = hidx(e[0] - (d == 0), e[1] - (d == 1), e[2] - (d == 2));
                        D[d] = h == 0 ? D[d] + g : fma(g, mono[h], D[d]);
                    }
            }
            S = fma((double)(2 * n + 1) * b[n + 1], Q, S);
#pragma unroll
            for (int d = 0; d < 3; ++d) acc[d] = fma(b[n], D[d], acc[d]);
        }
    }
    acc[0] = fma(-X, S, acc[0]);
    acc[1] = fma(-Y, S, acc[1]);
    acc[2] = fma(-Z, S, acc[2]);
}

// S[k] += b_n X^a Y^b Z^c for every term k = (n; a, b, c)
template <int L>
__device__ __forceinline__ void f64_accumulate(double X, double Y, double Z, const double (&b)[L + 1],
                                               double (&S)[far_nterms(L)])
{
    constexpr FarTerms FT = far_terms(L);
    S[0] += b[0];
    if constexpr (L > 0) {
        double mono[nherm(L)];
        f64_monomials<L>(X, Y, Z, mono);
#pragma unroll
        for (int k = 1; k < far_nterms(L); ++k) {
            const int h = hidx(FT.a[k], FT.b[k], FT.c[k]);
            S[k] = h == 0 ? S[k] + b[FT.n[k]] : fma(b[FT.n[k]], mono[h], S[k]);
        }
    }
}

// b_n of near interactions (lanes with `on`) of pairs whose far form comes from
// their cell's expansion: what the near form adds to it, zero from f64_far_T on.
// T >= F64_H_MIN (the cells that are expanded see to it).
template <int L>
__device__ __forceinline__ void f64_near_minus_far(double R2, double2 rc, bool on, const double *__restrict__ tab,
                                                   double (&b)[L + 1])
{
    on = on && f64_below(R2, rc.x, (float)f64_far_T(L));
    f64_near<L>(R2, rc.x, rc.y, on, tab + F64_TABLE, b);
#pragma unroll
    for (int n = 0; n <= L; ++n) b[n] = on ? b[n] : 0.0;
}

// b_n of one interaction per lane, near or far form by T; zero for lanes whose
// pair is `expanded` (their near part is left to f64_near_minus_far).
template <int L>
__device__ __forceinline__ void f64_terms(double R2, double2 rc, bool expanded, const double *__restrict__ tab,
                                          double (&b)[L + 1])
{
    const bool near = f64_below(R2, rc.x, (float)f64_far_T(L));
    if (__any_sync(0xffffffffu, near && !expanded)) {
        f64_near<L>(R2, rc.x, rc.y, near, tab, b);
        if (!__all_sync(0xffffffffu, near)) {
            double bf[L + 1];
            f64_far<L>(R2, bf);
#pragma unroll
            for (int n = 0; n <= L; ++n) b[n] = near ? b[n] : bf[n];
        }
    } else {
        f64_far<L>(R2, b);
    }
#pragma unroll
    for (int n = 0; n <= L; ++n) b[n] = expanded ? 0.0 : b[n];
}

}  // namespace pcm
