// Multipole far field of the PCM_FP64 integrals: orders, index maps and the map
// between Hermite components and the (n, mu) shifts of solid harmonics.
#pragma once
#include "common.cuh"

namespace pcm {

// highest order.  24 / 30: Fock correction of 300 s/sp atoms 114 / 88.7 ms, gradient of 180
// 141 / 114 (one thread per (l, m) in mp_p2m_kernel ends at 30)
constexpr int MP_P = 30;
constexpr int MP_NLM = (MP_P + 1) * (MP_P + 2) / 2; // (l, m >= 0)
// What an expansion may leave out of an interaction's n-th derivative, relative to it:
// 2n + 1 units of 2^-53, which R^-(2n+1) of the direct form rounds to by itself.
__host__ __device__ constexpr float mp_eps(int n) { return (float)(2 * n + 1) * 0x1p-53f; }
constexpr float MP_GAIN = 1.5f;                     // an expansion has to save this factor over its pairs

// Order of a cell's expansion for points at D or more from its centre and pairs within
// r = x D of it: the smallest p at which sum_{l > p} C(l, n) x^(l-n), what the n-th
// derivative of 1/R leaves out over its leading term (terms beyond p + 1 by the
// geometric series of their largest ratio), is below mp_eps; 0: none up to MP_P.
__host__ __device__ inline int mp_order_for(float x, int n)
{
    float t = (float)(n + 1) * x;                   // C(p + 1, n) x^(p + 1 - n) at p = n
    for (int p = n; p <= MP_P; ++p) {
        const float g = x * (float)(p + 2) / (float)(p + 2 - n);
        if (t <= mp_eps(n) * (1.f - g)) return p < 1 ? 1 : p;
        t *= g;
    }
    return 0;
}

// Classes by the derivatives they take: level 0 up to the second (ss, ps, pp, ds), level
// 1 the third and fourth (dp, dd).  A tile that is too close for a cell's level 1 but not
// for its level 0 is expanded for the latter's pairs, most of them, alone (one level:
// Fock correction of 300 s/p/d atoms 150 ms, two 130; gradient of 180 204 and 179).  An
// entry of the table of orders is the order, with MP_ALL if it holds for both levels.
constexpr int MP_LEVELS = 2;
__host__ __device__ constexpr int mp_level(int k) { return k >= 4 ? 1 : 0; }
constexpr unsigned char MP_ALL = 0x80;

// entries by columns m, l = m .. MP_P
__host__ __device__ constexpr int mp_col(int m) { return m * (MP_P + 1) - m * (m - 1) / 2; }
__host__ __device__ constexpr int mp_at(int l, int m) { return mp_col(m) + l - m; }
static_assert(mp_at(MP_P, MP_P) == MP_NLM - 1, "mp_at");

// c_mu of d_x^t d_y^u = sum_mu c_mu (shift m -> m + mu), with d_x = (d+ + d-)/2,
// d_y = (d+ - d-)/(2i), d+ R_l^m = -R_{l-1}^{m+1}, d- R_l^m = R_{l-1}^{m-1}
struct MpShift {
    double re, im;
};

__host__ __device__ constexpr MpShift mp_shift(int t, int u, int mu)
{
    auto binom = [](int n, int k) {
        double r = 1.0;
        for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
        return r;
    };
    double s = 0.0;
    for (int a = 0; a <= t; ++a)
        for (int b = 0; b <= u; ++b) {
            const int p = a + b, q = t + u - p;
            if (p - q != mu) continue;
            s += binom(t, a) * binom(u, b) * (((u - b) & 1) ? -1.0 : 1.0) * ((p & 1) ? -1.0 : 1.0);
        }
    for (int i = 0; i < t + u; ++i) s *= 0.5;
    // (1/i)^u
    switch (u & 3) {
    case 0: return MpShift{s, 0.0};
    case 1: return MpShift{0.0, -s};
    case 2: return MpShift{-s, 0.0};
    default: return MpShift{0.0, s};
    }
}

// set s = n^2 (mu = 0), n^2 + 2 mu - 1 (real part), n^2 + 2 mu (imaginary part);
// the nonzero weights B of Hermite component h = (t, u, v) in B_s, and V of V_s in W_tuv
struct MpMap {
    int h[320], s[320];
    double B[320], V[320];
    int count;
};

__host__ __device__ constexpr MpMap mp_map(int L)
{
    MpMap M{};
    int q = 0;
    for (int n = 0; n <= L; ++n)
        for (int t = n; t >= 0; --t)
            for (int u = n - t; u >= 0; --u)
                for (int mu = 0; mu <= t + u; ++mu) {
                    const MpShift c = mp_shift(t, u, mu);
                    for (int part = 0; part < 2; ++part) {
                        const double w = part == 0 ? c.re : c.im;
                        if (w == 0.0) continue;
                        M.h[q] = hidx(t, u, n - t - u);
                        M.s[q] = mu == 0 ? n * n : n * n + 2 * mu - 1 + part;
                        M.B[q] = w;
                        M.V[q] = mu == 0 ? w : (part == 0 ? 2.0 * w : -2.0 * w);
                        ++q;
                    }
                }
    M.count = q;
    return M;
}

}  // namespace pcm
