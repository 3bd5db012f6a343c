// Multipole far field of the PCM_FP64 integrals: orders, index maps and the map
// between Hermite components and the (n, mu) shifts of solid harmonics.
#pragma once
#include "common.cuh"

namespace pcm {

constexpr int MP_P = 24;                            // highest order
constexpr int MP_NLM = (MP_P + 1) * (MP_P + 2) / 2; // (l, m >= 0)
// first neglected term over the leading one, for pairs at the cell's rim (most lie
// well inside and their errors cancel).  Measured against the direct sums on 40 to
// 300 atoms: the Fock correction keeps 1.2e-15 relative down to 1e-10 (4e-15 at
// 1e-9), the gradient, with higher derivatives and larger cancellation, 1.1e-15 at
// 3e-13 (8e-15 at 1e-11, 2e-13 at 1e-10).
constexpr float MP_EPS = 1e-10f;
constexpr float MP_EPS_GRAD = 3e-13f;
constexpr float MP_GAIN = 1.5f;                     // an expansion has to save this factor over its pairs

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
