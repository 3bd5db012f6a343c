// Order along a Hilbert curve over a cubic grid, so that consecutive points or
// pairs lie together (Skilling, AIP Conf. Proc. 707, 381 (2004): axes to transposed
// index by Gray decoding of the exchanged bits).
#pragma once
#include "context.h"

namespace pcm {

template <int BITS>
__device__ __forceinline__ unsigned hilbert3(unsigned x, unsigned y, unsigned z)
{
    unsigned X[3] = {x, y, z};
    for (unsigned q = 1u << (BITS - 1); q > 1; q >>= 1) {
        const unsigned p = q - 1;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            if (X[i] & q) {
                X[0] ^= p;
            } else {
                const unsigned t = (X[0] ^ X[i]) & p;
                X[0] ^= t;
                X[i] ^= t;
            }
        }
    }
    X[1] ^= X[0];
    X[2] ^= X[1];
    unsigned t = 0;
    for (unsigned q = 1u << (BITS - 1); q > 1; q >>= 1)
        if (X[2] & q) t ^= q - 1;
    unsigned h = 0;
    for (int b = BITS - 1; b >= 0; --b)
        for (int i = 0; i < 3; ++i) h = (h << 1) | (((X[i] ^ t) >> b) & 1u);
    return h;
}

template <int BITS>
__device__ __forceinline__ unsigned curve_key(double x, double y, double z, const F64Box &b)
{
    const int top = (1 << BITS) - 1;
    const double s = (double)(1 << BITS) * b.inv;
    const int i = min(max((int)((x - b.lo[0]) * s), 0), top);
    const int j = min(max((int)((y - b.lo[1]) * s), 0), top);
    const int k = min(max((int)((z - b.lo[2]) * s), 0), top);
    return hilbert3<BITS>(i, j, k);
}

constexpr int CURVE_HBITS = 5;             // cells per side of the pairs' grid: 2^5
constexpr int CURVE_PBITS = 4;             // exponent bins

}  // namespace pcm
