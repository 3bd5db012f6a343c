// Stable least-significant-digit radix sort of (32-bit key, 32-bit value)
// pairs, eight bits per pass: digit counts per block of SORT_ITEMS keys, an
// exclusive scan of the counts over the blocks by a block per digit, and a
// scatter that adds the smaller digits' totals and in which every warp ranks its keys with match instructions, so that
// equal keys keep their order.
#include <algorithm>

#include "context.h"

namespace pcm {

constexpr int SORT_NT = 256;
constexpr int SORT_ROUNDS = 8;
constexpr int SORT_ITEMS = SORT_NT * SORT_ROUNDS;   // keys per block: warp w holds [256 w, 256 w + 256)

__global__ void __launch_bounds__(SORT_NT) sort_count_kernel(int n, int shift, const unsigned *__restrict__ key,
                                                             int nblk, int *__restrict__ cnt)
{
    __shared__ int h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    for (int r = 0; r < SORT_ROUNDS; ++r) {
        const int i = blockIdx.x * SORT_ITEMS + r * SORT_NT + threadIdx.x;
        if (i < n) atomicAdd(&h[(key[i] >> shift) & 255u], 1);
    }
    __syncthreads();
    cnt[threadIdx.x * nblk + blockIdx.x] = h[threadIdx.x];
}

// inclusive scan of a value per thread over a block of 256
__device__ __forceinline__ int scan256(int x, int *wsum)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    for (int k = 0; k < w; ++k) x += wsum[k];
    __syncthreads();
    return x;
}

// exclusive scan of a digit's counts over the blocks, in place, and its total: a
// block per digit (one block for all digits took 30 us for 300k keys; 4 now)
__global__ void __launch_bounds__(SORT_NT) sort_scan_kernel(int nblk, int *__restrict__ cnt, int *__restrict__ total)
{
    __shared__ int wsum[SORT_NT / 32], sum;
    int *v = cnt + (size_t)blockIdx.x * nblk;
    int carry = 0;
    for (int b0 = 0; b0 < nblk; b0 += SORT_NT) {
        const int i = b0 + threadIdx.x, x = i < nblk ? v[i] : 0;
        const int s = scan256(x, wsum);
        if (i < nblk) v[i] = carry + s - x;
        if (threadIdx.x == SORT_NT - 1) sum = s;
        __syncthreads();
        carry += sum;
        __syncthreads();
    }
    if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

__global__ void __launch_bounds__(SORT_NT) sort_scatter_kernel(int n, int shift, const unsigned *__restrict__ key,
                                                               const int *__restrict__ val, int nblk,
                                                               const int *__restrict__ off,
                                                               const int *__restrict__ total,
                                                               unsigned *__restrict__ okey, int *__restrict__ oval)
{
    __shared__ int c[SORT_NT / 32][256];
    __shared__ int wsum[SORT_NT / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int k = 0; k < SORT_NT / 32; ++k) c[k][threadIdx.x] = 0;
    __syncthreads();
    const int base = blockIdx.x * SORT_ITEMS + w * (32 * SORT_ROUNDS);
    for (int r = 0; r < SORT_ROUNDS; ++r) {
        const int i = base + 32 * r + lane;
        const unsigned d = i < n ? (key[i] >> shift) & 255u : 256u;
        const unsigned m = __match_any_sync(0xffffffffu, d);
        if (d < 256u && lane == __ffs(m) - 1) c[w][d] += __popc(m);
        __syncwarp();
    }
    __syncthreads();
    // keys of smaller digits, then of this digit in earlier blocks
    const int mine = total[threadIdx.x];
    int run = scan256(mine, wsum) - mine + off[threadIdx.x * nblk + blockIdx.x];
    for (int k = 0; k < SORT_NT / 32; ++k) {
        const int t = c[k][threadIdx.x];
        c[k][threadIdx.x] = run;
        run += t;
    }
    __syncthreads();
    for (int r = 0; r < SORT_ROUNDS; ++r) {
        const int i = base + 32 * r + lane;
        const unsigned kk = i < n ? key[i] : 0u;
        const unsigned d = i < n ? (kk >> shift) & 255u : 256u;
        const unsigned m = __match_any_sync(0xffffffffu, d);
        const int lead = __ffs(m) - 1;
        int pos = 0;
        if (d < 256u && lane == lead) {
            pos = c[w][d];
            c[w][d] = pos + __popc(m);
        }
        pos = __shfl_sync(0xffffffffu, pos, lead) + __popc(m & ((1u << lane) - 1u));
        if (i < n) {
            okey[pos] = kk;
            oval[pos] = val[i];
        }
        __syncwarp();
    }
}

// sort the first n entries of key (its low `bits` bits) and val; both are
// replaced by their sorted order (buffers may be swapped with the scratch)
int sort_pairs(pcm_ctx *c, int n, int bits, DBuf<unsigned> &key, DBuf<int> &val)
{
    if (n <= 1) return PCM_OK;
    const int nblk = (n + SORT_ITEMS - 1) / SORT_ITEMS;
    PCM_TRY(c->sort_key.alloc(n));
    PCM_TRY(c->sort_val.alloc(n));
    PCM_TRY(c->sort_cnt.alloc((size_t)256 * nblk + 256));   // counts, then the digits' totals
    int *total = c->sort_cnt.p + (size_t)256 * nblk;
    for (int shift = 0; shift < bits; shift += 8) {
        sort_count_kernel<<<nblk, SORT_NT, 0, c->stream>>>(n, shift, key.p, nblk, c->sort_cnt.p);
        PCM_LAUNCHED(c);
        sort_scan_kernel<<<256, SORT_NT, 0, c->stream>>>(nblk, c->sort_cnt.p, total);
        PCM_LAUNCHED(c);
        sort_scatter_kernel<<<nblk, SORT_NT, 0, c->stream>>>(n, shift, key.p, val.p, nblk, c->sort_cnt.p,
                                                             total, c->sort_key.p, c->sort_val.p);
        PCM_LAUNCHED(c);
        std::swap(key.p, c->sort_key.p);
        std::swap(key.n, c->sort_key.n);
        std::swap(val.p, c->sort_val.p);
        std::swap(val.n, c->sort_val.n);
    }
    return PCM_OK;
}

}  // namespace pcm
