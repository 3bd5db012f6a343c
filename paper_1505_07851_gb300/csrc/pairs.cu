// Basis set-up and the primitive-pair list with the Schwarz-type screening of
// Eq. 15 (Section 4a).
#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "context.h"

namespace pcm {

__host__ __device__ inline int class_index(int la, int lb) { return la * (la + 1) / 2 + lb; }

// coefficient x (2a/pi)^(3/4) (4a)^(l/2) / sqrt((2l-1)!!): normalisation of the
// x^l component; the other Cartesian components differ by comp_factor().
__global__ void cnorm_kernel(int nshell, const int *__restrict__ sh_l, const int *__restrict__ sh_nprim,
                             const int *__restrict__ sh_off, const double *__restrict__ exps,
                             const double *__restrict__ coefs, double *__restrict__ cnorm)
{
    // eight lanes per shell (a thread per shell: 23 us for three atoms, a pow at a time)
    const int s = (blockIdx.x * blockDim.x + threadIdx.x) / 8;
    if (s >= nshell) return;
    const int l = sh_l[s];
    double dfl = 1.0;
    for (int k = 2 * l - 1; k > 1; k -= 2) dfl *= k;
    for (int i = threadIdx.x % 8; i < sh_nprim[s]; i += 8) {
        const double a = exps[sh_off[s] + i];
        cnorm[sh_off[s] + i] = coefs[sh_off[s] + i] * pow(2.0 * a / PCM_PI, 0.75) * pow(4.0 * a, 0.5 * l) / sqrt(dfl);
    }
}

// sqrt((2l-1)!! / ((2lx-1)!! (2ly-1)!! (2lz-1)!!)) for l <= 2
__device__ inline double comp_factor(int l, int c)
{
    if (l < 2) return 1.0;
    return (c == 1 || c == 2 || c == 4) ? 1.7320508075688772935 : 1.0;  // xy, xz, yz
}

// (T-1)!! for even T >= 0
__device__ inline double dfact_even(int T)
{
    double r = 1.0;
    for (int k = T - 1; k > 1; k -= 2) r *= k;
    return r;
}

// what the screening reads of one class
struct PairSrc {
    int nsp;
    const long long *sp_cand;          // first candidate of each shell pair (nsp + 1)
    const int *spA, *spB, *sh_atom, *sh_nprim, *sh_off;
    const double *exps, *cnorm, *xyz;
};

// shell pair s in [lo, hi] and primitives i, j of candidate g
__device__ __forceinline__ void pair_locate(const PairSrc &p, long long g, int lo, int hi, int &s, int &i, int &j)
{
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.sp_cand[mid] <= g) lo = mid;
        else hi = mid - 1;
    }
    s = lo;
    int r = (int)(g - p.sp_cand[s]);
    const int A = p.spA[s], B = p.spB[s];
    if (A == B) {
        const int n = p.sh_nprim[A];
        i = 0;
        while (r >= n - i) {
            r -= n - i;
            ++i;
        }
        j = i + r;
    } else {
        const int nb = p.sh_nprim[B];
        i = r / nb;
        j = r - i * nb;
    }
}

struct PairValues {
    double P[3], p, pref, Q;
};

// Centre, exponent sum, prefactor and Schwarz bound of a primitive pair.  TS:
// arithmetic of the bound (FP64, or FP32 for PCM_MIXED, where a bound off by 1e-6
// relative only moves pairs at the cutoff whose contributions are of the cutoff's
// size); the pair data are FP64 either way.
template <int LA, int LB, typename TS>
__device__ __forceinline__ PairValues pair_values(const PairSrc &src, int A, int B, int i, int j)
{
    PairValues v;
    const double a = src.exps[src.sh_off[A] + i], b = src.exps[src.sh_off[B] + j];
    const double *RA = src.xyz + 3 * src.sh_atom[A], *RB = src.xyz + 3 * src.sh_atom[B];
    const double p = a + b;
    // one FP64 division per pair (the FP64 pipe runs at 1/64 of FP32 here)
    const double ip = 1.0 / p;
    double P[3], ab2 = 0.0;
    for (int d = 0; d < 3; ++d) {
        P[d] = (a * RA[d] + b * RB[d]) * ip;
        const double t = RA[d] - RB[d];
        ab2 += t * t;
    }
    const double K = exp(-a * b * ip * ab2);
    const double pref = 2.0 * PCM_PI * ip * K;

    // Schwarz bound |c_i c_j| max_{ab} N_a N_b [ab|ab]^(1/2) from the
    // McMurchie-Davidson diagonal two-electron integral at zero separation
    //   [ab|ab] = 2 pi^(5/2) / (p^2 sqrt(2p)) K^2
    //             sum_{tuv,t'u'v'} E_tuv E_t'u'v' (-1)^(t'+u'+v') R_{t+t',u+u',v+v'}(p/2, 0),
    // R_{TUV}(alpha, 0) = (-2 alpha)^((T+U+V)/2) (T-1)!!(U-1)!!(V-1)!! / (T+U+V+1)
    // for even T, U, V and 0 otherwise.
    E1T<LA, LB, TS> Ex, Ey, Ez;
    const TS inv2p = TS(0.5 * ip);
    // 2 pi^(5/2) / (p^2 sqrt(2 p)) K^2 (2 pi^(5/2) = 2 * 17.4934...)
    const double eri_pre = 2.0 * 17.493418327624862846 * ip * ip * sqrt(0.5 * ip) * K * K;
    hermite_E1T<LA, LB, TS>(TS(P[0] - RA[0]), TS(P[0] - RB[0]), inv2p, Ex);
    hermite_E1T<LA, LB, TS>(TS(P[1] - RA[1]), TS(P[1] - RB[1]), inv2p, Ey);
    hermite_E1T<LA, LB, TS>(TS(P[2] - RA[2]), TS(P[2] - RB[2]), inv2p, Ez);
    constexpr int LL = LA + LB;
    // (-2 alpha)^n with alpha = p / 2
    TS pw[LL + 1];
    pw[0] = TS(1);
#pragma unroll
    for (int n = 1; n <= LL; ++n) pw[n] = pw[n - 1] * TS(-p);
    double qmax = 0.0;
#pragma unroll
    for (int ca = 0; ca < ncart(LA); ++ca)
#pragma unroll
        for (int cb = 0; cb < ncart(LB); ++cb) {
            const int ax = cart_e(LA, ca, 0), ay = cart_e(LA, ca, 1), az = cart_e(LA, ca, 2);
            const int bx = cart_e(LB, cb, 0), by = cart_e(LB, cb, 1), bz = cart_e(LB, cb, 2);
            TS Gx[2 * LL + 1], Gy[2 * LL + 1], Gz[2 * LL + 1];
#pragma unroll
            for (int t = 0; t <= 2 * LL; ++t) Gx[t] = Gy[t] = Gz[t] = TS(0);
            // E_t vanishes for t > i + j, so the full loops add exact zeros there
#pragma unroll
            for (int t = 0; t <= LL; ++t)
#pragma unroll
                for (int t2 = 0; t2 <= LL; ++t2) {
                    const TS sg = (t2 & 1) ? TS(-1) : TS(1);
                    Gx[t + t2] += Ex.e[ax][bx][t] * Ex.e[ax][bx][t2] * sg;
                    Gy[t + t2] += Ey.e[ay][by][t] * Ey.e[ay][by][t2] * sg;
                    Gz[t + t2] += Ez.e[az][bz][t] * Ez.e[az][bz][t2] * sg;
                }
            TS sum = TS(0);
#pragma unroll
            for (int T = 0; T <= 2 * LL; T += 2)
#pragma unroll
                for (int U = 0; U <= 2 * LL - T; U += 2)
#pragma unroll
                    for (int V = 0; V <= 2 * LL - T - U; V += 2) {
                        const int n = (T + U + V) / 2;
                        const TS R = TS(dfact_even(T) * dfact_even(U) * dfact_even(V) / (T + U + V + 1)) * pw[n];
                        sum += Gx[T] * Gy[U] * Gz[V] * R;
                    }
            const double eri = eri_pre * (double)sum;
            const double f = comp_factor(LA, ca) * comp_factor(LB, cb);
            qmax = fmax(qmax, f * f * fabs(eri));
        }
    v.P[0] = P[0];
    v.P[1] = P[1];
    v.P[2] = P[2];
    v.p = p;
    v.pref = pref;
    v.Q = fabs(src.cnorm[src.sh_off[A] + i] * src.cnorm[src.sh_off[B] + j]) * sqrt(qmax);
    return v;
}

// FP32 value of a double from its high word (20 mantissa bits, towards zero; values
// below 2^-126 become that), without the conversion's FP64-pipe slot
__device__ __forceinline__ float trunc32(double v)
{
    const int h = __double2hiint(v);
    const int m = max(h & 0x7fffffff, 0x38100000);
    return __int_as_float((h & 0x80000000) | (min(m, 0x47efffff) - 0x38000000) << 3);
}

// log2 of an upper bound of the Schwarz bound from FP32 values: K = e^-x with
// x = ab R^2 / p and, for the sums over Hermite terms, |E_t| <= (R + 1/2p + 4)^(la + lb)
// and at most 2^14 terms of size max(1, p)^(la + lb)
template <int LA, int LB>
__device__ __forceinline__ float pair_bound_log2(const PairSrc &src, int A, int B, int i, int j)
{
    constexpr int LL = LA + LB;
    const float a = trunc32(src.exps[src.sh_off[A] + i]), b = trunc32(src.exps[src.sh_off[B] + j]);
    const double *RA = src.xyz + 3 * src.sh_atom[A], *RB = src.xyz + 3 * src.sh_atom[B];
    float R2 = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        // the truncated coordinates are off by up to 2^-20 of themselves
        const float u = trunc32(RA[d]), w = trunc32(RB[d]);
        const float t = fmaxf(fabsf(u - w) - 1e-6f * (fabsf(u) + fabsf(w)), 0.f);
        R2 = fmaf(t, t, R2);
    }
    const float p = a + b;
    if (!(p > 1e-30f && p < 1e30f)) return INFINITY;   // beyond FP32: no bound
    const float x = 0.9999f * (a / p * b) * R2;
    const float lp = __log2f(p);
    const float lc = __log2f(fabsf(trunc32(src.cnorm[src.sh_off[A] + i]))) +
                     __log2f(fabsf(trunc32(src.cnorm[src.sh_off[B] + j])));
    float lq = lc + 2.6f - 1.25f * lp - 1.4426950f * x + 1.f;
    if (LL > 0) lq += 0.5f * LL * fmaxf(lp, 0.f) + LL * __log2f(sqrtf(R2) + 0.5f / p + 4.1f) + 9.f;
    return lq;
}

// Candidates kept (Q >= thresh).  Nearly all candidates of a large molecule are far
// below the cutoff: the FP32 bound drops them before any FP64 work, which was all of
// this kernel's time (45 FP64 instructions per candidate; 1000 atoms, 40 M ss
// candidates: 3.3 ms).
template <int LA, int LB, typename TS>
__global__ void __launch_bounds__(128) pair_screen_kernel(long long ncand, PairSrc src, double thresh,
                                                          float log2_thresh, unsigned char *__restrict__ flag)
{
    __shared__ int range[2];
    const long long g0 = (long long)blockIdx.x * 128;
    const long long g = g0 + threadIdx.x;
    // the shell pairs of the block's first and last candidates bound every thread's search
    if (threadIdx.x < 2) {
        const long long t = threadIdx.x == 0 ? g0 : (g0 + 127 < ncand ? g0 + 127 : ncand - 1);
        int lo = 0, hi = src.nsp - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (src.sp_cand[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        range[threadIdx.x] = lo;
    }
    __syncthreads();
    if (g >= ncand) return;
    int s, i, j;
    pair_locate(src, g, range[0], range[1], s, i, j);
    const int A = src.spA[s], B = src.spB[s];
    bool keep = thresh <= 0.0;
    if (!keep && !(pair_bound_log2<LA, LB>(src, A, B, i, j) < log2_thresh))
        keep = pair_values<LA, LB, TS>(src, A, B, i, j).Q >= thresh;
    flag[g] = keep ? 1 : 0;
}

// the kept pairs of a class: list[0 .. n) are its kept candidates + base
template <int LA, int LB, typename TS>
__global__ void __launch_bounds__(128) pair_gather_kernel(int n, PairSrc src, const int *__restrict__ list, int base,
                                                          int *__restrict__ sp, int *__restrict__ ia,
                                                          int *__restrict__ ib, double *__restrict__ Px,
                                                          double *__restrict__ Py, double *__restrict__ Pz,
                                                          double *__restrict__ p, double *__restrict__ pref,
                                                          double *__restrict__ Q, float *__restrict__ P32)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    int s, i, j;
    pair_locate(src, list[r] - base, 0, src.nsp - 1, s, i, j);
    const PairValues v = pair_values<LA, LB, TS>(src, src.spA[s], src.spB[s], i, j);
    sp[r] = s;
    ia[r] = i;
    ib[r] = j;
    Px[r] = v.P[0];
    Py[r] = v.P[1];
    Pz[r] = v.P[2];
    p[r] = v.p;
    pref[r] = v.pref;
    Q[r] = v.Q;
    // FP32 hi/lo split of the centre: hi on a 2^-10 grid, so that differences of
    // hi parts are exact in FP32
    for (int d = 0; d < 3; ++d) {
        const double h = rint(v.P[d] * 1024.0) * (1.0 / 1024.0);
        P32[(size_t)d * n + r] = (float)h;
        P32[(size_t)(3 + d) * n + r] = (float)(v.P[d] - h);
    }
}

__device__ __forceinline__ int lower_bound(const int *__restrict__ v, int n, long long x)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (v[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

struct ClassBase {
    long long base[7];                 // first candidate of each class in the group's flags
};

// kept candidates before each class
__global__ void class_first_kernel(ClassBase b, const int *__restrict__ list, const int *__restrict__ count,
                                   int *__restrict__ first)
{
    if (threadIdx.x < 7) first[threadIdx.x] = lower_bound(list, *count, b.base[threadIdx.x]);
}

// first kept pair of each shell pair
__global__ void sp_start_kernel(int nsp, const long long *__restrict__ sp_cand, const int *__restrict__ list, int n,
                                int base, int *__restrict__ sp_start)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s <= nsp) sp_start[s] = lower_bound(list, n, base + sp_cand[s]);
}

static PairSrc pair_src(pcm_ctx *c, const PairClass &pc)
{
    PairSrc s;
    s.nsp = pc.nsp;
    s.sp_cand = pc.sp_cand.p;
    s.spA = pc.spA.p;
    s.spB = pc.spB.p;
    s.sh_atom = c->sh_atom.p;
    s.sh_nprim = c->sh_nprim.p;
    s.sh_off = c->sh_off.p;
    s.exps = c->exps.p;
    s.cnorm = c->cnorm.p;
    s.xyz = c->xyz.p;
    return s;
}

template <int LA, int LB>
static int screen_launch(pcm_ctx *c, const PairClass &pc, unsigned char *flag)
{
    if (pc.ncand == 0) return PCM_OK;
    const unsigned grid = (unsigned)((pc.ncand + 127) / 128);
    const double t = c->opt.schwarz;
    const float l = t > 0.0 ? (float)log2(t) : 0.f;
    if (c->opt.precision == PCM_MIXED)
        pair_screen_kernel<LA, LB, float><<<grid, 128, 0, c->stream>>>(pc.ncand, pair_src(c, pc), t, l, flag);
    else
        pair_screen_kernel<LA, LB, double><<<grid, 128, 0, c->stream>>>(pc.ncand, pair_src(c, pc), t, l, flag);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

template <int LA, int LB>
static int gather_launch(pcm_ctx *c, PairClass &pc, const int *list, int base)
{
    const int n = pc.npair;
    PCM_TRY(pc.sp.alloc(n));
    PCM_TRY(pc.ia.alloc(n));
    PCM_TRY(pc.ib.alloc(n));
    PCM_TRY(pc.Px.alloc(n));
    PCM_TRY(pc.Py.alloc(n));
    PCM_TRY(pc.Pz.alloc(n));
    PCM_TRY(pc.p.alloc(n));
    PCM_TRY(pc.pref.alloc(n));
    PCM_TRY(pc.Q.alloc(n));
    PCM_TRY(pc.Pxyz32.alloc(6 * (size_t)n));
    PCM_TRY(pc.sp_start.alloc(pc.nsp + 1));
    if (pc.nsp == 0) return PCM_OK;
    sp_start_kernel<<<(pc.nsp + 1 + 127) / 128, 128, 0, c->stream>>>(pc.nsp, pc.sp_cand.p, list, n, base,
                                                                    pc.sp_start.p);
    PCM_LAUNCHED(c);
    if (n == 0) return PCM_OK;
    if (c->opt.precision == PCM_MIXED)
        pair_gather_kernel<LA, LB, float><<<(n + 127) / 128, 128, 0, c->stream>>>(
            n, pair_src(c, pc), list, base, pc.sp.p, pc.ia.p, pc.ib.p, pc.Px.p, pc.Py.p, pc.Pz.p, pc.p.p, pc.pref.p,
            pc.Q.p, pc.Pxyz32.p);
    else
        pair_gather_kernel<LA, LB, double><<<(n + 127) / 128, 128, 0, c->stream>>>(
            n, pair_src(c, pc), list, base, pc.sp.p, pc.ia.p, pc.ib.p, pc.Px.p, pc.Py.p, pc.Pz.p, pc.p.p, pc.pref.p,
            pc.Q.p, pc.Pxyz32.p);
    PCM_LAUNCHED(c);
    return PCM_OK;
}

// Screening of the classes [k0, k1) together: flags of all their candidates, one
// compaction and one synchronisation, then the kept pairs' data.
static int screen_classes(pcm_ctx *c, int k0, int k1)
{
    ClassBase b;
    long long n = 0;
    for (int k = 0; k < 7; ++k) {
        b.base[k] = n;
        if (k >= k0 && k < k1) n += c->cls[k].ncand;
    }
    DBuf<unsigned char> &flag = c->su8[0];
    DBuf<int> &list = c->si[4];
    PCM_TRY(flag.alloc(std::max(1LL, n)));
    PCM_TRY(list.alloc(std::max(1LL, n)));
    for (int k = k0; k < k1; ++k) {
        unsigned char *f = flag.p + b.base[k];
        switch (k) {
        case 0: PCM_TRY((screen_launch<0, 0>(c, c->cls[k], f))); break;
        case 1: PCM_TRY((screen_launch<1, 0>(c, c->cls[k], f))); break;
        case 2: PCM_TRY((screen_launch<1, 1>(c, c->cls[k], f))); break;
        case 3: PCM_TRY((screen_launch<2, 0>(c, c->cls[k], f))); break;
        case 4: PCM_TRY((screen_launch<2, 1>(c, c->cls[k], f))); break;
        case 5: PCM_TRY((screen_launch<2, 2>(c, c->cls[k], f))); break;
        }
    }
    int first[7];
    PCM_TRY(compact_flags(c, flag.p, n, list.p, nullptr, c->iscal.p + 8));
    class_first_kernel<<<1, 32, 0, c->stream>>>(b, list.p, c->iscal.p + 8, c->iscal.p);
    PCM_LAUNCHED(c);
    PCM_CUDA(cudaMemcpyAsync(first, c->iscal.p, sizeof(first), cudaMemcpyDeviceToHost, c->stream));
    PCM_CUDA(cudaStreamSynchronize(c->stream));
    for (int k = k0; k < k1; ++k) {
        PairClass &pc = c->cls[k];
        pc.npair = first[k + 1] - first[k];
        const int *l = list.p + first[k];
        const int base = (int)b.base[k];
        switch (k) {
        case 0: PCM_TRY((gather_launch<0, 0>(c, pc, l, base))); break;
        case 1: PCM_TRY((gather_launch<1, 0>(c, pc, l, base))); break;
        case 2: PCM_TRY((gather_launch<1, 1>(c, pc, l, base))); break;
        case 3: PCM_TRY((gather_launch<2, 0>(c, pc, l, base))); break;
        case 4: PCM_TRY((gather_launch<2, 1>(c, pc, l, base))); break;
        case 5: PCM_TRY((gather_launch<2, 2>(c, pc, l, base))); break;
        }
    }
    return PCM_OK;
}

int basis_build(pcm_ctx *c, int nshell, const int *shell_atom, const int *shell_l, const int *shell_nprim,
                const double *exps, const double *coefs)
{
    // expand sp shells into an s and a p shell that share exponents; a basis that is
    // refused here leaves the context's own as it was
    std::vector<int> sh_atom, sh_l, sh_nprim, sh_off, sh_bf;
    std::vector<double> ex, co;
    int off = 0, coff = 0, bf = 0;
    for (int s = 0; s < nshell; ++s) {
        const int l = shell_l[s], n = shell_nprim[s];
        if (n <= 0 || shell_atom[s] < 0 || shell_atom[s] >= c->natom) {
            set_last_error("shell %d: bad atom index or primitive count", s);
            return PCM_ERR_ARG;
        }
        if (l > 2 || l < -1) {
            set_last_error("shell %d: angular momentum %d is not supported (s, p, d, sp only)", s, l);
            return PCM_ERR_UNSUPPORTED;
        }
        for (int i = 0; i < n; ++i)
            if (!(exps[off + i] > 0.0) || !std::isfinite(exps[off + i])) {
                set_last_error("shell %d: exponent %d is not a positive finite number", s, i);
                return PCM_ERR_ARG;
            }
        const int nparts = (l == -1) ? 2 : 1;
        for (int part = 0; part < nparts; ++part) {
            const int ll = (l == -1) ? part : l;
            sh_atom.push_back(shell_atom[s]);
            sh_l.push_back(ll);
            sh_nprim.push_back(n);
            sh_off.push_back((int)ex.size());
            sh_bf.push_back(bf);
            for (int i = 0; i < n; ++i) {
                ex.push_back(exps[off + i]);
                const double cf = coefs[coff + part * n + i];
                if (!std::isfinite(cf)) {
                    set_last_error("shell %d: contraction coefficient %d is not finite", s, i);
                    return PCM_ERR_ARG;
                }
                co.push_back(cf);
            }
            bf += ncart(ll);
        }
        off += n;
        coff += nparts * n;
    }
    c->h_sh_atom.swap(sh_atom);
    c->h_sh_l.swap(sh_l);
    c->h_sh_nprim.swap(sh_nprim);
    c->h_sh_off.swap(sh_off);
    c->h_sh_bf.swap(sh_bf);
    c->nshell = (int)c->h_sh_l.size();
    c->nbf = 0;                            // no basis until all of it is in place
    c->fock_ord.on = false;
    const int ns = c->nshell;
    PCM_TRY(c->sh_atom.alloc(ns));
    PCM_TRY(c->sh_l.alloc(ns));
    PCM_TRY(c->sh_nprim.alloc(ns));
    PCM_TRY(c->sh_off.alloc(ns));
    PCM_TRY(c->sh_bf.alloc(ns));
    PCM_TRY(c->exps.alloc(ex.size()));
    PCM_TRY(c->cnorm.alloc(ex.size()));
    DBuf<double> &dco = c->sd[4];
    PCM_TRY(dco.alloc(co.size()));
    PCM_CUDA(cudaMemcpyAsync(c->sh_atom.p, c->h_sh_atom.data(), ns * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    PCM_CUDA(cudaMemcpyAsync(c->sh_l.p, c->h_sh_l.data(), ns * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    PCM_CUDA(cudaMemcpyAsync(c->sh_nprim.p, c->h_sh_nprim.data(), ns * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    PCM_CUDA(cudaMemcpyAsync(c->sh_off.p, c->h_sh_off.data(), ns * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    PCM_CUDA(cudaMemcpyAsync(c->sh_bf.p, c->h_sh_bf.data(), ns * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    PCM_CUDA(cudaMemcpyAsync(c->exps.p, ex.data(), ex.size() * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    PCM_CUDA(cudaMemcpyAsync(dco.p, co.data(), co.size() * sizeof(double), cudaMemcpyHostToDevice, c->stream));
    cnorm_kernel<<<(ns + 15) / 16, 128, 0, c->stream>>>(ns, c->sh_l.p, c->sh_nprim.p, c->sh_off.p, c->exps.p, dco.p,
                                                         c->cnorm.p);
    PCM_LAUNCHED(c);

    // shell pairs by class (la >= lb); the higher-l shell (ties: lower index) comes
    // first.  They depend only on the shells' atoms, angular momenta and
    // primitive counts: a new geometry with the same shells (the next step of an
    // optimisation or a trajectory) reuses the lists already on the device.
    const bool same_layout = c->pair_layout_ok && c->pl_atom == c->h_sh_atom && c->pl_l == c->h_sh_l &&
                             c->pl_nprim == c->h_sh_nprim;
    if (!same_layout) {
        c->pair_layout_ok = false;
        for (int k = 0; k < 6; ++k) {
            c->cls[k].h_spA.clear();
            c->cls[k].h_spB.clear();
        }
        for (int sa = 0; sa < ns; ++sa)
            for (int sb = sa; sb < ns; ++sb) {
                int A = sa, B = sb;
                if (c->h_sh_l[sb] > c->h_sh_l[sa]) std::swap(A, B);
                const int k = class_index(c->h_sh_l[A], c->h_sh_l[B]);
                c->cls[k].h_spA.push_back(A);
                c->cls[k].h_spB.push_back(B);
            }
    }
    c->pairs_candidate = 0;
    c->pairs_kept = 0;
    PCM_TRY(c->iscal.alloc(64));
    static const int LA[6] = {0, 1, 1, 2, 2, 2}, LB[6] = {0, 0, 1, 0, 1, 2};
    for (int k = 0; k < 6; ++k) {
        PairClass &pc = c->cls[k];
        pc.la = LA[k];
        pc.lb = LB[k];
        pc.nsp = (int)pc.h_spA.size();
        if (!same_layout) {
            pc.csr_ready = false;
            std::vector<long long> cand(pc.nsp + 1, 0);
            for (int s = 0; s < pc.nsp; ++s) {
                const int A = pc.h_spA[s], B = pc.h_spB[s];
                const long long na = c->h_sh_nprim[A], nb = c->h_sh_nprim[B];
                cand[s + 1] = cand[s] + (A == B ? na * (na + 1) / 2 : na * nb);
            }
            pc.ncand = cand[pc.nsp];
            PCM_TRY(pc.spA.alloc(pc.nsp));
            PCM_TRY(pc.spB.alloc(pc.nsp));
            PCM_TRY(pc.sp_cand.alloc(pc.nsp + 1));
            if (pc.nsp > 0) {
                PCM_CUDA(cudaMemcpyAsync(pc.spA.p, pc.h_spA.data(), pc.nsp * sizeof(int), cudaMemcpyHostToDevice,
                                         c->stream));
                PCM_CUDA(cudaMemcpyAsync(pc.spB.p, pc.h_spB.data(), pc.nsp * sizeof(int), cudaMemcpyHostToDevice,
                                         c->stream));
            }
            PCM_CUDA(cudaMemcpyAsync(pc.sp_cand.p, cand.data(), (pc.nsp + 1) * sizeof(long long),
                                     cudaMemcpyHostToDevice, c->stream));
            // cand is read by the copy before it goes out of scope
            PCM_CUDA(cudaStreamSynchronize(c->stream));
        }
    }
    // all classes at once while their candidates can be numbered in 31 bits
    long long total = 0;
    for (int k = 0; k < 6; ++k) total += c->cls[k].ncand;
    if (total < (1LL << 31) - 1) {
        PCM_TRY(screen_classes(c, 0, 6));
    } else {
        for (int k = 0; k < 6; ++k) PCM_TRY(screen_classes(c, k, k + 1));
    }
    for (int k = 0; k < 6; ++k) {
        c->pairs_candidate += c->cls[k].ncand;
        c->pairs_kept += c->cls[k].npair;
    }
    if (!same_layout) {
        c->pl_atom = c->h_sh_atom;
        c->pl_l = c->h_sh_l;
        c->pl_nprim = c->h_sh_nprim;
        c->pair_layout_ok = true;
    }
    if (c->opt.precision == PCM_FP64) {
        PCM_TRY(f64_prepare(c));
    } else if (c->opt.fp32x2) {
        int first[7];
        const float *x32[6];
        for (int k = 0; k < 6; ++k) x32[k] = c->cls[k].Pxyz32.p;
        PCM_TRY(fock_order(c, kept_pairs(c, first), x32, c->fock_ord));
    }
    c->nbf = bf;
    return PCM_OK;
}

}  // namespace pcm
