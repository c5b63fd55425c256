// vs_kernels.cu -- load/read conversions, centrifuge, action, vortex check,
// re-unitarisation, hot-start generation and the exponential diagnostic.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include "vs_internal.h"
#include "vs_stout.cuh"

namespace vs {

namespace {

constexpr int kThreads = 256;

inline int nblocks(long long n, int threads = kThreads) { return (int)((n + threads - 1) / threads); }
// grid of the grid-stride kernels that first build a per-block table
constexpr int kTableGrid = 2048;

// ---------------------------------------------------------------------------
// Load / read
// ---------------------------------------------------------------------------

// Z_mu(x) = exp(2 pi i n / 3) I, Sec. I Eq. (centre_project).  One thread per link.
template <class T, int NC>
__global__ void __launch_bounds__(kThreads) k_load_labels(Geo g, const int8_t *__restrict__ lab, T *U, int8_t *ref) {
    // e^{2 pi i n / 3} for n = -1, 0, 1, three sincospi per block instead of one
    // per link (the FP64 sincospi made this kernel FP64-bound); labels outside
    // {-1, 0, 1} (possible only from device input) take the direct evaluation.
    __shared__ double zc[3], zs[3];
    if (threadIdx.x < 3) sincospi(2.0 * ((int)threadIdx.x - 1) / 3.0, &zs[threadIdx.x], &zc[threadIdx.x]);
    __syncthreads();
    for (long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x; l < 4ll * g.V;
         l += (long long)gridDim.x * blockDim.x) {
        int mu = (int)(l / g.V), s = (int)(l % g.V);
        int n = lab[l];
        Pt p = site_of_lex(g, s);
        int i = sidx(g, p);
        double sn, cs;
        if (n >= -1 && n <= 1) {
            sn = zs[n + 1];
            cs = zc[n + 1];
        } else {
            sincospi(2.0 * n / 3.0, &sn, &cs);
        }
        M3<T> z;
        m3_zero(z);
        z.re[0] = z.re[4] = z.re[8] = T(cs);
        z.im[0] = z.im[4] = z.im[8] = T(sn);
        store_link<T, NC>(U, g.P, mu, i, z);
        ref[(long long)mu * g.P + i] = (int8_t)n;
    }
}

// FP64 link matrices of the caller ([..][9] (re, im) pairs, 144 bytes per matrix)
// pass through shared memory on their way in and out: a warp's global accesses
// are then runs of 256 bytes, where one thread per matrix touches 32 sectors
// 144 bytes apart with every 8-byte access (read at 32^3x64: 1.02 ms that way,
// against the 0.27 ms that its 1.8 GB take at the copy rate).  The accesses stay
// 8 bytes wide because the caller's pointer need not be aligned to more.  A
// block takes kThreads consecutive sites of one direction (V is a multiple of
// 256: every extent is a multiple of 4).
template <class T>
__device__ __forceinline__ M3<T> staged_matrix(const double *__restrict__ in, double *sm, double &tr, double &ti) {
#pragma unroll
    for (int k = 0; k < 18; ++k) sm[k * kThreads + threadIdx.x] = in[k * kThreads + threadIdx.x];
    __syncthreads();
    const double2 *q = reinterpret_cast<const double2 *>(sm) + 9 * threadIdx.x;
    M3<T> m;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double2 v = q[k];
        m.re[k] = T(v.x);
        m.im[k] = T(v.y);
        if (k == 0) { tr = v.x; ti = v.y; }
        if (k == 4 || k == 8) { tr += v.x; ti += v.y; }
    }
    return m;
}

// The matrix at q, read by its own thread.
template <class T>
__device__ __forceinline__ M3<T> direct_matrix(const double *__restrict__ q, double &tr, double &ti) {
    M3<T> m;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        m.re[k] = T(q[2 * k]);
        m.im[k] = T(q[2 * k + 1]);
    }
    tr = q[0] + q[8] + q[16];
    ti = q[1] + q[9] + q[17];
    return m;
}

// Links from FP64 host layout; the reference label is the sector of arg Tr U of the FP64 input.
// A thread's 18 reads of its matrix find the line of the first in L1, so staging pays only
// for 18-real links in rows whose runs of 5 or 7 sites leave unused positions (FP64, us
// staged / direct: 20^3x40 111.3 / 119.6, 28^3x56 309 / 336, but 24^3x48 139.1 / 131.3,
// 12x40^3 154.5 / 143.5; 12 reals 16^3x32 29.3 / 27.8).
template <class T, int NC, bool STAGED>
__global__ void __launch_bounds__(kThreads) k_load_links(Geo g, const double *__restrict__ in, T *U, int8_t *ref) {
    __shared__ __align__(16) double sm[STAGED ? kThreads * 18 : 1];
    const int mu = blockIdx.y, s0 = blockIdx.x * kThreads;
    double tr, ti;
    const double *first = in + ((long long)mu * g.V + s0) * 18;
    M3<T> m;
    if constexpr (STAGED) m = staged_matrix<T>(first, sm, tr, ti);
    else m = direct_matrix<T>(first + 18 * threadIdx.x, tr, ti);
    const int i = sidx(g, site_of_lex(g, s0 + threadIdx.x));
    store_link<T, NC>(U, g.P, mu, i, m);
    ref[(long long)mu * g.P + i] = (int8_t)z3_label<double>(tr, ti);
}

template <class T, int NC>
__global__ void __launch_bounds__(kThreads) k_read_links(Geo g, const T *__restrict__ U, double *out) {
    __shared__ __align__(16) T sm[kThreads * 18];
    const int mu = blockIdx.y, s0 = blockIdx.x * kThreads;
    const M3<T> m = load_link<T, NC>(U, g.P, mu, sidx(g, site_of_lex(g, s0 + threadIdx.x)));
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        T *q = sm + 18 * threadIdx.x + 2 * k;
        if constexpr (sizeof(T) == 4) *reinterpret_cast<float2 *>(q) = make_float2(m.re[k], m.im[k]);
        else *reinterpret_cast<double2 *>(q) = make_double2(m.re[k], m.im[k]);
    }
    __syncthreads();
    double *o = out + ((long long)mu * g.V + s0) * 18;
#pragma unroll
    for (int k = 0; k < 18; ++k) o[k * kThreads + threadIdx.x] = double(sm[k * kThreads + threadIdx.x]);
}

__global__ void k_read_labels(Geo g, const int8_t *__restrict__ ref, int8_t *out) {
    long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= 4ll * g.V) return;
    int mu = (int)(l / g.V), s = (int)(l % g.V);
    out[l] = ref[(long long)mu * g.P + sidx(g, site_of_lex(g, s))];
}

// Links with a non-finite entry (NaN or Inf), one thread per link.
template <class T, int NC>
__global__ void k_count_nonfinite(Geo g, const T *__restrict__ U, unsigned long long *count) {
    long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    bool bad = false;
    if (l < 4ll * g.V) {
        const M3<T> m = load_link<T, NC>(U, g.P, (int)(l / g.V), sidx(g, site_of_index(g, (int)(l % g.V))));
#pragma unroll
        for (int k = 0; k < 9; ++k) bad |= !isfinite(m.re[k]) || !isfinite(m.im[k]);
    }
    const unsigned b = __ballot_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && b) atomicAdd(count, (unsigned long long)__popc(b));
}

// reference labels from lexicographic order into plane order (restore)
__global__ void k_store_ref(Geo g, const int8_t *__restrict__ lab, int8_t *ref) {
    long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= 4ll * g.V) return;
    int mu = (int)(l / g.V), s = (int)(l % g.V);
    ref[(long long)mu * g.P + sidx(g, site_of_lex(g, s))] = lab[l];
}

// One thread per link, one direction per grid row; a label needs the link's
// diagonal, so only the chunks that hold it are loaded (40 of 72 bytes).
template <class T, int NC>
__global__ void __launch_bounds__(kThreads) k_current_labels(Geo g, const T *__restrict__ U, int8_t *out) {
    const int mu = blockIdx.y, s = blockIdx.x * kThreads + threadIdx.x;
    const M3<T> m = load_link<T, NC>(U, g.P, mu, sidx(g, site_of_lex(g, s)));
    out[(long long)mu * g.V + s] = (int8_t)z3_label<T>(m.re[0] + m.re[4] + m.re[8], m.im[0] + m.im[4] + m.im[8]);
}

// ---------------------------------------------------------------------------
// Centrifuge preconditioning, Sec. IV
// ---------------------------------------------------------------------------

// m = sum_{nu != mu} [n_nu(x) + n_mu(x+nu) - n_nu(x+mu) - n_nu(x-nu) + n_mu(x-nu)
// + n_nu(x-nu+mu)] so that sigma = m 2 pi / 18; delta = omega (sigma - lambda)
// = omega pi (m - 6n) / 9.  Pair p = SplitMix64(seed, mu V + s) mod 3 picks
// (j,k) = (0,1), (1,2), (2,0): phase j gets lambda + delta, phase k lambda - delta.
// The phases take few values: pi (2n/3 + omega k/9) with n in {-1, 0, 1} and
// k = +-(m - 6n) in [-24, 24] (k = 0 is the untouched phase 2n/3).
// k_centrifuge_table evaluates them once, with the same FP64 expressions as the
// per-link form, so the links are bit-identical to it; values outside the table
// (labels outside {-1, 0, 1}, only from device input) are evaluated directly.
// The table is a kernel of its own: one warp per SM computes 32 entries in a
// microsecond or two, where a table per block kept every SM's FP64 pipe busy for
// ~10 us a block (0.16 of the 0.53 ms that the single kernel took at 32^3x64).
constexpr int kCtabK = 24, kCtabN = 3 * (2 * kCtabK + 1);

__device__ __forceinline__ double2 centrifuge_phase(double omega, int n, int k) {
    const double delta = omega * (double)k / 9.0;   // in units of pi
    double2 v;
    sincospi(2.0 * n / 3.0 + delta, &v.y, &v.x);
    return v;
}

__global__ void k_centrifuge_table(double omega, double2 *tab) {   // (cos, sin) at (n + 1)(2K + 1) + k + K
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < kCtabN) tab[e] = centrifuge_phase(omega, e / (2 * kCtabK + 1) - 1, e % (2 * kCtabK + 1) - kCtabK);
}

// One thread per site, its four links: 44 label reads at 21 positions, where a
// thread per link read 19 labels at 13 positions four times over.  At 32^3x64
// the links written (604 MB) take 0.09 ms at the copy rate.
template <class T, int NC>
__global__ void __launch_bounds__(kThreads) k_centrifuge(Geo g, const int8_t *__restrict__ ref, double omega,
                                                          uint64_t seed, T *U, const double2 *__restrict__ gtab) {
    using T2 = typename std::conditional<sizeof(T) == 4, float2, double2>::type;
    __shared__ T2 tab[kCtabN];
    for (int e = threadIdx.x; e < kCtabN; e += blockDim.x) {
        const double2 v = gtab[e];
        tab[e].x = T(v.x);
        tab[e].y = T(v.y);
    }
    __syncthreads();
    for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < g.V; d += gridDim.x * blockDim.x) {
        const Pt x = site_of_index(g, d);
        const int i = sidx(g, x), s = lexidx(g, x);
        int dp[4], dm[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            dp[a] = shift_delta(g, x, a, 1);
            dm[a] = shift_delta(g, x, a, -1);
        }
        const int8_t *lab[4] = {ref + i, ref + g.P + i, ref + 2 * g.P + i, ref + 3 * g.P + i};
        int n[4], m[4];
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            n[mu] = lab[mu][0];
            m[mu] = 0;
        }
#pragma unroll
        for (int mu = 0; mu < 4; ++mu)
#pragma unroll
            for (int j = 1; j < 4; ++j) {
                const int nu = (mu + j) & 3;
                m[mu] += n[nu] + (int)lab[mu][dp[nu]] - (int)lab[nu][dp[mu]] - (int)lab[nu][dm[nu]] +
                         (int)lab[mu][dm[nu]] + (int)lab[nu][dm[nu] + dp[mu]];
            }
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            const int k = m[mu] - 6 * n[mu];
            const uint64_t z64 = splitmix64(seed, (uint64_t)mu * (uint64_t)g.V + (uint64_t)s);
            // z64 mod 3, with 2^32 = 1 (mod 3)
            const int jj = (int)(((uint32_t)(z64 >> 32) % 3u + (uint32_t)z64 % 3u) % 3u), kk = jj == 2 ? 0 : jj + 1;
            const bool in_tab = n[mu] >= -1 && n[mu] <= 1 && k >= -kCtabK && k <= kCtabK;
            M3<T> z;
            m3_zero(z);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int kc = c == jj ? k : c == kk ? -k : 0;
                if (in_tab) {
                    const T2 v = tab[(n[mu] + 1) * (2 * kCtabK + 1) + kc + kCtabK];
                    z.re[4 * c] = v.x;
                    z.im[4 * c] = v.y;
                } else {
                    const double2 v = centrifuge_phase(omega, n[mu], kc);
                    z.re[4 * c] = T(v.x);
                    z.im[4 * c] = T(v.y);
                }
            }
            store_link<T, NC>(U, g.P, mu, i, z);
        }
    }
}

// ---------------------------------------------------------------------------
// Wilson action, Sec. V: sum_x sum_{mu<nu} (3 - Re Tr P_munu(x)); each
// plaquette in the storage precision, the sums in FP64 in a fixed order
// (block tree, then one block over the partials).
// ---------------------------------------------------------------------------

__device__ __forceinline__ double block_sum(double v) {
    __shared__ double sh[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int w = threadIdx.x >> 5, ln = threadIdx.x & 31;
    if (ln == 0) sh[w] = v;
    __syncthreads();
    v = 0;
    if (w == 0) {
        int nw = blockDim.x >> 5;
        v = ln < nw ? sh[ln] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    __syncthreads();
    return v;
}

// Sum of a few values of the storage precision as FP64 would give it.  FP32: an
// error-free transformation (Knuth's TwoSum), so that a site costs two
// conversions instead of an FP64 operation per value (GB300's FP64 pipe takes a
// warp instruction every 16 cycles; 18 per site were 60 us of k_action at
// 32^3x64).
template <class T> struct ShortSum;
template <> struct ShortSum<double> {
    double v = 0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ double value() const { return v; }
};
template <> struct ShortSum<float> {
    float hi = 0, lo = 0;
    __device__ __forceinline__ void add(float x) {
        const float s = hi + x, b = s - hi;
        lo += (hi - (s - b)) + (x - b);
        hi = s;
    }
    // an infinite sum leaves NaN in lo
    __device__ __forceinline__ double value() const { return lo == lo ? (double)hi + (double)lo : (double)hi; }
};

// Sum of 3 - Re Tr P over a site's six plaquettes.  FP64 adds the differences, which
// are exact near 3: a smooth field's small action keeps its digits, where 18 less the
// sum of the traces would round at the size of 18.  The FP32 sum of the traces is exact.
template <class T> struct PlaqSum;
template <> struct PlaqSum<double> {
    double v = 0;
    __device__ __forceinline__ void add(double retr) { v += 3.0 - retr; }
    __device__ __forceinline__ double value() const { return v; }
};
template <> struct PlaqSum<float> {
    ShortSum<float> tr;
    __device__ __forceinline__ void add(float retr) { tr.add(retr); }
    __device__ __forceinline__ double value() const { return 18.0 - tr.value(); }
};

// Blocks of the measurement kernels: kMeasThreads threads, one wave of resident
// blocks, grid-stride over the sites.  Both are bound by the latency and the
// L1/L2 rate of their link loads (1.5 and 6 KB per site), so what counts is warps
// per SM: 16 for the action (120 registers), 12 for the observables (168), where
// blocks of 256 threads left 8.  Per call at 32^3x64, FP32: action 395 -> 213 us
// (five blocks per SM spill: 295), observables 1174 -> 880 us (four: 980).  FP64: two
// blocks per SM at a time (up to 255 registers); the action takes eight in all, so that the
// last of its four rounds is short (28^3x56 2996 -> 2957 us).
constexpr int kMeasThreads = 128, kActionPerSM = 4, kObsPerSM = 3, kMeasFp64PerSM = 2, kActionFp64Blocks = 8;

template <class T, int NC>
__global__ void __launch_bounds__(kMeasThreads, sizeof(T) == 4 ? kActionPerSM : kMeasFp64PerSM)
    k_action(Geo g, const T *__restrict__ U, double *partials) {
    double acc = 0;
    for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < g.V; d += gridDim.x * blockDim.x) {
        const Pt x = site_of_index(g, d);
        const int i = sidx(g, x);
        PlaqSum<T> s;
#pragma unroll 1
        for (int mu = 0; mu < 3; ++mu) {
            const M3<T> Umu = load_link<T, NC>(U, g.P, mu, i);
            const int im = i + shift_delta(g, x, mu, 1);
#pragma unroll 1
            for (int nu = mu + 1; nu < 4; ++nu) {
                // P = (U_mu(x) U_nu(x+mu)) (U_nu(x) U_mu(x+nu))^dag
                const M3<T> X = m3_mul(Umu, load_link<T, NC>(U, g.P, nu, im));
                const M3<T> Y = m3_mul(load_link<T, NC>(U, g.P, nu, i),
                                       load_link<T, NC>(U, g.P, mu, i + shift_delta(g, x, nu, 1)));
                // Re Tr(X Y^dag) in the storage precision: the FP32 products
                // already carry FP32 rounding, and an FP64 dot (18 conversions
                // and FMAs on the slow FP64 pipe) made this kernel FP64-bound
                T re = T(0);
#pragma unroll
                for (int k = 0; k < 9; ++k) re = fma(X.re[k], Y.re[k], fma(X.im[k], Y.im[k], re));
                s.add(re);
            }
        }
        acc += s.value();
    }
    double b = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = b;
}

// ---------------------------------------------------------------------------
// Smoothness observables, Sec. V: clover F_munu (the mean of the four leaves of
// the plane at x, F = (C - C^dag)/(2i), traceless), per site
//   S(x)/beta   = 1/72 sum_{mu != nu} Re Tr(1 - P_munu)
//   S_R(x)/beta = 1/72 sum_{mu != nu} Tr(F_munu^2) / 2
//   q(x)        = [Tr(F01 F23) - Tr(F02 F13) + Tr(F03 F12)] / (4 pi^2)
// (the eps-sum of Eq. 1LTopQ collapsed to its three pairings x 8 / (32 pi^2)).
// ---------------------------------------------------------------------------

// F_munu(x) by its diagonal h[0..2] and upper entries h[3..8] (re, im).
template <class T, int NC>
__device__ __forceinline__ void clover_F(const Geo &g, const T *__restrict__ U, const Pt &x, int i, int mu, int nu,
                                         T h[9], T &plaq_retr) {
    const int pm = shift_delta(g, x, mu, 1), mm = shift_delta(g, x, mu, -1);
    const int pn = shift_delta(g, x, nu, 1), mn = shift_delta(g, x, nu, -1);
    M3<T> C, L;
    // leaf 1: +mu +nu -mu -nu
    L = m3_mul(load_link<T, NC>(U, g.P, mu, i), load_link<T, NC>(U, g.P, nu, i + pm));
    L = m3_mul_nd(L, load_link<T, NC>(U, g.P, mu, i + pn));
    L = m3_mul_nd(L, load_link<T, NC>(U, g.P, nu, i));
    plaq_retr = L.re[0] + L.re[4] + L.re[8];
    C = L;
    // leaf 2: +nu -mu -nu +mu
    L = m3_mul_nd(load_link<T, NC>(U, g.P, nu, i), load_link<T, NC>(U, g.P, mu, i + pn + mm));
    L = m3_mul_nd(L, load_link<T, NC>(U, g.P, nu, i + mm));
    m3_madd(C, L, load_link<T, NC>(U, g.P, mu, i + mm));
    // leaf 3: -mu -nu +mu +nu
    L = m3_mul_dn(load_link<T, NC>(U, g.P, mu, i + mm), m3_dag(load_link<T, NC>(U, g.P, nu, i + mm + mn)));
    L = m3_mul(L, load_link<T, NC>(U, g.P, mu, i + mm + mn));
    m3_madd(C, L, load_link<T, NC>(U, g.P, nu, i + mn));
    // leaf 4: -nu +mu +nu -mu
    L = m3_mul_dn(load_link<T, NC>(U, g.P, nu, i + mn), load_link<T, NC>(U, g.P, mu, i + mn));
    L = m3_mul(L, load_link<T, NC>(U, g.P, nu, i + mn + pm));
    L = m3_mul_nd(L, load_link<T, NC>(U, g.P, mu, i));
#pragma unroll
    for (int k = 0; k < 9; ++k) { C.re[k] += L.re[k]; C.im[k] += L.im[k]; }
    // F = (C - C^dag) / (2i) / 4, traceless
#pragma unroll
    for (int j = 0; j < 3; ++j) h[j] = T(0.125) * (C.im[4 * j] + C.im[4 * j]);
    const T tr = (h[0] + h[1] + h[2]) / T(3);
#pragma unroll
    for (int j = 0; j < 3; ++j) h[j] -= tr;
    h[3] = T(0.125) * (C.im[1] + C.im[3]); h[4] = -T(0.125) * (C.re[1] - C.re[3]);
    h[5] = T(0.125) * (C.im[2] + C.im[6]); h[6] = -T(0.125) * (C.re[2] - C.re[6]);
    h[7] = T(0.125) * (C.im[5] + C.im[7]); h[8] = -T(0.125) * (C.re[5] - C.re[7]);
}

// Tr(A B) for Hermitian A, B by diagonal and upper entries: sum_jk A_jk
// conj(B_jk), row by row, in the storage precision (its FP32 inputs already carry
// FP32 rounding; an FP64 dot made the kernel FP64-bound); the sums over sites run
// in FP64.
template <class T>
__device__ __forceinline__ T tr_herm(const T a[9], const T b[9]) {
    const T o01 = fma(a[3], b[3], a[4] * b[4]), o02 = fma(a[5], b[5], a[6] * b[6]), o12 = fma(a[7], b[7], a[8] * b[8]);
    T s = a[0] * b[0];
    s += o01;
    s += o02;
    s += o01;
    s += a[1] * b[1];
    s += o12;
    s += o02;
    s += o12;
    s += a[2] * b[2];
    return s;
}

template <class T, int NC>
__global__ void __launch_bounds__(kMeasThreads, sizeof(T) == 4 ? kObsPerSM : kMeasFp64PerSM)
    k_observables(Geo g, const T *__restrict__ U, double *partials, double *S_site, double *SR_site,
                  double *q_site) {
    double aS = 0, aSR = 0, aQ = 0;
    for (int d = blockIdx.x * blockDim.x + threadIdx.x; d < g.V; d += gridDim.x * blockDim.x) {
        const Pt x = site_of_index(g, d);
        const int i = sidx(g, x);
        PlaqSum<T> ss;
        ShortSum<T> ssr, sq;
        // the pairings (01, 23), (02, 13), (03, 12) with signs +, -, +, one plane
        // at a time so that the clover code exists once
        T fa[9];
#pragma unroll 1
        for (int p = 0; p < 6; ++p) {
            const int j = (p >> 1) + 1;                       // the partner of direction 0
            const int mu = p & 1 ? (j == 1 ? 2 : 1) : 0, nu = p & 1 ? (j == 3 ? 2 : 3) : j;
            T f[9], re;
            clover_F<T, NC>(g, U, x, i, mu, nu, f, re);
            ss.add(re);
            ssr.add(tr_herm(f, f));
            if (p & 1) {
                const T qq = tr_herm(fa, f);
                sq.add(j == 2 ? -qq : qq);
            }
#pragma unroll
            for (int k = 0; k < 9; ++k) fa[k] = f[k];
        }
        const double s = ss.value() * (2.0 / 72.0), sr = ssr.value() / 72.0,
                     q = sq.value() / (4.0 * 9.869604401089358);
        const int lx = lexidx(g, x);
        if (S_site) S_site[lx] = s;
        if (SR_site) SR_site[lx] = sr;
        if (q_site) q_site[lx] = q;
        aS += s;
        aSR += sr;
        aQ += q;
    }
    const double b0 = block_sum(aS), b1 = block_sum(aSR), b2 = block_sum(aQ);
    if (threadIdx.x == 0) {
        partials[3 * blockIdx.x] = b0;
        partials[3 * blockIdx.x + 1] = b1;
        partials[3 * blockIdx.x + 2] = b2;
    }
}

__global__ void k_sum_partials3(const double *__restrict__ partials, int n, double invV, double *out) {
    for (int c = 0; c < 3; ++c) {
        double acc = 0;
        for (int i = threadIdx.x; i < n; i += blockDim.x) acc += partials[3 * i + c];
        const double b = block_sum(acc);
        if (threadIdx.x == 0) out[c] = c < 2 ? b * invV : b;
    }
}

__global__ void k_sum_partials(const double *__restrict__ partials, int n, double scale, double *out) {
    double acc = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += partials[i];
    double b = block_sum(acc);
    if (threadIdx.x == 0) *out = b * scale;
}

// ---------------------------------------------------------------------------
// Correlation of two densities, Sec. VII Eq. (correlation_s):
//   C = <a b> / (sqrt<a^2> sqrt<b^2>)
// three FP64 sums in a fixed order (grid-stride loop over a fixed grid, block
// tree, then one block over the partials), so the result is bit-reproducible.
// ---------------------------------------------------------------------------

constexpr int kCorrGrid = 400;

__global__ void __launch_bounds__(kThreads) k_correlation(const double *__restrict__ a, const double *__restrict__ b,
                                                          long long n, double *partials) {
    double sab = 0, saa = 0, sbb = 0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const double x = a[i], y = b[i];
        sab = fma(x, y, sab);
        saa = fma(x, x, saa);
        sbb = fma(y, y, sbb);
    }
    sab = block_sum(sab);
    saa = block_sum(saa);
    sbb = block_sum(sbb);
    if (threadIdx.x == 0) {
        partials[3 * blockIdx.x] = sab;
        partials[3 * blockIdx.x + 1] = saa;
        partials[3 * blockIdx.x + 2] = sbb;
    }
}

// out[0] = C, out[1..3] = the three sums (a zero norm leaves C = NaN)
__global__ void k_correlation_finish(const double *__restrict__ partials, int nb, double *out) {
    double s[3];
    for (int c = 0; c < 3; ++c) {
        double acc = 0;
        for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += partials[3 * i + c];
        s[c] = block_sum(acc);
    }
    if (threadIdx.x == 0) {
        out[1] = s[0];
        out[2] = s[1];
        out[3] = s[2];
        // the means' 1/n cancels between numerator and denominator
        out[0] = (s[1] > 0 && s[2] > 0) ? s[0] / (sqrt(s[1]) * sqrt(s[2])) : __longlong_as_double(0x7ff8000000000000ll);
    }
}

// ---------------------------------------------------------------------------
// Vortex check
// ---------------------------------------------------------------------------

// One thread per site, its four links; in FP64 on fields of few sites (kLinkSites) one per
// link, direction blockIdx.y.  dz: per link (current - reference label)
// mod 3 in {0, 1, 2}, all that the charges need.  A warp's smallest margin goes
// to the global minimum only if it is below the value read there: with one
// 64-bit atomicMin per warp of links, all to one address, this kernel took
// 0.21 ms at 32^3x64 whatever it read.  Without a gauge only the diagonals are
// loaded (40 of 72 bytes per FP32 link, 335 MB: 0.05 ms at the copy rate).
template <class T, int NC, bool GAUGE, bool LINK>
__global__ void __launch_bounds__(kThreads) k_vortex_links(Geo g, const T *__restrict__ U,
                                                            const int8_t *__restrict__ ref, int8_t *dz,
                                                            unsigned long long *counts, unsigned long long *mbits,
                                                            const T *__restrict__ G) {
    const Pt x = site_of_index(g, blockIdx.x * kThreads + threadIdx.x);   // V is a multiple of kThreads
    const int i = sidx(g, x);
    int n_diff = 0, n_near = 0;
    double margin = 1e300;
#pragma unroll
    for (int j = 0; j < (LINK ? 1 : 4); ++j) {
        const int mu = LINK ? (int)blockIdx.y : j;
        const M3<T> m = load_link<T, NC>(U, g.P, mu, i);
        T a, b;
        if constexpr (GAUGE) vp_trace<T>(G, g.P, i, i + shift_delta(g, x, mu, 1), m, a, b);
        else vp_trace<T>((const T *)nullptr, g.P, i, i, m, a, b);
        const int d = z3_label<T>(a, b) - (int)ref[(long long)mu * g.P + i];
        dz[(long long)mu * g.P + i] = (int8_t)((d % 3 + 3) % 3);
        n_diff += d != 0;
        // angular distance of arg Tr U from the nearest sector edge (+-pi/3,
        // pi), in the field's precision: an FP32 trace is itself rounded to
        // ~1e-7, and an FP64 atan2 per link made this kernel FP64-bound
        double mg;
        if constexpr (sizeof(T) == 4) {
            const float argf = atan2f(b + 0.0f, a);
            const float pi3f = 1.04719755f;
            mg = (double)fminf(fminf(fabsf(argf - pi3f), fabsf(argf + pi3f)), 3.14159265f - fabsf(argf));
        } else {
            const double arg = atan2((double)b + 0.0, (double)a);
            const double pi3 = 1.0471975511965976;
            mg = fmin(fmin(fabs(arg - pi3), fabs(arg + pi3)), 3.141592653589793 - fabs(arg));
        }
        n_near += mg < 1e-5;
        margin = fmin(margin, mg);
    }
    if (__any_sync(0xffffffffu, n_diff | n_near)) {
        n_diff = __reduce_add_sync(0xffffffffu, n_diff);
        n_near = __reduce_add_sync(0xffffffffu, n_near);
        if ((threadIdx.x & 31) == 0) {
            if (n_diff) atomicAdd(&counts[0], (unsigned long long)n_diff);
            if (n_near) atomicAdd(&counts[2], (unsigned long long)n_near);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) margin = fmin(margin, __shfl_xor_sync(0xffffffffu, margin, o));
    if ((threadIdx.x & 31) == 0 && margin < 1e300) {
        const unsigned long long bits = (unsigned long long)__double_as_longlong(margin);
        if (bits < *(volatile unsigned long long *)mbits) atomicMin(mbits, bits);
    }
}

// Plaquettes whose centre charge p = n_mu(x) + n_nu(x+mu) - n_mu(x+nu) - n_nu(x)
// (mod 3) differs from the reference: those whose label differences dz do not
// cancel mod 3.  Where no label differs (every check of a vortex-preserving run)
// no charge can, and the kernel ends on the count that k_vortex_links left.
__global__ void __launch_bounds__(kThreads) k_vortex_charges(Geo g, const int8_t *__restrict__ dz,
                                                              unsigned long long *counts) {
    if (counts[0] == 0) return;
    const Pt x = site_of_index(g, blockIdx.x * kThreads + threadIdx.x);
    const int i = sidx(g, x);
    int here[4], nd = 0;
    const int8_t *lab[4] = {dz + i, dz + g.P + i, dz + 2 * g.P + i, dz + 3 * g.P + i};
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) here[mu] = lab[mu][0];
    int dp[4];
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) dp[mu] = shift_delta(g, x, mu, 1);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
#pragma unroll
        for (int nu = mu + 1; nu < 4; ++nu)
            nd += (here[mu] + (int)lab[nu][dp[mu]] - (int)lab[mu][dp[nu]] - here[nu] + 6) % 3 != 0;
    nd = __reduce_add_sync(0xffffffffu, nd);
    if ((threadIdx.x & 31) == 0 && nd) atomicAdd(&counts[1], (unsigned long long)nd);
}

// ---------------------------------------------------------------------------
// Re-unitarisation: r0 /= |r0|; r1 -= (r0^dag r1) r0; r1 /= |r1|;
// r2 = conj(r0 x r1), all in the storage precision.  For FP32 links the
// result is unitary to the rounding of the stored rows (a few 1e-7), the
// level the FP32 sweeps themselves leave; FP64 norms would buy nothing
// measurable and make the kernel FP64-bound (GB300's FP64 pipe runs at
// 1/64 of FP32) instead of HBM-bound.
// With ref != nullptr (vortex preservation on) a re-unitarised link whose
// Z(3) label would differ from the reference is left as it was, so every
// stored link keeps its original label.
// ---------------------------------------------------------------------------

template <class T, int NC>
__global__ void k_reunit(Geo g, T *U, const int8_t *__restrict__ ref, const T *__restrict__ G) {
    long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= 4ll * g.V) return;
    const int mu = (int)(l / g.V);
    const Pt x = site_of_index(g, (int)(l % g.V));
    const int i = sidx(g, x);
    M3<T> m = load_link<T, NC>(U, g.P, mu, i);
    T n0 = T(0);
#pragma unroll
    for (int b = 0; b < 3; ++b) n0 = fma(m.re[b], m.re[b], fma(m.im[b], m.im[b], n0));
    const T s0 = T(1) / sqrt(n0);
#pragma unroll
    for (int b = 0; b < 3; ++b) { m.re[b] *= s0; m.im[b] *= s0; }
    T pr = T(0), pi = T(0);  // r0^dag r1
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        pr = fma(m.re[b], m.re[3 + b], fma(m.im[b], m.im[3 + b], pr));
        pi = fma(m.re[b], m.im[3 + b], fma(-m.im[b], m.re[3 + b], pi));
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        m.re[3 + b] -= pr * m.re[b] - pi * m.im[b];
        m.im[3 + b] -= pr * m.im[b] + pi * m.re[b];
    }
    T n1 = T(0);
#pragma unroll
    for (int b = 0; b < 3; ++b) n1 = fma(m.re[3 + b], m.re[3 + b], fma(m.im[3 + b], m.im[3 + b], n1));
    const T s1 = T(1) / sqrt(n1);
#pragma unroll
    for (int b = 0; b < 3; ++b) { m.re[3 + b] *= s1; m.im[3 + b] *= s1; }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int j1 = (j + 1) % 3, j2 = (j + 2) % 3;
        T cr = m.re[j1] * m.re[3 + j2] - m.im[j1] * m.im[3 + j2] - (m.re[j2] * m.re[3 + j1] - m.im[j2] * m.im[3 + j1]);
        T ci = m.re[j1] * m.im[3 + j2] + m.im[j1] * m.re[3 + j2] - (m.re[j2] * m.im[3 + j1] + m.im[j2] * m.re[3 + j1]);
        m.re[6 + j] = cr;
        m.im[6 + j] = -ci;
    }
    if (ref) {
        T a, b;
        vp_trace<T>(G, g.P, i, G ? sidx(g, mv(g, x, mu, 1)) : i, m, a, b);
        if (z3_label<T>(a, b) != (int)ref[(long long)mu * g.P + i]) return;
    }
    store_link<T, NC>(U, g.P, mu, i, m);
}

// ---------------------------------------------------------------------------
// Exponential diagnostic: E = exp(X), X traceless anti-Hermitian, via H = -iX
// ---------------------------------------------------------------------------

template <class T>
__global__ void k_debug_expm(const double *__restrict__ X, int n, double *E) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const double *x = X + 18ll * t;
    // H_jk = -i X_jk -> re = Im X_jk, im = -Re X_jk
    auto hre = [&](int j, int k) { return T(x[2 * (3 * j + k) + 1]); };
    auto him = [&](int j, int k) { return T(-x[2 * (3 * j + k)]); };
    bool f64;
    M3<T> M = exp_iH<T>(hre(0, 0), hre(1, 1), hre(2, 2), hre(0, 1), him(0, 1), hre(0, 2), him(0, 2),
                        hre(1, 2), him(1, 2), f64);
    double *e = E + 18ll * t;
    for (int k = 0; k < 9; ++k) { e[2 * k] = double(M.re[k]); e[2 * k + 1] = double(M.im[k]); }
}

// ---------------------------------------------------------------------------
// Hot start and MaxReTr cooling (input generation)
// ---------------------------------------------------------------------------

// Haar SU(3) per link: 18 Gaussians by Box-Muller from SplitMix64 values
// 18 l .. 18 l + 17 of `seed` (pair k: radius from value 2k, angle from 2k+1),
// Z_jk = (g_{2(3j+k)} + i g_{2(3j+k)+1}) / sqrt 2, Gram-Schmidt on the columns
// (QR with positive diag R: Haar U(3), Mezzadri 2007), then divide by the
// principal cube root of det.
template <class T, int NC>
__global__ void k_haar(Geo g, uint64_t seed, T *U) {
    long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= 4ll * g.V) return;
    int mu = (int)(l / g.V), s = (int)(l % g.V);
    double zr[9], zi[9];
    const double inv53 = 1.0 / 9007199254740992.0;
    for (int k = 0; k < 9; ++k) {
        uint64_t c = (uint64_t)l * 18ull + 2ull * k;
        double u1 = 1.0 - (double)(splitmix64(seed, c) >> 11) * inv53;
        double u2 = (double)(splitmix64(seed, c + 1) >> 11) * inv53;
        double rad = sqrt(-2.0 * log(u1));
        double sn, cs;
        sincospi(2.0 * u2, &sn, &cs);
        zr[k] = rad * cs * 0.7071067811865476;
        zi[k] = rad * sn * 0.7071067811865476;
    }
    // Gram-Schmidt on columns c = 0, 1, 2 (entries (j, c) at index 3j + c)
    for (int c = 0; c < 3; ++c) {
        for (int p = 0; p < c; ++p) {
            double pr = 0, pi = 0;  // <q_p, z_c> = sum conj(q_jp) z_jc
            for (int j = 0; j < 3; ++j) {
                pr += zr[3 * j + p] * zr[3 * j + c] + zi[3 * j + p] * zi[3 * j + c];
                pi += zr[3 * j + p] * zi[3 * j + c] - zi[3 * j + p] * zr[3 * j + c];
            }
            for (int j = 0; j < 3; ++j) {
                zr[3 * j + c] -= pr * zr[3 * j + p] - pi * zi[3 * j + p];
                zi[3 * j + c] -= pr * zi[3 * j + p] + pi * zr[3 * j + p];
            }
        }
        double nn = 0;
        for (int j = 0; j < 3; ++j) nn += zr[3 * j + c] * zr[3 * j + c] + zi[3 * j + c] * zi[3 * j + c];
        nn = 1.0 / sqrt(nn);
        for (int j = 0; j < 3; ++j) { zr[3 * j + c] *= nn; zi[3 * j + c] *= nn; }
    }
    // det by expansion along row 0
    auto cm = [](double ar, double ai, double br, double bi, double &rr, double &ri) {
        rr = ar * br - ai * bi; ri = ar * bi + ai * br;
    };
    double dr = 0, di = 0;
    for (int k = 0; k < 3; ++k) {
        int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
        double pr, pi, qr, qi, mr, mi;
        cm(zr[3 + k1], zi[3 + k1], zr[6 + k2], zi[6 + k2], pr, pi);
        cm(zr[3 + k2], zi[3 + k2], zr[6 + k1], zi[6 + k1], qr, qi);
        cm(zr[k], zi[k], pr - qr, pi - qi, mr, mi);
        dr += mr; di += mi;
    }
    double ph = atan2(di, dr) / 3.0;
    double sn, cs;
    sincos(-ph, &sn, &cs);
    M3<T> m;
    for (int k = 0; k < 9; ++k) {
        m.re[k] = T(zr[k] * cs - zi[k] * sn);
        m.im[k] = T(zr[k] * sn + zi[k] * cs);
    }
    store_link<T, NC>(U, g.P, mu, sidx(g, site_of_lex(g, s)), m);
}

// Random gauge transformation (Sec. V.D): store G(x) (FP64 [V][3][3][2] in
// lexicographic site order) as 18 reals per site in the link layout, then
// U_mu(x) -> G(x) U_mu(x) G^dag(x + mu) for every link.
template <class T>
__global__ void __launch_bounds__(kThreads) k_store_gauge(Geo g, const double *__restrict__ Glex, T *Gs) {
    __shared__ __align__(16) double sm[kThreads * 18];
    const int s0 = blockIdx.x * kThreads;
    double tr, ti;
    const M3<T> m = staged_matrix<T>(Glex + 18ll * s0, sm, tr, ti);
    store_link<T, 18>(Gs, g.P, 0, sidx(g, site_of_lex(g, s0 + threadIdx.x)), m);
}

template <class T, int NC>
__global__ void k_gauge_links(Geo g, const T *__restrict__ Gs, T *U) {
    long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= 4ll * g.V) return;
    const int mu = (int)(l / g.V);
    const Pt x = site_of_index(g, (int)(l % g.V));
    const int i = sidx(g, x);
    const int iy = sidx(g, mv(g, x, mu, 1));
    M3<T> u = load_link<T, NC>(U, g.P, mu, i);
    u = m3_mul(load_link<T, 18>(Gs, g.P, 0, i), u);
    u = m3_mul_nd(u, load_link<T, 18>(Gs, g.P, 0, iy));
    store_link<T, NC>(U, g.P, mu, i, u);
}

// Z(3) projection of every link: reference label from arg Tr U, link -> exp(2 pi i n/3) I.
template <class T, int NC>
__global__ void k_project(Geo g, T *U, int8_t *ref) {
    long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= 4ll * g.V) return;
    const int mu = (int)(l / g.V);
    const int i = sidx(g, site_of_index(g, (int)(l % g.V)));
    M3<T> m = load_link<T, NC>(U, g.P, mu, i);
    int n = z3_label<T>(m.re[0] + m.re[4] + m.re[8], m.im[0] + m.im[4] + m.im[8]);
    double sn, cs;
    sincospi(2.0 * n / 3.0, &sn, &cs);
    M3<T> z;
    m3_zero(z);
    z.re[0] = z.re[4] = z.re[8] = T(cs);
    z.im[0] = z.im[4] = z.im[8] = T(sn);
    store_link<T, NC>(U, g.P, mu, i, z);
    ref[(long long)mu * g.P + i] = (int8_t)n;
}

}  // namespace

// ---------------------------------------------------------------------------
// Dispatch
// ---------------------------------------------------------------------------

static std::atomic<long long> g_launches{0};
void count_launches(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long launches() { return g_launches.load(std::memory_order_relaxed); }

#define VS_DISPATCH(prec, nc, KERNEL, ...)                                          \
    do {                                                                            \
        if ((prec) == 0 && (nc) == 18) { KERNEL<double, 18>__VA_ARGS__; }           \
        else if ((prec) == 1 && (nc) == 18) { KERNEL<float, 18>__VA_ARGS__; }       \
        else if ((prec) == 1 && (nc) == 12) { KERNEL<float, 12>__VA_ARGS__; }       \
        else return cudaErrorInvalidValue;                                          \
    } while (0)

cudaError_t launch_load_labels(int prec, int nc, const Geo &g, const int8_t *lab, void *U, int8_t *ref,
                               cudaStream_t st) {
    int b = std::min(nblocks(4ll * g.V), kTableGrid);
    if (prec == 0) k_load_labels<double, 18><<<b, kThreads, 0, st>>>(g, lab, (double *)U, ref);
    else if (nc == 18) k_load_labels<float, 18><<<b, kThreads, 0, st>>>(g, lab, (float *)U, ref);
    else k_load_labels<float, 12><<<b, kThreads, 0, st>>>(g, lab, (float *)U, ref);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_load_links(int prec, int nc, const Geo &g, const double *in, void *U, int8_t *ref,
                              cudaStream_t st) {
    const dim3 b(nblocks(g.V), 4);
    const bool staged = g.Qp != g.Q && g.Q % 2 && nc == 18;
    if (prec == 0 && staged) k_load_links<double, 18, true><<<b, kThreads, 0, st>>>(g, in, (double *)U, ref);
    else if (prec == 0) k_load_links<double, 18, false><<<b, kThreads, 0, st>>>(g, in, (double *)U, ref);
    else if (staged) k_load_links<float, 18, true><<<b, kThreads, 0, st>>>(g, in, (float *)U, ref);
    else if (nc == 18) k_load_links<float, 18, false><<<b, kThreads, 0, st>>>(g, in, (float *)U, ref);
    else k_load_links<float, 12, false><<<b, kThreads, 0, st>>>(g, in, (float *)U, ref);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_read_links(int prec, int nc, const Geo &g, const void *U, double *out, cudaStream_t st) {
    const dim3 b(nblocks(g.V), 4);
    if (prec == 0) k_read_links<double, 18><<<b, kThreads, 0, st>>>(g, (const double *)U, out);
    else if (nc == 18) k_read_links<float, 18><<<b, kThreads, 0, st>>>(g, (const float *)U, out);
    else k_read_links<float, 12><<<b, kThreads, 0, st>>>(g, (const float *)U, out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_count_nonfinite(int prec, int nc, const Geo &g, const void *U, unsigned long long *count,
                                   cudaStream_t st) {
    const int b = nblocks(4ll * g.V);
    if (prec == 0) k_count_nonfinite<double, 18><<<b, kThreads, 0, st>>>(g, (const double *)U, count);
    else if (nc == 18) k_count_nonfinite<float, 18><<<b, kThreads, 0, st>>>(g, (const float *)U, count);
    else k_count_nonfinite<float, 12><<<b, kThreads, 0, st>>>(g, (const float *)U, count);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_store_ref(const Geo &g, const int8_t *lab_lex, int8_t *ref, cudaStream_t st) {
    k_store_ref<<<nblocks(4ll * g.V), kThreads, 0, st>>>(g, lab_lex, ref);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_read_labels(const Geo &g, const int8_t *ref, int8_t *out, cudaStream_t st) {
    k_read_labels<<<nblocks(4ll * g.V), kThreads, 0, st>>>(g, ref, out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_current_labels(int prec, int nc, const Geo &g, const void *U, int8_t *out, cudaStream_t st) {
    const dim3 b(nblocks(g.V), 4);
    if (prec == 0) k_current_labels<double, 18><<<b, kThreads, 0, st>>>(g, (const double *)U, out);
    else if (nc == 18) k_current_labels<float, 18><<<b, kThreads, 0, st>>>(g, (const float *)U, out);
    else k_current_labels<float, 12><<<b, kThreads, 0, st>>>(g, (const float *)U, out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_centrifuge(int prec, int nc, const Geo &g, const int8_t *ref, double omega, uint64_t seed,
                              void *U, double *table, cudaStream_t st) {
    const int b = std::min(nblocks(g.V), kTableGrid);
    double2 *tab = reinterpret_cast<double2 *>(table);
    k_centrifuge_table<<<(kCtabN + 31) / 32, 32, 0, st>>>(omega, tab);
    if (prec == 0) k_centrifuge<double, 18><<<b, kThreads, 0, st>>>(g, ref, omega, seed, (double *)U, tab);
    else if (nc == 18) k_centrifuge<float, 18><<<b, kThreads, 0, st>>>(g, ref, omega, seed, (float *)U, tab);
    else k_centrifuge<float, 12><<<b, kThreads, 0, st>>>(g, ref, omega, seed, (float *)U, tab);
    count_launches(2);
    return cudaGetLastError();
}

// Blocks of a measurement kernel: per_sm for each SM, at most `most` (its partials), or a
// thread per site where `most` blocks suffice for that.
static int meas_blocks(const Geo &g, int per_sm, int most) {
    int dev = 0, n_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int all = nblocks(g.V, kMeasThreads);
    return all <= most ? all : std::min(n_sm * per_sm, most);
}

cudaError_t launch_action(int prec, int nc, const Geo &g, const void *U, double *partials, double *out,
                          cudaStream_t st) {
    int b = 0;
    const auto run = [&](auto kernel, auto *links) {
        b = meas_blocks(g, prec == 0 ? kActionFp64Blocks : kActionPerSM, kActionBlocks);
        kernel<<<b, kMeasThreads, 0, st>>>(g, links, partials);
    };
    if (prec == 0) run(k_action<double, 18>, (const double *)U);
    else if (nc == 18) run(k_action<float, 18>, (const float *)U);
    else run(k_action<float, 12>, (const float *)U);
    // <S>/beta = (1/V) sum_x (2/72) sum_{mu<nu} (3 - Re Tr P)
    k_sum_partials<<<1, 1024, 0, st>>>(partials, b, 2.0 / 72.0 / (double)g.V, out);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_observables(int prec, int nc, const Geo &g, const void *U, double *partials, double *out,
                               double *S_site, double *SR_site, double *q_site, cudaStream_t st) {
    int b = 0;
    const auto run = [&](auto kernel, auto *links) {
        b = meas_blocks(g, prec == 0 ? kMeasFp64PerSM : kObsPerSM, kObsBlocks);
        kernel<<<b, kMeasThreads, 0, st>>>(g, links, partials, S_site, SR_site, q_site);
    };
    if (prec == 0) run(k_observables<double, 18>, (const double *)U);
    else if (nc == 18) run(k_observables<float, 18>, (const float *)U);
    else run(k_observables<float, 12>, (const float *)U);
    k_sum_partials3<<<1, 1024, 0, st>>>(partials, b, 1.0 / (double)g.V, out);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_correlation(const double *a, const double *b, long long n, double *partials, double *out,
                               cudaStream_t st) {
    const int nb = (int)std::min<long long>(nblocks(n), kCorrGrid);
    k_correlation<<<nb, kThreads, 0, st>>>(a, b, n, partials);
    k_correlation_finish<<<1, 1024, 0, st>>>(partials, nb, out);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t preload_vortex_kernels() {
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, k_vortex_links<double, 18, false, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_vortex_links<double, 18, false, true>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_vortex_links<float, 18, false, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_vortex_links<float, 12, false, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_vortex_links<double, 18, true, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_vortex_links<double, 18, true, true>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_vortex_links<float, 18, true, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_vortex_links<float, 12, true, false>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_vortex_charges);
    return e;
}

// Up to this many sites an FP64 check takes a thread per link: a site's four atan2 in a row
// then last longer than the links' loads (us per check, per site / per link: 4^4 42.0 / 29.7,
// 12^3x24 67.1 / 55.3, 16^3x32 106.8 / 107.4, 24^3x48 403.6 / 458.0).
constexpr int kLinkSites = 65536;

template <class T, int NC, bool LINK = false>
static void vortex_links(const Geo &g, const void *U, const int8_t *ref, int8_t *dz, unsigned long long *counts,
                         unsigned long long *mbits, cudaStream_t st, const void *G) {
    const dim3 b(nblocks(g.V), LINK ? 4 : 1);
    if (G)
        k_vortex_links<T, NC, true, LINK><<<b, kThreads, 0, st>>>(g, (const T *)U, ref, dz, counts, mbits, (const T *)G);
    else
        k_vortex_links<T, NC, false, LINK><<<b, kThreads, 0, st>>>(g, (const T *)U, ref, dz, counts, mbits, nullptr);
}

cudaError_t launch_vortex(int prec, int nc, const Geo &g, const void *U, const int8_t *ref, int8_t *dz,
                          unsigned long long *counts, unsigned long long *mbits, cudaStream_t st,
                          const void *G) {
    if (prec == 0 && g.V <= kLinkSites) vortex_links<double, 18, true>(g, U, ref, dz, counts, mbits, st, G);
    else if (prec == 0) vortex_links<double, 18>(g, U, ref, dz, counts, mbits, st, G);
    else if (nc == 18) vortex_links<float, 18>(g, U, ref, dz, counts, mbits, st, G);
    else vortex_links<float, 12>(g, U, ref, dz, counts, mbits, st, G);
    k_vortex_charges<<<nblocks(g.V), kThreads, 0, st>>>(g, dz, counts);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_reunit(int prec, int nc, const Geo &g, void *U, const int8_t *ref, cudaStream_t st,
                          const void *G) {
    int b = nblocks(4ll * g.V);
    if (prec == 0) k_reunit<double, 18><<<b, kThreads, 0, st>>>(g, (double *)U, ref, (const double *)G);
    else if (nc == 18) k_reunit<float, 18><<<b, kThreads, 0, st>>>(g, (float *)U, ref, (const float *)G);
    else k_reunit<float, 12><<<b, kThreads, 0, st>>>(g, (float *)U, ref, (const float *)G);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_debug_expm(int prec, const double *X, int n, double *E, cudaStream_t st) {
    if (prec == 0) k_debug_expm<double><<<nblocks(n), kThreads, 0, st>>>(X, n, E);
    else k_debug_expm<float><<<nblocks(n), kThreads, 0, st>>>(X, n, E);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_haar(int prec, int nc, const Geo &g, uint64_t seed, void *U, cudaStream_t st) {
    int b = nblocks(4ll * g.V);
    if (prec == 0) k_haar<double, 18><<<b, kThreads, 0, st>>>(g, seed, (double *)U);
    else if (nc == 18) k_haar<float, 18><<<b, kThreads, 0, st>>>(g, seed, (float *)U);
    else k_haar<float, 12><<<b, kThreads, 0, st>>>(g, seed, (float *)U);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_aus_class(int prec, int nc, bool rect, int mu, const AusParams &p, cudaStream_t st) {
    if (prec == 0) return launch_aus_d18(rect, mu, p, st);
    if (nc == 18) return launch_aus_f18(rect, mu, p, st);
    return launch_aus_f12(rect, mu, p, st);
}

cudaError_t launch_gauge(int prec, int nc, const Geo &g, const double *G_lex, void *Gs, void *U,
                         cudaStream_t st) {
    if (prec == 0) {
        k_store_gauge<double><<<nblocks(g.V), kThreads, 0, st>>>(g, G_lex, (double *)Gs);
        k_gauge_links<double, 18><<<nblocks(4ll * g.V), kThreads, 0, st>>>(g, (const double *)Gs, (double *)U);
    } else {
        k_store_gauge<float><<<nblocks(g.V), kThreads, 0, st>>>(g, G_lex, (float *)Gs);
        if (nc == 18)
            k_gauge_links<float, 18><<<nblocks(4ll * g.V), kThreads, 0, st>>>(g, (const float *)Gs, (float *)U);
        else
            k_gauge_links<float, 12><<<nblocks(4ll * g.V), kThreads, 0, st>>>(g, (const float *)Gs, (float *)U);
    }
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_project(int prec, int nc, const Geo &g, void *U, int8_t *ref, cudaStream_t st) {
    int b = nblocks(4ll * g.V);
    if (prec == 0) k_project<double, 18><<<b, kThreads, 0, st>>>(g, (double *)U, ref);
    else if (nc == 18) k_project<float, 18><<<b, kThreads, 0, st>>>(g, (float *)U, ref);
    else k_project<float, 12><<<b, kThreads, 0, st>>>(g, (float *)U, ref);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace vs
