// vs_split.cuh -- FP32 class updates with three warps per 32 links, for launches
// that leave the chip idle.
//
// A class launch of a small lattice is bound by one thread's serial chain: the
// six (nu, s) units of the one-pass staple sum, ~1100 instructions each, then the
// update (~800), at the ~3.7 cycles per instruction of a lone warp.  The units are
// independent, so here warp w of a block takes one direction nu of the same 32
// links; the partial sums meet in the first warp's registers through the warps'
// own ring columns in shared memory, and that warp updates the links.  Six warps,
// one per unit, were no faster (5.4 us against 5.5 at 1024 links per launch, 22.5
// against 17.7 at 32,768): launch and update dominate by then.
#pragma once

#include "vs_ape.cuh"

namespace vs {

template <int V> struct Int { static constexpr int value = V; };

constexpr int kSplit = 3, kSplitThreads = 32 * kSplit;   // warps per 32 links

// Staple sum of link (x, mu) and the link, complete in the first warp (returns
// true there).  Every thread of the block calls it.
template <int NC, bool RECT>
__device__ __forceinline__ bool staple_sum_split(const Geo &g, const float *U, int mu, const Pt &x,
                                                 float c0, float c1, float4 *shared, M3<float> &sig, M3<float> &Ux) {
    constexpr int BT = kSplitThreads;
    const LinkRing<NC, BT> R = ring_of<NC, BT>(shared, reinterpret_cast<float2 *>(shared + 6 * (NC / 4) * BT));
    const int w = threadIdx.x >> 5;
    const bool first = w == 0;
    const long long P = g.P;
    const int nu = (mu + 1 + w) & 3;
    const float *Umu = U + (long long)mu * NC * P, *Unu = U + (long long)nu * NC * P;
    Around A;
    A.i0 = sidx(g, x);
    A.dmm1 = RECT ? shift_delta(g, x, mu, -1) : 0;
    A.dmp1 = shift_delta(g, x, mu, 1);
    A.dmp2 = RECT ? shift_delta(g, x, mu, 2) : 0;
    around_nu(g, x, nu, RECT, A);
    M3<float> F, Lp;
    m3_zero(F);
    m3_zero(sig);
    dep_wait_launch();
    const auto fetch = [&](auto sign, auto entry, auto slot) {
        const float *b;
        int q;
        u_link<decltype(sign)::value, decltype(entry)::value>(A, Umu, Unu, b, q);
        ring_fetch<NC, decltype(slot)::value>(R, b, P, q);
    };
    if constexpr (RECT) {
        // entries 0-5 of the first unit
        fetch(Int<1>(), Int<0>(), Int<0>()); fetch(Int<1>(), Int<1>(), Int<1>()); fetch(Int<1>(), Int<2>(), Int<2>());
        fetch(Int<1>(), Int<3>(), Int<3>()); fetch(Int<1>(), Int<4>(), Int<4>()); fetch(Int<1>(), Int<5>(), Int<5>());
        const M3<float> Lm = m3_dag(load_link<float, NC, kLive>(U, P, mu, A.i0 + A.dmm1));
        fused_unit<NC, 1>(R, F, sig, c0, c1, Lm, Umu, Unu, Unu, P, A, A, true, first);
        fused_unit<NC, -1>(R, F, sig, c0, c1, Lm, Umu, Unu, Unu, P, A, A, true, first);
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        if (first) {
            Lp = ring_read<NC, false, 4>(R);     // U_mu(x + mu) and U_mu(x): the spare entries
            Ux = ring_read<NC, false, 5>(R);
        }
    } else {
        fetch(Int<1>(), Int<0>(), Int<0>()); fetch(Int<1>(), Int<1>(), Int<1>()); fetch(Int<1>(), Int<9>(), Int<2>());
        fetch(Int<-1>(), Int<0>(), Int<3>()); fetch(Int<-1>(), Int<1>(), Int<4>()); fetch(Int<-1>(), Int<9>(), Int<5>());
        if (first) Ux = load_link<float, NC, kLive>(U, P, mu, A.i0);
        plain_unit<NC, 1>(R, sig, Umu, Unu, P, A, true);
        plain_unit<NC, -1>(R, sig, Umu, Unu, P, A, true);
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    // the partial sums through the warps' own ring columns
    constexpr int NQ = RECT ? 9 : 5;
    if (!first) {
        float4 *col = shared + threadIdx.x;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int e = 2 * q, f = 2 * q + 1;
            const auto at = [&](int k) {
                return k < 9 ? make_float2(sig.re[k % 9], sig.im[k % 9]) : make_float2(F.re[k % 9], F.im[k % 9]);
            };
            const float2 a = at(e), b = at(f);
            col[q * BT] = make_float4(a.x, a.y, b.x, b.y);
        }
    }
    __syncthreads();
    if (!first) return false;
#pragma unroll
    for (int v = 1; v < kSplit; ++v) {
        const float4 *col = shared + threadIdx.x + 32 * v;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 a = col[q * BT];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = 2 * q + h;
                const float re = h ? a.z : a.x, im = h ? a.w : a.y;
                if (k < 9) { sig.re[k % 9] += re; sig.im[k % 9] += im; }
                else if (RECT) { F.re[k % 9] += re; F.im[k % 9] += im; }
            }
        }
    }
    if constexpr (RECT) m3_axpy(sig, c1, m3_mul_nd(F, Lp));
    else if (c0 != 1.0f) m3_scale(sig, c0);
    return true;
}

// Site and direction of this lane: colour class (direction `arg`), or with colour < 0
// every link, `arg` blocks per direction.  Links per launch are a multiple of 64 (a
// quarter of V), so every warp is full.
__device__ __forceinline__ Pt split_site(const Geo &g, int colour, int arg, int &mu) {
    const int lane = threadIdx.x & 31, b = blockIdx.x;
    if (colour >= 0) {
        mu = arg;
        return class_site(g, mu, colour, b * 32 + lane);
    }
    mu = b / arg;
    return site_of_index(g, (b - mu * arg) * 32 + lane);
}

template <int NC, bool RECT>
__global__ void __launch_bounds__(kSplitThreads, 4) k_subsweep_split(SubsweepParams a, int arg) {
    extern __shared__ float4 split_dyn[];
    const Geo &g = a.g;
    int mu;
    const Pt x = split_site(g, a.colour, arg, mu);
    M3<float> sig, Ux;
    if (!staple_sum_split<NC, RECT>(g, static_cast<const float *>(a.Usrc), mu, x, a.c0_f, a.c1_f, split_dyn, sig, Ux))
        return;
    Update<float> u;
    stout_store<float, NC>(a, mu, x, sidx(g, x), sig, Ux, u);
    count_update<float>(a.counters, u);
}

template <int NC, bool RECT>
__global__ void __launch_bounds__(kSplitThreads, 4) k_aus_split(AusParams a, int mu) {
    extern __shared__ float4 split_dyn[];
    const Geo &g = a.g;
    const Pt x = class_site(g, mu, a.colour, blockIdx.x * 32 + (threadIdx.x & 31));
    M3<float> sig, Ux;
    if (!staple_sum_split<NC, RECT>(g, static_cast<const float *>(a.U), mu, x, a.c0_f, a.c1_f, split_dyn, sig, Ux))
        return;
    Update<float> u;
    aus_finish<float, NC>(a, mu, x, sidx(g, x), sig, Ux, u);
    count_update<float>(a.counters, u);
}

template <int NC, bool RECT>
__global__ void __launch_bounds__(kSplitThreads, 4) k_ape_split(ApeParams a, int arg) {
    extern __shared__ float4 split_dyn[];
    const Geo &g = a.g;
    int mu;
    const Pt x = split_site(g, a.colour, arg, mu);
    M3<float> sig, Ux;
    if (!staple_sum_split<NC, RECT>(g, static_cast<const float *>(a.Usrc), mu, x, a.c0_f, a.c1_f, split_dyn, sig, Ux))
        return;
    Update<float> u;
    ape_finish<float, NC>(a, mu, x, sidx(g, x), sig, Ux, u);
    count_update<float>(a.counters, u);
}

template <int NC, bool RECT>
__global__ void __launch_bounds__(kSplitThreads, 4) k_flow_split(FlowParams a, int arg) {
    extern __shared__ float4 split_dyn[];
    const Geo &g = a.g;
    int mu;
    const Pt x = split_site(g, -1, arg, mu);
    M3<float> sig, u;
    if (!staple_sum_split<NC, RECT>(g, static_cast<const float *>(a.Usrc), mu, x, a.c0_f, a.c1_f, split_dyn, sig, u))
        return;
    bool used64 = false;
    flow_finish<float, NC>(a, mu, sidx(g, x), sig, u, used64);
    flow_count(a, used64);
}

// Up to this many links per launch three warps share 32 links.  The time depends on the
// row as well as on the links: a class is a run of Lx/4 sites per x-row, and the shorter
// the run, the more lines every load visits.  us per class launch with one warp / three,
// 18 reals:
//   over-improved    rows of 12      16             20             32
//     3072-5120      15.7 / 6.5                     12.0 / 7.8     9.6 / 5.8
//     8192-9216      16.1 / 9.8      10.9 / 6.8                    10.0 / 6.4
//     11,520-12,288  16.3 / 16.1     11.0 / 9.2     12.5 / 12.4    10.2 / 8.2
//     15,360-16,384  16.5 / 16.4     11.3 / 9.7     12.9 / 12.7
//     20,480-24,576  29.1 / 20.3     15.5 / 12.3    20.0 / 15.9    14.3 / 13.0
//     28,672-32,768                  16.1 / 14.3                   14.7 / 17.7
//   plaquette staples
//     8192-11,520    6.2 / 4.3       4.3 / 3.3      5.0 / 4.7      4.0 / 3.1
//     12,288         6.2 / 7.3       4.5 / 4.5                     4.1 / 4.1
// (12 reals: 28,672 links in rows of 16 15.9 / 17.0, otherwise alike.)  Two warps, one per
// sign, run two code paths at a time and lose to either (1024 links 6.5, 10,368 13.0,
// 24,576 16.3).
constexpr int kSplitMost = 28672, kSplitMostPlain = 12288;

inline bool split_launch(bool rect, long long links) { return links <= (rect ? kSplitMost : kSplitMostPlain); }

// The launch of a smoother's plaquette-staple (0) or over-improved (1) kernel for a
// colour class of direction mu, or for every link of p.n_threads sites (mu < 0).
template <int NC, class P>
cudaError_t launch_split(void (*const kernels[2])(P, int), bool rect, int mu, const P &p,
                         std::atomic<unsigned long long> &attr_set, cudaStream_t st) {
    constexpr int sm = ring6_smem_bytes<NC, kSplitThreads>();
    once_per_device(attr_set, [&] {
        for (int k = 0; k < 2; ++k)
            cudaFuncSetAttribute(kernels[k], cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    });
    const int b = p.n_threads / 32;
    return launch_dependent(kernels[rect], mu < 0 ? 4 * b : b, kSplitThreads, (size_t)sm, st, p, mu < 0 ? b : mu);
}

}  // namespace vs
