// vs_sweep_inst.cuh -- instantiates the colour-class update kernel for one
// (precision, storage) pair.  Included by vs_sweep_f18.cu, vs_sweep_f12.cu and
// vs_sweep_d18.cu so the heavy instantiations compile in parallel.
#pragma once

#include "vs_internal.h"
#include "vs_split.cuh"

namespace vs {

// FP64 re-decision of the candidates the FP32 class launch just made left to it.
template <int NC, bool RECT>
void launch_redecide(int mu, const SubsweepParams &p, cudaStream_t st) {
    switch (mu) {
        case 0: k_redecide<NC, RECT, 0><<<16, 32, 0, st>>>(p); break;
        case 1: k_redecide<NC, RECT, 1><<<16, 32, 0, st>>>(p); break;
        case 2: k_redecide<NC, RECT, 2><<<16, 32, 0, st>>>(p); break;
        default: k_redecide<NC, RECT, 3><<<16, 32, 0, st>>>(p); break;
    }
    count_launches(1);
}

// FP32 stout: a colour class of direction mu, or every link (mu < 0: simultaneous
// sweeps; the re-decision list holds links of one direction, so with it each direction
// is a launch of its own, as it is on large lattices).
template <int NC>
cudaError_t launch_subsweep_tpl(bool rect, int mu, const SubsweepParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    if (mu < 0 && (p.defer_idx || !all_launch(rect, p.n_threads))) {
        cudaError_t e = cudaSuccess;
        for (int d = 0; e == cudaSuccess && d < 4; ++d) e = launch_subsweep_tpl<NC>(rect, d, p, st);
        return e;
    }
    cudaError_t e;
    if ((mu < 0 || p.colour >= 0) && split_launch(rect, mu < 0 ? 4ll * p.n_threads : p.n_threads)) {
        static void (*const kernels[2])(SubsweepParams, int) = {k_subsweep_split<NC, false>, k_subsweep_split<NC, true>};
        static std::atomic<unsigned long long> set{0};
        e = launch_split<NC>(kernels, rect, mu, p, set, st);
    } else if (mu < 0) {
        static void (*const kernels[2])(SubsweepParams) = {k_subsweep_all<NC, false>, k_subsweep_all<NC, true>};
        static std::atomic<unsigned long long> set{0};
        e = launch_all<NC>(kernels, rect, p, set, st);
    } else {
        static void (*const kernels[2][4])(SubsweepParams) = {
            {k_subsweep_pring<NC, 0>, k_subsweep_pring<NC, 1>, k_subsweep_pring<NC, 2>, k_subsweep_pring<NC, 3>},
            {k_subsweep_fused<NC, 0>, k_subsweep_fused<NC, 1>, k_subsweep_fused<NC, 2>, k_subsweep_fused<NC, 3>}};
        static std::atomic<unsigned long long> set[2] = {{0}, {0}};
        e = launch_ring<NC>(kernels[rect], mu, p, p.crowded ? 0 : kRingPerSM[rect], set[rect], st);
    }
    if (e == cudaSuccess && p.defer_idx) {
        if (rect) launch_redecide<NC, true>(mu, p, st);
        else launch_redecide<NC, false>(mu, p, st);
    }
    return e == cudaSuccess ? cudaGetLastError() : e;
}

template <class T, int NC>
cudaError_t launch_aus_tpl(bool rect, int mu, const AusParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    if constexpr (sizeof(T) == 8) {
        static void (*const kernels[2][4])(AusParams) = {{k_aus<false, 0>, k_aus<false, 1>, k_aus<false, 2>, k_aus<false, 3>},
                                                         {k_aus<true, 0>, k_aus<true, 1>, k_aus<true, 2>, k_aus<true, 3>}};
        return launch_links(kernels[rect][mu], p, st);
    } else if (split_launch(rect, p.n_threads)) {
        static void (*const kernels[2])(AusParams, int) = {k_aus_split<NC, false>, k_aus_split<NC, true>};
        static std::atomic<unsigned long long> set{0};
        return launch_split<NC>(kernels, rect, mu, p, set, st);
    } else {
        static void (*const kernels[2][4])(AusParams) = {
            {k_aus_pring<NC, 0>, k_aus_pring<NC, 1>, k_aus_pring<NC, 2>, k_aus_pring<NC, 3>},
            {k_aus_ring<NC, 0>, k_aus_ring<NC, 1>, k_aus_ring<NC, 2>, k_aus_ring<NC, 3>}};
        static std::atomic<unsigned long long> set[2] = {{0}, {0}};
        return launch_ring<NC>(kernels[rect], mu, p, p.crowded ? 0 : kRingPerSM[rect], set[rect], st);
    }
}

}  // namespace vs
