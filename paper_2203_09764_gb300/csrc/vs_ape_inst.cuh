// vs_ape_inst.cuh -- launches of the APE / UCP and Runge-Kutta kernels for one
// (precision, storage) pair.  Included by vs_ape_f18.cu, vs_ape_f12.cu and
// vs_ape_d18.cu.
#pragma once

#include "vs_split.cuh"

namespace vs {

// annealed classes and simultaneous sweeps alike
template <class T, int NC>
cudaError_t launch_ape_tpl(bool rect, int mu, const ApeParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    if constexpr (sizeof(T) == 8) {
        static void (*const kernels[2][4])(ApeParams) = {{k_ape<false, 0>, k_ape<false, 1>, k_ape<false, 2>, k_ape<false, 3>},
                                                         {k_ape<true, 0>, k_ape<true, 1>, k_ape<true, 2>, k_ape<true, 3>}};
        return launch_links(kernels[rect][mu], p, st);
    } else if (split_launch(rect, p.n_threads)) {
        static void (*const kernels[2])(ApeParams, int) = {k_ape_split<NC, false>, k_ape_split<NC, true>};
        static std::atomic<unsigned long long> set{0};
        return launch_split<NC>(kernels, rect, mu, p, set, st);
    } else {
        static void (*const kernels[2][4])(ApeParams) = {
            {k_ape_ring<NC, false, 0>, k_ape_ring<NC, false, 1>, k_ape_ring<NC, false, 2>, k_ape_ring<NC, false, 3>},
            {k_ape_ring<NC, true, 0>, k_ape_ring<NC, true, 1>, k_ape_ring<NC, true, 2>, k_ape_ring<NC, true, 3>}};
        static std::atomic<unsigned long long> set[2] = {{0}, {0}};
        return launch_ring(kernels[rect], mu, p, ring6_smem_bytes<NC>(), set[rect], st);
    }
}

template <class T, int NC>
cudaError_t launch_flow_tpl(bool rect, int mu, const FlowParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    if constexpr (sizeof(T) == 8) {
        static void (*const kernels[2][4])(FlowParams) = {
            {k_flow_stage<false, 0>, k_flow_stage<false, 1>, k_flow_stage<false, 2>, k_flow_stage<false, 3>},
            {k_flow_stage<true, 0>, k_flow_stage<true, 1>, k_flow_stage<true, 2>, k_flow_stage<true, 3>}};
        return launch_links(kernels[rect][mu], p, st);
    } else if (split_launch(rect, p.n_threads)) {
        static void (*const kernels[2])(FlowParams, int) = {k_flow_split<NC, false>, k_flow_split<NC, true>};
        static std::atomic<unsigned long long> set{0};
        return launch_split<NC>(kernels, rect, mu, p, set, st);
    } else {
        static void (*const kernels[2][4])(FlowParams) = {
            {k_flow_stage_ring<NC, false, 0>, k_flow_stage_ring<NC, false, 1>, k_flow_stage_ring<NC, false, 2>,
             k_flow_stage_ring<NC, false, 3>},
            {k_flow_stage_ring<NC, true, 0>, k_flow_stage_ring<NC, true, 1>, k_flow_stage_ring<NC, true, 2>,
             k_flow_stage_ring<NC, true, 3>}};
        static std::atomic<unsigned long long> set[2] = {{0}, {0}};
        return launch_ring(kernels[rect], mu, p, ring6_smem_bytes<NC>(), set[rect], st);
    }
}

}  // namespace vs
