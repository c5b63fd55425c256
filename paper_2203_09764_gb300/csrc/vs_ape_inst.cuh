// vs_ape_inst.cuh -- launches of the APE / UCP and Runge-Kutta kernels for one
// (precision, storage) pair.  Included by vs_ape_f18.cu, vs_ape_f12.cu and
// vs_ape_d18.cu.
#pragma once

#include "vs_split.cuh"

namespace vs {

// Whether a colour class with plaquette staples takes plain loads (k_ape) instead of the
// link ring.  Where a run of class sites has an odd number of positions, every 16-byte
// chunk run ends in half a 32-byte sector: the ring's copies pass the L1 cache by and fetch
// the other half again, plain loads find it there.  With four blocks per SM (58,369 to
// 77,824 links) all of a launch is resident and that decides; in narrow rows it decides
// elsewhere, too.  us per class launch, ring / plain loads, 18 reals: rows of 4, 33,792
// links 13.9 / 12.4, 64,000 24.5 / 19.4, 139,968 46.9 / 40.2; rows of 12, 60,480 20.3 /
// 16.7, 96,000 25.7 / 28.1, 139,968 39.0 / 37.0; rows of 36, 64,512 15.7 / 14.7, 96,768
// 20.8 / 25.4; rows of 28 (runs of seven in lines of eight), 64,512 14.8 / 15.6.  12 reals:
// rows of 4, 109,440 27.4 / 23.2; rows of 12, 67,584 16.2 / 14.5, 110,592 23.5 / 22.6; rows
// of 36, 64,512 13.4 / 14.4.
inline bool plain_ape(int nc, int Qp, int links) {
    int dev = 0, n_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int per_sm = ((links + VS_SUBSWEEP_THREADS - 1) / VS_SUBSWEEP_THREADS + n_sm - 1) / n_sm;
    if (Qp % 2 == 0 || per_sm < (Qp == 1 ? 2 : 4)) return false;
    if (Qp == 1) return true;
    if (nc == 12) return Qp == 3;
    return per_sm == 4 || (Qp == 3 && per_sm % 4 == 0);
}

// A colour class of direction mu, or every link (mu < 0: simultaneous sweeps).
template <class T, int NC>
cudaError_t launch_ape_tpl(bool rect, int mu, const ApeParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    if constexpr (sizeof(T) == 8) {
        static void (*const kernels[2][4])(ApeParams) = {
            {k_ape<T, NC, false, 0>, k_ape<T, NC, false, 1>, k_ape<T, NC, false, 2>, k_ape<T, NC, false, 3>},
            {k_ape<T, NC, true, 0>, k_ape<T, NC, true, 1>, k_ape<T, NC, true, 2>, k_ape<T, NC, true, 3>}};
        cudaError_t e = cudaSuccess;
        for (int d = mu < 0 ? 0 : mu; e == cudaSuccess && d <= (mu < 0 ? 3 : mu); ++d)
            e = launch_links(kernels[rect][d], p, st);
        return e;
    } else if (mu < 0 && !all_launch(rect, p.n_threads)) {
        cudaError_t e = cudaSuccess;
        for (int d = 0; e == cudaSuccess && d < 4; ++d) e = launch_ape_tpl<T, NC>(rect, d, p, st);
        return e;
    } else if ((mu < 0 || p.colour >= 0) && split_launch(rect, mu < 0 ? 4ll * p.n_threads : p.n_threads)) {
        static void (*const kernels[2])(ApeParams, int) = {k_ape_split<NC, false>, k_ape_split<NC, true>};
        static std::atomic<unsigned long long> set{0};
        return launch_split<NC>(kernels, rect, mu, p, set, st);
    } else if (mu < 0) {
        static void (*const kernels[2])(ApeParams) = {k_ape_all<NC, false>, k_ape_all<NC, true>};
        static std::atomic<unsigned long long> set{0};
        return launch_all<NC>(kernels, rect, p, set, st);
    } else if (!rect && p.colour >= 0 && plain_ape(NC, p.g.Qp, p.n_threads)) {
        static void (*const kernels[4])(ApeParams) = {k_ape<T, NC, false, 0>, k_ape<T, NC, false, 1>, k_ape<T, NC, false, 2>,
                                                      k_ape<T, NC, false, 3>};
        return launch_links(kernels[mu], p, st);
    } else {
        static void (*const kernels[2][4])(ApeParams) = {
            {k_ape_ring<NC, false, 0>, k_ape_ring<NC, false, 1>, k_ape_ring<NC, false, 2>, k_ape_ring<NC, false, 3>},
            {k_ape_ring<NC, true, 0>, k_ape_ring<NC, true, 1>, k_ape_ring<NC, true, 2>, k_ape_ring<NC, true, 3>}};
        static std::atomic<unsigned long long> set[2] = {{0}, {0}};
        return launch_ring<NC>(kernels[rect], mu, p, kRingPerSM[rect], set[rect], st);
    }
}

// One stage, every direction.
template <class T, int NC>
cudaError_t launch_flow_tpl(bool rect, const FlowParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    if constexpr (sizeof(T) == 8) {
        static void (*const kernels[2][4])(FlowParams) = {
            {k_flow_stage<false, 0>, k_flow_stage<false, 1>, k_flow_stage<false, 2>, k_flow_stage<false, 3>},
            {k_flow_stage<true, 0>, k_flow_stage<true, 1>, k_flow_stage<true, 2>, k_flow_stage<true, 3>}};
        for (int mu = 0; mu < 4; ++mu) {
            const cudaError_t e = launch_links(kernels[rect][mu], p, st);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    } else if (split_launch(rect, 4ll * p.n_threads)) {
        static void (*const kernels[2])(FlowParams, int) = {k_flow_split<NC, false>, k_flow_split<NC, true>};
        static std::atomic<unsigned long long> set{0};
        return launch_split<NC>(kernels, rect, -1, p, set, st);
    } else {
        static void (*const all[2])(FlowParams) = {k_flow_stage_ring<NC, false, -1>, k_flow_stage_ring<NC, true, -1>};
        static void (*const each[4])(FlowParams) = {k_flow_stage_ring<NC, true, 0>, k_flow_stage_ring<NC, true, 1>,
                                                    k_flow_stage_ring<NC, true, 2>, k_flow_stage_ring<NC, true, 3>};
        static std::atomic<unsigned long long> set[2] = {{0}, {0}};
        if (all_launch(rect, p.n_threads)) return launch_all<NC>(all, rect, p, set[0], st);
        cudaError_t e = cudaSuccess;
        for (int d = 0; e == cudaSuccess && d < 4; ++d)
            e = launch_ring<NC>(each, d, p, 0, set[1], st);
        return e;
    }
}

}  // namespace vs
