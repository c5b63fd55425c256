// FP64 arithmetic and storage (18 reals per link).
#include <algorithm>

#include "vs_rows.cuh"
#include "vs_sweep_inst.cuh"
namespace vs {

template <bool RECT>
static cudaError_t launch_stout(int mu, const SubsweepParams &p, cudaStream_t st) {
    int dev = 0, n_sm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (thread_layers<RECT>(p.n_threads, n_sm)) {
        static void (*const kernels[4])(SubsweepParams) = {k_subsweep<RECT, 0>, k_subsweep<RECT, 1>, k_subsweep<RECT, 2>,
                                                           k_subsweep<RECT, 3>};
        return launch_links(kernels[mu], p, st);
    }
    const RowPlan<RECT> r = row_plan<RECT>(p.n_threads, n_sm);
    const int US = r.sixes ? 6 : 2, b = r.n_whole + (r.rest + row_links(US) - 1) / row_links(US);
    // more than a block per SM: blocks of the next launch would double up with this
    // one's on some SMs' FP64 pipes (2048 links: 53 us instead of 39)
    if (r.sixes && b <= n_sm) return launch_dependent(k_subsweep_rows<RECT, false>, b, kRowThreads, 0, st, p, mu, 0);
    if (r.sixes) k_subsweep_rows<RECT, false><<<b, kRowThreads, 0, st>>>(p, mu, 0);
    else k_subsweep_rows<RECT, true><<<b, kRowThreads, 0, st>>>(p, mu, r.n_whole);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_subsweep_d18(bool rect, int mu, const SubsweepParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    cudaError_t e = cudaSuccess;   // mu < 0: a simultaneous sweep
    for (int d = std::max(mu, 0); e == cudaSuccess && d <= (mu < 0 ? 3 : mu); ++d)
        e = rect ? launch_stout<true>(d, p, st) : launch_stout<false>(d, p, st);
    return e;
}
cudaError_t launch_aus_d18(bool rect, int mu, const AusParams &p, cudaStream_t st) {
    return launch_aus_tpl<double, 18>(rect, mu, p, st);
}
}  // namespace vs
