// FP64 arithmetic and storage (18 reals per link).
#include <algorithm>

#include "vs_rows.cuh"
#include "vs_sweep_inst.cuh"
namespace vs {

// Plaquette staples at and above this many links per launch take a thread per link
// (k_subsweep): the update after the short staple sum, shared by a row's lanes, costs
// the row kernel 15 % more FP64 instructions (98,304 links: 338 us against 344 for a
// thread per link; 165,888: 563 against 517).
constexpr int kRowsMost = 131072;

// The links of a launch over blocks of 42 links (US = 1), 21 (2) and 7 (6).  A
// layer of one block per SM takes kLayer us of the FP64 pipe; the whole layers go
// to the first kind, what is left to whichever kind needs least.  Measured (us per
// class launch, over-improved / standard staples; before: one thread per link,
// 240 / 60 per started 38,912 links' half):
//   links       64      1024    3456    10368    32768     262144
//   before      241/60  483/120 485/121 485/121  484/121   3342/803
//   US = 1      94/30   97/31   98/32   170/49   491/135   3364/900
//   US = 2      55/21   57/23   94/31   182/58   472/140   3479/1013
//   US = 6      26/14   27/14   74/36   173/72   505/203   3919/1556
//   this rule   26/14   27/14   76/32   185/49   427/119   3303/797
template <bool RECT>
static void launch_rows(int mu, const SubsweepParams &p, cudaStream_t st) {
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const double layer[3] = {RECT ? 80.0 : 21.4, RECT ? 41.9 : 12.2, RECT ? 15.9 : 6.3};   // US = 1, 2, 6
    const auto layers = [&](int links, int us) { return (links + n_sm * row_links(us) - 1) / (n_sm * row_links(us)); };
    int n_whole = p.n_threads / (n_sm * row_links(1)) * n_sm;
    const int rest = p.n_threads - n_whole * row_links(1);
    const double c1 = layer[0], c2 = layer[1] * layers(rest, 2), c6 = layer[2] * layers(rest, 6);
    if (c1 <= c2 && c1 <= c6) n_whole += (rest + row_links(1) - 1) / row_links(1);
    const int left = std::max(0, p.n_threads - n_whole * row_links(1));
    if (c2 < c6) k_subsweep_rows<RECT, 2><<<n_whole + (left + row_links(2) - 1) / row_links(2), kRowThreads, 0, st>>>(
        p, mu, n_whole);
    else k_subsweep_rows<RECT, 6><<<n_whole + (left + row_links(6) - 1) / row_links(6), kRowThreads, 0, st>>>(
        p, mu, n_whole);
    count_launches(1);
}

cudaError_t launch_subsweep_d18(bool rect, int mu, const SubsweepParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    if (rect) {
        launch_rows<true>(mu, p, st);
    } else if (p.n_threads < kRowsMost) {
        launch_rows<false>(mu, p, st);
    } else {
        const int b = (p.n_threads + VS_SUBSWEEP_THREADS - 1) / VS_SUBSWEEP_THREADS;
        switch (mu) {
            case 0: k_subsweep<0><<<b, VS_SUBSWEEP_THREADS, 0, st>>>(p); break;
            case 1: k_subsweep<1><<<b, VS_SUBSWEEP_THREADS, 0, st>>>(p); break;
            case 2: k_subsweep<2><<<b, VS_SUBSWEEP_THREADS, 0, st>>>(p); break;
            default: k_subsweep<3><<<b, VS_SUBSWEEP_THREADS, 0, st>>>(p); break;
        }
        count_launches(1);
    }
    return cudaGetLastError();
}
cudaError_t launch_aus_d18(bool rect, int mu, const AusParams &p, cudaStream_t st) {
    return launch_aus_tpl<double, 18>(rect, mu, p, st);
}
}  // namespace vs
