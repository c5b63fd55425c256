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

// The links of a launch over blocks of 42 links (one lane per row), 21 (two) and 7
// (six).  A layer of one block per SM takes layer[] us of the FP64 pipe: whole layers
// go to the first kind and what is left to the cheaper of the first two (they sum in
// the same order, so that equal links of a launch come out bit-identical), unless
// blocks of 7 are cheaper for all of it.  Measured (us per class launch, over-improved
// / plaquette staples; before: a thread per link in blocks of 256):
//   links              64      1024    3456    10368    32768     262144
//   before             241/60  483/120 485/121 485/121  484/121   3342/803
//   one lane           94/30   97/31   98/32   170/49   491/135   3364/900
//   two                55/21   57/23   94/31   182/58   472/140   3479/1013
//   six                26/14   27/14   74/36   173/72   505/203   3919/1556
template <bool RECT>
static void launch_rows(int mu, const SubsweepParams &p, cudaStream_t st) {
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    constexpr double layer[3] = {RECT ? 80.0 : 21.4, RECT ? 41.9 : 12.2, RECT ? 15.9 : 6.3};
    const auto blocks = [](int links, int us) { return (links + row_links(us) - 1) / row_links(us); };
    const auto layers = [&](int links, int us) { return (blocks(links, us) + n_sm - 1) / n_sm; };
    const int whole = p.n_threads / (n_sm * row_links(1));            // whole layers
    int n_whole = whole * n_sm;
    const int rest = p.n_threads - n_whole * row_links(1);
    const double c2 = layer[1] * layers(rest, 2), mixed = layer[0] * whole + std::min(layer[0], c2);
    if (layer[2] * layers(p.n_threads, 6) < mixed) {
        const int b = blocks(p.n_threads, 6);
        // more than a block per SM: blocks of the next launch would double up with
        // this one's on some SMs' FP64 pipes (2048 links: 53 us instead of 39)
        if (b <= n_sm) {
            launch_dependent(k_subsweep_rows<RECT, false>, b, kRowThreads, 0, st, p, mu, 0);
            return;
        }
        k_subsweep_rows<RECT, false><<<b, kRowThreads, 0, st>>>(p, mu, 0);
    } else {
        if (layer[0] <= c2) n_whole += blocks(rest, 1);
        const int left = std::max(0, p.n_threads - n_whole * row_links(1));
        k_subsweep_rows<RECT, true><<<n_whole + blocks(left, 2), kRowThreads, 0, st>>>(p, mu, n_whole);
    }
    count_launches(1);
}

cudaError_t launch_subsweep_d18(bool rect, int mu, const SubsweepParams &p, cudaStream_t st) {
    if (p.n_threads <= 0) return cudaSuccess;
    if (mu < 0) {   // simultaneous sweep
        cudaError_t e = cudaSuccess;
        for (int d = 0; e == cudaSuccess && d < 4; ++d) e = launch_subsweep_d18(rect, d, p, st);
        return e;
    }
    if (rect) {
        launch_rows<true>(mu, p, st);
    } else if (p.n_threads < kRowsMost) {
        launch_rows<false>(mu, p, st);
    } else {
        static void (*const kernels[4])(SubsweepParams) = {k_subsweep<0>, k_subsweep<1>, k_subsweep<2>, k_subsweep<3>};
        return launch_links(kernels[mu], p, st);
    }
    return cudaGetLastError();
}
cudaError_t launch_aus_d18(bool rect, int mu, const AusParams &p, cudaStream_t st) {
    return launch_aus_tpl<double, 18>(rect, mu, p, st);
}
}  // namespace vs
