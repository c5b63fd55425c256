// vs_rows.cuh -- the FP64 stout class update, three lanes (one per matrix row)
// and up to six units (nu, s) of lanes per link.
//
// Every path of the staple sum is a product A B C ..., and row r of the product
// needs row r of A only.  So a lane carries row r of every chain
// (row-times-matrix products, 36 FMAs each, no communication) and the full
// products of the FP64 path split over three lanes for nothing: same FMAs per
// link, a third of the registers (a chain holds 6 reals, not 18), three times
// the lanes.  On GB300 a warp's FP64 instruction takes its SM sub-partition's
// pipe for 64 cycles, whatever its active lanes: a class launch lasts as long as
// the longest queue of warp instructions on one of the 608 sub-partitions.  With
// a thread per link that was 240 us for one warp however small the lattice; here
// it is a third of it, and where the lattice leaves sub-partitions idle the six
// (nu, s) units of a link also go to two or six lanes of their own.
#pragma once

#include <algorithm>

#include "vs_stout.cuh"

namespace vs {

struct Row {      // a row of a 3x3 matrix
    double re[3], im[3];
};

// A link as the right factor of a row product: entry (k, j) of it, or of its
// adjoint, is at p[k rs + j cs], the imaginary part with the sign bit flipped
// by m.  Both orientations are the same code, so lanes may differ in s.
struct RowLink {
    const double2 *p;
    int rs, cs;
    unsigned m;
};

__device__ __forceinline__ RowLink row_link(const double *base, int i, bool dag) {
    RowLink L;
    L.p = blk_double2(base, i);
    L.rs = dag ? 16 : 48;
    L.cs = dag ? 48 : 16;
    L.m = dag ? 0x80000000u : 0u;
    return L;
}

__device__ __forceinline__ double2 row_entry(const RowLink &L, int k, int j) {
    double2 v = load_vec<kLive>(L.p + k * L.rs + j * L.cs);
    v.y = __hiloint2double(__double2hiint(v.y) ^ (int)L.m, __double2loint(v.y));
    return v;
}

__device__ __forceinline__ Row row_of(const RowLink &L, int r) {
    Row x;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double2 v = row_entry(L, r, j);
        x.re[j] = v.x;
        x.im[j] = v.y;
    }
    return x;
}

// acc += x L
__device__ __forceinline__ void row_madd(Row &acc, const Row &x, const RowLink &L) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double2 b = row_entry(L, k, j);
            acc.re[j] = fma(x.re[k], b.x, acc.re[j]);
            acc.re[j] = fma(-x.im[k], b.y, acc.re[j]);
            acc.im[j] = fma(x.re[k], b.y, acc.im[j]);
            acc.im[j] = fma(x.im[k], b.x, acc.im[j]);
        }
}

__device__ __forceinline__ Row row_mul(const Row &x, const RowLink &L) {
    Row y = {{0, 0, 0}, {0, 0, 0}};
    row_madd(y, x, L);
    return y;
}

// Sites x + a nu + b mu around a link, for the unit's direction nu and sign s.
struct RowUnit {
    int i0, dm[4];          // position of x; shifts along mu by -1, 0, 1, 2
    int f0, f1, s1, s2;     // shifts along nu: the sites whose nu-link is one and two steps out, and s, 2s
};

// The units u = u0, u0 + du, ... (UNITS of them) of link (x, mu) for row r added
// to the rows of the sums sig and F of the one-pass form
//   Sigma = c1 F U_mu^dag(x+mu) + sum [c1 U_mu^dag(x-mu) G H B + c0 A B + c1 A T0 T1 T2] C
// (without rectangles sig = sum A B C, unscaled).
template <bool RECT, int UNITS>
__device__ __forceinline__ void row_units(const Geo &g, const double *U, const Pt &x, int i0, int mu,
                                          int u0, int du, int r, double c0, double c1, Row &sig, Row &F) {
    RowUnit S;
    S.i0 = i0;
    S.dm[0] = RECT ? shift_delta(g, x, mu, -1) : 0;
    S.dm[1] = 0;
    S.dm[2] = shift_delta(g, x, mu, 1);
    S.dm[3] = RECT ? shift_delta(g, x, mu, 2) : 0;
    const long long plane = 18 * g.P;
    const double *Um = U + mu * plane;
    Row lm;
    if constexpr (RECT) lm = row_of(row_link(Um, i0 + S.dm[0], true), r);
#pragma unroll 1
    for (int n = 0; n < UNITS; ++n) {
        const int u = u0 + n * du;
        const int nu = (mu + 1 + (u >> 1)) & 3;
        const bool neg = u & 1;
        S.s1 = shift_delta(g, x, nu, neg ? -1 : 1);
        S.f0 = neg ? S.s1 : 0;
        const double *Un = U + nu * plane;
        const Row a = row_of(row_link(Un, i0 + S.f0, neg), r);
        const RowLink B = row_link(Um, i0 + S.s1, false);
        const RowLink C = row_link(Un, i0 + S.f0 + S.dm[2], !neg);
        Row K = row_mul(a, B);
        if constexpr (RECT) {
            S.s2 = shift_delta(g, x, nu, neg ? -2 : 2);
            S.f1 = neg ? S.s2 : S.s1;
            Row W = row_mul(lm, row_link(Un, i0 + S.f0 + S.dm[0], neg));
            W = row_mul(W, row_link(Um, i0 + S.s1 + S.dm[0], false));
            W = row_mul(W, B);
            row_madd(F, row_mul(K, row_link(Um, i0 + S.s1 + S.dm[2], false)),
                     row_link(Un, i0 + S.f0 + S.dm[3], !neg));
            Row T = row_mul(a, row_link(Un, i0 + S.f1, neg));
            T = row_mul(T, row_link(Um, i0 + S.s2, false));
            row_madd(W, T, row_link(Un, i0 + S.f1 + S.dm[2], !neg));
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                K.re[j] = fma(c1, W.re[j], c0 * K.re[j]);
                K.im[j] = fma(c1, W.im[j], c0 * K.im[j]);
            }
        }
        row_madd(sig, K, C);
    }
}

// The six reals of a row (component c: entry c / 2, real or imaginary part c % 2)
// spread over the US lanes of a row: lane u holds and computes components u,
// u + US, ...  A warp instruction costs the FP64 pipe the same whatever its
// active lanes, so after the staple sum the lanes share the update instead of
// leaving it to one of them.
template <int US>
struct Part {
    double v[6 / US];
};

template <int US>
__device__ __forceinline__ int part_comp(int n, int u) { return US == 1 ? n : n * US + u; }

// Shared memory of a block, [..][link].
template <int US, int LPB>
struct RowShared {
    double part[3][US == 1 ? 12 : 6 * US][LPB];   // partial rows of the lanes, then whole rows
    double om[18][LPB];            // Omega
    double hf[15][LPB];            // H (diagonal, upper entries) and the exponential's coefficients
    double2 un[9][LPB];            // the candidate
    bool keep[LPB];
};

// Sum over a row's lanes of their partial rows: this lane's components of it.
template <int US, int LPB>
__device__ __forceinline__ Part<US> part_sum(const Row &x, double (*buf)[LPB], int u, int l, bool on) {
    Part<US> y;
    if constexpr (US == 1) {
#pragma unroll
        for (int c = 0; c < 6; ++c) y.v[c] = c & 1 ? x.im[c >> 1] : x.re[c >> 1];
    } else {
        __syncthreads();
        if (on)
#pragma unroll
            for (int c = 0; c < 6; ++c) buf[u * 6 + c][l] = c & 1 ? x.im[c >> 1] : x.re[c >> 1];
        __syncthreads();
#pragma unroll
        for (int n = 0; n < 6 / US; ++n) {
            const int c = part_comp<US>(n, u);
            double s = buf[c][l];
#pragma unroll
            for (int k = 1; k < US; ++k) s += buf[6 * k + c][l];
            y.v[n] = s;
        }
    }
    return y;
}

// The whole row from its lanes' components.
template <int US, int LPB>
__device__ __forceinline__ Row part_gather(const Part<US> &x, double (*buf)[LPB], int u, int l, bool on) {
    if constexpr (US > 1) {
        __syncthreads();
        if (on)
#pragma unroll
            for (int n = 0; n < 6 / US; ++n) buf[part_comp<US>(n, u)][l] = x.v[n];
        __syncthreads();
    }
    Row y;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        const double v = US > 1 ? buf[c][l] : x.v[US > 1 ? 0 : c];
        if (c & 1) y.im[c >> 1] = v;
        else y.re[c >> 1] = v;
    }
    return y;
}

// Components of x L.
template <int US>
__device__ __forceinline__ Part<US> part_mul(const Row &x, const RowLink &L, int u) {
    Part<US> y;
#pragma unroll
    for (int n = 0; n < 6 / US; ++n) {
        const int c = part_comp<US>(n, u), j = c >> 1;
        double s = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const double2 b = row_entry(L, k, j);
            s = fma(x.re[k], c & 1 ? b.y : b.x, s);
            s = fma(x.im[k], c & 1 ? b.x : -b.y, s);
        }
        y.v[n] = s;
    }
    return y;
}

// Coefficient f_which of exp(iH) = f0 + f1 H + f2 H^2 by the series of ch_exp_coeffs
// (H by its diagonal and upper entries): three operations per term where all three
// coefficients take five.
__device__ __forceinline__ void exp_coefficient(const double h[9], int which, double &re, double &im) {
    const double a01 = h[3] * h[3] + h[4] * h[4], a02 = h[5] * h[5] + h[6] * h[6], a12 = h[7] * h[7] + h[8] * h[8];
    const double tau = 0.5 * (h[0] * h[0] + h[1] * h[1] + h[2] * h[2]) + a01 + a02 + a12;
    const double pr = h[3] * h[7] - h[4] * h[8], pi = h[3] * h[8] + h[4] * h[7];
    const double delta = h[0] * h[1] * h[2] + 2.0 * (pr * h[5] + pi * h[6]) - h[0] * a12 - h[1] * a02 - h[2] * a01;
    const double r4 = 4.0 * tau * tau;
    double sr = 0, si = 0, cm = 0, c = 0, cp = 1, w = 1, bound = 1;   // c_{n-1}, c_n, c_{n+1} at n = 1; 1 / n!
    const auto pick = [&] { return which == 0 ? cm : which == 1 ? cp : c; };
    const auto next = [&] {
        const double v = fma(tau, c, delta * cm);
        cm = c;
        c = cp;
        cp = v;
    };
#pragma unroll
    for (int g4 = 0; g4 < 12; ++g4) {
        const int n = 4 * g4 + 1;
        w *= 1.0 / n;
        si = fma(w, pick(), si);                              // i^n = i, -1, -i, 1
        next();
        w *= 1.0 / (n + 1);
        sr = fma(-w, pick(), sr);
        next();
        w *= 1.0 / (n + 2);
        si = fma(-w, pick(), si);
        next();
        w *= 1.0 / (n + 3);
        sr = fma(w, pick(), sr);
        next();
        bound *= r4 * (1.0 / ((double)n * (n + 1) * (n + 2) * (n + 3)));
        if (bound < Tol<double>::eps()) break;
    }
    re = which == 0 ? fma(delta, sr, 1.0) : sr;
    im = which == 0 ? delta * si : si;
}

// Update of LPB links t0 .. t0 + LPB - 1 of a class launch by one block: blocks of
// four warps (one per SM sub-partition; three warps leave one idle), LPB =
// 128 / (3 US) links of 3 US lanes each, thread (r US + u) LPB + link.
constexpr int kRowThreads = 128;
__host__ __device__ constexpr int row_links(int US) { return kRowThreads / (3 * US); }

template <bool RECT, int US>
__device__ __forceinline__ void rows_block(const SubsweepParams &a, int mu, int t0, int t1, void *shared) {
    constexpr int LPB = row_links(US);
    RowShared<US, LPB> &sh = *static_cast<RowShared<US, LPB> *>(shared);
    const Geo &g = a.g;
    const int part = threadIdx.x / LPB, l = threadIdx.x % LPB;
    const int r = min(part / US, 2), u = part % US;
    const int t = t0 + l;
    const bool work = part < 3 * US && t < t1;
    const bool own = work && u == 0;                  // one lane per row of a link
    const double *Us = static_cast<const double *>(a.Usrc);
    double(*buf)[LPB] = sh.part[r];
    Pt x = {0, 0, 0, 0};
    int i = 0;
    Row sig = {{0, 0, 0}, {0, 0, 0}}, F = sig;
    if (work) {
        if (a.colour >= 0)
            x = class_site(g, mu, a.colour, t);
        else
            x = dir_site(g, mu, t);
        i = sidx(g, x);
    }
    dep_wait_launch();
    if (work) {
        if constexpr (US == 1) {
            // the forward units, then the backward ones on their own: the sum that
            // two lanes per row form, bit for bit, so that a launch can mix both
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                row_units<RECT, 3>(g, Us, x, i, mu, h, 2, r, a.c0, a.c1, sig, F);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    if (h == 0) {
                        buf[j][l] = sig.re[j]; buf[3 + j][l] = sig.im[j];
                        buf[6 + j][l] = F.re[j]; buf[9 + j][l] = F.im[j];
                        sig.re[j] = sig.im[j] = F.re[j] = F.im[j] = 0;
                    } else {
                        sig.re[j] += buf[j][l]; sig.im[j] += buf[3 + j][l];
                        F.re[j] += buf[6 + j][l]; F.im[j] += buf[9 + j][l];
                    }
                }
            }
        } else {
            // two lanes: the signs; six: one unit each
            row_units<RECT, 6 / US>(g, Us, x, i, mu, u, US, r, a.c0, a.c1, sig, F);
        }
    }
    // From here on idle lanes compute on the link at position 0 and write
    // nothing, so that every barrier sees the whole block.
    const double *Umu = Us + (long long)mu * 18 * g.P;
    Part<US> ps = part_sum<US, LPB>(sig, buf, u, l, work);
    if constexpr (RECT) {
        const Row Fs = part_gather<US, LPB>(part_sum<US, LPB>(F, buf, u, l, work), buf, u, l, work);
        const Part<US> t1 = part_mul<US>(Fs, row_link(Umu, i + shift_delta(g, x, mu, 1), true), u);
#pragma unroll
        for (int n = 0; n < 6 / US; ++n) ps.v[n] = fma(a.c1, t1.v[n], ps.v[n]);
    } else {
#pragma unroll
        for (int n = 0; n < 6 / US; ++n) ps.v[n] *= a.c0;
    }
    {   // row r of Omega = Sigma U^dag
        const Part<US> om = part_mul<US>(part_gather<US, LPB>(ps, buf, u, l, work), row_link(Umu, i, true), u);
        if (work)
#pragma unroll
            for (int n = 0; n < 6 / US; ++n) sh.om[6 * r + part_comp<US>(n, u)][l] = om.v[n];
    }
    __syncthreads();
    const double third = 1.0 / 3.0, hr2 = 0.5 * a.rho;
    // H as in stout_H: component k of its diagonal (0-2) and upper entries (3-8)
    const auto h_comp = [&](int k) {
        if (k < 3) {
            const double d = sh.om[8 * k + 1][l], d1 = sh.om[k == 0 ? 9 : 1][l], d2 = sh.om[k == 2 ? 9 : 17][l];
            return a.rho * ((2.0 * d - d1 - d2) * third);
        }
        const int q = (k - 3) >> 1;                           // (0,1), (0,2), (1,2): entries 1, 2, 5 and 3, 6, 7
        const int up = q == 0 ? 1 : q == 1 ? 2 : 5, dn = q == 0 ? 3 : q == 1 ? 6 : 7;
        return k & 1 ? hr2 * (sh.om[2 * up + 1][l] + sh.om[2 * dn + 1][l])
                     : -hr2 * (sh.om[2 * up][l] - sh.om[2 * dn][l]);
    };
    if constexpr (US == 6) {
        // one of the 18 lanes per component, then each row sums one coefficient
        if (work && part < 9) sh.hf[part][l] = h_comp(part);
        __syncthreads();
        if (own) {
            double h[9], re, im;
#pragma unroll
            for (int k = 0; k < 9; ++k) h[k] = sh.hf[k][l];
            exp_coefficient(h, r, re, im);
            sh.hf[9 + 2 * r][l] = re;
            sh.hf[10 + 2 * r][l] = im;
        }
    } else if (r == 0 && own) {
        // once per link, not once per row
        double h[9], f[6];
#pragma unroll
        for (int k = 0; k < 9; ++k) h[k] = h_comp(k);
        ch_exp_coeffs<double, 12>(h[0], h[1], h[2], h[3], h[4], h[5], h[6], h[7], h[8], 1e300, f);
#pragma unroll
        for (int k = 0; k < 9; ++k) sh.hf[k][l] = h[k];
#pragma unroll
        for (int k = 0; k < 6; ++k) sh.hf[9 + k][l] = f[k];
    }
    __syncthreads();
    // row r of exp(iH) = f0 + f1 H + f2 H^2: with y = f1 e_r + f2 H_r, the row is f0 e_r + y H
    Part<US> un;
    {
        const double h0 = sh.hf[0][l], h1 = sh.hf[1][l], h2 = sh.hf[2][l], ar = sh.hf[3][l], ai = sh.hf[4][l], br = sh.hf[5][l],
                     bi = sh.hf[6][l], cr = sh.hf[7][l], ci = sh.hf[8][l];
        const double Hr[9] = {h0, ar, br, ar, h1, cr, br, cr, h2};
        const double Hi[9] = {0.0, ai, bi, -ai, 0.0, ci, -bi, -ci, 0.0};
        const double f2r = sh.hf[13][l], f2i = sh.hf[14][l];
        const auto entry = [&](const double m[9], int k) {   // entry (r, k) of a matrix in registers
            const double c0 = r == 0 ? m[0] : r == 1 ? m[3] : m[6], c1 = r == 0 ? m[1] : r == 1 ? m[4] : m[7],
                         c2 = r == 0 ? m[2] : r == 1 ? m[5] : m[8];
            return k == 0 ? c0 : k == 1 ? c1 : c2;
        };
        Row y;
        if constexpr (US == 6) {
            Part<US> yp;
            const int k = u >> 1;
            const double xr = entry(Hr, k), xi = entry(Hi, k);
            yp.v[0] = u & 1 ? f2r * xi + f2i * xr : f2r * xr - f2i * xi;
            if (k == r) yp.v[0] += sh.hf[11 + (u & 1)][l];
            y = part_gather<US, LPB>(yp, buf, u, l, work);
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double xr = entry(Hr, k), xi = entry(Hi, k);
                y.re[k] = f2r * xr - f2i * xi;
                y.im[k] = f2r * xi + f2i * xr;
                if (k == r) { y.re[k] += sh.hf[11][l]; y.im[k] += sh.hf[12][l]; }
            }
        }
        Part<US> m;
#pragma unroll
        for (int n = 0; n < 6 / US; ++n) {
            const int c = part_comp<US>(n, u), j = c >> 1;
            double s = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double hr = j == 0 ? Hr[3 * k] : j == 1 ? Hr[3 * k + 1] : Hr[3 * k + 2];
                const double hi = j == 0 ? Hi[3 * k] : j == 1 ? Hi[3 * k + 1] : Hi[3 * k + 2];
                s = fma(y.re[k], c & 1 ? hi : hr, s);
                s = fma(y.im[k], c & 1 ? hr : -hi, s);
            }
            if (j == r) s += c & 1 ? sh.hf[10][l] : sh.hf[9][l];
            m.v[n] = s;
        }
        un = part_mul<US>(part_gather<US, LPB>(m, buf, u, l, work), row_link(Umu, i, false), u);
    }
    if (work)
#pragma unroll
        for (int n = 0; n < 6 / US; ++n) {
            const int c = part_comp<US>(n, u);
            double2 &e = sh.un[3 * r + (c >> 1)][l];
            if (c & 1) e.y = un.v[n];
            else e.x = un.v[n];
        }
    __syncthreads();
    {
        Update<double> up;
        if (own && r == 0) {
            M3<double> Un;
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                const double2 v = sh.un[e][l];
                Un.re[e] = v.x;
                Un.im[e] = v.y;
            }
            double tr_re, tr_im;
            vp_trace<double>(static_cast<const double *>(a.G), g.P, i, a.G ? sidx(g, mv(g, x, mu, 1)) : i, Un, tr_re,
                             tr_im);
            vp_decide<double>(a.vp, a.counters != nullptr, (int)a.ref[(long long)mu * g.P + i], tr_re, tr_im, up);
            sh.keep[l] = !up.reject;
        }
        count_update<double>(a.counters, up);
    }
    __syncthreads();
    if (own) {
        // a rejected link keeps its value: nothing to write in place (annealed),
        // the old link into the destination when that is another buffer
        double2 *dst = const_cast<double2 *>(blk_double2(static_cast<double *>(a.U) + (long long)mu * 18 * g.P, i));
#pragma unroll
        for (int e = 3 * r; e < 3 * r + 3; ++e) {
            if (sh.keep[l]) dst[16 * e] = sh.un[e][l];
            else if (a.U != a.Usrc) dst[16 * e] = load_vec<kLive>(blk_double2(Umu, i) + 16 * e);
        }
    }
}

// Class launch (or every link of direction mu, colour < 0).  WHOLE: blocks below
// n_whole take 42 links with a lane per row, the rest of the links go to blocks of
// 21 with two lanes per row, so that the last, partial layer of blocks over the SMs
// is short.  Otherwise blocks of 7 links with six lanes per row (n_whole = 0).
template <bool RECT, bool WHOLE>
__global__ void __launch_bounds__(kRowThreads, 3) k_subsweep_rows(SubsweepParams a, int mu, int n_whole) {
    constexpr int US = WHOLE ? 2 : 6;
    constexpr size_t s1 = sizeof(RowShared<1, row_links(1)>), s2 = sizeof(RowShared<US, row_links(US)>);
    __shared__ __align__(16) unsigned char shared[WHOLE && s1 > s2 ? s1 : s2];
    const int b = blockIdx.x;
    if constexpr (WHOLE)
        if (b < n_whole) {
            rows_block<RECT, 1>(a, mu, b * row_links(1), a.n_threads, shared);
            return;
        }
    rows_block<RECT, US>(a, mu, n_whole * row_links(1) + (b - n_whole) * row_links(US), a.n_threads, shared);
}

// A launch of n links as blocks of 42 links (one lane per row), 21 (two) and 7 (six), or a
// thread per link.  A layer of one block per SM takes layer[] us of the FP64 pipe: whole
// layers go to the first kind and what is left to the cheaper of the first two (they sum in
// the same order, so that equal links of a launch come out bit-identical), unless blocks of
// 7 are cheaper for all of it.  Measured (us per class launch, over-improved / plaquette
// staples; a thread per link in blocks of 128, the last row):
//   links       64      1024    3456    10368    18432    32768    36864    57600    262144
//   one lane    94/30   97/31   98/32   170/49   253/73   491/135  495/137  773/213  3364/900
//   two         55/21   57/23   94/31   182/58            472/140                    3479/1013
//   six         26/14   27/14   74/36   173/72            505/203                    3919/1556
//   thread      247/62  247/62  247/62  247/62   247/62   482/117  483/118  726/176      /793
// A thread per link takes layers of 19,456 links and wins where the last one is nearly
// full: thread_layers() compares the two by their layers' times and a launch's own (before,
// the row kernel took every over-improved launch and every plaquette launch below 131,072
// links: 38,400 links 533/149 where a thread per link takes 485/120).
template <bool RECT>
struct RowPlan {
    static constexpr double layer[3] = {RECT ? 80.0 : 21.4, RECT ? 41.9 : 12.2, RECT ? 15.9 : 6.3};
    int n_whole;       // blocks of 42 links
    int rest;          // links left to blocks of 21, or all of them to blocks of 7
    bool sixes;
    double us;
};

template <bool RECT>
inline RowPlan<RECT> row_plan(int n, int n_sm) {
    using R = RowPlan<RECT>;
    const auto blocks = [](int links, int us) { return (links + row_links(us) - 1) / row_links(us); };
    const auto layers = [&](int links, int us) { return (blocks(links, us) + n_sm - 1) / n_sm; };
    R r;
    const int whole = n / (n_sm * row_links(1));   // whole layers
    r.n_whole = whole * n_sm;
    r.rest = n - r.n_whole * row_links(1);
    const double c2 = R::layer[1] * layers(r.rest, 2), c6 = R::layer[2] * layers(n, 6);
    r.us = R::layer[0] * whole + std::min(R::layer[0], c2);
    r.sixes = c6 < r.us;
    if (r.sixes) {
        r.us = c6;
        r.n_whole = 0;
        r.rest = n;
    } else if (R::layer[0] <= c2) {
        r.n_whole += blocks(r.rest, 1);
        r.rest = std::max(0, n - r.n_whole * row_links(1));
    }
    return r;
}

// Whether a thread per link is faster: 237.2 us per layer and 9.6 per launch over-improved,
// 56.0 and 5.8 with plaquette staples, against the row kernel's plan and 12 or 8 us.
template <bool RECT>
inline bool thread_layers(int n, int n_sm) {
    const int layers = (n + VS_SUBSWEEP_THREADS * n_sm - 1) / (VS_SUBSWEEP_THREADS * n_sm);
    const double thread = (RECT ? 237.2 : 56.0) * layers + (RECT ? 9.6 : 5.8);
    return thread < row_plan<RECT>(n, n_sm).us + (RECT ? 12.0 : 8.0);
}

}  // namespace vs
