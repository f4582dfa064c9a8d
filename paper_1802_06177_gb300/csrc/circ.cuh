// Symmetric circulant transforms of short lines, y[d] = sum_m t[|d - m|] v[m] (t[k] = t[n - k]), the two factors
// of the separable hopping exponential [Suppl. Eq. (S2)], in FP64.
//
// The factor is given less the identity, which a value's own term adds exactly: exp(dtau t C) is close to the
// identity, every slice multiplies by the same coefficients, and the rounding of a diagonal of 1.1 would add up over the
// N L factors of a determinant.
//
// FP64 issue bounds every kernel that applies them (two FMAs per clock per SM, 65 cycles of latency), so the
// n^2 FMAs of the direct sum are folded by the symmetries of the line: reflection about site 0 splits v into
// even and odd halves, and for even n the map m -> n/2 - m splits each half again. A line of 12 then takes
// 38 FMAs and 40 additions instead of 144 FMAs, one of 16 takes 66 and 56 instead of 256. The length is a
// template parameter, so every index is a constant; with a runtime length each product sat behind its own
// test and its load of t (3-4 thousand cycles for a line of 4).
#pragma once

namespace slmc {
namespace circ {

constexpr int kMaxN = 32;
constexpr __host__ __device__ bool two_level(int n) { return n >= 4 && n % 2 == 0; }

// Block sizes: even half (plus, minus), odd half (plus, minus); one level: (even, 0, odd, 0).
struct Sizes {
    int p, m, q, r;
};
constexpr __host__ __device__ Sizes sizes(int n) {
    const int h = n / 2;
    if (!two_level(n)) return Sizes{h + 1, 0, (n - 1) / 2, 0};
    return Sizes{(h + 1) / 2 + (h % 2 == 0 ? 1 : 0), (h + 1) / 2, (h - 1) / 2 + (h % 2 == 0 ? 1 : 0), (h - 1) / 2};
}
constexpr __host__ __device__ int ncoef(int n) {
    return sizes(n).p * sizes(n).p + sizes(n).m * sizes(n).m + sizes(n).q * sizes(n).q + sizes(n).r * sizes(n).r;
}

// Coefficients of the folded transform of length n from tab (t[0..n-1] less the identity); by nt threads, thread tid.
__device__ inline void build(double* coef, const double* tab, int n, int tid, int nt) {
    const Sizes z = sizes(n);
    const int h = n / 2, n0 = z.p * z.p, n1 = n0 + z.m * z.m, n2 = n1 + z.q * z.q, n3 = n2 + z.r * z.r;
    const bool two = two_level(n);
    auto t = [&](int k) { return tab[((k % n) + n) % n]; };
    auto ce = [&](int d, int m) { return (m == 0 || 2 * m == n) ? t(d - m) : 0.5 * (t(d - m) + t(d + m)); };
    auto co = [&](int d, int m) { return 0.5 * (t(d - m) - t(d + m)); };
    for (int i = tid; i < n3; i += nt) {
        double v;
        if (i < n0) {
            const int d = i / z.p, m = i % z.p;
            v = (two && m < z.m) ? 0.5 * (ce(d, m) + ce(d, h - m)) : ce(d, m);
        } else if (i < n1) {
            const int d = (i - n0) / z.m, m = (i - n0) % z.m;
            v = 0.5 * (ce(d, m) - ce(d, h - m));
        } else if (i < n2) {
            const int d = (i - n1) / z.q + 1, m = (i - n1) % z.q + 1;
            v = (two && m <= z.r) ? 0.5 * (co(d, m) + co(d, h - m)) : co(d, m);
        } else {
            const int d = (i - n2) / z.r + 1, m = (i - n2) % z.r + 1;
            v = 0.5 * (co(d, m) - co(d, h - m));
        }
        coef[i] = v;
    }
}

// x 2^-k by integer operations (an FP64 multiplication would take the pipe that bounds the transforms). Infinities and
// NaN stay as they are; values below 2^(k - 1022) become zero.
template <int k>
__device__ __forceinline__ double scaled(double x) {
    if (k == 0) return x;
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    const bool tiny = e <= k;
    return __hiloint2double(tiny ? 0 : (e == 0x7ff ? hi : hi - (k << 20)), tiny ? 0 : __double2loint(x));
}

// y = c x plus the identity's part of the block: 2^-H x, but 2^-H0 x for the first K0 values and 2^-H1 x for the last K1.
template <int K, int H, int K0 = 0, int H0 = 0, int K1 = 0, int H1 = 0>
__device__ __forceinline__ void block(const double* __restrict__ c, const double (&x)[K > 0 ? K : 1],
                                      double (&y)[K > 0 ? K : 1]) {
#pragma unroll
    for (int d = 0; d < K; ++d)
        y[d] = fma(c[d * K], x[0], d < K0 ? scaled<H0>(x[d]) : (d >= K - K1 ? scaled<H1>(x[d]) : scaled<H>(x[d])));
#pragma unroll
    for (int m = 1; m < K; ++m)
#pragma unroll
        for (int d = 0; d < K; ++d) y[d] = fma(c[d * K + m], x[m], y[d]);
}

// v <- (folded transform of length n with coefficients c) v.
template <int n>
__device__ __forceinline__ void line(const double* __restrict__ c, double (&v)[n]) {
    constexpr Sizes z = sizes(n);
    constexpr int h = n / 2, hm = (n - 1) / 2;
    const double* cm = c + z.p * z.p;
    const double* cq = cm + z.m * z.m;
    const double* cr = cq + z.q * z.q;
    double e[h + 1], o[hm > 0 ? hm : 1];  // o[m - 1]: odd part of site m
    e[0] = v[0];
    if (n % 2 == 0) e[h] = v[h];
#pragma unroll
    for (int m = 1; m <= hm; ++m) {
        e[m] = v[m] + v[n - m];
        o[m - 1] = v[m] - v[n - m];
    }
    double s[h + 1], a[hm > 0 ? hm : 1];
    if constexpr (!two_level(n)) {
        // sites 0 and n / 2 are their own mirror images (weight 1), every other one shares a pair (1/2)
        block<h + 1, 1, 1, 0, n % 2 == 0 ? 1 : 0, 0>(c, e, s);
        if constexpr (hm > 0) block<hm, 1>(cq, o, a);
    } else {
        double ep[z.p], sp[z.p], em[z.m], sm[z.m];
#pragma unroll
        for (int m = 0; m < z.m; ++m) {
            ep[m] = e[m] + e[h - m];
            em[m] = e[m] - e[h - m];
        }
        if constexpr (z.p > z.m) ep[z.m] = e[h / 2];
        // the same weights halved again, but for the middle value, its own mirror image in the second fold
        block<z.p, 2, 1, 1, z.p - z.m, 1>(c, ep, sp);
        block<z.m, 2, 1, 1>(cm, em, sm);
#pragma unroll
        for (int d = 0; d < z.m; ++d) {
            s[d] = sp[d] + sm[d];
            s[h - d] = sp[d] - sm[d];
        }
        if constexpr (z.p > z.m) s[h / 2] = sp[z.m];
        if constexpr (z.q > 0) {
            double op[z.q], ap[z.q], om[z.r > 0 ? z.r : 1], am[z.r > 0 ? z.r : 1];
#pragma unroll
            for (int m = 1; m <= z.r; ++m) {
                op[m - 1] = o[m - 1] + o[h - m - 1];
                om[m - 1] = o[m - 1] - o[h - m - 1];
            }
            if constexpr (z.q > z.r) op[z.r] = o[h / 2 - 1];
            block<z.q, 2, 0, 0, z.q - z.r, 1>(cq, op, ap);
            if constexpr (z.r > 0) block<z.r, 2>(cr, om, am);
#pragma unroll
            for (int d = 1; d <= z.r; ++d) {
                a[d - 1] = ap[d - 1] + am[d - 1];
                a[h - d - 1] = ap[d - 1] - am[d - 1];
            }
            if constexpr (z.q > z.r) a[h / 2 - 1] = ap[z.r];
        }
    }
    v[0] = s[0];
    if (n % 2 == 0) v[h] = s[h];
#pragma unroll
    for (int d = 1; d <= hm; ++d) {
        v[d] = s[d] + a[d - 1];
        v[n - d] = s[d] - a[d - 1];
    }
}

// The line g[0], g[stride], ... in place, with optional input scales in_sc[m in_st] and output scales
// out_sc[d out_st] (times *mul if given).
template <int n>
__device__ __forceinline__ void apply(double* g, int stride, const double* __restrict__ c, const double* in_sc, int in_st,
                                      const double* out_sc, int out_st, const double* mul) {
    double v[n];
#pragma unroll
    for (int m = 0; m < n; ++m) v[m] = g[m * stride];
    if (in_sc)
#pragma unroll
        for (int m = 0; m < n; ++m) v[m] *= in_sc[m * in_st];
    line<n>(c, v);
    if (out_sc) {
        if (mul) {
            const double f = *mul;
#pragma unroll
            for (int m = 0; m < n; ++m) v[m] *= out_sc[m * out_st] * f;
        } else {
#pragma unroll
            for (int m = 0; m < n; ++m) v[m] *= out_sc[m * out_st];
        }
    }
#pragma unroll
    for (int m = 0; m < n; ++m) g[m * stride] = v[m];
}

// Length n <= LMAX at run time (one call site per kernel: every length is expanded there).
template <int LMAX>
__device__ __forceinline__ void apply_any(int n, double* g, int stride, const double* __restrict__ c, const double* in_sc,
                                          int in_st, const double* out_sc, int out_st,
                                          const double* mul = nullptr) {
#define SLMC_CIRC(k)                                                                             \
    case k:                                                                                      \
        if constexpr (k <= LMAX) apply<k>(g, stride, c, in_sc, in_st, out_sc, out_st, mul); \
        break;
    switch (n) {
        SLMC_CIRC(2) SLMC_CIRC(3) SLMC_CIRC(4) SLMC_CIRC(5) SLMC_CIRC(6) SLMC_CIRC(7) SLMC_CIRC(8) SLMC_CIRC(9)
        SLMC_CIRC(10) SLMC_CIRC(11) SLMC_CIRC(12) SLMC_CIRC(13) SLMC_CIRC(14) SLMC_CIRC(15) SLMC_CIRC(16)
        SLMC_CIRC(17) SLMC_CIRC(18) SLMC_CIRC(19) SLMC_CIRC(20) SLMC_CIRC(21) SLMC_CIRC(22) SLMC_CIRC(23)
        SLMC_CIRC(24) SLMC_CIRC(25) SLMC_CIRC(26) SLMC_CIRC(27) SLMC_CIRC(28) SLMC_CIRC(29) SLMC_CIRC(30)
        SLMC_CIRC(31) SLMC_CIRC(32)
    }
#undef SLMC_CIRC
}

}  // namespace circ
}  // namespace slmc
