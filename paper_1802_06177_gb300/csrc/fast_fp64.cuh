// Short FP64 square root and quotient for latency-bound chains (a warp runs one FP64 instruction per 64 cycles: the
// library's root and quotient take about 660 and 390 cycles, these 390 and 325).
#pragma once

#include <stdint.h>

namespace slmc {

// Square root and quotient of normal numbers of moderate exponent (others take the library's) by Newton steps from an
// FP32 estimate of the significand: Goldschmidt's coupled iteration for the root with a final residual correction,
// Newton's for the reciprocal and Markstein's correction of the quotient. Six and five FP64 instructions; results
// are within one unit in the last place of the correctly rounded ones, for any FP32 estimate within the documented two
// units of rsqrtf (tests/test_fast_fp64.py).
__device__ __forceinline__ double fast_sqrt(double a) {
    const int hi = __double2hiint(a), ex = (hi >> 20) - 1023;
    if (ex < -900 || ex > 900) return sqrt(a);
    const int k = ex >> 1;  // a = m 4^k, m in [1, 4)
    const double m = __hiloint2double(hi - (k << 21), __double2loint(a));
    const float mf = __int_as_float(((hi - (k << 21) - 0x38000000) << 3) | ((uint32_t)__double2loint(a) >> 29));
    const float y = rsqrtf(mf);
    const double yd = __hiloint2double((int)(__float_as_uint(y) >> 3) + 0x38000000, (int)(__float_as_uint(y) << 29));
    double g = m * yd, h = __hiloint2double(__double2hiint(yd) - 0x00100000, __double2loint(yd));
    const double r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    h = fma(h, r, h);
    g = fma(fma(-g, g, m), h, g);
    return __hiloint2double(__double2hiint(g) + (k << 20), __double2loint(g));
}
__device__ __forceinline__ double fast_div(double n, double d) {
    const int hd = __double2hiint(d), ex = ((hd >> 20) & 0x7ff) - 1023;
    const int en = ((__double2hiint(n) >> 20) & 0x7ff) - 1023;
    if (ex < -400 || ex > 400 || en < -400 || en > 400) return n / d;
    const int sh = ex << 20;  // d = s 2^ex, |s| in [1, 2)
    const double sd = __hiloint2double(hd - sh, __double2loint(d));
    const float sf = __int_as_float((int)((hd & 0x80000000u) | ((((hd & 0x7fffffff) - sh - 0x38000000) << 3) |
                                                                ((uint32_t)__double2loint(d) >> 29))));
    const float y = __frcp_rn(sf);
    const uint32_t yu = __float_as_uint(y) & 0x7fffffffu;
    double yd = __hiloint2double((int)((yu >> 3) + 0x38000000u) | (hd & (int)0x80000000), (int)(yu << 29));
    yd = fma(fma(-sd, yd, 1.0), yd, yd);
    double q = n * yd;
    q = fma(fma(-sd, q, n), yd, q);
    return __hiloint2double(__double2hiint(q) - (q == 0.0 ? 0 : sh), __double2loint(q));
}

}  // namespace slmc
