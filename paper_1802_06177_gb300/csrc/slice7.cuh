// Fixed-point slicing of FP64 values into seven 7-bit digits that BF16 holds exactly, for the
// FP64-accurate products on the tensor cores (T update of the UDT chain, trailing updates of the
// blocked QR). A row or column with largest magnitude in [2^e, 2^(e+1)) is written as
//   v = 2^(e - 6) sum_{s=0..6} d_s 2^(-7 s) + r,   |d_0| <= 128, |d_s| <= 64 (s >= 1), |r| <= 2^(e - 49),
// with integer arithmetic only (the FP64 pipe is the scarce unit). Products of two such operands
// summed per level a + b are exact in FP32 accumulators while the level's sum of absolute terms
// stays below 2^24 (after Ozaki, Ogita, Oishi, Rump 2012).
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace slmc {
namespace s7 {

constexpr int kS = 7;  // slices per operand

__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// |v| as an ordered integer (the bit pattern without the sign), and its warp maximum.
__device__ __forceinline__ long long abs_bits(double v) { return __double_as_longlong(v) & 0x7fffffffffffffffll; }

__device__ __forceinline__ long long warp_max_bits(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Power of two of the largest |v| from its bit pattern (0 for a zero row or column).
__device__ __forceinline__ int exponent_of_bits(long long m) {
    return m == 0 ? 0 : (int)((m >> 52) & 0x7ff) - 1023;
}

// The seven slices of v in units of 2^(e - 6 - 42), with integer arithmetic only (the FP64 pipe
// is the scarce unit, and the integer-to-float conversions share its issue): v is rounded once to
// n = round(v 2^(48 - e)) (|n| <= 2^49, half away from zero) and n is written in balanced base-128 digits
// d_6..d_1 in [-64, 63] and d_0 = the rest, |d_0| <= 128, so v ~ 2^(e - 6) sum_s d_s 2^(-7 s). Adding 64 at every
// place below the top makes the digits plain bit fields (plus 64); each is placed in the significand of
// 1.5 2^23 and freed by one exact FP32 subtraction. The results are small integers as FP32, exact in BF16 (the
// upper half of their bits).
__device__ __forceinline__ void slice7(double v, int e, float (&q)[kS]) {
    const long long bits = __double_as_longlong(v);
    const int ex = (int)((bits >> 52) & 0x7ff);
    long long n = 0;
    const int r = 1027 + e - ex;  // right shift of the 53-bit significand; >= 4 whenever |v| < 2^(e + 1)
    if (ex != 0 && r < 63) {
        const long long m = (bits & 0xfffffffffffffll) | 0x10000000000000ll;
        n = r > 0 ? (m + (1ll << (r - 1))) >> r : m;
        if (bits < 0) n = -n;
    }
    constexpr long long kBias = 64ll * (1 + 128 * (1 + 128 * (1 + 128 * (1 + 128ll * (1 + 128ll)))));
    n += kBias;
#pragma unroll
    for (int s = kS - 1; s >= 1; --s)
        q[s] = __int_as_float(0x4B400000 | ((int)(n >> (7 * (kS - 1 - s))) & 127)) - 12582976.f;
    q[0] = __int_as_float(0x4B400000 + (int)(n >> (7 * (kS - 1)))) - 12582912.f;
}

// BF16 bits of an exact small integer, and of two adjacent ones.
__device__ __forceinline__ __nv_bfloat16 bf16_of(float q) {
    return __ushort_as_bfloat16((unsigned short)(__float_as_uint(q) >> 16));
}
__device__ __forceinline__ uint32_t bf16x2_of(float q0, float q1) {
    return __byte_perm(__float_as_uint(q0), __float_as_uint(q1), 0x7632);
}

// (hi 2^28 + lo) 2^k rounded once to FP64 (to nearest, ties to even), assembled with integer operations: the two
// conversions, the FMA and the scaling of an FP64 combination take 64 issue cycles of the FP64 pipe per warp, the bound of
// the epilogues that combine level sums. |hi| < 2^50, |lo| < 2^60.
__device__ __forceinline__ double combine(long long hi, long long lo, int k) {
    unsigned long long l = (unsigned long long)hi << 28;
    const unsigned long long sum = l + (unsigned long long)lo;
    long long h = (hi >> 36) + (lo >> 63) + (sum < l ? 1 : 0);
    l = sum;
    const bool neg = h < 0;
    if (neg) {
        l = 0ull - l;
        h = ~h + (l == 0ull ? 1 : 0);
    }
    const int up = h == 0 ? 0 : 64 - __clzll(h);  // bits above the low word (at most 15)
    unsigned long long m = l;
    uint32_t sticky = 0u;
    int nb;
    if (up) {
        sticky = (uint32_t)l & ((1u << up) - 1u);
        m = (l >> up) | ((unsigned long long)h << (64 - up));
        nb = 64 + up;
    } else {
        if (l == 0ull) return 0.0;
        const int z = __clzll((long long)l);
        m = l << z;
        nb = 64 - z;
    }
    const uint32_t frac = (uint32_t)m & 0x7ffu;
    unsigned long long mant = m >> 11;
    if (frac > 0x400u || (frac == 0x400u && (sticky || (mant & 1ull)))) ++mant;
    const int E = nb - 1 + k + 1023;
    if (E < 1 || E > 2046)  // out of the normal range: the FP64 operations round as they did
        return fma(__ll2double_rn(hi), 268435456.0, __ll2double_rn(lo)) * pow2d(k);
    const long long r = ((long long)(E - 1) << 52) + (long long)mant;
    return __longlong_as_double(neg ? r | (long long)0x8000000000000000ull : r);
}

}  // namespace s7
}  // namespace slmc
