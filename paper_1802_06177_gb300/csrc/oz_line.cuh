// Transforms of short lines by a symmetric circulant factor, FP64-accurate, on the warp-level tensor
// instruction (mma.sync, BF16): the slices of the FP64 mode and of the DQMC chains.
// Also the rank-16 updates of the DQMC moves (rank_update).
//
// The transforms are FP64-issue bound (one warp instruction per 16-19 cycles per SM; 6.5 to 8 per value and pass even
// when folded, circ.cuh), and a line of at most 16 values is one K step of an MMA whose operands never leave the
// registers. Lines of up to 16 values: 16 of them (the same line of 16 columns) are the rows of A, cut per row into
// eight 7-bit digits against the row's power of two (as slice7.cuh with one digit more: 56 bits, so the slicing
// error is 2^-56 of the row's largest value, below the FP64 sum's own rounding); the factor's digits, less the
// identity (build), are B, laid out in fragment order once per CTA. The 36 products a + b <= 7 of a tile are summed per
// level in FP32, exactly (at most 41 thousand per index of K <= 16), combined in two 64-bit integers and rounded once
// with integer operations: about 50 integer and FP32 instructions per value and pass, no FP64. tcgen05 would need the
// digits in shared memory and the sums back from tensor memory for 36 instructions of K = 16.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "slmc_internal.cuh"

namespace slmc {
namespace oz {

constexpr int kD = 8;         // digits per operand
constexpr int kMaxLine = 16;  // one K step

__host__ __device__ constexpr int ntiles(int n) { return (n + 7) / 8; }
// bytes of the fragments of a factor of length n: [ntiles][kD][32 lanes] pairs of registers
__host__ __device__ constexpr int frag_bytes(int n) { return ntiles(n) * kD * 32 * 8; }

// The eight digits of v in units of 2^(e - 6 - 7 s), as small integers in FP32 (see slice7.cuh): v is rounded to
// n 2^(e - 55) (half away from zero) in 32-bit words -- the variable 64-bit shifts and the conversions were most of
// this function -- and the balanced digits of n are bit fields of n plus 64 at every place below the top.
// Returns n with its sign.
__device__ __forceinline__ long long digits(double v, int e, float (&q)[kD]) {
    const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
    const int ex = (int)((h >> 20) & 0x7ffu);
    const uint32_t mh = ex ? (h & 0xfffffu) | 0x100000u : 0u;  // a subnormal counts as zero
    // 2 n before rounding: significand 2^4 shifted right by r >= 0
    const int r = min(1023 + e - ex, 63);
    const uint32_t Mh = __funnelshift_l(ex ? l : 0u, mh, 4), Ml = (ex ? l : 0u) << 4;
    const uint32_t H = r >= 32 ? 0u : Mh, L = r >= 32 ? Mh : Ml;
    const uint32_t yh = H >> (r & 31), yl = __funnelshift_r(L, H, r & 31);
    long long n = (long long)((((unsigned long long)yh << 32) | yl) + 1ull) >> 1;
    const long long sg = (long long)((int)h >> 31);
    constexpr long long kBias = 64ll * (1 + 128 * (1 + 128 * (1 + 128 * (1 + 128ll * (1 + 128ll * (1 + 128ll))))));
    const long long ns = (n ^ sg) - sg;
    n = ns + kBias;
    const uint32_t nl = (uint32_t)n;
    const int nh = (int)(n >> 32);
    auto low = [](uint32_t d) { return __uint_as_float(0x4B400000u | (d & 127u)) - 12582976.f; };
    q[7] = low(nl);
    q[6] = low(nl >> 7);
    q[5] = low(nl >> 14);
    q[4] = low(nl >> 21);
    q[3] = low(__funnelshift_r(nl, (uint32_t)nh, 28));
    q[2] = low((uint32_t)nh >> 3);
    q[1] = low((uint32_t)nh >> 10);
    q[0] = __int_as_float(0x4B400000 + (nh >> 17)) - 12582912.f;
    return ns;
}

// Power of two of the largest of |v| from the upper words of their bits (1024 if one is not finite).
__device__ __forceinline__ int exponent_of_hi(int h) { return (h >> 20) - 1023; }

__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack(float q0, float q1) {
    return __byte_perm(__float_as_uint(q0), __float_as_uint(q1), 0x7632);
}

// sum_l w_l 128^(7 - l) 2^k from the level sums w_l of at most 96 products per pair of digits (|w_l| < 2^22; the sum
// then fits 62 bits without its lowest 8, which are rounded off first), plus add 2^(k + 8), rounded to nearest.
__device__ __forceinline__ double value(const float (&w)[kD], int k, long long add = 0) {
    int i[kD];
#pragma unroll
    for (int l = 0; l < kD; ++l) i[l] = __float_as_int(w[l] + 12582912.f) - 0x4B400000;
    const long long hi = (long long)((i[0] << 7) + i[1]) * 16384 + (long long)((i[2] << 7) + i[3]);
    const long long lo = (long long)((i[4] << 7) + i[5]) * 16384 + (long long)((i[6] << 7) + i[7]);
    const long long t = (hi << 20) + ((lo + 128) >> 8) + add;
    const unsigned long long m = t < 0 ? (unsigned long long)-t : (unsigned long long)t;
    const int z = __clzll((long long)m);
    const int E = 62 - z + k + 8 + 1023;  // biased exponent - 1; the significand's leading bit adds the 1
    const unsigned long long mm = m << (z & 63);
    long long r = ((long long)E << 52) + (long long)((mm >> 11) + ((mm >> 10) & 1ull));
    if (m == 0ull || E < 0) r = 0;  // zero, or below the normal range
    if (E > 2045) r = 0x7ff0000000000000ll;
    return __longlong_as_double(r | (t & (long long)0x8000000000000000ull));
}

// Fragments for MMAs with B[k][c] = t[(c - k) mod n] of a circulant factor given less the identity (tab[0..n-1]), by nt
// threads; returns their exponent eB, and in sh whether they hold the factor less the identity (sh >= 0) or all of it
// (sh < 0). exp(dtau t C) is close to the identity, and its digits are the same in every slice: cut at 2^-56 of the
// diagonal, their rounding adds up over N L factors (ln det against 64-bit-mantissa arithmetic, rms of 16 fields: 16x16,
// L = 160, 6.0e-12 whole, 2.6e-12 less the identity; 12x12, L = 120, 2.7e-12 / 2.2e-12). The lines' own integers, shifted by
// sh = -2 - eB to the sums' unit, add the identity exactly; sh is at most 4, so that the sum keeps within 62 bits.
__device__ inline int build(uint2* frag, const double* __restrict__ tab, int n, int tid, int nt, int& sh) {
    int h = 0;
    for (int d = 0; d < n; ++d) h = max(h, __double2hiint(tab[d]) & 0x7fffffff);
    int e = max(exponent_of_hi(h), -6);
    sh = -2 - e;
    const double one = sh >= 0 ? 0.0 : 1.0;  // what the fragments add to the diagonal
    if (sh < 0) {
        h = 0;
        for (int d = 0; d < n; ++d) h = max(h, __double2hiint(tab[d] + (d == 0 ? 1.0 : 0.0)) & 0x7fffffff);
        e = exponent_of_hi(h);
    }
    const int total = ntiles(n) * 32;
    for (int i = tid; i < total; i += nt) {
        const int lane = i & 31, j = i >> 5;
        const int c = 8 * j + (lane >> 2), k0 = 2 * (lane & 3);
        float q[4][kD];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = k0 + (u & 1) + 8 * (u >> 1);
            digits(c < n && k < n ? tab[c >= k ? c - k : c - k + n] + (c == k ? one : 0.0) : 0.0, e, q[u]);
        }
#pragma unroll
        for (int s = 0; s < kD; ++s)
            frag[(j * kD + s) * 32 + lane] = make_uint2(pack(q[0][s], q[1][s]), pack(q[2][s], q[3][s]));
    }
    return e;
}

// One tile: the line g[0], g[stride], .. (n <= 8 NTL values) of 16 columns (row r of the tile at g + r rstep, rows
// r < rows used) times the factor, in place; optional input and output scales of the sites (in_sc[m sstep]). All lanes
// of the warp take part.
template <int NTL>
__device__ __forceinline__ void tile(double* g, int rstep, int rows, int stride, int n, const uint2* __restrict__ frag, int eB,
                                     int sh, const double* in_sc, const double* out_sc, int sstep) {
    const int lane = threadIdx.x & 31, r0 = lane >> 2, t2 = 2 * (lane & 3);
    uint32_t a[kD][4];
    long long own[8];  // the thread's values as integers: at the positions of its results
    int e0, e1;
    {
        double v[8];
        int h0 = 0, h1 = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = t2 + (u & 1) + 8 * (u >> 1);
            double x0 = 0.0, x1 = 0.0;
            if (k < n) {
                if (r0 < rows) x0 = g[r0 * rstep + k * stride];
                if (r0 + 8 < rows) x1 = g[(r0 + 8) * rstep + k * stride];
                if (in_sc) {
                    x0 *= in_sc[k * sstep];
                    x1 *= in_sc[k * sstep];
                }
            }
            v[u] = x0;
            v[4 + u] = x1;
            h0 = max(h0, __double2hiint(x0) & 0x7fffffff);
            h1 = max(h1, __double2hiint(x1) & 0x7fffffff);
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            h0 = max(h0, __shfl_xor_sync(0xffffffffu, h0, o));
            h1 = max(h1, __shfl_xor_sync(0xffffffffu, h1, o));
        }
        e0 = exponent_of_hi(h0);
        e1 = exponent_of_hi(h1);
#pragma unroll
        for (int u = 0; u < 4; u += 2) {
            float q0[kD], q1[kD], p0[kD], p1[kD];
            own[u] = digits(v[u], e0, q0);
            own[u + 1] = digits(v[u + 1], e0, q1);
            own[4 + u] = digits(v[4 + u], e1, p0);
            own[5 + u] = digits(v[5 + u], e1, p1);
#pragma unroll
            for (int s = 0; s < kD; ++s) {
                a[s][u] = pack(q0[s], q1[s]);
                a[s][u + 1] = pack(p0[s], p1[s]);
            }
        }
    }
    __syncwarp();  // every lane has read its values
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll 1
    for (int j = 0; j < NTL; ++j) {
        float c[kD][4];
#pragma unroll
        for (int l = 0; l < kD; ++l)
#pragma unroll
            for (int u = 0; u < 4; ++u) c[l][u] = 0.f;
#pragma unroll
        for (int b = 0; b < kD; ++b) {
            const uint2 f = frag[(j * kD + b) * 32 + lane];
#pragma unroll
            for (int s = 0; s + b < kD; ++s) mma(c[s + b], a[s], f.x, f.y);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int col = 8 * j + t2 + (u & 1), r = r0 + 8 * (u >> 1), e = u < 2 ? e0 : e1;
            if (col >= n || r >= rows) continue;
            float w[kD];
#pragma unroll
            for (int l = 0; l < kD; ++l) w[l] = c[l][u];
            // a line with a value that is not finite becomes NaN, as its sums would
            const int at = (u & 1) + 4 * (u >> 1);
            const long long o = j == 0 ? own[at] : own[at + 2];
            double y = e == 1024 ? nan : value(w, e + eB - 61, sh >= 0 ? o << sh : 0);
            if (out_sc) y *= out_sc[col * sstep];
            g[r * rstep + col * stride] = y;
        }
    }
}

// C (row-major, row stride ldc) += sum_{q < cnt} A_q B_q^T, A_q and B_q the N-vectors at Ad + q N and Bd + q N,
// cnt <= 16: one K step, 16 x 8 tiles, digits per row of A and per column of B, each entry's sum rounded once and added
// in FP64: against 64-bit-mantissa arithmetic, the entries of G after a batch are off by 4e-17 (median, relative)
// where 16 rounded FMAs leave 1.2e-16 (9x8 and 12x12 lattices, L = 40 and 80). By the warps of a CTA (warp of
// nw); kChunk column tiles share a row tile's digits.
__device__ __forceinline__ void rank_update(double* C, int ldc, const double* Ad, const double* Bd, int cnt, int N, int warp,
                                            int nw) {
    constexpr int kChunk = 6;
    const int lane = threadIdx.x & 31, r0 = lane >> 2, t2 = 2 * (lane & 3);
    const int CT = (N + 7) / 8, nch = (CT + kChunk - 1) / kChunk, units = (N + 15) / 16 * nch;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    for (int unit = warp; unit < units; unit += nw) {
        const int j0 = unit / nch * 16, c0 = unit % nch * kChunk, c1 = min(CT, c0 + kChunk);
        uint32_t a[kD][4];
        int eA[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + r0 + 8 * h;
            double v[4];
            int m = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = t2 + (u & 1) + 8 * (u >> 1);
                v[u] = (k < cnt && j < N) ? Ad[k * N + j] : 0.0;
                m = max(m, __double2hiint(v[u]) & 0x7fffffff);
            }
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
            eA[h] = exponent_of_hi(m);
            float q[4][kD];
#pragma unroll
            for (int u = 0; u < 4; ++u) digits(v[u], eA[h], q[u]);
#pragma unroll
            for (int s = 0; s < kD; ++s) {
                a[s][h] = pack(q[0][s], q[1][s]);
                a[s][2 + h] = pack(q[2][s], q[3][s]);
            }
        }
#pragma unroll 1
        for (int ct = c0; ct < c1; ++ct) {
            const int col = 8 * ct + r0;
            double v[4];
            int m = 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = t2 + (u & 1) + 8 * (u >> 1);
                v[u] = (k < cnt && col < N) ? Bd[k * N + col] : 0.0;
                m = max(m, __double2hiint(v[u]) & 0x7fffffff);
            }
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
            const int eB = exponent_of_hi(m);
            float c[kD][4];
#pragma unroll
            for (int l = 0; l < kD; ++l)
#pragma unroll
                for (int u = 0; u < 4; ++u) c[l][u] = 0.f;
            {
                float q[4][kD];
#pragma unroll
                for (int u = 0; u < 4; ++u) digits(v[u], eB, q[u]);
#pragma unroll
                for (int b = 0; b < kD; ++b) {
                    const uint32_t f0 = pack(q[0][b], q[1][b]), f1 = pack(q[2][b], q[3][b]);
#pragma unroll
                    for (int s = 0; s + b < kD; ++s) mma(c[s + b], a[s], f0, f1);
                }
            }
            const int eC[2] = {__shfl_sync(0xffffffffu, eB, 4 * t2), __shfl_sync(0xffffffffu, eB, 4 * t2 + 4)};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int m2 = 8 * ct + t2 + (u & 1), j = j0 + r0 + 8 * (u >> 1), e1 = eA[u >> 1], e2 = eC[u & 1];
                if (m2 >= N || j >= N) continue;
                float w[kD];
#pragma unroll
                for (int l = 0; l < kD; ++l) w[l] = c[l][u];
                C[j * ldc + m2] += (e1 == 1024 || e2 == 1024) ? nan : value(w, e1 + e2 - 61);
            }
        }
    }
}

// Length n <= kMaxLine at run time; frag built for that n.
__device__ __forceinline__ void tile_any(double* g, int rstep, int rows, int stride, int n, const uint2* __restrict__ frag,
                                         int eB, int sh, const double* in_sc, const double* out_sc, int sstep) {
    if (n <= 8) tile<1>(g, rstep, rows, stride, n, frag, eB, sh, in_sc, out_sc, sstep);
    else tile<2>(g, rstep, rows, stride, n, frag, eB, sh, in_sc, out_sc, sstep);
}

}  // namespace oz
}  // namespace slmc
