// Blocked Householder QR of the UDT stabilisation with its trailing updates on the tensor cores,
// FP64-accurate.
//
// The pre-pivoted blocked QR (see k_qrb.cu) spends about half of its FP64 issue slots on the
// trailing updates C <- (I - V S^T V^T) C = C - V W', W' = S^T W, W = V^T C, after each panel of BP
// reflectors. Here the panels are factored as before (FP64, one CTA per field, k_qrt_panel), and the
// two products of each trailing update run on the tensor cores in exact fixed-point BF16 slices
// (the same Ozaki-style splitting as the T update): every operand row or column is cut into seven
// 7-bit digits (slice7.cuh) against its own power of two, the products of digit slices a, b with
// a + b <= 6 are summed per level a + b in FP32 accumulators in tensor memory -- exactly, because a
// level's sum of absolute terms stays below 2^24 by construction (at most 36864 per K index, and
// the K range of one accumulator is at most 448) -- and the epilogue combines the levels in two
// 64-bit integers and rounds once to FP64. Each product entry is then the correctly rounded value
// of the sliced operands' product; the slicing (rounding at 2^-48 of each row's / column's largest
// entry) and the dropped levels 7..12 leave an error below 2^-44 K max_k|a_ik| max_k|b_kj| per
// entry: normwise the size of the FP64 loop's own rounding, which is what the backward stability of
// the Householder update needs (errors relative to each column of C, each reflector, each row of
// W').
//
// Per panel t (p = t BP), on the caller's stream:
//   k_qrt_panel<BP>  factor the panel (shared panel_step); write its outputs; slice V twice: per
//                    reflector over the rows (B operand of W^T = C^T V) and per row over the
//                    reflectors (A operand of V W');
//   k_qrt_slice_C    slice the trailing columns of C (rows p..N-1), one exponent per column;
//   k_qrt_gemm1<BP>  W^T = C^T V on the tensor cores (M = trailing columns, N = BP, K = rows), then
//                    W'^T = W^T S and its slices, one exponent per trailing column;
//   k_qrt_gemm2<BP>  C -= V W' on the tensor cores (M = rows, N = 32 trailing columns, K = BP), the
//                    FP64 read-modify-write of C in the epilogue.
// The same kernels form Q in FP64 and, in the chains of DQMC, the trailing updates with eight digits (56 bits) per
// operand and levels 0..7, which leaves the error of FP64 FMAs (Dig, launch_form_q).
// Outputs are those of k_qrb (packed QR, tau, perm, new ln D, sgnU, the panels' S). All waits are
// clock-bounded and set SLMC_EBIT_TIMEOUT; a CTA that gives up drains its copies and frees its
// tensor memory.
#include <algorithm>

#include "oz_line.cuh"
#include "qr_panel.cuh"
#include "slice7.cuh"
#include "tc_ptx.cuh"

namespace {

using namespace slmc::tc;
using slmc::s7::abs_bits;
using slmc::s7::bf16_of;
using slmc::s7::bf16x2_of;
using slmc::s7::combine;
using slmc::s7::exponent_of_bits;
using slmc::s7::slice7;
using slmc::s7::warp_max_bits;

constexpr int kQT = 320;                     // GEMM threads: 8 epilogue warps, TMA warp, MMA warp
constexpr uint32_t kTileA = 128 * 128;       // 128 rows x 64 BF16 (one 128-byte swizzle row each)
constexpr int kMaxN = 896;                   // 14 K chunks: two accumulator sets of seven
constexpr int kVRows = 32;                   // rows of the V1 slice buffer per field (BP <= 32)
// W^T = C^T V streams the seven C slices of a K chunk through a ring of three tiles (tile a is
// released once its products with the seven V slices are issued), so two CTAs fit on an SM: one's
// FP64 epilogue then overlaps the other's copies and products.
constexpr int kRing = 3;
constexpr int kDMax = 8;

// What depends on the number of digits D per operand: seven (49 bits, the trailing updates) or eight (56 bits, Q in
// FP64 and the trailing updates of the DQMC chains; oz_line.cuh's digits). Products a + b <= D - 1 in D levels.
template <int D>
struct Dig {
    // K chunks (64 rows) per accumulator set of W^T = C^T V: a level's sum of absolute terms is at most 36864 per K
    // index with seven digits, 40960 with eight, and stays below 2^24. Tensor memory holds two sets of eight levels of 32
    // reflectors (panels of 32 end at N = 667, eleven chunks) or four of 16 (three needed at N = 896)
    static constexpr int kSegChunks = D == 7 ? 7 : 6;
    // the digits' units 2^(e - 6) per operand and the level weights 2^(-7 level)
    static constexpr int kUnitShift = 2 * 6 + 7 * (D - 1);
    // tiles of the first product's A ring: two leave room for two CTAs per SM beside eight slices of 32 reflectors
    static constexpr __host__ __device__ int ring1(int BP) { return D == 8 && BP == 32 ? 2 : kRing; }
};

template <int D>
__device__ __forceinline__ void cut(double v, int e, float (&q)[D]) {
    if constexpr (D == 7) slice7(v, e, q);
    else slmc::oz::digits(v, e, q);
}

// Level sums (FP32 integers) of one accumulator entry -> hi 2^28 + lo as 64-bit integers.
template <int D>
__device__ __forceinline__ void levels_to_int(const uint32_t (&v)[D], long long& hi, long long& lo) {
    hi = (long long)__float2int_rn(__uint_as_float(v[0]));
#pragma unroll
    for (int lv = 1; lv < D - 4; ++lv) hi = hi * 128 + (long long)__float2int_rn(__uint_as_float(v[lv]));
    lo = (long long)__float2int_rn(__uint_as_float(v[D - 4]));
#pragma unroll
    for (int lv = D - 3; lv < D; ++lv) lo = lo * 128 + (long long)__float2int_rn(__uint_as_float(v[lv]));
}

// The same for sums below 2^22 (K <= 32 indices: at most 40960 * 32 < 2^21): one exact FP32 addition places the
// integer in the significand, where the conversion instruction would take the FP64 pipe's issue.
__device__ __forceinline__ int small_int(uint32_t v) {
    return __float_as_int(__uint_as_float(v) + 12582912.f) - 0x4B400000;
}
template <int D>
__device__ __forceinline__ void small_levels_to_int(const uint32_t (&v)[D], long long& hi, long long& lo) {
    hi = small_int(v[0]);
    if constexpr (D == 8) hi = hi * 128 + (long long)small_int(v[1]);
    hi = hi * 16384 + (long long)((small_int(v[D - 6]) << 7) + small_int(v[D - 5]));
    lo = (long long)((small_int(v[D - 4]) << 7) + small_int(v[D - 3])) * 16384 +
         (long long)((small_int(v[D - 2]) << 7) + small_int(v[D - 1]));
}

// Compact-WY triangle S of BP reflectors from their Gram matrix G (row stride ldg) and tau, by the 256
// threads of the 8 epilogue warps (named barrier 1), in blocks: S is the inverse of the upper
// triangular T with T_cc = 1 / tau_c and T_qc = G_qc (q < c), so the four diagonal blocks of BP/4
// columns follow the column recurrence S_cc = tau_c, S[., c] = -tau_c S[., <c] G[<c, c] (one warp
// each), and blocks merge as S12 = -S11 T12 S22 (T12 = G of the two blocks; no division by tau, so a
// trivial reflector, tau = 0, gives its zero column as the recurrence does). The recurrence of one
// warp over all BP columns was a chain of BP dependent steps. tmp holds BP x BP doubles.
template <int BP>
__device__ __forceinline__ void wy_triangle_blocked(const double* G, int ldg, const double* tau, double* S, double* tmp,
                                                    int tid) {
    constexpr int B4 = BP / 4, B2 = BP / 2;
    const int warp = tid >> 5, lane = tid & 31;
    for (int idx = tid; idx < BP * BP; idx += 256) S[idx] = 0.0;
    slmc::tc::named_sync(1, 256);
    if (warp < 4) {  // diagonal block b = warp: rows and columns o .. o + B4 - 1
        const int o = warp * B4;
        for (int c = 0; c < B4; ++c) {
            double v = 0.0;
            if (lane < c) {
                for (int q = lane; q < c; ++q) v = fma(S[(o + lane) * BP + o + q], G[(o + q) * ldg + o + c], v);
                v = -tau[o + c] * v;
            } else if (lane == c) {
                v = tau[o + c];
            }
            if (lane <= c) S[(o + lane) * BP + o + c] = v;
            __syncwarp();
        }
    }
    slmc::tc::named_sync(1, 256);
    {  // two merges of block pairs (2m, 2m + 1) into B2 x B2 triangles: U = T12 S22, then S12 = -S11 U
        const int m = tid / (B4 * B4), e = tid % (B4 * B4), r = e / B4, c = e % B4;
        const int o1 = m * B2, o2 = o1 + B4;
        if (m < 2) {
            double u = 0.0;
            for (int k = 0; k <= c; ++k) u = fma(G[(o1 + r) * ldg + o2 + k], S[(o2 + k) * BP + o2 + c], u);
            tmp[m * B4 * B4 + e] = u;
        }
        slmc::tc::named_sync(1, 256);
        if (m < 2) {
            double v = 0.0;
            for (int k = r; k < B4; ++k) v = fma(S[(o1 + r) * BP + o1 + k], tmp[m * B4 * B4 + k * B4 + c], v);
            S[(o1 + r) * BP + o2 + c] = -v;
        }
        slmc::tc::named_sync(1, 256);
    }
    for (int e = tid; e < B2 * B2; e += 256) {  // the last merge: U = T12 S22 over the two halves
        const int r = e / B2, c = e % B2;
        double u = 0.0;
        for (int k = 0; k <= c; ++k) u = fma(G[r * ldg + B2 + k], S[(B2 + k) * BP + B2 + c], u);
        tmp[e] = u;
    }
    slmc::tc::named_sync(1, 256);
    for (int e = tid; e < B2 * B2; e += 256) {  // S12 = -S11 U
        const int r = e / B2, c = e % B2;
        double v = 0.0;
        for (int k = r; k < B2; ++k) v = fma(S[r * BP + k], tmp[k * B2 + c], v);
        S[r * BP + B2 + c] = -v;
    }
    slmc::tc::named_sync(1, 256);
}

// ---- panel ----------------------------------------------------------------------------------
// The panel is a chain of column steps (dot products, warp reductions, square root and divisions, one block
// barrier each), so what counts is how many panels an SM works on at once, beside the trailing updates of the
// other sub-batches: 8 warps per field, and shared memory for rows p.. only (PanelSmem; 77 KB for the first
// panel of N = 256, 42 KB for the fifth; with 16 warps and 102 KB whatever the panel a 16x16 evaluation of 512 fields took
// 294 ms, with these 283). With at most one field per SM nothing shares it, and 16 warps shorten the chain (24x24, 32
// fields: 656 against 665 ms per evaluation).

// Shared memory of panel t: V (rows p.. of the panel), the last panel's S and Gram matrix, the scales, the first
// panel's ordering keys, tau, beta, the permutation.
template <int BP>
struct PanelSmem {
    __host__ __device__ static size_t doubles(int N, int p, bool last) {
        return (size_t)(N - p) * (BP + 1) + (last ? 2 * BP * BP : 0) + 3 * (size_t)N + (p == 0 ? N : 0) + 2 * BP;
    }
    static size_t bytes(int N, int p, bool last) { return sizeof(double) * doubles(N, p, last) + sizeof(int) * (size_t)N; }
};

// Slices of the clean reflectors V (row r at Vp + r (BP + 1), rows p..N-1) of one field: per reflector over the
// rows (V1) and per row over the reflectors (V2), with their exponents.
template <int BP, int NT, int D>
__device__ __forceinline__ void slice_V(const double* Vp, __nv_bfloat16* __restrict__ V1, int* __restrict__ eV1,
                                        __nv_bfloat16* __restrict__ V2, int* __restrict__ eV2, int N, int p, int gf, int kpad,
                                        int mpad, size_t plane1, size_t plane2) {
    constexpr int BPS = BP + 1, kW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // V1: reflector m over rows p..N-1 (K-major, K chunks from the one holding row p)
    const int kstart = (p / 64) * 64;
    for (int m = warp; m < BP; m += kW) {
        long long mx = 0;
        for (int r = p + lane; r < N; r += 32) mx = max(mx, abs_bits(Vp[r * BPS + m]));
        const int e = exponent_of_bits(warp_max_bits(mx));
        if (lane == 0) eV1[(size_t)gf * kVRows + m] = e;
        __nv_bfloat16* dst = V1 + ((size_t)gf * kVRows + m) * kpad;
        for (int k = kstart + 2 * lane; k < kpad; k += 64) {  // two adjacent rows per lane (multiples of 64)
            float q0[D], q1[D];
            cut<D>((k >= p && k < N) ? Vp[k * BPS + m] : 0.0, e, q0);
            cut<D>((k + 1 >= p && k + 1 < N) ? Vp[(k + 1) * BPS + m] : 0.0, e, q1);
#pragma unroll
            for (int s = 0; s < D; ++s)
                *reinterpret_cast<uint32_t*>(dst + (size_t)s * plane1 + k) = bf16x2_of(q0[s], q1[s]);
        }
    }
    // V2: row r over the reflectors (K = the BP reflectors, padded to 64 with zeros set at init),
    // rows of the first row tile that holds row p onward
    for (int r = (p / 128) * 128 + warp; r < mpad; r += kW) {
        const double v = (r >= p && r < N && lane < BP) ? Vp[r * BPS + lane] : 0.0;
        const int e = exponent_of_bits(warp_max_bits(abs_bits(v)));
        if (lane == 0) eV2[(size_t)gf * mpad + r] = e;
        if (lane < BP) {
            float q[D];
            cut<D>(v, e, q);
#pragma unroll
            for (int s = 0; s < D; ++s) V2[(size_t)s * plane2 + ((size_t)gf * mpad + r) * 64 + lane] = bf16_of(q[s]);
        }
    }
}

template <int BP, int kPT, int D>
__global__ void __launch_bounds__(kPT, kPT == 256 ? 3 : 1)
    k_qrt_panel(double* __restrict__ Yall, double* __restrict__ lnD_all, double* __restrict__ QRall,
                double* __restrict__ tau_all, int* __restrict__ perm_all, int* __restrict__ sgnU,
                double* __restrict__ Sall, unsigned int* __restrict__ err, int N, int t, double* __restrict__ lnDn_ws,
                int* __restrict__ ntriv_ws, __nv_bfloat16* __restrict__ V1, int* __restrict__ eV1,
                __nv_bfloat16* __restrict__ V2, int* __restrict__ eV2, int kpad, int mpad, size_t plane1,
                size_t plane2, int fbase) {
    constexpr int BPS = BP + 1, kPW = kPT / 32;
    const int f = blockIdx.x, gf = fbase + f;
    const size_t NN = (size_t)N * N;
    double* __restrict__ Y = Yall + f * NN;
    double* __restrict__ QR = QRall + f * NN;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int p = t * BP, nb = min(BP, N - p), npanels = (N + BP - 1) / BP;
    const bool last = t == npanels - 1;
    double* Vst = reinterpret_cast<double*>(smraw);
    double* Vp = Vst - (size_t)p * BPS;  // row r of the panel at r BPS, rows p.. stored
    double* Ssm = Vst + (size_t)(N - p) * BPS;
    double* Gsm = Ssm + BP * BP;  // (last panel only)
    double* s_lnd = Ssm + (last ? 2 * BP * BP : 0);
    double* s_lnDn = s_lnd + N;
    double* s_g = s_lnDn + N;
    double* s_tau = s_g + N;
    double* s_beta = s_tau + BP;
    double* s_key = s_beta + BP;  // (first panel only)
    int* s_perm = reinterpret_cast<int*>(s_key + (p == 0 ? N : 0));
    __shared__ double s_mx;
    __shared__ int s_ntriv, s_wide;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    for (int j = tid; j < N; j += kPT) s_lnd[j] = lnD_all[(size_t)f * N + j];
    if (tid == 0) {
        s_ntriv = 0;
        s_wide = 0;
    }
    __syncthreads();
    if (t == 0) {  // scaled column norms and the pre-pivoting order, as in k_qrb
        if (warp == 0) {
            double mx = -DBL_MAX;
            for (int j = lane; j < N; j += 32) mx = fmax(mx, s_lnd[j]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (lane == 0) s_mx = mx;
        }
        __syncthreads();
        for (int j = warp; j < N; j += kPW) {
            double a = 0.0;
            for (int i = lane; i < N; i += 32) {
                const double y = Y[(size_t)j * N + i];
                a = fma(y, y, a);
            }
            a = slmc::warp_allsum(a);
            if (lane == 0) s_key[j] = a;
        }
        __syncthreads();
        for (int j = tid; j < N; j += kPT) {  // a column per lane: an exponential is about 20 FP64 instructions
            const double key = s_key[j] * exp(2.0 * (s_lnd[j] - s_mx));
            s_key[j] = (key >= 0.0) ? key : -1.0;
        }
        __syncthreads();
        for (int j = tid; j < N; j += kPT) {
            // keys are >= +0 or -1: their bit patterns as 64-bit integers order as the values do, and
            // the integer compares leave the FP64 pipe to the factorisation
            const long long kj = __double_as_longlong(s_key[j]);
            int r = 0;
            for (int i = 0; i < N; ++i) {
                const long long ki = __double_as_longlong(s_key[i]);
                r += (ki > kj) || (ki == kj && i < j);
            }
            s_perm[r] = j;
        }
        __syncthreads();
        for (int j = tid; j < N; j += kPT) perm_all[(size_t)f * N + j] = s_perm[j];
    } else {
        for (int j = tid; j < N; j += kPT) s_perm[j] = perm_all[(size_t)f * N + j];
        for (int i = tid; i < p; i += kPT) {
            const double l = lnDn_ws[(size_t)gf * N + i];
            s_lnDn[i] = l;
            s_g[i] = exp(-l);
            if (fabs(l) > 600.0) s_wide = 1;
        }
    }
    for (int k = tid; k < N; k += kPT)
        if (fabs(s_lnd[k]) > 600.0) s_wide = 1;
    __syncthreads();

    // the Gram matrix and S of every panel but the last are formed on the tensor cores (k_qrt_gemm1)
    panel_step<BP, kPT>(Y, QR, tau_all + (size_t)f * N, Sall + (size_t)f * N * BP, Vp, Ssm, Gsm, s_lnd, s_lnDn, s_g, s_tau,
                        s_beta, s_perm, &s_ntriv, &s_wide, N, p, nb, last);
    __syncthreads();
    if (tid < nb) lnDn_ws[(size_t)gf * N + p + tid] = s_lnDn[p + tid];
    if (tid == 0) {  // reflectors with tau != 0 so far (their parity is the sign of det U)
        const int ntriv = (t == 0 ? 0 : ntriv_ws[gf]) + s_ntriv;
        if (t == npanels - 1) sgnU[f] = (ntriv & 1) ? -1 : 1;
        else ntriv_ws[gf] = ntriv;
    }
    if (t == npanels - 1) {  // every scale is known: publish ln D'
        bool bad = false;
        for (int k = tid; k < N; k += kPT) {
            lnD_all[(size_t)f * N + k] = s_lnDn[k];
            bad |= !isfinite(s_lnDn[k]);
        }
        if (bad) atomicOr(err, SLMC_EBIT_NONFINITE);
        return;
    }
    slice_V<BP, kPT, D>(Vp, V1, eV1, V2, eV2, N, p, gf, kpad, mpad, plane1, plane2);
}

// ---- slices of the trailing columns ---------------------------------------------------------
// Warp w of block x slices trailing column jj = 8 x + w (logical column j0 + jj; no permutation in the formation of
// Q) over rows p..N-1.
template <int D>
__global__ void __launch_bounds__(256) k_qrt_slice_C(const double* __restrict__ Yall, const int* __restrict__ perm_all,
                                                     __nv_bfloat16* __restrict__ Cs, int* __restrict__ eC, int N,
                                                     int p, int j0, int kpad, int jpad, size_t plane, int fbase) {
    const int f = blockIdx.y, gf = fbase + f, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int jj = blockIdx.x * 8 + warp, j = j0 + jj;
    if (j >= N) return;
    const double* col = Yall + (size_t)f * N * N + (size_t)(perm_all ? perm_all[(size_t)f * N + j] : j) * N;
    long long mx = 0;
    for (int r = p + lane; r < N; r += 32) mx = max(mx, abs_bits(col[r]));
    const int e = exponent_of_bits(warp_max_bits(mx));
    if (lane == 0) eC[(size_t)gf * jpad + jj] = e;
    __nv_bfloat16* dst = Cs + ((size_t)gf * jpad + jj) * kpad;
    for (int k = (p / 64) * 64 + 2 * lane; k < kpad; k += 64) {  // two adjacent rows per lane (multiples of 64)
        float q0[D], q1[D];
        cut<D>((k >= p && k < N) ? col[k] : 0.0, e, q0);
        cut<D>((k + 1 >= p && k + 1 < N) ? col[k + 1] : 0.0, e, q1);
#pragma unroll
        for (int s = 0; s < D; ++s)
            *reinterpret_cast<uint32_t*>(dst + (size_t)s * plane + k) = bf16x2_of(q0[s], q1[s]);
    }
}

// The reflectors of panel p of a finished QR (below the diagonal of its packed output), sliced again for the
// formation of Q.
template <int BP, int D>
__global__ void __launch_bounds__(256) k_qrt_slice_V(const double* __restrict__ QRall, __nv_bfloat16* __restrict__ V1,
                                                     int* __restrict__ eV1, __nv_bfloat16* __restrict__ V2,
                                                     int* __restrict__ eV2, int N, int p, int kpad, int mpad, size_t plane1,
                                                     size_t plane2, int fbase) {
    constexpr int BPS = BP + 1;
    extern __shared__ __align__(16) unsigned char smraw[];
    double* Vp = reinterpret_cast<double*>(smraw) - (size_t)p * BPS;  // rows p.. stored
    const int f = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double* QR = QRall + (size_t)f * N * N;
    for (int c = warp; c < BP; c += 8) {
        const int k = p + c;
        for (int r = p + lane; r < N; r += 32)
            Vp[r * BPS + c] = k < N ? (r > k ? QR[(size_t)k * N + r] : (r == k ? 1.0 : 0.0)) : 0.0;
    }
    __syncthreads();
    slice_V<BP, 256, D>(Vp, V1, eV1, V2, eV2, N, p, fbase + f, kpad, mpad, plane1, plane2);
}

// ---- [G; W^T] = [V C]^T V, S from G, then W'^T = W^T S and its slices -----------------------
// CTA = the BP reflectors plus 128 - BP trailing columns of one field: each 128-row A tile holds the
// slices of V's columns (rows 0..BP-1, from the reflector slice buffer) above those of the CTA's
// trailing columns of C, so the product's first BP rows are the panel's Gram matrix G = V^T V. The
// epilogue forms the compact-WY triangle S from G (the panel kernel no longer does; CTA 0 writes it
// out for the formation of Q), then W' = S^T W. TMA streams per 64-row K chunk the D A slices
// through a ring of tiles and the D V slices double-buffered; products (a, b), a + b <= D - 1, go to
// the accumulator of level a + b of the chunk's segment (Dig<D>::kSegChunks chunks per segment).
// kForm: the step of the formation of Q, whose panels need W' = S W with the S the QR left in Sall (the Gram rows
// of the product are not used).
template <int BP, bool kForm, int D>
__global__ void __launch_bounds__(kQT, 2)
    k_qrt_gemm1(const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmV,
                const int* __restrict__ eC, const int* __restrict__ eV1, const double* __restrict__ tau_all,
                double* __restrict__ Sall, __nv_bfloat16* __restrict__ Ws, int* __restrict__ eW, int N, int p,
                int n_t, int kpad, int jpad, int wpad, size_t planeW, int fbase, unsigned int* __restrict__ err) {
    constexpr uint32_t kTileB = BP * 128;
    constexpr int kRing = Dig<D>::ring1(BP), kSegChunks = Dig<D>::kSegChunks;
    constexpr uint32_t kChunkB = D * kTileB;
    constexpr int WS = BP + 1;
    constexpr int kMC = 128 - BP;  // trailing columns per CTA
    const int mt = blockIdx.x, f = blockIdx.y, gf = fbase + f;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kc0 = p / 64, nkc = kpad / 64 - kc0;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[kRing], bar_empty[kRing], bar_bfull[2], bar_bempty[2], bar_acc, bar_done;
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_sh;
    __shared__ int eV_sh[BP];
    __shared__ double tau_sh[BP];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t bbuf = base, aring = base + 2 * kChunkB;
    // after the MMAs: stage of [G; W] [128][WS], W' [128][WS] and S [BP][BP] over the B buffers and the ring
    double* stW = reinterpret_cast<double*>(smem_raw + (bbuf - raw));
    double* stWp = stW + 128 * WS;
    double* Ssh = stWp + 128 * WS;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kRing; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_bfull[b]), 1);
            mbar_init(smem_u32(&bar_bempty[b]), 1);
        }
        mbar_init(smem_u32(&bar_acc), 1);
        mbar_init(smem_u32(&bar_done), 1);
        abort_sh = 0;
        fence_barrier_init();
    }
    if (threadIdx.x < BP) {
        eV_sh[threadIdx.x] = eV1[(size_t)gf * kVRows + threadIdx.x];
        if (!kForm) tau_sh[threadIdx.x] = tau_all[(size_t)f * N + p + threadIdx.x];
    }
    const int nseg = (nkc + kSegChunks - 1) / kSegChunks;
    const uint32_t tcols = nseg == 1 ? 256u : 512u;  // D levels x BP columns per accumulator set
    if (warp == 9) {
        tmem_alloc(smem_u32(&tmem_base_sh), tcols);
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;

    if (warp == 8) {
        if (lane == 0) {
            int issued_a = 0, issued_b = 0;
            for (int u = 0; u < nkc && !abort_sh; ++u) {
                const int kc = kc0 + u, bs = u & 1;
                if (u >= 2 && !mbar_wait(smem_u32(&bar_bempty[bs]), ((u >> 1) - 1) & 1, err)) {
                    abort_sh = 1;
                    break;
                }
                const uint32_t bb = smem_u32(&bar_bfull[bs]);
                mbar_expect_tx(bb, kChunkB);
                for (int b = 0; b < D; ++b) tma_load_3d(bbuf + bs * kChunkB + b * kTileB, &tmV, kc * 64, gf * kVRows, b, bb);
                issued_b = u + 1;
                for (int a = 0; a < D; ++a) {
                    const int q = u * D + a, slot = q % kRing;
                    if (q >= kRing && !mbar_wait(smem_u32(&bar_empty[slot]), ((q / kRing) - 1) & 1, err)) {
                        abort_sh = 1;
                        break;
                    }
                    const uint32_t fb = smem_u32(&bar_full[slot]);
                    mbar_expect_tx(fb, kTileA);  // BP rows of V + kMC rows of C
                    tma_load_3d(aring + slot * kTileA, &tmV, kc * 64, gf * kVRows, a, fb);
                    tma_load_3d(aring + slot * kTileA + kTileB, &tmC, kc * 64, gf * jpad + mt * kMC, a, fb);
                    issued_a = q + 1;
                }
                if (abort_sh) break;
            }
            for (int q = issued_a - 1; q >= 0 && q >= issued_a - kRing; --q)
                mbar_wait(smem_u32(&bar_full[q % kRing]), (q / kRing) & 1, err);
            for (int u = issued_b - 1; u >= 0 && u >= issued_b - 2; --u)
                mbar_wait(smem_u32(&bar_bfull[u & 1]), (u >> 1) & 1, err);
        }
    } else if (warp == 9) {
        if (lane == 0) {
            bool ok = true;
            Ring ring;
            const uint64_t da0 = smem_desc_sw128(aring), db0 = smem_desc_sw128(bbuf);
            const uint32_t full0 = smem_u32(bar_full), empty0 = smem_u32(bar_empty);
            for (int u = 0; u < nkc && ok; ++u) {
                const int bs = u & 1, seg = u / kSegChunks;
                if (!mbar_wait(smem_u32(&bar_bfull[bs]), (u >> 1) & 1, err) || abort_sh) {
                    ok = false;
                    break;
                }
                const uint64_t db = db0 + (uint64_t)bs * desc_step(kChunkB);
                const bool first = u == seg * kSegChunks;
#pragma unroll
                for (int a = 0; a < D; ++a) {
                    if (!ok || !mbar_wait(full0 + 8 * ring.slot, ring.phase, err) || abort_sh) {
                        ok = false;
                        continue;
                    }
                    tc_fence_after();
                    const uint64_t da = da0 + (uint64_t)ring.slot * desc_step(kTileA);
                    // slices b = 0 .. D - 1 - a of V into the levels a .. D - 1: adjacent operand rows and adjacent
                    // accumulators, so one instruction of N = (D - a) BP per step of K
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        mma_bf16(tmem + (uint32_t)((seg * D + a) * BP), da + desc_step(ks * 32), db + desc_step(ks * 32),
                                 idesc_f32acc(1, 128, (D - a) * BP), (a | ks) != 0 || !first ? 1u : 0u);
                    mma_commit(empty0 + 8 * ring.slot);
                    ring.next(kRing);
                }
                if (ok) mma_commit(smem_u32(&bar_bempty[bs]));
            }
            if (ok) mma_commit(smem_u32(&bar_acc));
            else abort_sh = 1;
            mma_commit(smem_u32(&bar_done));
            mbar_wait(smem_u32(&bar_done), 0, err);
        }
    } else {
        // ---- epilogue: warp w drains rows 32 (w % 4).. for reflectors (w / 4) BP/2 .. ----
        // row r < BP: G[r][.] (exponents of the reflectors); row r >= BP: W of trailing column
        // jj = mt kMC + r - BP
        constexpr int HC = BP / 2;
        const int q4 = warp & 3, h = warp >> 2, r = 32 * q4 + lane, jj = mt * kMC + r - BP;
        constexpr int SPT = BP * BP / 256;
        double s_in[SPT];  // kForm: S (rows beyond the last reflector are zero), loaded before the products are waited for
        if (kForm)
#pragma unroll
            for (int q = 0; q < SPT; ++q) {
                const int idx = threadIdx.x + 256 * q;
                s_in[q] = p + idx / BP < N ? Sall[((size_t)f * N + p) * BP + idx] : 0.0;
            }
        const bool bad = !mbar_wait(smem_u32(&bar_acc), 0, err) || abort_sh;
        if (!named_sync_or(1, 256, bad)) {
            tc_fence_after();
            const int er = r < BP ? eV_sh[r] : (jj < n_t ? eC[(size_t)gf * jpad + jj] : 0);
#pragma unroll
            for (int c0 = 0; c0 < HC; c0 += 8) {
                long long hi[8], lo[8];
#pragma unroll
                for (int c = 0; c < 8; ++c) hi[c] = lo[c] = 0;
                for (int sg = 0; sg < nseg; ++sg) {
                    uint32_t v[D][8];
                    const uint32_t tl = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(sg * D * BP + h * HC + c0);
#pragma unroll
                    for (int lv = 0; lv < D; ++lv) tmem_ld8(tl + (uint32_t)(lv * BP), v[lv]);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        uint32_t w[D];
#pragma unroll
                        for (int lv = 0; lv < D; ++lv) w[lv] = v[lv][c];
                        long long a, b;
                        levels_to_int<D>(w, a, b);
                        hi[c] += a;
                        lo[c] += b;
                    }
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int m = h * HC + c0 + c;
                    stW[r * WS + m] = combine(hi[c], lo[c], er + eV_sh[m] - Dig<D>::kUnitShift);
                }
            }
        }
        named_sync(1, 256);
        if (kForm) {
            if (!bad)
#pragma unroll
                for (int q = 0; q < SPT; ++q) Ssh[threadIdx.x + 256 * q] = s_in[q];
            named_sync(1, 256);
        } else if (!bad) {
            wy_triangle_blocked<BP>(stW, WS, tau_sh, Ssh, stWp, threadIdx.x);  // S from G = rows 0..BP-1
        }
        if (!bad) {
            if (!kForm && mt == 0)  // S of the panel for the formation of Q
                for (int idx = threadIdx.x; idx < BP * BP; idx += 256)
                    Sall[((size_t)f * N + p) * BP + idx] = Ssh[idx];
            // W'[m] = sum_{q <= m} S[q][m] W[q]  (S upper triangular); thread (row, half)
            const int rr = BP + (threadIdx.x & 127) % kMC, hh = threadIdx.x >> 7;
            if ((threadIdx.x & 127) < kMC)
                for (int m = hh * HC; m < hh * HC + HC; ++m) {
                    double a = 0.0;
                    if (kForm)
                        for (int q = m; q < BP; ++q) a = fma(Ssh[m * BP + q], stW[rr * WS + q], a);
                    else
                        for (int q = 0; q <= m; ++q) a = fma(Ssh[q * BP + m], stW[rr * WS + q], a);
                    stWp[rr * WS + m] = a;
                }
        }
        named_sync(1, 256);
        if (!bad) {
            // slices of W', one row (trailing column) per warp at a time, lane = reflector: the row's
            // exponent by a warp reduction, each plane's row one coalesced store
            for (int t = warp; t < kMC; t += 8) {
                const int rr = BP + t, j2 = mt * kMC + t;
                if (j2 >= n_t) break;
                const double v = lane < BP ? stWp[rr * WS + lane] : 0.0;
                const int e = exponent_of_bits(warp_max_bits(abs_bits(v)));
                if (lane == 0) eW[(size_t)gf * wpad + j2] = e;
                if (lane < BP) {
                    float q[D];
                    cut<D>(v, e, q);
                    __nv_bfloat16* dst = Ws + ((size_t)gf * wpad + j2) * 64 + lane;
#pragma unroll
                    for (int s = 0; s < D; ++s) dst[(size_t)s * planeW] = bf16_of(q[s]);
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 9) tmem_dealloc(tmem, tcols);
}

// ---- C -= V W' -----------------------------------------------------------------------------
// CTA = 128 rows (row tile p/128 + blockIdx.y) x kNC trailing columns of one field; one K chunk (BP
// reflectors): the D W' slices resident, the D V slices streamed through the 3-tile ring.
// 32 columns keep the accumulators at D x 32 <= 256 tensor-memory columns, so two CTAs share an SM.
constexpr int kNC = 32;

template <int BP, int D>
__global__ void __launch_bounds__(kQT, 2)
    k_qrt_gemm2(const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmW,
                const int* __restrict__ eV2, const int* __restrict__ eW, const int* __restrict__ perm_all,
                double* __restrict__ Yall, int N, int p, int j0, int n_t, int mpad, int wpad, int fbase,
                unsigned int* __restrict__ err) {
    constexpr uint32_t kTileW = kNC * 128;
    const int nt = blockIdx.x, mt = p / 128 + blockIdx.y, f = blockIdx.z, gf = fbase + f;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[kRing], bar_empty[kRing], bar_bfull, bar_acc, bar_done;
    __shared__ uint32_t tmem_base_sh;
    __shared__ volatile int abort_sh;
    __shared__ int eW_sh[kNC];
    __shared__ int col_sh[kNC];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const uint32_t bbuf = base, aring = base + D * kTileW;

    if (threadIdx.x == 0) {
        for (int q = 0; q < kRing; ++q) {
            mbar_init(smem_u32(&bar_full[q]), 1);
            mbar_init(smem_u32(&bar_empty[q]), 1);
        }
        mbar_init(smem_u32(&bar_bfull), 1);
        mbar_init(smem_u32(&bar_acc), 1);
        mbar_init(smem_u32(&bar_done), 1);
        abort_sh = 0;
        fence_barrier_init();
    }
    if (threadIdx.x < kNC) {
        const int jj = nt * kNC + threadIdx.x;
        eW_sh[threadIdx.x] = jj < n_t ? eW[(size_t)gf * wpad + jj] : 0;
        col_sh[threadIdx.x] = jj < n_t ? (perm_all ? perm_all[(size_t)f * N + j0 + jj] : j0 + jj) : 0;
    }
    if (warp == 9) {
        tmem_alloc(smem_u32(&tmem_base_sh), 256);
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;

    if (warp == 8) {
        if (lane == 0) {
            const uint32_t bb = smem_u32(&bar_bfull);
            mbar_expect_tx(bb, D * kTileW);
            for (int b = 0; b < D; ++b) tma_load_3d(bbuf + b * kTileW, &tmW, 0, gf * wpad + nt * kNC, b, bb);
            int issued = 0;
            for (int a = 0; a < D; ++a) {
                const int slot = a % kRing;
                if (a >= kRing && !mbar_wait(smem_u32(&bar_empty[slot]), ((a / kRing) - 1) & 1, err)) break;
                const uint32_t fb = smem_u32(&bar_full[slot]);
                mbar_expect_tx(fb, kTileA);
                tma_load_3d(aring + slot * kTileA, &tmV, 0, gf * mpad + mt * 128, a, fb);
                issued = a + 1;
            }
            // (bounded) the copies have landed before the CTA can exit
            mbar_wait(bb, 0, err);
            for (int a = issued - 1; a >= 0 && a >= issued - kRing; --a)
                mbar_wait(smem_u32(&bar_full[a % kRing]), (a / kRing) & 1, err);
        }
    } else if (warp == 9) {
        if (lane == 0) {
            bool ok = mbar_wait(smem_u32(&bar_bfull), 0, err);
            const uint64_t da0 = smem_desc_sw128(aring), db0 = smem_desc_sw128(bbuf);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const int slot = a % kRing;
                if (!ok || !mbar_wait(smem_u32(&bar_full[slot]), (a / kRing) & 1, err)) {
                    ok = false;
                    continue;
                }
                tc_fence_after();
#pragma unroll
                for (int ks = 0; ks < BP / 16; ++ks)
                    mma_bf16(tmem + (uint32_t)(a * kNC), da0 + desc_step(slot * kTileA + ks * 32), db0 + desc_step(ks * 32),
                             idesc_f32acc(1, 128, (D - a) * kNC), (a | ks) != 0 ? 1u : 0u);
                mma_commit(smem_u32(&bar_empty[slot]));
            }
            if (ok) mma_commit(smem_u32(&bar_acc));
            else abort_sh = 1;
            mma_commit(smem_u32(&bar_done));
            mbar_wait(smem_u32(&bar_done), 0, err);
        }
    } else {
        // ---- epilogue: warp w: rows 32 (w % 4).. of the tile, columns 16 (w / 4)..; C -= V W' ----
        constexpr int HC = kNC / 2;
        const int q4 = warp & 3, h = warp >> 2, r = mt * 128 + 32 * q4 + lane;
        const bool row_ok = r >= p && r < N;
        const int ev = row_ok ? eV2[(size_t)gf * mpad + r] : 0;
        double* Yf = Yall + (size_t)f * N * N + r;
        // the entries of C for a block of 8 columns are loaded together, the first block's before the products are
        // waited for (one at a time behind the stores of the last, their latencies were most of the epilogue)
        double y[8];
        auto fetch = [&](int c0) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int cc = HC * h + c0 + c;
                y[c] = (row_ok && nt * kNC + cc < n_t) ? Yf[(size_t)col_sh[cc] * N] : 0.0;
            }
        };
        fetch(0);
        const bool bad = !mbar_wait(smem_u32(&bar_acc), 0, err) || abort_sh;
        if (!named_sync_or(1, 256, bad)) {
            tc_fence_after();
#pragma unroll
            for (int c0 = 0; c0 < HC; c0 += 8) {
                uint32_t v[D][8];
                const uint32_t tl = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(HC * h + c0);
#pragma unroll
                for (int lv = 0; lv < D; ++lv) tmem_ld8(tl + (uint32_t)(lv * kNC), v[lv]);
                if (c0 > 0) fetch(c0);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int cc = HC * h + c0 + c;
                    if (!row_ok || nt * kNC + cc >= n_t) continue;
                    uint32_t w[D];
#pragma unroll
                    for (int lv = 0; lv < D; ++lv) w[lv] = v[lv][c];
                    long long hi, lo;
                    small_levels_to_int<D>(w, hi, lo);
                    Yf[(size_t)col_sh[cc] * N] = y[c] - combine(hi, lo, ev + eW_sh[cc] - Dig<D>::kUnitShift);
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 9) tmem_dealloc(tmem, 256);
}

template <int D>
size_t gemm1_smem(int BP) { return 1024 + 2 * (size_t)D * BP * 128 + (size_t)Dig<D>::ring1(BP) * kTileA; }
template <int D>
size_t gemm2_smem() { return 1024 + (size_t)D * kNC * 128 + (size_t)kRing * kTileA; }

struct QrtArgs {
    int N, kpad, mpad, wpad, jpad;
    size_t plane1, plane2, planeC, planeW;
    __nv_bfloat16 *V1, *V2, *Cs, *Ws;
};

QrtArgs qrt_args(const slmc_ctx* c) {
    QrtArgs a;
    a.N = c->N;
    a.kpad = c->qt_kpad;
    a.mpad = c->qt_mpad;
    a.wpad = c->qt_wpad;
    a.jpad = c->qt_mpad;
    const size_t F = c->max_fields;
    a.plane1 = F * kVRows * a.kpad;
    a.plane2 = F * a.mpad * 64;
    a.planeC = F * a.jpad * a.kpad;
    a.planeW = F * a.wpad * 64;
    a.V1 = reinterpret_cast<__nv_bfloat16*>(c->qt_V1);
    a.V2 = reinterpret_cast<__nv_bfloat16*>(c->qt_V2);
    a.Cs = reinterpret_cast<__nv_bfloat16*>(c->qt_C);
    a.Ws = reinterpret_cast<__nv_bfloat16*>(c->qt_W);
    return a;
}

template <int BP, int kPT, int D>
cudaError_t launch_panel(slmc_ctx* c, int nf, int t, cudaStream_t s) {
    const QrtArgs a = qrt_args(c);
    const int p = t * BP;
    const size_t smP = PanelSmem<BP>::bytes(a.N, p, p + BP >= a.N);
    cudaError_t e = slmc::allow_smem(k_qrt_panel<BP, kPT, D>, smP);
    if (e != cudaSuccess) return e;
    k_qrt_panel<BP, kPT, D><<<nf, kPT, smP, s>>>(c->Y, c->lnD, c->QR, c->tau, c->perm, c->sgnU, c->Sws, c->err, a.N, t,
                                              c->qt_lnDn, c->qt_ntriv, a.V1, c->qt_eV1, a.V2, c->qt_eV2, a.kpad,
                                              a.mpad, a.plane1, a.plane2, c->fbase);
    return cudaGetLastError();
}

// Trailing update of panel t (t < last panel): slices of C, W'^T = (C^T V) S, C -= V W'.
template <int BP, int D>
cudaError_t launch_trailing(slmc_ctx* c, int nf, int t, cudaStream_t s) {
    const QrtArgs a = qrt_args(c);
    const size_t sm1 = gemm1_smem<D>(BP), sm2 = gemm2_smem<D>();
    cudaError_t e = slmc::allow_smem(k_qrt_gemm1<BP, false, D>, sm1);
    if (e == cudaSuccess) e = slmc::allow_smem(k_qrt_gemm2<BP, D>, sm2);
    if (e != cudaSuccess) return e;
    const CUtensorMap& mapV1 = BP == 32 ? c->qt_mapV1_32 : c->qt_mapV1_16;
    const int N = a.N, p = t * BP, j0 = p + BP, n_t = N - j0;
    k_qrt_slice_C<D><<<dim3((n_t + 7) / 8, nf), 256, 0, s>>>(c->Y, c->perm, a.Cs, c->qt_eC, N, p, j0, a.kpad, a.jpad,
                                                          a.planeC, c->fbase);
    const CUtensorMap& mapC = BP == 32 ? c->qt_mapC96 : c->qt_mapC112;
    k_qrt_gemm1<BP, false, D><<<dim3((n_t + 127 - BP) / (128 - BP), nf), kQT, sm1, s>>>(
        mapC, mapV1, c->qt_eC, c->qt_eV1, c->tau, c->Sws, a.Ws, c->qt_eW, N, p, n_t, a.kpad, a.jpad, a.wpad, a.planeW,
        c->fbase, c->err);
    k_qrt_gemm2<BP, D><<<dim3((n_t + kNC - 1) / kNC, a.mpad / 128 - p / 128, nf), kQT, sm2, s>>>(
        c->qt_mapV2, c->qt_mapW, c->qt_eV2, c->qt_eW, c->perm, c->Y, N, p, j0, n_t, a.mpad, a.wpad, c->fbase, c->err);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_qrt_identity(double* __restrict__ U, int N) {
    double* Uf = U + (size_t)blockIdx.y * N * N;
    for (int idx = blockIdx.x * 256 + threadIdx.x; idx < N * N; idx += gridDim.x * 256) Uf[idx] = idx % (N + 1) == 0 ? 1.0 : 0.0;
}

// Q = Q_0 Q_1 ... accumulated backwards into U: per panel, columns and rows p.. of U take I - V S V^T through the
// products of the trailing update (slices of V and of U's columns, W = V^T U, W' = S W, U -= V W'), with eight digits:
// Q then is as near to the exact one as by FP64 FMAs, and G errs by the QR's and the T update's 49 bits only (T by FMAs,
// error of G against extended precision: 18x18, L = 30 1.41e-13 with FMAs or eight digits, 1.71e-13 with
// seven; 18x10, L = 37 2.07 / 2.07 / 2.15e-13; 12x12, L = 40 1.38 / 1.38 / 1.44e-13). On the FP64 pipe
// (k_formq_b) the 4/3 N^3 flops were 30-45 % of an FP64 evaluation: 12x12, L = 120, 256 fields with G take 62 ms that
// way, 53.0 with eight digits and 51.7 with seven; 18x10, L = 37, 50 fields 13.3, 11.3 and 11.2 ms.
template <int BP>
cudaError_t launch_form_q(slmc_ctx* c, int nf, cudaStream_t s) {
    const QrtArgs a = qrt_args(c);
    const int N = a.N;
    const size_t sm1 = gemm1_smem<8>(BP), sm2 = gemm2_smem<8>(), smV = sizeof(double) * (size_t)N * (BP + 1);
    cudaError_t e = slmc::allow_smem(k_qrt_gemm1<BP, true, 8>, sm1);
    if (e == cudaSuccess) e = slmc::allow_smem(k_qrt_gemm2<BP, 8>, sm2);
    if (e == cudaSuccess) e = slmc::allow_smem(k_qrt_slice_V<BP, 8>, smV);
    if (e != cudaSuccess) return e;
    const CUtensorMap& mapV1 = BP == 32 ? c->qt_mapV1_32 : c->qt_mapV1_16;
    const CUtensorMap& mapC = BP == 32 ? c->qt_mapC96 : c->qt_mapC112;
    k_qrt_identity<<<dim3(std::min(64, (N * N + 1023) / 1024), nf), 256, 0, s>>>(c->U, N);
    for (int p = (N - 1) / BP * BP; p >= 0; p -= BP) {
        const int n_t = N - p;
        k_qrt_slice_V<BP, 8><<<nf, 256, sizeof(double) * (size_t)n_t * (BP + 1), s>>>(
            c->QR, a.V1, c->qt_eV1, a.V2, c->qt_eV2, N, p, a.kpad, a.mpad, a.plane1, a.plane2, c->fbase);
        k_qrt_slice_C<8><<<dim3((n_t + 7) / 8, nf), 256, 0, s>>>(c->U, nullptr, a.Cs, c->qt_eC, N, p, p, a.kpad, a.jpad, a.planeC,
                                                              c->fbase);
        k_qrt_gemm1<BP, true, 8><<<dim3((n_t + 127 - BP) / (128 - BP), nf), kQT, sm1, s>>>(
            mapC, mapV1, c->qt_eC, c->qt_eV1, c->tau, c->Sws, a.Ws, c->qt_eW, N, p, n_t, a.kpad, a.jpad, a.wpad, a.planeW,
            c->fbase, c->err);
        k_qrt_gemm2<BP, 8><<<dim3((n_t + kNC - 1) / kNC, a.mpad / 128 - p / 128, nf), kQT, sm2, s>>>(
            c->qt_mapV2, c->qt_mapW, c->qt_eV2, c->qt_eW, nullptr, c->U, N, p, p, n_t, a.mpad, a.wpad, c->fbase, c->err);
    }
    return cudaGetLastError();
}

}  // namespace

namespace slmc {

bool qrt_supported(int N) { return N >= 2 && N <= kMaxN; }

// Sizes of the slice buffers (BF16 elements) and exponent arrays of a context with F fields.
void qrt_sizes(int N, int F, size_t* bf16_elems, size_t* int_elems) {
    const size_t kpad = (N + 63) / 64 * 64, mpad = (N + 127) / 128 * 128, wpad = kpad;
    *bf16_elems = (size_t)kDMax * F * (mpad * kpad + kVRows * kpad + mpad * 64 + wpad * 64);
    *int_elems = (size_t)F * (mpad + kVRows + mpad + wpad + 1);
}

// Carves the buffers allocated by slmc_init, zeroes them (the padding is never written again) and
// encodes the TMA descriptors.
cudaError_t qrt_init(slmc_ctx* c, void* bf16_base, int* int_base) {
    const int N = c->N;
    const size_t F = c->max_fields;
    c->qt_kpad = (N + 63) / 64 * 64;
    c->qt_mpad = (N + 127) / 128 * 128;
    c->qt_wpad = c->qt_kpad;
    const size_t kpad = c->qt_kpad, mpad = c->qt_mpad, wpad = c->qt_wpad;
    __nv_bfloat16* b = reinterpret_cast<__nv_bfloat16*>(bf16_base);
    c->qt_C = b;
    b += (size_t)kDMax * F * mpad * kpad;
    c->qt_V1 = b;
    b += (size_t)kDMax * F * kVRows * kpad;
    c->qt_V2 = b;
    b += (size_t)kDMax * F * mpad * 64;
    c->qt_W = b;
    b += (size_t)kDMax * F * wpad * 64;
    c->qt_eC = int_base;
    c->qt_eV1 = c->qt_eC + F * mpad;
    c->qt_eV2 = c->qt_eV1 + F * kVRows;
    c->qt_eW = c->qt_eV2 + F * mpad;
    c->qt_ntriv = c->qt_eW + F * wpad;
    size_t nb16 = 0, nint = 0;
    qrt_sizes(N, (int)F, &nb16, &nint);
    cudaError_t e = cudaMemset(bf16_base, 0, nb16 * sizeof(__nv_bfloat16));
    if (e == cudaSuccess) e = cudaMemset(int_base, 0, nint * sizeof(int));
    if (e != cudaSuccess) return e;
    if (!make_map_sw128(&c->qt_mapC96, c->qt_C, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, kpad, F * mpad, kDMax, 96) ||
        !make_map_sw128(&c->qt_mapC112, c->qt_C, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, kpad, F * mpad, kDMax, 112) ||
        !make_map_sw128(&c->qt_mapV1_32, c->qt_V1, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, kpad, F * kVRows, kDMax, 32) ||
        !make_map_sw128(&c->qt_mapV1_16, c->qt_V1, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, kpad, F * kVRows, kDMax, 16) ||
        !make_map_sw128(&c->qt_mapV2, c->qt_V2, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 64, F * mpad, kDMax, 128) ||
        !make_map_sw128(&c->qt_mapW, c->qt_W, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, 64, F * wpad, kDMax, kNC))
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

// From three panels on, four launches a panel against one in all: with few fields FP64 FMAs are faster up to about 100
// sites, with many the products from 66 on. The path may not depend on the number of fields (the split into batches
// leaves results as they are), so the line lies where what either side loses is even. FP64 evaluations with G, L = 40, FMAs
// / products, 1, 64, 152, 512 fields: N = 72 3.56 / 3.86, 4.01 / 4.39, 5.23 / 5.42, 11.6 / 11.2 ms; N = 81 4.16 / 4.44,
// 4.68 / 4.98, 6.13 / 6.27, 14.2 / 13.4; N = 100 5.88 / 6.12, 6.82 / 6.91, 9.15 / 8.76, 21.1 / 19.2; N = 132 7.59 / 7.71,
// 9.75 / 9.45, 14.2 / 13.2, 37.2 / 32.9.
constexpr int kFormQMinN = 81;

bool qrt_active(const slmc_ctx* c) { return c->qt_C && c->qr_path == 0 && qrt_supported(c->N); }

// The formation of Q in FP64 on the tensor cores: 4 launches per panel.
bool qrt_form_q_active(const slmc_ctx* c) { return qrt_active(c) && c->N >= kFormQMinN; }
int qrt_form_q_launches(const slmc_ctx* c) { return 1 + 4 * qrt_panels(c); }
cudaError_t qrt_form_q(slmc_ctx* c, int nf, cudaStream_t s) {
    return qr_panel_width(c) == 32 ? launch_form_q<32>(c, nf, s) : launch_form_q<16>(c, nf, s);
}

int qrt_panels(const slmc_ctx* c) {
    const int BP = qr_panel_width(c);
    return (c->N + BP - 1) / BP;
}

namespace {
template <int D>
cudaError_t panel(slmc_ctx* c, int nf, int t, cudaStream_t s) {
    if (nf <= c->num_sms)
        return qr_panel_width(c) == 32 ? launch_panel<32, 512, D>(c, nf, t, s) : launch_panel<16, 512, D>(c, nf, t, s);
    return qr_panel_width(c) == 32 ? launch_panel<32, 256, D>(c, nf, t, s) : launch_panel<16, 256, D>(c, nf, t, s);
}
template <int D>
cudaError_t trailing(slmc_ctx* c, int nf, int t, cudaStream_t s) {
    return qr_panel_width(c) == 32 ? launch_trailing<32, D>(c, nf, t, s) : launch_trailing<16, D>(c, nf, t, s);
}
}  // namespace

cudaError_t qrt_panel(slmc_ctx* c, int nf, int t, cudaStream_t s, bool eight) {
    return eight ? panel<8>(c, nf, t, s) : panel<7>(c, nf, t, s);
}

cudaError_t qrt_trailing(slmc_ctx* c, int nf, int t, cudaStream_t s, bool eight) {
    return eight ? trailing<8>(c, nf, t, s) : trailing<7>(c, nf, t, s);
}

}  // namespace slmc
