// Device code of the small-lattice FP64 path (N <= 64): one CTA carries one field's whole stabilised
// product in shared memory -- slices, pre-pivoted Householder QR, Q, T, and the final LU and solve --
// so a determinant is one launch instead of several per slice group, and nothing goes through global memory
// but the field and the result.
//
// What bounds it: for N <= 36 the chain of column steps; for N = 64 the FP64 pipe (an SM issues one FP64 warp
// instruction per 16 to 19 cycles). One warp issues one per 64 cycles, however many lanes are active and however
// independent they are, so the chain is as long as the number of FP64 instructions one warp runs in sequence. Columns
// are held in registers by groups of G lanes: thread G j + g owns rows g, g + G, ... of column j, so a dot product is a
// run of FMAs per thread and log2 G additions across the group (a column per warp would spend five of every nine on the
// reduction); square root and divisions are short Newton forms, the two divisions of a reflector in neighbouring lanes
// of one instruction stream; and a group's slice scales are exponentiated together before its slices. With G, L = 40,
// 64 fields of 4x4 take 242 us (general kernels, a launch per step: 784), 16 of 2x32 2.3 ms (5.0), although the instance
// for lines of 17 to 32 sites spills (2.7 KB of registers per thread).
//
// Matrices in shared memory: element (r, c) of a column-major one at c * ld + r, of a row-major one at
// r * ld + c, ld = NMAX + 1; rows and columns beyond N are zero.
#pragma once

#include <cfloat>

#include "circ.cuh"
#include "fast_fp64.cuh"
#include "slmc_internal.cuh"

namespace slmc {
namespace sm {

template <int NMAX>
struct Dim {
    static constexpr int G = 8;  // lanes per column
    static constexpr int ld = NMAX + 1, mat = NMAX * ld, threads = G * NMAX, rpt = NMAX / G, cpw = 32 / G;
};
constexpr int kScMax = 16;  // slices whose scales are formed together

constexpr int kSmallCoef = 481;  // circ::ncoef of the longest line (31: one level; 32 folds twice)
static_assert(circ::ncoef(31) <= kSmallCoef && circ::ncoef(32) <= kSmallCoef && circ::ncoef(30) <= kSmallCoef, "");

// Vectors of one field in shared memory.
template <int NMAX>
struct Vecs {
    double lnd[NMAX], lnn[NMAX];   // ln D, new ln D
    double key[NMAX], e1[NMAX], e2[NMAX], tau[NMAX], beta[NMAX];
    double sc[kScMax][NMAX];       // slice scales of a group
    double cx[kSmallCoef], cy[kSmallCoef];  // folded coefficients of E_x, E_y
    double lbuf[2][NMAX];          // multipliers of the current / next LU step
    int perm[NMAX];
    int src[NMAX];                 // row interchanges as a permutation
    int piv[2];
    int ntriv, wide, neg, sing;
};

template <int G>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One pass of a transform over short lines (n <= 8, the 4x4 class): two lanes per line, each half of the outputs by
// direct sums (t: the factor less the identity). At this size the folded transform's chain (18 FP64 instructions for a
// line of 4 on two warps) is longer than eight direct ones on four.
template <int n>
__device__ __forceinline__ void half_line(double* g, int stride, const double* __restrict__ t, int half,
                                          const double* out_sc, bool on) {
    constexpr int nh = (n + 1) / 2;
    double v[n], y[nh];
#pragma unroll
    for (int m = 0; m < n; ++m) v[m] = g[m * stride];
#pragma unroll
    for (int o = 0; o < nh; ++o) {
        const int d = half * nh + o;
        y[o] = fma(t[d < n ? d : 0], v[0], half ? v[nh + o < n ? nh + o : 0] : v[o]);
#pragma unroll
        for (int m = 1; m < n; ++m) y[o] = fma(t[d >= m ? (d < n ? d - m : 0) : d - m + n], v[m], y[o]);
        if (out_sc) y[o] *= out_sc[(d < n ? d : 0) * stride];
    }
    __syncwarp();
#pragma unroll
    for (int o = 0; o < nh; ++o)
        if (on && half * nh + o < n) g[(half * nh + o) * stride] = y[o];
}

template <int NMAX>
__device__ __forceinline__ void short_pass(double* P, const double* __restrict__ t, const double* out_sc, int N,
                                           int n, int lines, int step_l, int stride) {
    constexpr int ld = Dim<NMAX>::ld, NT = Dim<NMAX>::threads;
    for (int q0 = 0; q0 < 2 * N * lines; q0 += NT) {  // uniform trip count: the halves meet at a warp barrier
        const int q = q0 + threadIdx.x, li = (q >> 1) / N, jj = (q >> 1) - li * N, o = li * step_l;
        const bool on = q < 2 * N * lines;
        double* g = P + (on ? jj * ld + o : 0);
#define SLMC_SHORT(k) \
    case k: half_line<k>(g, stride, t, q & 1, out_sc ? out_sc + (on ? o : 0) : nullptr, on); break;  // off lanes: no store
        switch (n) {
            SLMC_SHORT(2) SLMC_SHORT(3) SLMC_SHORT(4) SLMC_SHORT(5) SLMC_SHORT(6) SLMC_SHORT(7) SLMC_SHORT(8)
        }
#undef SLMC_SHORT
    }
}

// P <- B_{c1} ... B_{c0} P for the field columns c0 .. c1 - 1 in order: circulant transforms along the x and the y lines
// of every column, then the slice's scales.
// v.cx, v.cy: folded coefficients, or the factors less the identity for NMAX = 16 (short_pass).
template <int NMAX, int LMAX>
__device__ __forceinline__ void slices(double* P, Vecs<NMAX>& v, const double* __restrict__ xf, int N, int Lx, int Ly,
                                       int L, int c0, int c1, double dtlam, double emu) {
    constexpr int ld = Dim<NMAX>::ld, NT = Dim<NMAX>::threads;
    const int tid = threadIdx.x;
    for (int b0 = c0; b0 < c1; b0 += kScMax) {
        const int nb = min(kScMax, c1 - b0);  // field columns of this batch, in the order of the slices
        for (int idx = tid; idx < nb * N; idx += NT) {
            const int i = idx / nb, k = idx - i * nb;
            v.sc[k][i] = exp(-dtlam * xf[(size_t)i * L + b0 + k]) * emu;
        }
        __syncthreads();
        for (int k = 0; k < nb; ++k)
            for (int pass = 0; pass < 2; ++pass) {
                const int lines = pass ? Lx : Ly, step_l = pass ? 1 : Lx, stride = pass ? Lx : 1, n = pass ? Ly : Lx;
                const double* out_sc = pass ? v.sc[k] : nullptr;
                if constexpr (NMAX == 16) {
                    short_pass<NMAX>(P, pass ? v.cy : v.cx, out_sc, N, n, lines, step_l, stride);
                } else {
                    for (int q = tid; q < N * lines; q += NT) {
                        const int li = q / N, jj = q - li * N, o = li * step_l;
                        circ::apply_any<LMAX>(n, P + jj * ld + o, stride, pass ? v.cy : v.cx, nullptr, 0,
                                              out_sc ? out_sc + o : nullptr, stride);
                    }
                }
                __syncthreads();
            }
    }
}

// The transform's coefficients into v.cx, v.cy (caller synchronises).
template <int NMAX>
__device__ __forceinline__ void load_factors(Vecs<NMAX>& v, const double* __restrict__ kron, int Lx, int Ly) {
    constexpr int NT = Dim<NMAX>::threads;
    if constexpr (NMAX == 16) {
        if (threadIdx.x < 8) {
            v.cx[threadIdx.x] = kron[kKronMaxLine + threadIdx.x];
            v.cy[threadIdx.x] = kron[2 * kKronTab + kKronMaxLine + threadIdx.x];
        }
    } else {
        circ::build(v.cx, kron + kKronMaxLine, Lx, threadIdx.x, NT);
        circ::build(v.cy, kron + 2 * kKronTab + kKronMaxLine, Ly, threadIdx.x, NT);
    }
}

// Reflector of column j = k (its group calls it; rows before G kq are final): beta, tau, v into the packed column k
// of A (R above the diagonal, beta on it, v below).
template <int NMAX>
__device__ __forceinline__ void reflector(double (&a)[Dim<NMAX>::rpt], int kq, int kg, int k, int N, int g, bool mine,
                                          double* A, Vecs<NMAX>& v) {
    constexpr int ld = Dim<NMAX>::ld, RPT = Dim<NMAX>::rpt, G = Dim<NMAX>::G;
    double alpha = 0.0, sig = 0.0;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        if (q < kq || G * q >= N) continue;
        if (q == kq) {
            if (g == kg) alpha = a[q];
            if (g > kg) sig = a[q] * a[q];
        } else {
            sig = fma(a[q], a[q], sig);
        }
    }
    sig = group_sum<G>(sig);
    alpha = __shfl_sync(0xffffffffu, alpha, (threadIdx.x & (32 - G)) + kg);
    double tau = 0.0, beta = alpha, scal = 0.0;
    const bool refl = mine && sig != 0.0;
    if (refl) {
        const double nrm = fast_sqrt(fma(alpha, alpha, sig));
        beta = (alpha >= 0.0) ? -nrm : nrm;
        // tau = (beta - alpha) / beta in the even lanes, scal = 1 / (alpha - beta) in the odd ones
        const double d = beta - alpha;
        const double r = fast_div((g & 1) ? -1.0 : d, (g & 1) ? d : beta);
        const double o = __shfl_xor_sync(((1u << G) - 1u) << (threadIdx.x & (32 - G)), r, 1);
        tau = (g & 1) ? o : r;
        scal = (g & 1) ? r : o;
    }
    if (mine) {
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = G * q + g;
            if (r < N) A[k * ld + r] = r < k ? a[q] : (r == k ? beta : a[q] * scal);
        }
        if (g == 0) {
            v.tau[k] = tau;
            v.beta[k] = beta;
            if (tau != 0.0) v.ntriv += 1;
        }
    }
}

// Pre-pivoted Householder QR of P (column-major) with the columns in the order of ||p_j|| D_j: packed factors
// into A (logical order), tau, beta, perm, new ln D in v.lnn; the scaled factor D'^-1 R D P replaces R in A
// (unit diagonal signs). Returns the parity count of reflectors in v.ntriv.
template <int NMAX>
__device__ void qr(const double* P, double* A, Vecs<NMAX>& v, int N) {
    constexpr int ld = Dim<NMAX>::ld, NT = Dim<NMAX>::threads, RPT = Dim<NMAX>::rpt, G = Dim<NMAX>::G;
    constexpr int CPW = Dim<NMAX>::cpw;
    const int tid = threadIdx.x, j = tid / G, g = tid % G, lane = tid & 31;
    double a[RPT];
    if (tid == 0) {
        v.ntriv = 0;
        v.wide = 0;
    }
    {   // squared norms and keys
        double mx = -DBL_MAX;
        for (int i = lane; i < N; i += 32) mx = fmax(mx, v.lnd[i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = G * q + g;
            const double p = (j < N && r < N) ? P[j * ld + r] : 0.0;
            s = fma(p, p, s);
        }
        s = group_sum<G>(s);
        const double key = s * exp(2.0 * ((j < N ? v.lnd[j] : 0.0) - mx));
        if (j < N && g == 0) v.key[j] = (key >= 0.0) ? key : -1.0;  // NaN sorts last and keeps ranks unique
    }
    __syncthreads();
    if (tid < N) {
        const long long kj = __double_as_longlong(v.key[tid]);
        int r = 0;
        for (int i = 0; i < N; ++i) {
            const long long ki = __double_as_longlong(v.key[i]);
            r += (ki > kj) || (ki == kj && i < tid);
        }
        v.perm[r] = tid;
        if (fabs(v.lnd[tid]) > 600.0) v.wide = 1;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int r = G * q + g;
        a[q] = (j < N && r < N) ? P[v.perm[j < N ? j : 0] * ld + r] : 0.0;
    }
    if (tid < 32) reflector<NMAX>(a, 0, 0, 0, N, g, j == 0, A, v);
    __syncthreads();
    // step k applies reflector k to the columns right of it; the warp of column k + 1 then forms reflector k + 1
    // (one barrier per step)
#pragma unroll
    for (int kq = 0; kq < RPT; ++kq) {
        if (G * kq >= N) break;
        for (int kg = 0; kg < G; ++kg) {
            const int k = G * kq + kg;
            if (k + 1 >= N) break;
            const int jlast = (tid | 31) / G;  // last column of the warp
            if (jlast > k) {
                const double tau = v.tau[k];
                double vv[RPT], d = 0.0;
#pragma unroll
                for (int q = kq; q < RPT; ++q) {
                    if (G * q >= N) continue;
                    const int r = G * q + g;
                    vv[q] = (r < N) ? A[k * ld + r] : 0.0;
                    if (q == kq) vv[q] = g == kg ? 1.0 : (g > kg ? vv[q] : 0.0);
                    d = fma(vv[q], a[q], d);
                }
                d = group_sum<G>(d) * tau;
                if (j > k) {
#pragma unroll
                    for (int q = kq; q < RPT; ++q) {
                        if (G * q >= N) continue;
                        a[q] = fma(-d, vv[q], a[q]);
                    }
                }
                if ((k + 1) / CPW == tid >> 5) {  // the warp that holds column k + 1
                    const int g1 = (kg + 1) % G;
                    if (kg < G - 1) reflector<NMAX>(a, kq, g1, k + 1, N, g, j == k + 1, A, v);
                    else reflector<NMAX>(a, kq + 1, g1, k + 1, N, g, j == k + 1, A, v);
                }
            }
            __syncthreads();
        }
    }
    if (tid < N) {
        const int pc = v.perm[tid];
        const double l = log(fabs(v.beta[tid])) + v.lnd[pc];
        v.lnn[tid] = l;
        v.e1[tid] = exp(v.lnd[pc]);
        v.e2[tid] = exp(-l);
        if (fabs(l) > 600.0) v.wide = 1;
    }
    __syncthreads();
    const bool wide = v.wide != 0;
    for (int idx = tid; idx < N * N; idx += NT) {
        const int k = idx / N, i = idx - k * N;
        if (i > k) continue;
        double& e = A[k * ld + i];
        if (i == k) e = v.beta[k] >= 0.0 ? 1.0 : -1.0;
        else e = wide ? e * exp(v.lnd[v.perm[k]] - v.lnn[i]) : e * v.e1[k] * v.e2[i];
    }
    __syncthreads();
}

// T <- Rt P^T T in place (T row-major, Rt in the upper triangle of A): TX x TY entries per thread.
template <int NMAX>
__device__ void t_update(const double* A, double* T, const Vecs<NMAX>& v, int N) {
    constexpr int ld = Dim<NMAX>::ld, NTH = Dim<NMAX>::threads;
    constexpr int TX = NMAX * NMAX / NTH >= 16 ? 4 : (NMAX * NMAX / NTH >= 4 ? 2 : 1), TY = NMAX * NMAX / NTH / TX;
    static_assert(TX * TY * NTH == NMAX * NMAX && TY >= 1, "one tile per thread");
    constexpr int TT = NMAX / TY;
    const int i0 = threadIdx.x / TT * TX, j0 = threadIdx.x % TT * TY;
    const bool on = i0 < N && j0 < N;
    double acc[TX][TY];
#pragma unroll
    for (int x = 0; x < TX; ++x)
#pragma unroll
        for (int y = 0; y < TY; ++y) acc[x][y] = 0.0;
    if (on)
        for (int k = i0; k < N; ++k) {
            double a[TX], b[TY];
            const double* Tk = T + v.perm[k] * ld + j0;
#pragma unroll
            for (int x = 0; x < TX; ++x) a[x] = (i0 + x <= k) ? A[k * ld + i0 + x] : 0.0;
#pragma unroll
            for (int y = 0; y < TY; ++y) b[y] = Tk[y];
#pragma unroll
            for (int x = 0; x < TX; ++x)
#pragma unroll
                for (int y = 0; y < TY; ++y) acc[x][y] = fma(a[x], b[y], acc[x][y]);
        }
    __syncthreads();
    if (on)
#pragma unroll
        for (int x = 0; x < TX; ++x)
#pragma unroll
            for (int y = 0; y < TY; ++y)
                if (i0 + x < N && j0 + y < N) T[(i0 + x) * ld + j0 + y] = acc[x][y];
}

// Q (column-major) from the packed reflectors of A, accumulated backwards; a group per column, no barriers.
template <int NMAX>
__device__ void form_q(const double* A, double* Q, const Vecs<NMAX>& v, int N) {
    constexpr int ld = Dim<NMAX>::ld, RPT = Dim<NMAX>::rpt, G = Dim<NMAX>::G;
    const int tid = threadIdx.x, j = tid / G, g = tid % G;
    double x[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) x[q] = (G * q + g == j) ? 1.0 : 0.0;
    const int jlast = (tid | 31) / G;
#pragma unroll
    for (int kq = RPT - 1; kq >= 0; --kq) {
        if (G * kq >= N) continue;
        for (int kg = G - 1; kg >= 0; --kg) {
            const int k = G * kq + kg;
            if (k >= N || k > jlast) continue;  // columns left of k are still unit vectors
            double vv[RPT], d = 0.0;
#pragma unroll
            for (int q = kq; q < RPT; ++q) {
                if (G * q >= N) continue;
                const int r = G * q + g;
                vv[q] = (r < N) ? A[k * ld + r] : 0.0;
                if (q == kq) vv[q] = g == kg ? 1.0 : (g > kg ? vv[q] : 0.0);
                d = fma(vv[q], x[q], d);
            }
            d = group_sum<G>(d) * v.tau[k];
#pragma unroll
            for (int q = kq; q < RPT; ++q) {
                if (G * q >= N) continue;
                x[q] = fma(-d, vv[q], x[q]);
            }
        }
    }
    if (j < N)
#pragma unroll
        for (int q = 0; q < RPT; ++q)
            if (G * q + g < N) Q[j * ld + G * q + g] = x[q];
}

// Pivot search and multipliers of column k of M (column-major) by one warp: rows k.. of the column, the chosen row,
// the interchanged multipliers into v.lbuf[k & 1]; the column itself is written back factored.
template <int NMAX>
__device__ __forceinline__ void lu_column(double* M, Vecs<NMAX>& v, int k, int N, int lane) {
    constexpr int ld = Dim<NMAX>::ld, R = (NMAX + 31) / 32;
    double* col = M + k * ld;
    double c[R];
    long long bv = -1;
    int bi = N;
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int r = lane + 32 * t;
        c[t] = (r < N) ? col[r] : 0.0;
        if (r >= k && r < N) {  // bit patterns of |c| order as the values do; NaN never wins a comparison in FP64
            const double m = fabs(c[t]);
            const long long b = (m == m) ? __double_as_longlong(m) : -1;
            if (b > bv) {
                bv = b;
                bi = r;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > bv || (ov == bv && oi < bi)) {
            bv = ov;
            bi = oi;
        }
    }
    if (bi >= N) bi = k;  // no comparable entry (NaN column): no interchange
    double pval = col[bi], top = col[k];
    const double rinv = (pval != 0.0) ? fast_div(1.0, pval) : 0.0;
    __syncwarp();
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int r = lane + 32 * t;
        if (r < k || r >= N) continue;
        const double e = r == bi ? top : c[t];
        const double l = r == k ? pval : e * rinv;
        col[r] = l;
        v.lbuf[k & 1][r] = l;
    }
    if (lane == 0) {
        v.piv[k & 1] = bi;
        if (pval == 0.0) v.sing = 1;
        v.key[k] = pval;
        v.neg ^= (pval < 0.0) ^ (bi != k);
        const int t = v.src[k];
        v.src[k] = v.src[bi];
        v.src[bi] = t;
    }
}

// LU with partial pivoting of M (column-major) in place: warps own columns, the warp of column k + 1 factors it
// right after its update (one barrier per step). v.src: row of the right-hand side that lands in each row;
// v.key: the pivots; v.neg / v.sing: sign and singularity.
template <int NMAX>
__device__ void lu(double* M, Vecs<NMAX>& v, int N) {
    constexpr int ld = Dim<NMAX>::ld, NW = Dim<NMAX>::threads / 32, R = (NMAX + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < N; i += Dim<NMAX>::threads) v.src[i] = i;
    if (threadIdx.x == 0) {
        v.neg = 0;
        v.sing = 0;
    }
    __syncthreads();
    if (warp == 0) lu_column<NMAX>(M, v, 0, N, lane);
    __syncthreads();
    for (int k = 0; k < N; ++k) {
        const int p = v.piv[k & 1];
        double l[R];
#pragma unroll
        for (int t = 0; t < R; ++t) {
            const int r = lane + 32 * t;
            l[t] = (r > k && r < N) ? v.lbuf[k & 1][r] : 0.0;
        }
        // the column of the next step first: its warp factors it while the others still update
        const int next = k + 1;
        if (next < N && next % NW == warp) {
            double* col = M + next * ld;
            const double u = col[p], t0 = col[k];
            __syncwarp();
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const int r = lane + 32 * t;
                if (r < k || r >= N) continue;
                const double e = r == p ? t0 : col[r];
                col[r] = r == k ? u : fma(-l[t], u, e);
            }
            __syncwarp();
            lu_column<NMAX>(M, v, next, N, lane);
        }
        // the warp's other columns, two at a time (independent loads); earlier ones only take the interchange
        for (int c0 = warp; c0 < N; c0 += 2 * NW) {
            double u[2], e[2][R];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = c0 + h * NW;
                if (c >= N || c == k || c == next) continue;
                const double* col = M + c * ld;
                u[h] = col[p];
                const double t0 = col[k];
#pragma unroll
                for (int t = 0; t < R; ++t) {
                    const int r = lane + 32 * t;
                    e[h][t] = (r < k || r >= N) ? 0.0 : (r == p ? t0 : col[r]);
                }
            }
            __syncwarp();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = c0 + h * NW;
                if (c >= N || c == k || c == next) continue;
                double* col = M + c * ld;
#pragma unroll
                for (int t = 0; t < R; ++t) {
                    const int r = lane + 32 * t;
                    if (r < k || r >= N) continue;
                    col[r] = r == k ? u[h] : (c < k ? e[h][t] : fma(-l[t], u[h], e[h][t]));
                }
            }
        }
        __syncthreads();
    }
}

// Right-hand side column j in group registers (row G q + g in x[q]): x <- U'^-1 L^-1 x with the factors in M and
// the reciprocal pivots rd.
template <int NMAX>
__device__ __forceinline__ void lu_solve(const double* M, const double* rd, double (&x)[Dim<NMAX>::rpt], int N) {
    constexpr int ld = Dim<NMAX>::ld, RPT = Dim<NMAX>::rpt, G = Dim<NMAX>::G;
    const int g = threadIdx.x % G, q0 = threadIdx.x & (32 - G);
#pragma unroll
    for (int kq = 0; kq < RPT; ++kq) {
        if (G * kq >= N) break;
        for (int kg = 0; kg < G; ++kg) {
            const int k = G * kq + kg;
            if (k >= N) break;
            const double xk = __shfl_sync(0xffffffffu, x[kq], q0 + kg);
#pragma unroll
            for (int q = kq; q < RPT; ++q) {
                const int r = G * q + g;
                if (G * q >= N) continue;
                if (r > k && r < N) x[q] = fma(-M[k * ld + r], xk, x[q]);
            }
        }
    }
#pragma unroll
    for (int kq = RPT - 1; kq >= 0; --kq) {
        if (G * kq >= N) continue;
        for (int kg = G - 1; kg >= 0; --kg) {
            const int k = G * kq + kg;
            if (k >= N) continue;
            const double xk = __shfl_sync(0xffffffffu, x[kq], q0 + kg) * rd[k];
            if (g == kg) x[kq] = xk;
#pragma unroll
            for (int q = 0; q <= kq; ++q) {
                const int r = G * q + g;
                if (r < k) x[q] = fma(-M[k * ld + r], xk, x[q]);
            }
        }
    }
}

}  // namespace sm
}  // namespace slmc
