// Device code of the small-lattice FP64 path (N <= 64): one CTA carries one field's whole stabilised
// product in shared memory -- slices, pre-pivoted Householder QR, Q, T, and the final LU and solve --
// so a determinant is one launch instead of several per slice group, and nothing goes through global memory
// but the field and the result.
//
// What bounds it: for N <= 36 the chain of column steps (barriers, square roots, divisions); for N = 64 the
// FP64 pipe (two FMAs per clock per SM). Columns are held in registers by quads: thread 4 j + g owns rows g,
// g + 4, ... of column j, so a dot product is a run of FMAs per thread and two additions across the quad; a
// column per warp would spend five of every nine FP64 slots on the reduction at these sizes.
//
// Matrices in shared memory: element (r, c) of a column-major one at c * ld + r, of a row-major one at
// r * ld + c, ld = NMAX + 1; rows and columns beyond N are zero.
#pragma once

#include <cfloat>

#include "circ.cuh"
#include "slmc_internal.cuh"

namespace slmc {
namespace sm {

template <int NMAX>
struct Dim {
    static constexpr int ld = NMAX + 1, mat = NMAX * ld, threads = 4 * NMAX, rpt = NMAX / 4;
};

constexpr int kSmallCoef = 481;  // circ::ncoef of the longest line (31: one level; 32 folds twice)
static_assert(circ::ncoef(31) <= kSmallCoef && circ::ncoef(32) <= kSmallCoef && circ::ncoef(30) <= kSmallCoef, "");

// Vectors of one field in shared memory.
template <int NMAX>
struct Vecs {
    double lnd[NMAX], lnn[NMAX];   // ln D, new ln D
    double key[NMAX], e1[NMAX], e2[NMAX], tau[NMAX], beta[NMAX];
    double sc[NMAX];               // slice scales
    double cx[kSmallCoef], cy[kSmallCoef];  // folded coefficients of E_x, E_y
    double lbuf[2][NMAX];          // multipliers of the current / next LU step
    double logabs;
    int perm[NMAX];
    int src[NMAX];                 // row interchanges as a permutation
    int piv[2];
    int ntriv, wide, neg, sing;
};

__device__ __forceinline__ double quad_sum(double v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// P <- B_{c1} ... B_{c0} P (plain) for the field columns c0 .. c1 - 1 in order, or with trans the transposed
// slices E diag(s) from c1 - 1 down to c0: circulant transforms along the x and the y lines of every column.
template <int NMAX, int LMAX, bool kTrans>
__device__ __forceinline__ void slices(double* P, Vecs<NMAX>& v, const double* __restrict__ xf, int N, int Lx, int Ly,
                                       int L, int c0, int c1, double dtlam, double emu) {
    constexpr int ld = Dim<NMAX>::ld, NT = Dim<NMAX>::threads;
    const int tid = threadIdx.x;
    // the field column of the next slice is loaded a slice ahead (N <= NT: one site per thread)
    double xv = tid < N ? xf[(size_t)tid * L + (kTrans ? c1 - 1 : c0)] : 0.0;
    for (int step = 0; step < c1 - c0; ++step) {
        if (tid < N) v.sc[tid] = exp(-dtlam * xv) * emu;
        if (tid < N && step + 1 < c1 - c0) xv = xf[(size_t)tid * L + (kTrans ? c1 - 2 - step : c0 + step + 1)];
        if (kTrans) __syncthreads();  // the x pass scales its input; plain slices use sc after the next barrier
        for (int pass = 0; pass < 2; ++pass) {
            const int lines = pass ? Lx : Ly, step_l = pass ? 1 : Lx, stride = pass ? Lx : 1;
            for (int q = tid; q < N * lines; q += NT) {
                const int li = q / N, jj = q - li * N, o = li * step_l;
                circ::apply_any<LMAX>(pass ? Ly : Lx, P + jj * ld + o, stride, pass ? v.cy : v.cx,
                                      kTrans && pass == 0 ? v.sc + o : nullptr, stride,
                                      !kTrans && pass == 1 ? v.sc + o : nullptr, stride, 1.0);
            }
            __syncthreads();
        }
    }
}

// Reflector of column j = k (its quad calls it; rows q < kq are final): beta, tau, v into the packed column k of
// A (R above the diagonal, beta on it, v below).
template <int NMAX>
__device__ __forceinline__ void reflector(double (&a)[NMAX / 4], int kq, int kg, int k, int N, int g, bool mine, double* A,
                                          Vecs<NMAX>& v) {
    constexpr int ld = Dim<NMAX>::ld, RPT = NMAX / 4;
    double alpha = 0.0, sig = 0.0;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        if (q < kq || 4 * q >= N) continue;
        if (q == kq) {
            if (g == kg) alpha = a[q];
            if (g > kg) sig = a[q] * a[q];
        } else {
            sig = fma(a[q], a[q], sig);
        }
    }
    sig = quad_sum(sig);
    alpha = __shfl_sync(0xffffffffu, alpha, (threadIdx.x & 28) + kg);
    double tau = 0.0, beta = alpha, scal = 0.0;
    if (mine && sig != 0.0) {
        const double nrm = sqrt(fma(alpha, alpha, sig));
        beta = (alpha >= 0.0) ? -nrm : nrm;
        tau = (beta - alpha) / beta;
        scal = 1.0 / (alpha - beta);
    }
    if (mine) {
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = 4 * q + g;
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
    constexpr int ld = Dim<NMAX>::ld, NT = Dim<NMAX>::threads, RPT = NMAX / 4;
    const int tid = threadIdx.x, j = tid >> 2, g = tid & 3, lane = tid & 31;
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
            const int r = 4 * q + g;
            const double p = (j < N && r < N) ? P[j * ld + r] : 0.0;
            s = fma(p, p, s);
        }
        s = quad_sum(s);
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
        const int r = 4 * q + g;
        a[q] = (j < N && r < N) ? P[v.perm[j < N ? j : 0] * ld + r] : 0.0;
    }
    if (tid < 32) reflector<NMAX>(a, 0, 0, 0, N, g, j == 0, A, v);
    __syncthreads();
    // step k applies reflector k to the columns right of it; the warp of column k + 1 then forms reflector k + 1
    // (one barrier per step)
#pragma unroll
    for (int kq = 0; kq < RPT; ++kq) {
        if (4 * kq >= N) break;
        for (int kg = 0; kg < 4; ++kg) {
            const int k = 4 * kq + kg;
            if (k + 1 >= N) break;
            const int jlast = (tid | 31) >> 2;  // last column of the warp
            if (jlast > k) {
                const double tau = v.tau[k];
                double vv[RPT], d = 0.0;
#pragma unroll
                for (int q = kq; q < RPT; ++q) {
                    if (4 * q >= N) continue;
                    const int r = 4 * q + g;
                    vv[q] = (r < N) ? A[k * ld + r] : 0.0;
                    if (q == kq) vv[q] = g == kg ? 1.0 : (g > kg ? vv[q] : 0.0);
                    d = fma(vv[q], a[q], d);
                }
                d = quad_sum(d) * tau;
                if (j > k) {
#pragma unroll
                    for (int q = kq; q < RPT; ++q) {
                        if (4 * q >= N) continue;
                        a[q] = fma(-d, vv[q], a[q]);
                    }
                }
                if ((k + 1) >> 3 == tid >> 5) {  // the warp that holds column k + 1
                    const int g1 = (kg + 1) & 3;
                    if (kg < 3) reflector<NMAX>(a, kq, g1, k + 1, N, g, j == k + 1, A, v);
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

// T <- Rt P^T T in place (T row-major, Rt in the upper triangle of A): 4 x 4 entries per thread.
template <int NMAX>
__device__ void t_update(const double* A, double* T, const Vecs<NMAX>& v, int N) {
    constexpr int ld = Dim<NMAX>::ld, TT = NMAX / 4, NTH = Dim<NMAX>::threads;
    constexpr int PASS = (TT * TT + NTH - 1) / NTH;
    static_assert(PASS == 1, "one tile per thread");
    const int ti = threadIdx.x / TT, tj = threadIdx.x % TT;
    const bool on = threadIdx.x < TT * TT && 4 * ti < N && 4 * tj < N;
    double acc[4][4];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = 0.0;
    if (on)
        for (int k = 4 * ti; k < N; ++k) {
            double a[4], b[4];
            const double* Tk = T + v.perm[k] * ld + 4 * tj;
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                a[x] = (4 * ti + x <= k) ? A[k * ld + 4 * ti + x] : 0.0;
                b[x] = Tk[x];
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fma(a[x], b[y], acc[x][y]);
        }
    __syncthreads();
    if (on)
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y)
                if (4 * ti + x < N && 4 * tj + y < N) T[(4 * ti + x) * ld + 4 * tj + y] = acc[x][y];
}

// Q (column-major) from the packed reflectors of A, accumulated backwards; a quad per column, no barriers.
template <int NMAX>
__device__ void form_q(const double* A, double* Q, const Vecs<NMAX>& v, int N) {
    constexpr int ld = Dim<NMAX>::ld, RPT = NMAX / 4;
    const int tid = threadIdx.x, j = tid >> 2, g = tid & 3;
    double x[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) x[q] = (4 * q + g == j) ? 1.0 : 0.0;
    const int jlast = (tid | 31) >> 2;
#pragma unroll
    for (int kq = RPT - 1; kq >= 0; --kq) {
        if (4 * kq >= N) continue;
        for (int kg = 3; kg >= 0; --kg) {
            const int k = 4 * kq + kg;
            if (k >= N || k > jlast) continue;  // columns left of k are still unit vectors
            double vv[RPT], d = 0.0;
#pragma unroll
            for (int q = kq; q < RPT; ++q) {
                if (4 * q >= N) continue;
                const int r = 4 * q + g;
                vv[q] = (r < N) ? A[k * ld + r] : 0.0;
                if (q == kq) vv[q] = g == kg ? 1.0 : (g > kg ? vv[q] : 0.0);
                d = fma(vv[q], x[q], d);
            }
            d = quad_sum(d) * v.tau[k];
#pragma unroll
            for (int q = kq; q < RPT; ++q) {
                if (4 * q >= N) continue;
                x[q] = fma(-d, vv[q], x[q]);
            }
        }
    }
    if (j < N)
#pragma unroll
        for (int q = 0; q < RPT; ++q)
            if (4 * q + g < N) Q[j * ld + 4 * q + g] = x[q];
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
    const double rinv = (pval != 0.0) ? 1.0 / pval : 0.0;
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
        // the column of the next step first
        const int next = k + 1;
        const int start = next < N && next % NW == warp ? next : -1;
        for (int it = -1, j = warp; j < N || it < 0; ++it) {
            int c;
            if (it < 0) {
                if (start < 0) continue;
                c = start;
            } else {
                c = j;
                j += NW;
                if (c == start || c == k) continue;
            }
            double* col = M + c * ld;
            const double u = col[p], t0 = col[k];
            __syncwarp();
            if (c < k) {  // earlier columns only take the interchange
                if (lane == 0 && p != k) {
                    col[k] = u;
                    col[p] = t0;
                }
                __syncwarp();
                continue;
            }
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const int r = lane + 32 * t;
                if (r < k || r >= N) continue;
                const double e = r == p ? t0 : col[r];
                col[r] = r == k ? u : fma(-l[t], u, e);
            }
            __syncwarp();
            if (c == start) lu_column<NMAX>(M, v, next, N, lane);
        }
        __syncthreads();
    }
}

// Right-hand side column j in quad registers (row 4 q + g in x[q]): x <- U'^-1 L^-1 x with the factors in M and
// the reciprocal pivots rd.
template <int NMAX>
__device__ __forceinline__ void lu_solve(const double* M, const double* rd, double (&x)[NMAX / 4], int N) {
    constexpr int ld = Dim<NMAX>::ld, RPT = NMAX / 4;
    const int g = threadIdx.x & 3, q0 = threadIdx.x & 28;
#pragma unroll
    for (int kq = 0; kq < RPT; ++kq) {
        if (4 * kq >= N) break;
        for (int kg = 0; kg < 4; ++kg) {
            const int k = 4 * kq + kg;
            if (k >= N) break;
            const double xk = __shfl_sync(0xffffffffu, x[kq], q0 + kg);
#pragma unroll
            for (int q = kq; q < RPT; ++q) {
                const int r = 4 * q + g;
                if (4 * q >= N) continue;
                if (r > k && r < N) x[q] = fma(-M[k * ld + r], xk, x[q]);
            }
        }
    }
#pragma unroll
    for (int kq = RPT - 1; kq >= 0; --kq) {
        if (4 * kq >= N) continue;
        for (int kg = 3; kg >= 0; --kg) {
            const int k = 4 * kq + kg;
            if (k >= N) continue;
            const double xk = __shfl_sync(0xffffffffu, x[kq], q0 + kg) * rd[k];
            if (g == kg) x[kq] = xk;
#pragma unroll
            for (int q = 0; q <= kq; ++q) {
                const int r = 4 * q + g;
                if (r < k) x[q] = fma(-M[k * ld + r], xk, x[q]);
            }
        }
    }
}

}  // namespace sm
}  // namespace slmc
