// FP64 determinant and Green's function of small lattices (N <= 64) in one launch, one CTA per field
// (small.cuh holds the steps and what bounds them): the general kernels are launch latency at these sizes, about 28
// launches for a determinant of 4x4, L = 40.
#include <algorithm>

#include "small.cuh"

namespace {

using namespace slmc::sm;

// ln|det|, sign and error flags of M from its pivots (warp 0 of the CTA, after lu).
template <int NMAX>
__device__ __forceinline__ void publish_det(Vecs<NMAX>& v, double* __restrict__ lndet, int* __restrict__ sign,
                                            unsigned int* __restrict__ err, int N, int sgn) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int k = lane; k < N; k += 32) s += log(fabs(v.key[k])) + fmax(v.lnd[k], 0.0);
    s = slmc::warp_allsum(s);
    if (lane == 0) {
        const bool ok = !v.sing && isfinite(s);
        *lndet = ok ? s : __longlong_as_double(0x7ff8000000000000ll);
        *sign = ok ? sgn * (v.neg ? -1 : 1) : 0;
        if (v.sing) atomicOr(err, SLMC_EBIT_SINGULAR);
        else if (!ok) atomicOr(err, SLMC_EBIT_NONFINITE);
    }
}

template <int NMAX, int LMAX>
__global__ void __launch_bounds__(Dim<NMAX>::threads, NMAX == 16 ? 4 : (NMAX == 32 ? 2 : 1)) k_small_logdet(const double* __restrict__ x, const double* __restrict__ kron,
                                                           double* __restrict__ lndet, int* __restrict__ sign,
                                                           double* __restrict__ Gout, unsigned int* __restrict__ err, int N,
                                                           int Lx, int Ly, int L, int n_s, double dtlam, double emu) {
    constexpr int ld = Dim<NMAX>::ld, NT = Dim<NMAX>::threads, RPT = Dim<NMAX>::rpt, G = Dim<NMAX>::G;
    extern __shared__ __align__(16) double dsm[];
    double* A = dsm;                       // packed QR, then M and its LU
    double* B = A + Dim<NMAX>::mat;        // U
    double* T = B + Dim<NMAX>::mat;
    Vecs<NMAX>& v = *reinterpret_cast<Vecs<NMAX>*>(T + Dim<NMAX>::mat);
    const int f = blockIdx.x, tid = threadIdx.x;
    const double* xf = x + (size_t)f * N * L;
    for (int idx = tid; idx < Dim<NMAX>::mat; idx += NT) {
        const double e = idx % (ld + 1) == 0 ? 1.0 : 0.0;
        B[idx] = e;
        T[idx] = e;
    }
    load_factors<NMAX>(v, kron, Lx, Ly);
    if (tid < N) v.lnd[tid] = 0.0;
    __syncthreads();
    bool bad = false;
    for (int l0 = 0; l0 < L; l0 += n_s) {
        slices<NMAX, LMAX>(B, v, xf, N, Lx, Ly, L, l0, min(L, l0 + n_s), dtlam, emu);
        qr<NMAX>(B, A, v, N);
        t_update<NMAX>(A, T, v, N);
        form_q<NMAX>(A, B, v, N);
        if (tid < N) {
            v.lnd[tid] = v.lnn[tid];
            bad |= !isfinite(v.lnn[tid]);
        }
        __syncthreads();
    }
    if (bad) atomicOr(err, SLMC_EBIT_NONFINITE);
    // M = D_b^-1 U^T + D_s T
    if (tid < N) {
        v.e1[tid] = exp(-fmax(v.lnd[tid], 0.0));
        v.e2[tid] = exp(fmin(v.lnd[tid], 0.0));
    }
    __syncthreads();
    for (int idx = tid; idx < N * N; idx += NT) {
        const int j = idx / N, i = idx - j * N;
        A[j * ld + i] = fma(v.e1[i], B[i * ld + j], v.e2[i] * T[i * ld + j]);
    }
    __syncthreads();
    lu<NMAX>(A, v, N);
    if (tid < 32) publish_det<NMAX>(v, lndet + f, sign + f, err, N, (v.ntriv & 1) ? -1 : 1);
    if (!Gout) return;
    if (tid < N) v.beta[tid] = 1.0 / A[tid * ld + tid];
    __syncthreads();
    const int j = tid / G, g = tid % G;
    double b[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int r = G * q + g;
        const int sr = r < N ? v.src[r] : 0;
        b[q] = (j < N && r < N) ? v.e1[sr] * B[sr * ld + j] : 0.0;
    }
    lu_solve<NMAX>(A, v.beta, b, N);
    if (j < N)
#pragma unroll
        for (int q = 0; q < RPT; ++q)
            if (G * q + g < N) Gout[(size_t)f * N * N + (size_t)(G * q + g) * N + j] = b[q];
}

// The final step of the general kernels at these sizes: M assembled (or given in Yall), its LU in place, ln|det|
// and sign; src[r] = row of the right-hand side that lands in row r. The blocked LU spent 297 us on 43 fields of
// 8x8 (panels, interchanges and updates of one or two blocks, four block barriers per column), this
// 132 us; the solve 122 and 90 us.
template <int NMAX>
__global__ void __launch_bounds__(Dim<NMAX>::threads) k_small_lu(const double* __restrict__ Uall, const double* __restrict__ Tall,
                                                                 const double* __restrict__ lnD_all, double* __restrict__ Yall,
                                                                 int* __restrict__ src_all, const int* __restrict__ sgnU,
                                                                 double* __restrict__ lndet, int* __restrict__ sign,
                                                                 unsigned int* __restrict__ err, int N, int assemble) {
    constexpr int ld = Dim<NMAX>::ld, NT = Dim<NMAX>::threads;
    extern __shared__ __align__(16) double dsm[];
    double* A = dsm;
    Vecs<NMAX>& v = *reinterpret_cast<Vecs<NMAX>*>(A + Dim<NMAX>::mat);
    const int f = blockIdx.x, tid = threadIdx.x;
    double* Y = Yall + (size_t)f * N * N;
    const double* U = Uall + (size_t)f * N * N;
    const double* T = Tall + (size_t)f * N * N;
    if (tid < N) {
        const double l = lnD_all[(size_t)f * N + tid];
        v.lnd[tid] = l;
        v.e1[tid] = exp(-fmax(l, 0.0));
        v.e2[tid] = exp(fmin(l, 0.0));
    }
    __syncthreads();
    for (int idx = tid; idx < N * N; idx += NT) {  // j fastest: U and T are read along rows i
        const int i = idx / N, j = idx - i * N;
        if (assemble) A[j * ld + i] = fma(v.e1[i], U[idx], v.e2[i] * T[idx]);
        else A[i * ld + j] = Y[idx];
    }
    __syncthreads();
    lu<NMAX>(A, v, N);
    if (tid < 32) publish_det<NMAX>(v, lndet + f, sign + f, err, N, sgnU[f]);
    for (int idx = tid; idx < N * N; idx += NT) Y[idx] = A[idx / N * ld + idx % N];
    if (tid < N) src_all[(size_t)f * N + tid] = v.src[tid];
}

// G = M^-1 D_b^-1 U^T with the factors of k_small_lu, a group of lanes per column.
template <int NMAX>
__global__ void __launch_bounds__(Dim<NMAX>::threads) k_small_greens(const double* __restrict__ Yall,
                                                                     const int* __restrict__ src_all,
                                                                     const double* __restrict__ Uall,
                                                                     const double* __restrict__ lnD_all,
                                                                     double* __restrict__ Gall, int N) {
    constexpr int ld = Dim<NMAX>::ld, NT = Dim<NMAX>::threads, RPT = Dim<NMAX>::rpt, G = Dim<NMAX>::G;
    extern __shared__ __align__(16) double dsm[];
    double* A = dsm;
    double* rd = A + Dim<NMAX>::mat;  // reciprocal pivots
    double* e1 = rd + NMAX;           // D_b^-1
    const int f = blockIdx.x, tid = threadIdx.x;
    const size_t NN = (size_t)N * N;
    for (int idx = tid; idx < N * N; idx += NT) A[idx / N * ld + idx % N] = Yall[f * NN + idx];
    if (tid < N) e1[tid] = exp(-fmax(lnD_all[(size_t)f * N + tid], 0.0));
    __syncthreads();
    if (tid < N) rd[tid] = 1.0 / A[tid * ld + tid];
    __syncthreads();
    const int j = tid / G, g = tid % G;
    double b[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int r = G * q + g, sr = r < N ? src_all[(size_t)f * N + r] : 0;
        b[q] = (j < N && r < N) ? e1[sr] * Uall[f * NN + (size_t)sr * N + j] : 0.0;
    }
    lu_solve<NMAX>(A, rd, b, N);
    if (j < N)
#pragma unroll
        for (int q = 0; q < RPT; ++q)
            if (G * q + g < N) Gall[f * NN + (size_t)(G * q + g) * N + j] = b[q];
}

template <int NMAX>
cudaError_t launch_small_lu(slmc_ctx* c, int nf, double* lndet, int* sign, cudaStream_t s, bool assemble) {
    const size_t smem = (size_t)Dim<NMAX>::mat * sizeof(double) + sizeof(Vecs<NMAX>);
    cudaError_t e = slmc::allow_smem(k_small_lu<NMAX>, smem);
    if (e != cudaSuccess) return e;
    k_small_lu<NMAX><<<nf, Dim<NMAX>::threads, smem, s>>>(c->U, c->Ta, c->lnD, c->Y, c->piv, c->sgnU, lndet, sign, c->err,
                                                         c->N, assemble ? 1 : 0);
    return cudaGetLastError();
}

template <int NMAX>
cudaError_t launch_small_greens(slmc_ctx* c, int nf, double* G, cudaStream_t s) {
    const size_t smem = ((size_t)Dim<NMAX>::mat + 2 * NMAX) * sizeof(double);
    cudaError_t e = slmc::allow_smem(k_small_greens<NMAX>, smem);
    if (e != cudaSuccess) return e;
    k_small_greens<NMAX><<<nf, Dim<NMAX>::threads, smem, s>>>(c->Y, c->piv, c->U, c->lnD, G, c->N);
    return cudaGetLastError();
}

template <int NMAX, int LMAX>
cudaError_t launch_small(slmc_ctx* c, const double* x, int nf, double* lndet, int* sign, double* G, cudaStream_t s) {
    const size_t smem = 3 * (size_t)Dim<NMAX>::mat * sizeof(double) + sizeof(Vecs<NMAX>);
    cudaError_t e = slmc::allow_smem(k_small_logdet<NMAX, LMAX>, smem);
    if (e != cudaSuccess) return e;
    k_small_logdet<NMAX, LMAX><<<nf, Dim<NMAX>::threads, smem, s>>>(x, c->kron, lndet, sign, G, c->err, c->N, c->p.Lx, c->p.Ly, c->L,
                                                         c->p.n_s, c->p.dtau * c->p.lambda, exp(c->p.dtau * c->p.mu));
    return cudaGetLastError();
}

}  // namespace

namespace slmc {

cudaError_t small_final_lu(slmc_ctx* c, int nf, double* lndet, int* sign, cudaStream_t s, bool assemble) {
    if (c->N <= 16) return launch_small_lu<16>(c, nf, lndet, sign, s, assemble);
    if (c->N <= 32) return launch_small_lu<32>(c, nf, lndet, sign, s, assemble);
    return launch_small_lu<64>(c, nf, lndet, sign, s, assemble);
}

cudaError_t small_final_greens(slmc_ctx* c, int nf, double* G, cudaStream_t s) {
    if (c->N <= 16) return launch_small_greens<16>(c, nf, G, s);
    if (c->N <= 32) return launch_small_greens<32>(c, nf, G, s);
    return launch_small_greens<64>(c, nf, G, s);
}

bool small_active(const slmc_ctx* c) {
    return c->N <= kSmallN && c->kron && c->p.precision == SLMC_PREC_FP64 && c->p.qr_mode == SLMC_QR_PREPIVOT &&
           c->qr_path == 0 && c->tt_path == 0 && !c->dense_slices && c->tune_qr_panel == 0 &&
           c->tune_qr_cluster == 0 && !c->nsub_set;
}

cudaError_t small_logdet(slmc_ctx* c, const double* x, int nf, double* lndet, int* sign, double* G, cudaStream_t s) {
    const int lm = std::max(c->p.Lx, c->p.Ly);  // at most N / 2: 8, 16 and 32 in the three size classes
    if (c->N <= 16) return launch_small<16, 8>(c, x, nf, lndet, sign, G, s);
    if (c->N <= 32)
        return lm <= 8 ? launch_small<32, 8>(c, x, nf, lndet, sign, G, s) : launch_small<32, 16>(c, x, nf, lndet, sign, G, s);
    if (lm <= 8) return launch_small<64, 8>(c, x, nf, lndet, sign, G, s);
    return lm <= 16 ? launch_small<64, 16>(c, x, nf, lndet, sign, G, s) : launch_small<64, 32>(c, x, nf, lndet, sign, G, s);
}

}  // namespace slmc
