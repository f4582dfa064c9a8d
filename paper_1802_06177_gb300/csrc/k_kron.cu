// FP64 slice-group products through the separable hopping exponential [Suppl. Eq. (S2)].
//
// On the periodic Lx x Ly lattice exp(-dtau K) = e^{dtau mu} E_x kron E_y exactly (the
// hopping along x and along y commute; E_x, E_y are symmetric circulant). Applying it to a
// column of the running product therefore takes N (Lx + Ly) FMAs, a circulant transform
// along every x line and every y line of the column, instead of the N^2 of a dense product:
// 8x fewer at 16 x 16. FP64 issue is the scarce resource of the FP64 path on this GPU, so
// this is the slice kernel of the FP64 mode.
//
//   plain:       Y = B_{l0+nsl} ... B_{l0+1} U,          B_l   = diag(s_l) E
//   transposed:  Y = B_{l0+1}^T ... B_{l0+nsl}^T U,      B_l^T = E diag(s_l)
// with s_l = exp(-dtau lambda x[:, l-1]). The transposed chain accumulates the products
// B(L, g0)^T = B_{g0+1}^T ... B_L^T that the DQMC updates combine with B(g0, 0) to obtain
// G(g0) without a full chain per recomputation.
//
// One CTA owns a panel of columns of one field in shared memory for all nsl slices (as the dense panel kernel does);
// within a slice, one pass transforms the x lines and one the y lines of every column. Two forms:
//   k_slice_oz    longer side 9..16: a warp takes the same line of 16 columns at a time through the tensor-instruction
//                 transform of oz_line.cuh;
//   k_slice_kron  other sides: a thread takes a line through the folded FP64 sums of circ.cuh, consecutive lanes the
//                 same line of consecutive columns.
// 12x12, L = 120, 256 fields: 65 ms of slice products by direct FP64 sums, 21.0 folded, 17.7 on the tensor
// instructions (16 lines and 16 outputs fill its tile best at sides 9..16). 18x10, L = 37, 50 fields: 7.8 ms direct, 2.1
// folded, 3.3 on the tensor instructions (two K steps, three column tiles for a line of 18); 8x8: half of each
// K step and tile would be padding.
// Layout: column-major N x N, element (i, j) at j*N + i, site i = ix + Lx iy; the panel's columns at the odd stride
// N | 1, so neither pass meets a bank conflict.
#include "circ.cuh"
#include "oz_line.cuh"
#include "slmc_internal.cuh"

namespace {

constexpr int kThreads = 128;
// Columns per CTA of the folded form: 32, a lane per column. From 27 x 32 sites on a panel of 32 columns, the slice
// scales and the coefficients of the two factors outgrow the 227 KB of a CTA; 24 columns fit up to 32 x 32.
constexpr int kNBF = 32, kNBFLarge = 24;

template <bool kTrans>
__global__ void __launch_bounds__(kThreads) k_slice_oz(const double* __restrict__ U, double* __restrict__ Y,
                                                         const double* __restrict__ x,
                                                         const double* __restrict__ kron, int Lx, int Ly, int L,
                                                         int l0, int nsl, double dtlam, double emu, int NB) {
    extern __shared__ __align__(16) double sm[];
    const int N = Lx * Ly, ld = N | 1;
    uint2* fx = reinterpret_cast<uint2*>(sm);  // digit fragments of E_x, E_y
    uint2* fy = fx + slmc::oz::frag_bytes(Lx) / 8;
    double* P = reinterpret_cast<double*>(fy + slmc::oz::frag_bytes(Ly) / 8);  // [NB][ld] panel, column-major
    double* sc = P + NB * ld;                                                  // [N] e^{dtau mu} s_l
    const int f = blockIdx.y, j0 = blockIdx.x * NB, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = min(NB, N - j0), groups = (nb + 15) / 16;
    const size_t NN = (size_t)N * N;
    const double* Uf = U + f * NN + (size_t)j0 * N;
    int shx, shy;
    const int ex = slmc::oz::build(fx, kron + slmc::kKronMaxLine, Lx, tid, kThreads, shx);
    const int ey = slmc::oz::build(fy, kron + 2 * slmc::kKronTab + slmc::kKronMaxLine, Ly, tid, kThreads, shy);
    for (int jj = warp; jj < nb; jj += kThreads / 32)
        for (int i = lane; i < N; i += 32) P[jj * ld + i] = Uf[(size_t)jj * N + i];
    const double* xf = x + (size_t)f * N * L;
    for (int step = 0; step < nsl; ++step) {
        const int c = kTrans ? l0 + nsl - 1 - step : l0 + step;  // field column of the slice
        for (int i = tid; i < N; i += kThreads) sc[i] = exp(-dtlam * xf[(size_t)i * L + c]) * emu;
        __syncthreads();
        // pass 0: x lines (contiguous; the transposed slice scales its input); pass 1: y lines (stride Lx; the
        // plain slice scales its output)
        for (int pass = 0; pass < 2; ++pass) {
            const int lines = pass ? Lx : Ly, step_l = pass ? 1 : Lx, stride = pass ? Lx : 1;
            for (int q = warp; q < lines * groups; q += kThreads / 32) {
                const int li = q / groups, j16 = (q - li * groups) * 16, o = li * step_l;
                slmc::oz::tile_any(P + j16 * ld + o, ld, min(16, nb - j16), stride, pass ? Ly : Lx, pass ? fy : fx,
                                      pass ? ey : ex, pass ? shy : shx, kTrans && pass == 0 ? sc + o : nullptr,
                                      !kTrans && pass == 1 ? sc + o : nullptr, stride);
            }
            __syncthreads();
        }
    }
    double* Yf = Y + f * NN + (size_t)j0 * N;
    for (int jj = warp; jj < nb; jj += kThreads / 32)
        for (int i = lane; i < N; i += 32) Yf[(size_t)jj * N + i] = P[jj * ld + i];
}

template <bool kTrans>
cudaError_t launch_oz(slmc_ctx* c, const double* x, int nf, int l0, int nsl, cudaStream_t s) {
    const int N = c->N;
    // columns per CTA: the widest of 64, 48, 32 that pads N least (each CTA forms the slice's scales again) and leaves
    // room for two CTAs per SM
    const size_t fixed = (size_t)slmc::oz::frag_bytes(c->p.Lx) + slmc::oz::frag_bytes(c->p.Ly) + N * sizeof(double);
    int NB = 32;
    for (int w = 48; w <= 64; w += 16)
        if ((N + w - 1) / w * w <= (N + NB - 1) / NB * NB && fixed + (size_t)w * (N | 1) * sizeof(double) <= 112 * 1024) NB = w;
    const size_t smem = fixed + (size_t)NB * (N | 1) * sizeof(double);
    cudaError_t e = slmc::allow_smem(k_slice_oz<kTrans>, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((N + NB - 1) / NB, nf);
    k_slice_oz<kTrans><<<grid, kThreads, smem, s>>>(c->U, c->Y, x, c->kron, c->p.Lx, c->p.Ly, c->L, l0, nsl,
                                                         c->p.dtau * c->p.lambda, exp(c->p.dtau * c->p.mu), NB);
    return cudaGetLastError();
}

template <int LMAX, bool kTrans>
__global__ void __launch_bounds__(kThreads) k_slice_kron(const double* __restrict__ U, double* __restrict__ Y,
                                                         const double* __restrict__ x,
                                                         const double* __restrict__ kron, int Lx, int Ly, int L,
                                                         int l0, int nsl, double dtlam, double emu, int NB) {
    extern __shared__ double sm[];
    const int N = Lx * Ly, ld = N | 1;
    double* P = sm;                // [NB][ld] panel, column-major
    double* sc = sm + NB * ld;     // [N] e^{dtau mu} s_l
    double* cx = sc + N;            // folded coefficients of E_x, E_y
    double* cy = cx + slmc::circ::ncoef(Lx);
    const int f = blockIdx.y, j0 = blockIdx.x * NB, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = min(NB, N - j0);
    const size_t NN = (size_t)N * N;
    const double* Uf = U + f * NN + (size_t)j0 * N;
    slmc::circ::build(cx, kron + slmc::kKronMaxLine, Lx, tid, kThreads);
    slmc::circ::build(cy, kron + 2 * slmc::kKronTab + slmc::kKronMaxLine, Ly, tid, kThreads);
    for (int jj = warp; jj < nb; jj += kThreads / 32)
        for (int i = lane; i < N; i += 32) P[jj * ld + i] = Uf[(size_t)jj * N + i];
    const double* xf = x + (size_t)f * N * L;
    double* Pl = P + lane * ld;  // this lane's column
    for (int step = 0; step < nsl; ++step) {
        const int c = kTrans ? l0 + nsl - 1 - step : l0 + step;  // field column of the slice
        for (int i = tid; i < N; i += kThreads) sc[i] = exp(-dtlam * xf[(size_t)i * L + c]) * emu;
        __syncthreads();
        // pass 0: x lines (contiguous; the transposed slice scales its input); pass 1: y lines (stride Lx; the
        // plain slice scales its output)
        for (int pass = 0; pass < 2; ++pass) {
            const int lines = pass ? Lx : Ly, step_l = pass ? 1 : Lx, stride = pass ? Lx : 1;
            if (lane < nb)
                for (int q = warp; q < lines; q += kThreads / 32) {
                    const int o = q * step_l;
                    slmc::circ::apply_any<LMAX>(pass ? Ly : Lx, Pl + o, stride, pass ? cy : cx,
                                                kTrans && pass == 0 ? sc + o : nullptr, stride,
                                                !kTrans && pass == 1 ? sc + o : nullptr, stride);
                }
            __syncthreads();
        }
    }
    double* Yf = Y + f * NN + (size_t)j0 * N;
    for (int jj = warp; jj < nb; jj += kThreads / 32)
        for (int i = lane; i < N; i += 32) Yf[(size_t)jj * N + i] = P[jj * ld + i];
}

template <int LMAX, bool kTrans>
cudaError_t launch_kron(slmc_ctx* c, const double* x, int nf, int l0, int nsl, cudaStream_t s) {
    const int N = c->N;
    const size_t fixed = (size_t)N + slmc::circ::ncoef(c->p.Lx) + slmc::circ::ncoef(c->p.Ly);
    const int NB = (fixed + (size_t)kNBF * (N | 1)) * sizeof(double) <= 227 * 1024 ? kNBF : kNBFLarge;
    const size_t smem = (fixed + (size_t)NB * (N | 1)) * sizeof(double);
    cudaError_t e = slmc::allow_smem(k_slice_kron<LMAX, kTrans>, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((N + NB - 1) / NB, nf);
    k_slice_kron<LMAX, kTrans><<<grid, kThreads, smem, s>>>(c->U, c->Y, x, c->kron, c->p.Lx, c->p.Ly, c->L, l0, nsl,
                                                            c->p.dtau * c->p.lambda, exp(c->p.dtau * c->p.mu), NB);
    return cudaGetLastError();
}

// LMAX: registers grow with the longest line expanded.
template <bool kTrans>
cudaError_t dispatch_kron(slmc_ctx* c, const double* x, int nf, int l0, int nsl, cudaStream_t s) {
    const int lm = c->p.Lx > c->p.Ly ? c->p.Lx : c->p.Ly;
    if (lm <= 8) return launch_kron<8, kTrans>(c, x, nf, l0, nsl, s);
    if (lm <= slmc::oz::kMaxLine) return launch_oz<kTrans>(c, x, nf, l0, nsl, s);
    return launch_kron<32, kTrans>(c, x, nf, l0, nsl, s);
}

}  // namespace

namespace slmc {

cudaError_t slice_group_kron(slmc_ctx* c, const double* x, int nf, int l0, int nsl, bool transposed, cudaStream_t s) {
    if (!c->kron) return cudaErrorInvalidValue;
    return transposed ? dispatch_kron<true>(c, x, nf, l0, nsl, s) : dispatch_kron<false>(c, x, nf, l0, nsl, s);
}

}  // namespace slmc
