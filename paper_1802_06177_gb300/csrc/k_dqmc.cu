// Conventional DQMC updates of the phonon field [Supplemental Material, Eqs. (S3)-(S6) and
// the block update described after them], the baseline the self-learning method is compared
// with.
//
// Local updates: at time slice l the equal-time Green's function G(l) (row-major, one chain
// per CTA) decides the move of x_{i,l-1} through the fast ratio R = 1 + (1 - G_ii) Delta_ii,
// Delta_ii = exp(-dtau lam d) - 1 (Eq. (S5)); with both spin species the weight ratio is
// R^2 exp(d ln w_bose). An accepted move updates G by Sherman-Morrison,
// G -= (Delta_ii / R) G[:, i] (e_i - G[i, :]) (Eq. (S6)). Between slices G(l) = B_l G(l-1) B_l^-1
// with B_l = diag(s) exp(-dtau K); at the start of every group of n_s slices G is recomputed
// from two stabilised products (dqmc_combine below).
//
// FP64 issue is the scarce resource on this GPU (about two FMAs per clock per SM), so the
// kernel spends it only on the arithmetic the method needs:
//  * exp(-dtau K) of the periodic square lattice factorises exactly into
//    e^{dtau mu} (E_x kron E_y), E_x and E_y symmetric circulant (the hopping along x and
//    along y commute); the mu factors of B_l and B_l^-1 cancel, and the wrap becomes four
//    in-place circulant transforms along the lines of G, folded by the factor's symmetry
//    (circ.cuh): about N^2 (Lx + Ly) FP64 operations instead of the 4 N^3 of two dense products;
//  * G stays in shared memory when it and the vectors beside it fit in 227 KB (up to N = 165), else in global memory
//    (L2-resident). For N > 64 the accepted moves of a slice are delayed in batches (Ad, Bd in shared memory, with the
//    running diagonal of G for the decisions) where there is room for them (up to N = 147): each new move needs only
//    the current column and row of G, and the batch is added to G in one pass. With G in shared memory a batch is 16 moves, one K step of the tensor-instruction update of oz_line.cuh
//    (each entry's sum of 16 products rounded once, 56-bit digits): the N^2 FMAs per move were most of the kernel
//    (40 slices, 128 chains, immediate / batched: 12x12 34.2 / 23.8 ms, 10x10 16.7 / 12.8, 9x8 8.6 / 7.9, 8x8 5.6 /
//    6.0, where moves stay immediate). With G in global memory it is up to 32 moves, added by FMAs in the order of
//    immediate updates (the same bits), for one read and write of G per batch instead of per move;
//  * the proposal, Delta_ii, exp(d ln w_bose) and both uniforms of every site of a slice are
//    computed in parallel before the slice's sites are visited; one warp then takes the decisions
//    (u < R^2 exp(d ln w_bose), the same test as ln(R^2) + d ln w_bose compared with ln u up to rounding) of the
//    next 32 sites at once, of which the first accepted one and the rejections before it stand.
//    The reciprocal runs beside the column and row of G. (Every thread deciding every site spent six FP64
//    instructions of eight warps per site and eight reciprocals per move: 40 slices of 128 chains of 12x12 23.8 ms
//    instead of 21.3, 8x8 5.6 / 4.8, 4x4 1.06 / 0.84.)
// Sites of a slice are visited in order; the proposal x' = x + U[-Delta, Delta] and the
// acceptance uniform come from Philox counter (i L + l - 1, sweep, chain, 3). The new field is
// rounded step by step as in the oracle, so accepted moves leave identical fields.
//
// Block updates reflect one site's whole column (x -> -x) and are accepted with the ratio of
// full weights (computed by the determinant path); the site and the uniform come from Philox
// counter (k, sweep, chain, 4).
#include "circ.cuh"
#include "oz_line.cuh"
#include "slmc_internal.cuh"

#include <algorithm>

namespace {

constexpr int kThreads = 256;

// G0 += sum_{q < cnt} A_q B_q^T in place (rows by warps, 4 columns per lane per pass), each entry by the
// FMA chain of cnt immediate rank-1 updates in their order: the result equals theirs bit for bit, for
// one read and one write of G per batch instead of per accepted move.
__device__ __forceinline__ void dqmc_flush(double* G, const double* Ad, const double* Bd, int cnt, int N, int lane,
                                           int warp) {
    for (int j = warp; j < N; j += kThreads / 32) {
        double* Gj = G + (size_t)j * N;
        for (int m0 = 0; m0 < N; m0 += 128) {
            double acc[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int m = m0 + lane + 32 * t;
                acc[t] = m < N ? Gj[m] : 0.0;
            }
            for (int q = 0; q < cnt; ++q) {
                const double aj = Ad[q * N + j];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int m = m0 + lane + 32 * t;
                    if (m < N) acc[t] = fma(aj, Bd[q * N + m], acc[t]);
                }
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int m = m0 + lane + 32 * t;
                if (m < N) Gj[m] = acc[t];
            }
        }
    }
}

template <int LMAX>
__global__ void __launch_bounds__(kThreads) k_dqmc_slices(double* __restrict__ x, double* __restrict__ Gall, int Lx,
                                                          int Ly, int L, int l0, int nsl, double dtau,
                                                          const double* __restrict__ kron,
                                                          double lam, double w02, double delta, uint32_t key0,
                                                          uint32_t key1, uint32_t sweep, int chain0, int g_in_smem,
                                                          int kd, unsigned long long* __restrict__ n_acc) {
    extern __shared__ double dsm[];
    constexpr int QMAX = (LMAX * LMAX + 31) / 32;  // columns per lane in the rank-1 update
    constexpr int JMAX = (LMAX * LMAX + kThreads - 1) / kThreads;  // columns per thread
    constexpr int kDecider = kThreads / 32 - 1;                    // has no column while N <= 224
    const int N = Lx * Ly;
    const int f = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t NN = (size_t)N * N;
    double* G = g_in_smem ? dsm : Gall + f * NN;
    // row stride: odd in shared memory, so that walks down a column (the wrap's right factors with a row per
    // lane, a move's column of G) meet no bank conflicts
    const int ldg = g_in_smem ? N | 1 : N;
    double* p = g_in_smem ? dsm + (size_t)N * ldg : dsm;
    double* s = p;                 // [N] slice scales exp(-dtau lam x_{i,l-1})
    double* sinv = p + N;          // [N] 1 / s
    double* xn = p + 2 * N;        // [N] proposed field
    double* dl = p + 3 * N;        // [N] Delta_ii
    double* eb = p + 4 * N;        // [N] exp(d ln w_bose)
    double* ua = p + 5 * N;        // [N] acceptance uniform
    double* ac = p + 6 * N;        // [N] -(Delta_ii / R) G[:, i]
    double* rw = p + 7 * N;        // [N] e_i - G[i, :]
    const int kx = slmc::circ::ncoef(Lx), ky = slmc::circ::ncoef(Ly);
    double* ex = p + 8 * N;        // folded coefficients (circ.cuh) of E_x, E_x^-1, E_y, E_y^-1
    double* exi = ex + kx;
    double* ey = exi + kx;
    double* eyi = ey + ky;
    // delayed updates (kd > 0, G in global memory): accepted moves q < cnt of the current batch as
    // G = G0 + sum_q A_q B_q^T, A_q = -(Delta/R) G[:, i_q], B_q = e_i - G[i_q, :] ([kd][N] each), and the
    // running diagonal of G
    double* Ad = eyi + ky;
    double* Bd = Ad + (size_t)kd * N;
    double* dg = Bd + (size_t)kd * N;
    double* s_a = dg + (kd > 0 ? N : 0);  // Delta / R of the next accepted site, and the site
    int* s_next = reinterpret_cast<int*>(s_a + 1);
    double* xf = x + (size_t)f * N * L;
    const uint32_t chain = (uint32_t)(chain0 + f);

    const double* less1 = kron + slmc::kKronMaxLine;  // the factors less the identity
    slmc::circ::build(ex, less1, Lx, tid, kThreads);
    slmc::circ::build(exi, less1 + slmc::kKronTab, Lx, tid, kThreads);
    slmc::circ::build(ey, less1 + 2 * slmc::kKronTab, Ly, tid, kThreads);
    slmc::circ::build(eyi, less1 + 3 * slmc::kKronTab, Ly, tid, kThreads);
    if (g_in_smem) {
        for (int j = warp; j < N; j += kThreads / 32)
            for (int m = lane; m < N; m += 32) G[j * ldg + m] = Gall[f * NN + (size_t)j * N + m];
    }
    int accepted = 0;
    for (int l = l0 + 1; l <= l0 + nsl; ++l) {
        const int c = l - 1;
        const int cu = c + 1 == L ? 0 : c + 1, cd = c == 0 ? L - 1 : c - 1;
        for (int i = tid; i < N; i += kThreads) {
            const double v = xf[(size_t)i * L + c];
            const slmc::u32x4 w = slmc::philox4x32_10(slmc::u32x4{(uint32_t)(i * L + c), sweep, chain, 3u}, key0, key1);
            const double u1 = slmc::uniform53(w.x, w.y);
            const double xp = __dadd_rn(v, __dmul_rn(delta, __dadd_rn(__dmul_rn(2.0, u1), -1.0)));
            const double up = xf[(size_t)i * L + cu], dn = xf[(size_t)i * L + cd];
            const double kin = ((up - xp) * (up - xp) + (xp - dn) * (xp - dn) - (up - v) * (up - v) -
                                (v - dn) * (v - dn)) / (2.0 * dtau * dtau);
            const double dlb = dtau * lam * (xp - v) - dtau * (0.5 * w02 * (xp * xp - v * v) + kin);
            s[i] = exp(-dtau * lam * v);
            sinv[i] = exp(dtau * lam * v);
            xn[i] = xp;
            dl[i] = exp(-dtau * lam * (xp - v)) - 1.0;
            eb[i] = exp(dlb);
            ua[i] = slmc::uniform53(w.z, w.w);
        }
        __syncthreads();
        // wrap: G <- diag(s) (E_x kron E_y) G (E_x kron E_y)^-1 diag(1/s), site i = ix + Lx iy
        // passes: right factor along y (lines (i, jx)), along x (lines (i, jy)), left factor along x (lines (iy, j)),
        // along y (lines (ix, j)) with the scales; consecutive threads take neighbouring rows or columns of G
        for (int pass = 0; pass < 4; ++pass) {
            const bool left = pass >= 2, alongx = pass == 1 || pass == 2;
            const int lines = alongx ? Ly : Lx, n = alongx ? Lx : Ly;
            const int unit = left ? ldg : 1, stride = (alongx ? 1 : Lx) * unit;
            const double* cf = left ? (alongx ? ex : ey) : (alongx ? exi : eyi);
            for (int q = tid; q < lines * N; q += kThreads) {
                const int li = q / N, o = q - li * N;  // line, and the row (right factors) or column (left) it belongs to
                const int at = (alongx ? li * Lx : li) * unit + o * (left ? 1 : ldg);
                slmc::circ::apply_any<LMAX>(n, G + at, stride, cf, nullptr, 0, pass == 3 ? s + li : nullptr, Lx,
                                            sinv + o);
            }
            __syncthreads();
        }
        if (kd > 0) {
            for (int j = tid; j < N; j += kThreads) dg[j] = G[(size_t)j * ldg + j];
            __syncthreads();
        }
        int cnt = 0;  // delayed moves of the current batch (block-uniform)
        for (int i0 = 0;;) {
            // the last warp finds the next accepted site, 32 sites at a time: G and the diagonal stay as they are up to it
            double R = 1.0;
            int i = N;
            if (warp == kDecider) {
                for (int b = i0; b < N && i == N; b += 32) {
                    const int k = min(b + lane, N - 1);
                    const double gkk = kd > 0 ? dg[k] : G[(size_t)k * ldg + k];
                    R = __dadd_rn(1.0, __dmul_rn(__dadd_rn(1.0, -gkk), dl[k]));
                    const unsigned m = __ballot_sync(0xffffffffu, b + lane < N && ua[k] < R * R * eb[k]);
                    if (m) {
                        i = b + __ffs(m) - 1;
                        R = __shfl_sync(0xffffffffu, R, __ffs(m) - 1);
                    }
                }
                if (lane == 0) *s_next = i;
                if (kd == 0 && i < N && lane == 0) *s_a = dl[i] * __drcp_rn(R);
            }
            __syncthreads();
            i = *s_next;
            if (i >= N) break;
            i0 = i + 1;
            if (kd > 0) {
                // the current column G[:, i] and row G[i, :] from G0 and the batch, each entry by the
                // same FMA chain the immediate update would have applied to it; the deciding warp's
                // reciprocal meanwhile
                if (warp == kDecider && lane == 0) *s_a = dl[i] * __drcp_rn(R);
                double cj[JMAX], rj[JMAX];
#pragma unroll
                for (int t = 0; t < JMAX; ++t) {
                    const int j = tid + t * kThreads;
                    if (j >= N) break;
                    cj[t] = G[(size_t)j * ldg + i], rj[t] = G[(size_t)i * ldg + j];
                    for (int q = 0; q < cnt; ++q) {
                        cj[t] = fma(Ad[q * N + j], Bd[q * N + i], cj[t]);
                        rj[t] = fma(Ad[q * N + i], Bd[q * N + j], rj[t]);
                    }
                }
                __syncthreads();
                const double a = *s_a;
#pragma unroll
                for (int t = 0; t < JMAX; ++t) {
                    const int j = tid + t * kThreads;
                    if (j >= N) break;
                    const double aj = -a * cj[t];
                    const double bj = (j == i ? 1.0 : 0.0) - rj[t];
                    Ad[cnt * N + j] = aj;
                    Bd[cnt * N + j] = bj;
                    dg[j] = fma(aj, bj, dg[j]);
                }
                if (tid == 0) {
                    xf[(size_t)i * L + c] = xn[i];
                    ++accepted;
                }
                __syncthreads();
                if (++cnt == kd) {
                    if (g_in_smem) slmc::oz::rank_update(G, ldg, Ad, Bd, cnt, N, warp, kThreads / 32);
                    else dqmc_flush(G, Ad, Bd, cnt, N, lane, warp);
                    cnt = 0;
                    __syncthreads();
                }
                continue;
            }
            const double a = *s_a;
            for (int j = tid; j < N; j += kThreads) {
                ac[j] = -a * G[(size_t)j * ldg + i];
                rw[j] = (j == i ? 1.0 : 0.0) - G[(size_t)i * ldg + j];
            }
            if (tid == 0) {
                xf[(size_t)i * L + c] = xn[i];
                ++accepted;
            }
            __syncthreads();
            // rank-1 update, one row per warp at a time: the row's coefficient is loaded once and
            // the lane's entries of e_i - G[i, :] stay in registers (N <= LMAX^2 = 32 QMAX)
            double r[QMAX];
#pragma unroll
            for (int q = 0; q < QMAX; ++q) r[q] = lane + 32 * q < N ? rw[lane + 32 * q] : 0.0;
            for (int j = warp; j < N; j += kThreads / 32) {
                const double cj = ac[j];
                double* Gj = G + (size_t)j * ldg;
#pragma unroll
                for (int q = 0; q < QMAX; ++q)
                    if (lane + 32 * q < N) Gj[lane + 32 * q] = fma(cj, r[q], Gj[lane + 32 * q]);
            }
            __syncthreads();
        }
        if (cnt > 0) {  // the slice's last batch
            if (g_in_smem) slmc::oz::rank_update(G, ldg, Ad, Bd, cnt, N, warp, kThreads / 32);
            else dqmc_flush(G, Ad, Bd, cnt, N, lane, warp);
        }
        __syncthreads();
    }
    if (tid == 0 && n_acc) n_acc[f] += (unsigned long long)accepted;
}

// Block update k: reflect the whole column of one site of every chain (in place) and draw the
// acceptance uniform u[f].
__global__ void k_block_propose(double* __restrict__ x, int N, int L, uint32_t key0, uint32_t key1, uint32_t sweep,
                                uint32_t k, int chain0, double* __restrict__ u) {
    const int f = blockIdx.x;
    const slmc::u32x4 w = slmc::philox4x32_10(slmc::u32x4{k, sweep, (uint32_t)(chain0 + f), 4u}, key0, key1);
    const int s0 = (int)(slmc::uniform53(w.x, w.y) * (double)N);
    const int site = s0 < N - 1 ? s0 : N - 1;
    double* xs = x + ((size_t)f * N + site) * L;
    for (int l = threadIdx.x; l < L; l += blockDim.x) xs[l] = -xs[l];
    if (threadIdx.x == 0) u[f] = slmc::uniform53(w.z, w.w);
}

// G(g0) from two stabilised products. With B(g0, 0) = U_R D_R T_R (the running chain of the
// slices already visited in this sweep) and B(L, g0)^T = U_L D_L T_L (the transposed chain of
// the slices still to come, kept from the start of the sweep), D = D_b D_s (D_b = max(D, 1),
// D_s = min(D, 1)):
//   I + B(g0, 0) B(L, g0) = U_R D_bR M D_bL U_L^T,
//   M = D_bR^-1 (U_R^T U_L) D_bL^-1 + D_sR (T_R T_L^T) D_sL,
//   G(g0) = U_L D_bL^-1 M^-1 D_bR^-1 U_R^T,
// M bounded entry-wise by the scale split, so its LU carries no exponentially large or small
// numbers (the same split as the final step of the determinant path).
struct GemmTerm {
    const double* A;   // A(i, k): A[i N + k] (kAik) or A[k N + i]
    const double* B;   // B(k, j): B[j N + k] (kBjk) or B[k N + j]
    const double* ra;  // optional row scales of A, [nf][sstride]
    const double* sk;  // optional scales of the summation index, applied to B
    const double* cb;  // optional column scales of B
};
struct GemmArgs {
    GemmTerm t[2];
    int nterms;
};

// C = sum over terms of diag(ra) A diag(sk) B diag(cb), one field per blockIdx.z, a TM x TM tile per CTA, 16 x 16
// per warp, on the warp-level tensor instruction.
//
// As FP64 FMAs (4 x 4 outputs per thread) these products ran at the FP64 issue limit. Here rows of A and columns of B
// (with sk) are cut into eight 7-bit digits against the power of two of their largest value (oz_line.cuh); the CTA cuts
// each 16-column step once into fragments in shared memory, the next step's values already loaded, and the 36 products
// a + b <= 7 accumulate exactly in FP32 for kSeg steps (a level's sum stays below 2^22), then as integers rounded once
// to FP64: of 36 MMAs per 16 x 8 x 16 block, two cycles each, instead of 64 FMA warp instructions of 16 to 19 cycles.
// G of a run of 40 slices (products, LU and solve), FP64 FMAs / digits: 128 chains of 12x12 18.8 / 12.0 ms, 10x10 10.5 /
// 6.4, 8x8 1.84 / 1.15, 4x4 0.35 / 0.26; 64 of 16x16, L = 20, 22.5 / 13.6. Against 64-bit-mantissa arithmetic (4x4, 9x8 and
// 12x12, L = 40 and 80), Frobenius norm, FMAs / digits: M 0.9e-16 to 3.8e-16 / 0.4e-16 to 1.1e-16, U_L (..) 0.8e-16 to
// 3.0e-16 / 0.7e-16 to 2.3e-16, smaller for every field.
template <int TM, bool kAik, bool kBjk, bool kCrow>
__global__ void __launch_bounds__(TM * TM / 8, TM == 32 ? 3 : 1) k_gemm_oz(GemmArgs g, double* __restrict__ C,
                                                                                         int N, int sstride) {
    namespace oz = slmc::oz;
    constexpr int WT = TM / 16, NW = WT * WT, NT = 32 * NW, kD = oz::kD, kSeg = 6;
    constexpr int kItems = TM * 16, P = (kItems + NT - 1) / NT;  // pairs (k, k + 1) of A and B in a step, per thread
    __shared__ uint4 Af[WT][kD][32];
    __shared__ uint2 Bf[2 * WT][kD][32];
    __shared__ int hi[2 * TM];  // upper words of the largest |a| of each row and |b| of each column
    const int f = blockIdx.z, i0 = blockIdx.y * TM, j0 = blockIdx.x * TM, KT = (N + 15) / 16;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wr = warp / WT, wc = warp % WT;
    const int r0 = lane >> 2, t2 = 2 * (lane & 3);
    const size_t NN = (size_t)N * N;
    double out[2][4];
#pragma unroll
    for (int ct = 0; ct < 2; ++ct)
#pragma unroll
        for (int u = 0; u < 4; ++u) out[ct][u] = 0.0;
#pragma unroll 1
    for (int t = 0; t < g.nterms; ++t) {
        const double* A = (t ? g.t[1].A : g.t[0].A) + f * NN;
        const double* B = (t ? g.t[1].B : g.t[0].B) + f * NN;
        const double* ra = t ? g.t[1].ra : g.t[0].ra;
        const double* sk = t ? g.t[1].sk : g.t[0].sk;
        const double* cb = t ? g.t[1].cb : g.t[0].cb;
        if (ra) ra += (size_t)f * sstride;
        if (sk) sk += (size_t)f * sstride;
        if (cb) cb += (size_t)f * sstride;
        auto val_a = [&](int r, int k) {
            const int i = i0 + r;
            return i < N && k < N ? (kAik ? A[(size_t)i * N + k] : A[(size_t)k * N + i]) : 0.0;
        };
        auto val_b = [&](int r, int k) {
            const int j = j0 + r;
            double v = j < N && k < N ? (kBjk ? B[(size_t)j * N + k] : B[(size_t)k * N + j]) : 0.0;
            if (sk && k < N) v *= sk[k];
            return v;
        };
        // item q of a step: pair kp of row r of A (r < TM) or of column r - TM of B, ordered along the operand's
        // contiguous index
        auto place = [&](int q, int& r, int& kp) {
            const bool b = q >= TM * 8;
            const int p = b ? q - TM * 8 : q;
            if (b ? kBjk : kAik) {
                r = p >> 3, kp = p & 7;
            } else {
                r = (p >> 5) % (TM / 8) * 8 + (p & 7), kp = (p >> 5) / (TM / 8) * 4 + ((p >> 3) & 3);
            }
            if (b) r += TM;
        };
        double v[P][2];
        auto load = [&](int k0) {
#pragma unroll
            for (int m = 0; m < P; ++m) {
                const int q = tid + m * NT;
                int r, kp;
                place(q, r, kp);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    v[m][h] = q >= kItems ? 0.0 : r < TM ? val_a(r, k0 + 2 * kp + h) : val_b(r - TM, k0 + 2 * kp + h);
            }
        };
        load(0);
        __syncthreads();  // the fragments and maxima of the previous term are read
        for (int r = tid; r < 2 * TM; r += NT) hi[r] = 0;
        __syncthreads();
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            auto bits = [&](int r, int k) { return __double2hiint(o ? val_b(r, k) : val_a(r, k)) & 0x7fffffff; };
            if (o ? kBjk : kAik) {
                for (int r = warp; r < TM; r += NW) {
                    int m = 0;
                    for (int k = lane; k < N; k += 32) m = max(m, bits(r, k));
                    m = __reduce_max_sync(0xffffffffu, m);
                    if (lane == 0) hi[o * TM + r] = m;
                }
            } else {
                constexpr int KS = NT / TM;  // rows of k per pass
                const int r = tid % TM;
                int m = 0;
                if (tid < KS * TM)
                    for (int k = tid / TM; k < N; k += KS) m = max(m, bits(r, k));
                atomicMax(&hi[o * TM + r], m);
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int s0 = 0; s0 < KT; s0 += kSeg) {
            float c[2][kD][4];
#pragma unroll
            for (int ct = 0; ct < 2; ++ct)
#pragma unroll
                for (int l = 0; l < kD; ++l)
#pragma unroll
                    for (int u = 0; u < 4; ++u) c[ct][l][u] = 0.f;
#pragma unroll 1
            for (int ks = s0; ks < min(KT, s0 + kSeg); ++ks) {
#pragma unroll
                for (int m = 0; m < P; ++m) {
                    const int q = tid + m * NT;
                    if (q >= kItems) break;
                    int r, kp;
                    place(q, r, kp);
                    const int e = oz::exponent_of_hi(hi[r]), ln = 4 * (r & 7) + (kp & 3);
                    float d0[kD], d1[kD];
                    oz::digits(v[m][0], e, d0);
                    oz::digits(v[m][1], e, d1);
                    uint32_t* w = r < TM ? reinterpret_cast<uint32_t*>(&Af[r >> 4][0][ln]) + ((r >> 3) & 1) + 2 * (kp >> 2)
                                         : reinterpret_cast<uint32_t*>(&Bf[(r - TM) >> 3][0][ln]) + (kp >> 2);
                    const int step = r < TM ? 128 : 64;
#pragma unroll
                    for (int s = 0; s < kD; ++s) w[s * step] = oz::pack(d0[s], d1[s]);
                }
                __syncthreads();
                if (ks + 1 < KT) load(16 * (ks + 1));
#pragma unroll
                for (int ct = 0; ct < 2; ++ct) {
                    uint2 b[kD];
#pragma unroll
                    for (int l = 0; l < kD; ++l) b[l] = Bf[2 * wc + ct][l][lane];
#pragma unroll
                    for (int l = 0; l < kD; ++l) {
                        const uint4 q = Af[wr][l][lane];
                        const uint32_t a[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                        for (int m = 0; l + m < kD; ++m) oz::mma(c[ct][l + m], a, b[m].x, b[m].y);
                    }
                }
                __syncthreads();
            }
#pragma unroll
            for (int ct = 0; ct < 2; ++ct)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    float w[kD];
#pragma unroll
                    for (int l = 0; l < kD; ++l) w[l] = c[ct][l][u];
                    const int ea = oz::exponent_of_hi(hi[16 * wr + r0 + 8 * (u >> 1)]);
                    const int eb = oz::exponent_of_hi(hi[TM + 16 * wc + 8 * ct + t2 + (u & 1)]);
                    double y = oz::value(w, ea + eb - 61);
                    // a row or column with a value that is not finite becomes NaN, as its sums would
                    if (ea == 1024 || eb == 1024) y = __longlong_as_double(0x7ff8000000000000ll);
                    const int i = min(i0 + 16 * wr + r0 + 8 * (u >> 1), N - 1);
                    const int j = min(j0 + 16 * wc + 8 * ct + t2 + (u & 1), N - 1);
                    if (ra) y *= ra[i];
                    if (cb) y *= cb[j];
                    out[ct][u] += y;
                }
        }
    }
#pragma unroll
    for (int ct = 0; ct < 2; ++ct)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + 16 * wr + r0 + 8 * (u >> 1), j = j0 + 16 * wc + 8 * ct + t2 + (u & 1);
            if (i < N && j < N) C[f * NN + (kCrow ? (size_t)i * N + j : (size_t)j * N + i)] = out[ct][u];
        }
}

// S[f] = [D_bR^-1 | D_sR | D_bL^-1 | D_sL], each [N], from the ln D of both products
__global__ void k_split_scales(const double* __restrict__ lnR, const double* __restrict__ lnL, double* __restrict__ S,
                               int N) {
    const int f = blockIdx.x;
    double* Sf = S + (size_t)f * 4 * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const double r = lnR[(size_t)f * N + i], l = lnL[(size_t)f * N + i];
        Sf[i] = exp(-fmax(r, 0.0));
        Sf[N + i] = exp(fmin(r, 0.0));
        Sf[2 * N + i] = exp(-fmax(l, 0.0));
        Sf[3 * N + i] = exp(fmin(l, 0.0));
    }
}

template <int TM, bool kAik, bool kBjk, bool kCrow>
cudaError_t launch_gemm(const GemmArgs& g, double* C, int N, int nf, int sstride, cudaStream_t s) {
    dim3 grid((N + TM - 1) / TM, (N + TM - 1) / TM, nf);
    k_gemm_oz<TM, kAik, kBjk, kCrow><<<grid, TM * TM / 8, 0, s>>>(g, C, N, sstride);
    return cudaGetLastError();
}

// One tile per field while N fits (32, 48 or 64), else tiles of 32, three CTAs per SM: one CTA's cutting then runs beside
// another's products (G of the 12x12 run above 12.0 ms with 32, 12.6 with 48, which pads nothing; 16x16 the same with
// 32 and 64; one tile of 48 or 64 against four of 32: 6x6 0.73 / 0.85 ms, 8x8 1.15 / 1.24).
template <bool kAik, bool kBjk, bool kCrow>
cudaError_t gemm_oz(const GemmArgs& g, double* C, int N, int nf, int sstride, cudaStream_t s) {
    if (N > 32 && N <= 48) return launch_gemm<48, kAik, kBjk, kCrow>(g, C, N, nf, sstride, s);
    if (N > 48 && N <= 64) return launch_gemm<64, kAik, kBjk, kCrow>(g, C, N, nf, sstride, s);
    return launch_gemm<32, kAik, kBjk, kCrow>(g, C, N, nf, sstride, s);
}

size_t dqmc_smem_bytes(int N, int ncoef, bool g_in_smem, int kd = 0) {
    return ((g_in_smem ? (size_t)N * (N | 1) : 0) + 8 * (size_t)N + ncoef + (kd > 0 ? (2 * (size_t)kd + 1) * N : 0) + 2) *
           sizeof(double);
}

constexpr int kDelayMax = 32;  // accepted moves per delayed batch (G in global memory)
constexpr int kDelaySmem = 16, kDelayMinN = 65;  // the same with G in shared memory

bool dqmc_supported(const slmc_ctx* c) { return c->L >= 2 && c->kron != nullptr; }

template <int LMAX>
cudaError_t launch_slices(slmc_ctx* c, double* x, double* G, int nf, int chain0, int l0, int nsl, uint64_t sweep,
                          long long* n_acc, cudaStream_t s) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const int nc = 2 * (slmc::circ::ncoef(c->p.Lx) + slmc::circ::ncoef(c->p.Ly));
    const bool in_smem = dqmc_smem_bytes(c->N, nc, true) <= (size_t)optin;
    // Batches of up to kd accepted moves (delayed updates). G in shared memory: 16 moves are one K step of the
    // tensor-instruction update, where there is room for them and N is large enough for the update to outweigh the
    // batch's bookkeeping (N = 72 gains 8%, N = 64 loses 6%, above); else, and from N = 150 on, where no room is left for
    // the batch, moves are applied at once (batches flushed by FP64 FMAs measured slower than that:
    // the same FMAs and the columns on top). G in global memory: batches of 32 by FMAs, one pass over G each.
    int kd = 0;
    if (in_smem) {
        if (c->N >= kDelayMinN && dqmc_smem_bytes(c->N, nc, true, kDelaySmem) <= (size_t)optin) kd = kDelaySmem;
    } else {
        kd = kDelayMax;
        while (kd > 1 && dqmc_smem_bytes(c->N, nc, false, kd) > (size_t)optin) kd /= 2;
        if (dqmc_smem_bytes(c->N, nc, false, kd) > (size_t)optin) kd = 0;
    }
    const size_t bytes = dqmc_smem_bytes(c->N, nc, in_smem, kd);
    e = slmc::allow_smem(k_dqmc_slices<LMAX>, bytes);
    if (e != cudaSuccess) return e;
    k_dqmc_slices<LMAX><<<nf, kThreads, bytes, s>>>(
        x, G, c->p.Lx, c->p.Ly, c->L, l0, nsl, c->p.dtau, c->kron, c->p.lambda, c->p.omega0 * c->p.omega0,
        c->p.sweep_delta, (uint32_t)(c->p.seed & 0xffffffffu), (uint32_t)(c->p.seed >> 32), (uint32_t)sweep, chain0,
        in_smem ? 1 : 0, kd, reinterpret_cast<unsigned long long*>(n_acc));
    return cudaGetLastError();
}

}  // namespace

namespace slmc {

bool dqmc_ok(const slmc_ctx* c) { return dqmc_supported(c); }

cudaError_t dqmc_combine(slmc_ctx* c, const double* Ul, const double* lnDl, const double* Tl, int nf, double* G,
                         double* lndet_scratch, int* sign_scratch, cudaStream_t s) {
    const int N = c->N;
    double* S = c->Sws;  // [nf][4][N]: free between the steps of a chain
    k_split_scales<<<nf, 256, 0, s>>>(c->lnD, lnDl, S, N);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    GemmArgs m{};
    m.nterms = 2;
    m.t[0] = GemmTerm{c->U, Ul, S, nullptr, S + 2 * N};     // D_bR^-1 U_R^T U_L D_bL^-1
    m.t[1] = GemmTerm{c->Ta, Tl, S + N, nullptr, S + 3 * N};  // D_sR T_R T_L^T D_sL
    e = gemm_oz<true, true, false>(m, c->Y, N, nf, 4 * N, s);  // M column-major, as the LU expects
    if (e != cudaSuccess) return e;
    e = final_lu(c, nf, lndet_scratch, sign_scratch, s);
    if (e != cudaSuccess) return e;
    e = final_greens(c, nf, c->Tb, s);  // X = M^-1 D_bR^-1 U_R^T, row-major, in the idle T buffer
    if (e != cudaSuccess) return e;
    GemmArgs gg{};
    gg.nterms = 1;
    gg.t[0] = GemmTerm{Ul, c->Tb, nullptr, S + 2 * N, nullptr};  // U_L D_bL^-1 X
    return gemm_oz<false, false, true>(gg, G, N, nf, 4 * N, s);
}

cudaError_t dqmc_slices(slmc_ctx* c, double* x, double* G, int nf, int chain0, int l0, int nsl, uint64_t sweep,
                        long long* n_acc, cudaStream_t s) {
    const int lm = std::max(c->p.Lx, c->p.Ly);
    if (lm <= 8) return launch_slices<8>(c, x, G, nf, chain0, l0, nsl, sweep, n_acc, s);
    if (lm <= 12) return launch_slices<12>(c, x, G, nf, chain0, l0, nsl, sweep, n_acc, s);
    if (lm <= 16) return launch_slices<16>(c, x, G, nf, chain0, l0, nsl, sweep, n_acc, s);
    return launch_slices<32>(c, x, G, nf, chain0, l0, nsl, sweep, n_acc, s);
}

cudaError_t dqmc_block_propose(slmc_ctx* c, double* x, int nf, int chain0, uint64_t sweep, int k, double* u,
                               cudaStream_t s) {
    k_block_propose<<<nf, 128, 0, s>>>(x, c->N, c->L, (uint32_t)(c->p.seed & 0xffffffffu), (uint32_t)(c->p.seed >> 32),
                                       (uint32_t)sweep, (uint32_t)k, chain0, u);
    return cudaGetLastError();
}

}  // namespace slmc
