// Bosonic parts of the weight, the symmetric effective model and its Markov chain, the
// cumulative-update acceptance, the CDW structure factor and the E_eff regression.
//
//   ln w       = 2 ln|det| + dtau lam sum x - dtau sum [w0^2 x^2/2 + (x_{l+1}-x_l)^2/(2 dtau^2)]
//                                                             [Sec. "Model", Suppl. Eq. (S2)]
//   ln w_eff   = -dtau (E0 + J_k F_k + J_p F_p + J_p' F_p' + J_nn F_nn + J_nn' F_nn')
//                                                             [Eq. (4) / (S7)]
//   acceptance = min{1, [w(x')/w(x)] [w_eff(x)/w_eff(x')]}   [Eq. (6)]
//   S(pi,pi)   = (1/N) sum_ij s_i s_j [4 (1-G_ii)(1-G_jj) + 2 (d_ij - G_ji) G_ij]  [Sec. "Results"]
//   fit        = least squares of ln w on [1, F]               [Eq. (5)]
//
// Site i = ix + Lx iy, field element (i, l) at i*L + l. All reductions use a fixed
// order (per-thread strided partial sums, then a shared-memory tree), so results are
// reproducible run to run.
#include <algorithm>
#include <cfloat>

#include "slmc_internal.cuh"

namespace {

constexpr int kThreads = 256;

template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* red /* [NV][kThreads] */) {
#pragma unroll
    for (int q = 0; q < NV; ++q) red[q * kThreads + threadIdx.x] = v[q];
    __syncthreads();
    for (int h = kThreads / 2; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) {
#pragma unroll
            for (int q = 0; q < NV; ++q) red[q * kThreads + threadIdx.x] += red[q * kThreads + threadIdx.x + h];
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = red[q * kThreads];
}

__global__ void __launch_bounds__(kThreads) k_bose(const double* __restrict__ x, int N, int L, double dtau, double lam,
                                                   double w02, const double* __restrict__ lndet, double* __restrict__ lnw) {
    __shared__ double red[kThreads];
    const int f = blockIdx.x;
    const double* xf = x + (size_t)f * N * L;
    const double inv2dt2 = 1.0 / (2.0 * dtau * dtau);
    double acc[1] = {0.0};
    for (int idx = threadIdx.x; idx < N * L; idx += kThreads) {
        const int i = idx / L, l = idx - i * L;
        const double v = xf[idx];
        const double vn = xf[(size_t)i * L + (l + 1 == L ? 0 : l + 1)];
        const double d = vn - v;
        acc[0] += dtau * lam * v - dtau * (0.5 * w02 * v * v + d * d * inv2dt2);
    }
    block_sum<1>(acc, red);
    if (threadIdx.x == 0) lnw[f] = (lndet ? 2.0 * lndet[f] : 0.0) + acc[0];
}

// n / d for the divisors of a lattice (half the slices, Lx) by one multiply-high: exact while n d < 2^32
// (q = floor(n ceil(2^32 / d) / 2^32)); magic 0 selects the division.
__device__ __forceinline__ int fast_div(int n, int d, uint32_t magic) {
    return magic ? (int)__umulhi((uint32_t)n, magic) : n / d;
}

// Feature sums of one field per CTA, eleven FP64 operations per value, the bound from a few thousand values on: a
// field of 12x12, L = 120 has 46 us of FP64 issue. Threads take values 256 apart, whatever rows they lie in (the site and
// slice advance by additions, the neighbours' rows come from a table), and load four values' operands before they use
// them; 152 / 1000 fields of 12x12, L = 120 take 61 / 364 us, of 4x4, L = 40 12 / 23 us, of 16x16, L = 160 132 / 846 us.
// With a row per warp and its lanes on the slices they took 104 / 686, 16 / 54 and 130 / 870 us: only row lengths of
// a multiple of 128 filled the unrolled loop.
__global__ void __launch_bounds__(kThreads) k_features(const double* __restrict__ x, int Lx, int Ly, int L, uint32_t ml,
                                                       uint32_t mlx, int di, double a2, double dtau, const double* __restrict__ J,
                                                       double* __restrict__ F, int ldF, double* __restrict__ lnw_eff) {
    constexpr int U = 4;  // values in flight
    __shared__ double red[5][kThreads], feat[5];
    __shared__ int nbx[SLMC_MAX_N], nby[SLMC_MAX_N];  // first element of the rows of a site's neighbours
    const int f = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int N = Lx * Ly, NL = N * L;
    const double* xf = x + (size_t)f * NL;
    for (int i = threadIdx.x; i < N; i += kThreads) {
        const int iy = fast_div(i, Lx, mlx), ix = i - iy * Lx;
        nbx[i] = (i + (ix + 1 == Lx ? 1 - Lx : 1)) * L;
        nby[i] = (iy + 1 == Ly ? ix : i + Lx) * L;
    }
    __syncthreads();
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const double h2 = -0.5 * a2, h4 = -0.25 * a2;
    const int dl = kThreads - di * L;  // di = kThreads / L
    int i = fast_div(threadIdx.x, L, ml), l = threadIdx.x - i * L;
    for (unsigned w0 = threadIdx.x & ~31u; w0 < (unsigned)NL; w0 += U * kThreads) {  // first value of the warp
        double v[U], vt[U], vx[U], vy[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            v[u] = vt[u] = vx[u] = vy[u] = 0.0;  // adds nothing
            if (i < N) {
                const double* xi = xf + i * L;
                v[u] = xi[l];
                vt[u] = xi[l + 1 == L ? 0 : l + 1];
                vx[u] = xf[nbx[i] + l];
                vy[u] = xf[nby[i] + l];
            }
            i += di;
            l += dl;
            if (l >= L) {
                l -= L;
                ++i;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (w0 + u * kThreads >= (unsigned)NL) break;
            const double nb = vx[u] + vy[u];
            const double v2 = v[u] * v[u], v4 = v2 * v2, d = vt[u] - v[u];
            acc[0] = fma(d, d, acc[0]);
            acc[1] = fma(v2, fma(0.25, v2, h2), acc[1]);
            acc[2] = fma(v4, fma(1.0 / 6.0, v2, h4), acc[2]);
            acc[3] = fma(v[u], nb, acc[3]);
            acc[4] = fma(v[u], vt[u], acc[4]);
        }
    }
    // one warp per sum: over the warps first, then over the lanes (13 additions of five warps)
#pragma unroll
    for (int q = 0; q < 5; ++q) red[q][threadIdx.x] = acc[q];
    __syncthreads();
    if (warp < 5) {
        double t = red[warp][lane];
#pragma unroll
        for (int w = 1; w < kThreads / 32; ++w) t += red[warp][lane + 32 * w];
        t = slmc::warp_allsum(t);
        if (lane == 0) feat[warp] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (F)
            for (int q = 0; q < 5; ++q) F[(size_t)f * ldF + q] = feat[q];
        if (lnw_eff) {
            const double e = J[0] + J[1] * feat[0] + J[2] * feat[1] + J[3] * feat[2] + J[4] * feat[3] + J[5] * feat[4];
            lnw_eff[f] = -dtau * e;
        }
    }
}

// Terms of E0 + J.F that contain one site value v.
__device__ __forceinline__ double local_energy(const double* J, double a2, double v, double up, double dn, double nb) {
    const double v2 = v * v;
    const double du = up - v, dd = v - dn;
    return J[1] * (du * du + dd * dd) + J[2] * (v2 * v2 * 0.25 - a2 * v2 * 0.5) +
           J[3] * (v2 * v2 * v2 * (1.0 / 6.0) - a2 * v2 * v2 * 0.25) + J[4] * v * nb + J[5] * v * (up + dn);
}

// Loads of the field: plain (cached) in the per-colour kernels, L2-only (ld.global.cg) in the
// persistent queue kernel, whose CTAs read values that other CTAs of the same launch wrote.
template <bool kL2>
__device__ __forceinline__ double ldx(const double* p) {
    if (kL2) return __ldcg(p);
    return *p;
}

// FP32 value of v rounded toward zero, by integer operations: the conversion instruction shares the
// FP64 pipe, whose two lanes per clock bound the sweeps when every site converts its seven operands
// there. |v| below 2^-126 gives 0; above the FP32 range, infinities and NaN give infinity (the caller's
// finiteness test then sends the site to the FP64 rule).
__device__ __forceinline__ float trunc_f32(double v) {
    const int hi = __double2hiint(v);
    const int t = (hi & 0x7fffffff) - 0x38000000;  // exponent rebased from FP64 to FP32
    uint32_t m = __funnelshift_l((uint32_t)__double2loint(v), (uint32_t)t, 3);
    if (t < 0x00100000) m = 0u;
    if (t >= 0x0ff00000) m = 0x7f800000u;
    return __uint_as_float((m & 0x7fffffffu) | ((uint32_t)hi & 0x80000000u));
}

// Couplings and constants of one chain's sweeps, FP64 for the exact rule and FP32 for the fast test, kept in
// shared memory.
struct SweepConst {
    double J[6];
    double dtau, a2, delta, ds;  // ds = delta 2^-52
    float Jf[6];
    float Jm[6];  // magnitudes
    float dtauf, a2f, deltaf;
    int plain;  // delta too small for ds to be normal: the proposal step by step
};

// Filled by the threads of one warp or more (caller synchronises).
__device__ __forceinline__ void sweep_const_init(SweepConst& C, const double* __restrict__ Jg, double dtau, double a2,
                                                 double delta) {
    if (threadIdx.x < 6) {
        const double j = Jg[threadIdx.x];
        C.J[threadIdx.x] = j;
        C.Jf[threadIdx.x] = (float)j;
        C.Jm[threadIdx.x] = fabsf((float)j);
    }
    if (threadIdx.x == 0) {
        C.dtau = dtau;
        C.a2 = a2;
        C.delta = delta;
        C.ds = delta * (1.0 / 4503599627370496.0);
        C.dtauf = (float)dtau;
        C.a2f = (float)a2;
        C.deltaf = (float)delta;
        C.plain = !(delta == 0.0 || delta > 1e-250);
    }
}

// Metropolis update of site pair s of colour c in one chain's field (thread s of the half-sweep
// owns site i = s / (L/2) and the slice l of colour c in the pair (2 (s mod L/2), 2 (s mod L/2) + 1)).
// ld is the row stride of the field. Returns 1 if the move was accepted (and written).
//
// Three FP64 operations per site (the proposal), everything else on the FP32 and integer pipes: with the
// operands converted and the uniforms formed in FP64 the kernel was bound by that pipe (two lanes per clock
// per SM): a half-sweep of 512 chains of 16x16, L = 160 took 524 us that way and takes 150 us now.
template <bool kL2>
__device__ __forceinline__ int site_update(double* xfield, int Lx, int Ly, int L, int ld, uint32_t mhalf, uint32_t mlx,
                                           const SweepConst& C, uint32_t key0, uint32_t key1, uint32_t sweep, int c, int s,
                                           uint32_t chain) {
    const int half = L >> 1;
    const int i = fast_div(s, half, mhalf), lp = s - i * half;
    const int iy = fast_div(i, Lx, mlx), ix = i - iy * Lx;
    const int l = 2 * lp + ((ix + iy + c) & 1);
    double* xi = xfield + (size_t)i * ld;
    const double v = ldx<kL2>(xi + l);
    const double up = ldx<kL2>(xi + (l + 1 == L ? 0 : l + 1));
    const double dn = ldx<kL2>(xi + (l == 0 ? L - 1 : l - 1));
    const int xp = (ix + 1 == Lx ? 0 : ix + 1) + Lx * iy, xm = (ix == 0 ? Lx - 1 : ix - 1) + Lx * iy;
    const int yp = ix + Lx * (iy + 1 == Ly ? 0 : iy + 1), ym = ix + Lx * (iy == 0 ? Ly - 1 : iy - 1);
    const double n0 = ldx<kL2>(xfield + (size_t)xp * ld + l), n1 = ldx<kL2>(xfield + (size_t)xm * ld + l);
    const double n2 = ldx<kL2>(xfield + (size_t)yp * ld + l), n3 = ldx<kL2>(xfield + (size_t)ym * ld + l);
    const slmc::u32x4 w = slmc::philox4x32_10(slmc::u32x4{(uint32_t)(i * L + l), sweep, chain, 0u}, key0, key1);
    // x' = x + delta (2 u1 - 1), rounded step by step (no contraction) as in the oracle. With u1 = r 2^-53,
    // 2 u1 - 1 = (r - 2^52) 2^-52 is exact: r mod 2^52 is placed in the significand of 2^52 and 2^52 or 2^53 is
    // subtracted (exact), and delta 2^-52 times it rounds as delta times (2 u1 - 1) does.
    double xn;
    if (!C.plain) {
        const double big = __hiloint2double(0x43300000 | (int)((w.x >> 11) & 0xfffffu),
                                            (int)(((w.x << 21) & 0xfc000000u) | (w.y >> 6)));
        const double off = __hiloint2double(0x43400000 - (int)((w.x >> 31) << 20), 0);
        xn = __dadd_rn(v, __dmul_rn(C.ds, __dadd_rn(big, -off)));
    } else {
        const double u1 = slmc::uniform53(w.x, w.y);
        xn = __dadd_rn(v, __dmul_rn(C.delta, __dadd_rn(__dmul_rn(2.0, u1), -1.0)));
    }
    // Fast decision in FP32: dE = d [2 J_k (s - up - dn) + s (J_p ((x'^2 + x^2)/4 - a^2/2)
    //   + J_p' ((x'^4 + x'^2 x^2 + x^4)/6 - a^2 (x'^2 + x^2)/4)) + J_nn nb + J_nn' (up + dn)],
    // d = x' - x, s = x' + x (the exact difference of the local energies, factored), from truncated
    // operands (relative error 2^-23) and d = delta (2 u1 - 1) from the top 23 bits of u1 (absolute
    // error 2^-22 delta, entering the bracket too: at most 5 2^-22 delta in all; and the rounding of
    // x' to FP64, 2^-53 |x'|). The FP32 verdict is used only
    // when the log-ratio is further from log u than a margin bounding (i) the FP32 rounding of the
    // bracket (1e-5 of the sum of the magnitudes of its terms, about 170 units of FP32 rounding),
    // (ii) the error of d, (iii) the truncation of u to 23 bits (log u is known to within 2^-23 / u)
    // and (iv) the hardware logarithm (documented: 2^-21.41 absolute on [0.5, 2], 3 units elsewhere;
    // |log u| < 16, so below 4e-6); otherwise the exact FP64 rule of the oracle decides.
    const float vf = trunc_f32(v), upf = trunc_f32(up), dnf = trunc_f32(dn);
    const float f0 = trunc_f32(n0), f1 = trunc_f32(n1), f2 = trunc_f32(n2), f3 = trunc_f32(n3);
    const float nbf = (f0 + f1) + (f2 + f3), nbm = (fabsf(f0) + fabsf(f1)) + (fabsf(f2) + fabsf(f3));
    const float d = C.deltaf * fmaf(2.f, __uint_as_float(0x3f800000u | (w.x >> 9)), -3.f);
    const float xf = vf + d;
    const float sm = xf + vf, x2 = xf * xf, v2 = vf * vf, q2 = x2 + v2, q4 = fmaf(x2, q2, v2 * v2);
    const float ud = upf + dnf, am = fabsf(upf) + fabsf(dnf), sa = fabsf(xf) + fabsf(vf);
    const float tk = 2.f * C.Jf[1] * (sm - ud);
    const float tp = C.Jf[2] * fmaf(0.25f, q2, -0.5f * C.a2f) + C.Jf[3] * (q4 * (1.f / 6.f) - 0.25f * C.a2f * q2);
    const float tn = C.Jf[4] * nbf + C.Jf[5] * ud;
    const float mag = 2.f * C.Jm[1] * (sa + am) + sa * (C.Jm[2] * (q2 + C.a2f) + C.Jm[3] * (q4 + C.a2f * q2)) +
                      C.Jm[4] * nbm + C.Jm[5] * am;
    const float dlnw32 = -C.dtauf * d * (tk + fmaf(sm, tp, tn));
    const float uf = __uint_as_float(0x3f800000u | (w.z >> 9)) - 1.f;  // top 23 bits of the acceptance uniform
    const float lu = __logf(uf);
    const float margin = 1.4e-5f + C.dtauf * mag * (1e-5f * fabsf(d) + 1.2e-6f * C.deltaf + 1e-14f * sa) +
                         __fdividef(1.3e-7f, uf);
    // uf = 0 makes the margin infinite, an operand out of FP32 range makes mag infinite: both comparisons fail
    int acc = dlnw32 > lu + margin;
    const bool decided = (acc || dlnw32 < lu - margin) && fabsf(dlnw32) < 3e38f;
    if (!decided) {  // exact FP64 rule of the oracle
        const double nb = ((n0 + n1) + n2) + n3;
        const double u2 = slmc::uniform53(w.z, w.w);
        const double dE = local_energy(C.J, C.a2, xn, up, dn, nb) - local_energy(C.J, C.a2, v, up, dn, nb);
        const double dlnw = -C.dtau * dE;
        acc = (dlnw >= 0.0 || u2 < exp(dlnw)) ? 1 : 0;
    }
    if (acc) xi[l] = xn;
    return acc;
}

// One checkerboard half-sweep over all chains: thread s of chain f updates site pair s.
__global__ void __launch_bounds__(kThreads) k_half_sweep(double* __restrict__ x, int Lx, int Ly, int L, uint32_t mhalf,
                                                         uint32_t mlx, const double* __restrict__ Jg, double dtau, double a2,
                                                         double delta, uint32_t key0, uint32_t key1, uint32_t sweep_arg,
                                                         int colour, const int* __restrict__ colour_pc, int cxor,
                                                         int chain0, unsigned long long* __restrict__ n_acc,
                                                         const unsigned long long* __restrict__ dctr, int nsweeps) {
    __shared__ SweepConst C;
    __shared__ int s_cnt;
    sweep_const_init(C, Jg, dtau, a2, delta);
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const int f = blockIdx.y;
    const int N = Lx * Ly, half = L / 2;
    const int s = blockIdx.x * kThreads + threadIdx.x;
    // cumulative updates: sweep counter (update * nsweeps + sweep_arg), update from the device counter
    const uint32_t sweep = dctr ? (uint32_t)((*dctr) * (unsigned long long)nsweeps + sweep_arg) : sweep_arg;
    int accepted = 0;
    if (s < N * half) {
        const int c = colour_pc ? (colour_pc[f] ^ cxor) : colour;
        accepted = site_update<false>(x + (size_t)f * N * L, Lx, Ly, L, L, mhalf, mlx, C, key0, key1, sweep, c, s,
                                      (uint32_t)(chain0 + f));
    }
    const unsigned int ballot = __ballot_sync(0xffffffffu, accepted);
    if ((threadIdx.x & 31) == 0 && ballot) atomicAdd(&s_cnt, __popc(ballot));
    __syncthreads();
    if (threadIdx.x == 0 && n_acc && s_cnt) atomicAdd(n_acc + f, (unsigned long long)s_cnt);
}

// Modified Wolff cluster update of E_eff [Sec. "Wolff update of the effective Hamiltonian",
// Eq. (S9)], one CTA per chain. Bond term b = 2i, (i, i + x^), or 2i + 1, (i, i + y^), of J_nn F_nn
// is activated with probability max(0, 1 - exp(t_b)), t_b = 2 dtau J_nn sum_l x_il x_jl: reflecting
// the whole column of one endpoint multiplies the term's weight by exp(t_b). The sum runs over l
// in order with products and sums rounded separately (as in the oracle, so both take the same
// decisions); the uniform is that of Philox counter (b, ctr, chain, 2), the seed site that of
// (2N, ctr, chain, 2), ctr = (sweep counter) * nwolff + k. The seed's connected component over
// the activated bonds is found by label propagation in shared memory (marks only go from 0 to 1,
// so at most N + 1 rounds) and its columns are reflected, x -> -x. Every other term of E_eff is
// invariant under reflecting whole columns: the move is always accepted.
// One Wolff cluster update of one chain's field xf by the whole CTA (blockDim.x threads); act and
// in_c are 2N and N bytes of shared memory; counter ctr, Philox chain index chain.
template <bool kL2>
__device__ __forceinline__ void wolff_chain(double* xf, int Lx, int Ly, int L, int ld, const double* Jg,
                                            double dtau, uint32_t key0, uint32_t key1, uint32_t ctr, uint32_t chain,
                                            unsigned char* act, unsigned char* in_c, int* s_seed, int* s_cnt,
                                            unsigned long long* __restrict__ n_sites) {
    const int N = Lx * Ly, tid = threadIdx.x;
    const double cfac = __dmul_rn(__dmul_rn(2.0, dtau), Jg[4]);
    for (int b = tid; b < 2 * N; b += blockDim.x) {
        const int i = b >> 1, ix = i % Lx, iy = i / Lx;
        const int j = (b & 1) ? ix + Lx * (iy + 1 == Ly ? 0 : iy + 1) : (ix + 1 == Lx ? 0 : ix + 1) + Lx * iy;
        const double* xi = xf + (size_t)i * ld;
        const double* xj = xf + (size_t)j * ld;
        double sb = 0.0;
        for (int l = 0; l < L; ++l) sb = __dadd_rn(sb, __dmul_rn(ldx<kL2>(xi + l), ldx<kL2>(xj + l)));
        const double t = __dmul_rn(cfac, sb);
        unsigned char a = 0;
        if (t < 0.0) {
            const slmc::u32x4 w = slmc::philox4x32_10(slmc::u32x4{(uint32_t)b, ctr, chain, 2u}, key0, key1);
            a = slmc::uniform53(w.x, w.y) < __dadd_rn(1.0, -exp(t));
        }
        act[b] = a;
    }
    if (tid == 0) {
        const slmc::u32x4 w = slmc::philox4x32_10(slmc::u32x4{(uint32_t)(2 * N), ctr, chain, 2u}, key0, key1);
        const int s0 = (int)(slmc::uniform53(w.x, w.y) * (double)N);
        *s_seed = s0 < N - 1 ? s0 : N - 1;
        *s_cnt = 0;
    }
    __syncthreads();
    for (int i = tid; i < N; i += blockDim.x) in_c[i] = (i == *s_seed);
    __syncthreads();
    for (int round = 0; round <= N; ++round) {
        int changed = 0;
        for (int b = tid; b < 2 * N; b += blockDim.x) {
            if (!act[b]) continue;
            const int i = b >> 1, ix = i % Lx, iy = i / Lx;
            const int j = (b & 1) ? ix + Lx * (iy + 1 == Ly ? 0 : iy + 1) : (ix + 1 == Lx ? 0 : ix + 1) + Lx * iy;
            if (in_c[i] != in_c[j]) {
                in_c[i] = 1;
                in_c[j] = 1;
                changed = 1;
            }
        }
        if (!__syncthreads_or(changed)) break;
    }
    int cnt = 0;
    for (int i = tid; i < N; i += blockDim.x) cnt += in_c[i];
    const int lane = tid & 31;
    for (int i = tid >> 5; i < N; i += blockDim.x >> 5)
        if (in_c[i])
            for (int l = lane; l < L; l += 32) xf[(size_t)i * ld + l] = -ldx<kL2>(xf + (size_t)i * ld + l);
    if (n_sites) {
        atomicAdd(s_cnt, cnt);
        __syncthreads();
        if (tid == 0) atomicAdd(n_sites, (unsigned long long)*s_cnt);
    }
}

__global__ void __launch_bounds__(256) k_wolff(double* __restrict__ x, int Lx, int Ly, int L,
                                               const double* __restrict__ Jg, double dtau, uint32_t key0,
                                               uint32_t key1, uint32_t sweep_arg,
                                               const unsigned long long* __restrict__ dctr, int nsweeps, int nwolff,
                                               int k, int chain0, unsigned long long* __restrict__ n_sites) {
    extern __shared__ unsigned char wsm[];
    const int N = Lx * Ly;
    __shared__ int s_seed, s_cnt;
    const int f = blockIdx.x;
    const uint32_t sweep = dctr ? (uint32_t)((*dctr) * (unsigned long long)nsweeps + sweep_arg) : sweep_arg;
    const uint32_t ctr = sweep * (uint32_t)nwolff + (uint32_t)k;
    wolff_chain<false>(x + (size_t)f * N * L, Lx, Ly, L, L, Jg, dtau, key0, key1, ctr, (uint32_t)(chain0 + f), wsm,
                       wsm + 2 * N, &s_seed, &s_cnt, n_sites);
}

// Every sweep of a call for one chain per CTA, the chain's field in shared memory from the first
// half-sweep to the last: one launch and one read and write of the field for nsweeps sweeps, block
// barriers between the colours and the Wolff updates. A small chain's half-sweep is shorter than its
// launch, and the many launches of the kernel-per-half-sweep path were its time. Rows are padded to the odd stride
// L + 1, so the Wolff bond sums (a column per lane) meet no bank conflicts. Site and Wolff arithmetic and
// random numbers are those of k_half_sweep / k_wolff: bit-identical chains.
__global__ void __launch_bounds__(1024) k_chain_sweeps(double* __restrict__ x, int Lx, int Ly, int L, uint32_t mhalf,
                                                       uint32_t mlx, const double* __restrict__ Jg, double dtau, double a2,
                                                       double delta, uint32_t key0, uint32_t key1, uint32_t sweep_arg,
                                                       int nsweeps, int colour, const int* __restrict__ colour_pc,
                                                       int chain0, int nwolff, unsigned long long* __restrict__ n_acc,
                                                       unsigned long long* __restrict__ n_sites,
                                                       const unsigned long long* __restrict__ dctr, int ctr_mul) {
    extern __shared__ double csm[];
    __shared__ SweepConst C;
    __shared__ int s_cnt, s_seed, s_wcnt;
    const int f = blockIdx.x, N = Lx * Ly, ld = L + 1, sites = N * (L / 2), tid = threadIdx.x;
    unsigned char* act = reinterpret_cast<unsigned char*>(csm + (size_t)N * ld);
    double* xf = x + (size_t)f * N * L;
    sweep_const_init(C, Jg, dtau, a2, delta);
    if (tid == 0) s_cnt = 0;
    for (int i = tid >> 5; i < N; i += blockDim.x >> 5)
        for (int l = tid & 31; l < L; l += 32) csm[i * ld + l] = xf[(size_t)i * L + l];
    const uint32_t sweep0 = dctr ? (uint32_t)((*dctr) * (unsigned long long)ctr_mul + sweep_arg) : sweep_arg;
    const int first = colour_pc ? colour_pc[f] : colour;
    const uint32_t chain = (uint32_t)(chain0 + f);
    int accepted = 0;
    __syncthreads();
    for (int sw = 0; sw < nsweeps; ++sw) {
        const uint32_t sweep = sweep0 + (uint32_t)sw;
        for (int h = 0; h < 2; ++h) {
            if (h == 1)
                for (int k = 0; k < nwolff; ++k) {
                    wolff_chain<false>(csm, Lx, Ly, L, ld, C.J, dtau, key0, key1, sweep * (uint32_t)nwolff + (uint32_t)k,
                                       chain, act, act + 2 * N, &s_seed, &s_wcnt, n_sites);
                    __syncthreads();
                }
            for (int s = tid; s < sites; s += blockDim.x)
                accepted += site_update<false>(csm, Lx, Ly, L, ld, mhalf, mlx, C, key0, key1, sweep, first ^ h, s, chain);
            __syncthreads();
        }
    }
    accepted = __reduce_add_sync(0xffffffffu, accepted);
    if ((tid & 31) == 0 && accepted) atomicAdd(&s_cnt, accepted);
    for (int i = tid >> 5; i < N; i += blockDim.x >> 5)
        for (int l = tid & 31; l < L; l += 32) xf[(size_t)i * L + l] = csm[i * ld + l];
    __syncthreads();
    if (tid == 0 && n_acc && s_cnt) atomicAdd(n_acc + f, (unsigned long long)s_cnt);
}

// Persistent E_eff sweep queue: the half-sweep slabs and Wolff updates of every chain of several
// lattice classes, pulled in queue order by the CTAs of one launch. The queue lists, phase after
// phase (colour 0, the Wolff updates, colour 1 of each sweep), the items of every chain in order of
// decreasing N L (longest first), so every item depends only on earlier ones: item q of chain g
// waits until g's completion counter reaches its count of g's earlier items. A CTA takes an item
// only while it runs, so all items it waits on are held by running CTAs, and the launch cannot
// deadlock whatever the grid size. Values written by other CTAs of the launch are read through L2
// (__ldcg); a CTA publishes an item after a barrier and a device-scope fence. The arithmetic of a
// site update or a Wolff update is the one of k_half_sweep / k_wolff (shared device functions), so
// the chains are bit-identical to the kernel-per-half-sweep path.
//
// Every wait is bounded: after wait_cycles the CTA sets SLMC_EBIT_TIMEOUT in the error word of
// every class and the abort word ctl[1]; every CTA stops taking items once it sees the abort.
__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__global__ void __launch_bounds__(kThreads) k_sweep_queue(const slmc::QueueClass* __restrict__ cls, int ncls,
                                                          const int4* __restrict__ items, int nitems,
                                                          unsigned int* __restrict__ done, unsigned int* __restrict__ ctl,
                                                          uint32_t u, long long wait_cycles) {
    extern __shared__ unsigned char qsm[];
    __shared__ SweepConst K;
    __shared__ int s_item, s_cnt, s_seed, s_wcnt;
    for (;;) {
        if (threadIdx.x == 0) {
            int q = -1;
            if (ld_acquire_u32(ctl + 1) == 0u) q = (int)atomicAdd(ctl, 1u);
            if (q >= nitems) q = -1;
            if (q >= 0) {
                const int4 it = items[q];
                const slmc::QueueClass& C = cls[it.x >> 24];
                const unsigned int* cnt = done + C.done0 + (it.x & 0xffffff);
                const long long t0 = clock64();
                while (ld_acquire_u32(cnt) < (unsigned int)it.w) {
                    if (ld_acquire_u32(ctl + 1) != 0u) {
                        q = -1;
                        break;
                    }
                    if (clock64() - t0 > wait_cycles) {
                        for (int k = 0; k < ncls; ++k) atomicOr(cls[k].err, SLMC_EBIT_TIMEOUT);
                        atomicExch(ctl + 1, 1u);
                        q = -1;
                        break;
                    }
                    __nanosleep(100);
                }
            }
            s_item = q;
            s_cnt = 0;
        }
        __syncthreads();
        const int q = s_item;
        if (q < 0) break;
        const int4 it = items[q];
        const slmc::QueueClass& C = cls[it.x >> 24];
        const int f = it.x & 0xffffff;
        sweep_const_init(K, C.J, C.dtau, C.a2, C.delta);
        __syncthreads();
        const int N = C.Lx * C.Ly;
        double* xf = C.x + (size_t)f * N * C.L;
        const int sw = it.y >> 8, sub = it.y & 0x7f;
        const uint32_t chain = (uint32_t)f;
        const uint32_t sweep = (uint32_t)((*C.dctr) * (unsigned long long)C.nsweeps +
                                          (unsigned long long)u * C.nsweeps + sw);
        if (it.y & 0x80) {
            const uint32_t ctr = sweep * (uint32_t)C.nwolff + (uint32_t)sub;
            wolff_chain<true>(xf, C.Lx, C.Ly, C.L, C.L, K.J, C.dtau, C.key0, C.key1, ctr, chain, qsm, qsm + 2 * N, &s_seed,
                              &s_wcnt, C.wolff_sites);
        } else {
            const int sites = N * (C.L / 2);
            const int c = C.first_colour[f] ^ sub;
            int accepted = 0;
            for (int j = 0; j < slmc::kQueueSlab / kThreads; ++j) {
                const int st = it.z * slmc::kQueueSlab + j * kThreads + threadIdx.x;
                if (st < sites)
                    accepted += site_update<true>(xf, C.Lx, C.Ly, C.L, C.L, C.mhalf, C.mlx, K, C.key0, C.key1, sweep,
                                                  c, st, chain);
            }
            if (accepted) atomicAdd(&s_cnt, accepted);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            if (!(it.y & 0x80) && C.n_acc && s_cnt) atomicAdd(C.n_acc + f, (unsigned long long)s_cnt);
            __threadfence();
            atomicAdd(done + C.done0 + f, 1u);
        }
    }
}

__global__ void k_update_draws(int nf, int chain0, uint32_t u_off, const unsigned long long* __restrict__ dctr,
                               uint32_t key0, uint32_t key1, int* __restrict__ first, double* __restrict__ u) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nf) return;
    const uint32_t update = (uint32_t)(*dctr + u_off);
    const slmc::u32x4 w = slmc::philox4x32_10(slmc::u32x4{update, 0u, (uint32_t)(chain0 + f), 1u}, key0, key1);
    first[f] = (int)(w.x & 1u);
    u[f] = slmc::uniform53(w.z, w.w);
}

__global__ void k_accept(int nf, const double* __restrict__ lnw_new, const double* __restrict__ lnweff_old,
                         const double* __restrict__ lnweff_new, const double* __restrict__ u, double* __restrict__ lnw,
                         int* __restrict__ accepted, unsigned long long* __restrict__ n_acc) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= nf) return;
    const double lnA = (lnw_new[f] - lnw[f]) - (lnweff_new[f] - lnweff_old[f]);
    const bool acc = lnA >= 0.0 || u[f] < exp(lnA);
    accepted[f] = acc ? 1 : 0;
    if (acc) {
        lnw[f] = lnw_new[f];
        if (n_acc) n_acc[f] += 1ull;
    }
}

__global__ void k_restore(double* __restrict__ x, const double* __restrict__ x_old, const int* __restrict__ accepted,
                          int NL) {
    const int f = blockIdx.y;
    if (accepted[f]) return;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < NL; idx += gridDim.x * blockDim.x)
        x[(size_t)f * NL + idx] = x_old[(size_t)f * NL + idx];
}

__global__ void __launch_bounds__(kThreads) k_cdw(const double* __restrict__ G, int Lx, int Ly, double* __restrict__ S,
                                                  const int* __restrict__ only_if, double* __restrict__ obs) {
    __shared__ double red[3 * kThreads];
    const int f = blockIdx.x;
    const int N = Lx * Ly;
    const size_t NN = (size_t)N * N;
    const bool update = !only_if || only_if[f];
    if (update) {
        const double* Gf = G + f * NN;
        double acc[3] = {0.0, 0.0, 0.0};  // sum s_i (1 - G_ii), sum G_ii, sum s_i s_j G_ij G_ji
        for (int i = threadIdx.x; i < N; i += kThreads) {
            const double si = (((i % Lx) + (i / Lx)) & 1) ? -1.0 : 1.0;
            const double g = Gf[(size_t)i * N + i];
            acc[0] += si * (1.0 - g);
            acc[1] += g;
        }
        for (size_t idx = threadIdx.x; idx < NN; idx += kThreads) {
            const int i = (int)(idx / N), j = (int)(idx - (size_t)i * N);
            const double sij = ((((i % Lx) + (i / Lx)) ^ ((j % Lx) + (j / Lx))) & 1) ? -1.0 : 1.0;
            acc[2] += sij * Gf[idx] * Gf[(size_t)j * N + i];
        }
        block_sum<3>(acc, red);  // block-uniform branch: `update` depends on f only
        if (threadIdx.x == 0) S[f] = (4.0 * acc[0] * acc[0] + 2.0 * acc[1] - 2.0 * acc[2]) / N;
    }
    if (obs && threadIdx.x == 0) obs[f] = S[f];
}

// ---- regression: Givens-rotation QR of the rows [1, (F - F_ref)/sc, y - y_ref] into a 7x7 R ----
// fitR layout: R[7][7] row-major (0..48), ref[6] (49..54: F_ref[5], y_ref), flag (55), count (56).
__global__ void k_fit_begin(double* __restrict__ R) {
    for (int q = threadIdx.x; q < 64; q += blockDim.x) R[q] = 0.0;
}

// Absorbs one row (lane m < 7 holds its element m) into the triangular factor held by the warp
// (lane m holds column m of every row of R) with Givens rotations.
__device__ __forceinline__ void givens_absorb(double (&Rrow)[7], double a, int lane) {
    for (int k = 0; k < 7; ++k) {
        const double ak = __shfl_sync(0xffffffffu, a, k);
        const double rkk = __shfl_sync(0xffffffffu, Rrow[k], k);
        if (ak == 0.0) continue;
        const double r = hypot(rkk, ak);
        const double cs = rkk / r, sn = ak / r;
        if (lane == k) {
            Rrow[k] = r;
            a = 0.0;
        } else if (lane > k && lane < 7) {
            const double rk = Rrow[k];
            Rrow[k] = cs * rk + sn * a;
            a = -sn * rk + cs * a;
        }
    }
}

// Absorbs nconf rows into the triangle, up to 2048 per pass, by Householder reflections of [R; rows] in one CTA:
// the rows stay in registers (up to four per thread), and the reflector of column k touches row k of R and the rows
// only. The products of column k with itself and with the columns right of it are reduced together (one block
// reduction per column); scaling by the reflector's normalisation comes after. Row k of R takes the sign that
// makes its diagonal non-negative, as the Givens merge below leaves it. A fit of 4x4, L = 40 takes
// 60 us with 6 to 100 rows, 103 with 500, 128 with 2000 (512 threads whatever the rows: 100 with 6, 192 with 2000).
// Couplings against quad precision, geometric mean of 120 fits: 1.6e-13.
constexpr int kFitThreads = 512, kFitMinThreads = 224 /* a warp per column */, kFitPer = 4;

__global__ void __launch_bounds__(kFitThreads) k_fit_accumulate(double* __restrict__ R, const double* __restrict__ feat,
                                                                int ldF, const double* __restrict__ lnw, int nconf,
                                                                double sc) {
    __shared__ double sR[49], ref[6], part[7][kFitThreads / 32], dot[7], par[2];  // par: tau, scal
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x, NW = T / 32;
    if (tid == 0 && R[55] == 0.0) {
        for (int q = 0; q < 5; ++q) R[49 + q] = feat[q];
        R[54] = lnw[0];
        R[55] = 1.0;
    }
    __syncthreads();
    if (tid < 49) sR[tid] = R[tid];
    if (tid >= 64 && tid < 70) ref[tid - 64] = R[49 + tid - 64];
    __syncthreads();
    const double inv = 1.0 / sc;
    for (int c0 = 0; c0 < nconf; c0 += kFitPer * T) {
        double a[kFitPer][7];
        const int left = nconf - c0 - 32 * warp, nr = left <= 0 ? 0 : min(kFitPer, (left + T - 1) / T);  // the warp's rows
#pragma unroll
        for (int r = 0; r < kFitPer; ++r) {
            const int c = c0 + r * T + tid;
            const bool on = c < nconf;
            a[r][0] = on ? 1.0 : 0.0;
#pragma unroll
            for (int q = 0; q < 5; ++q) a[r][q + 1] = on ? (feat[(size_t)c * ldF + q] - ref[q]) * inv : 0.0;
            a[r][6] = on ? lnw[c] - ref[5] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < 7; ++k) {
#pragma unroll
            for (int m = k; m < 7; ++m) {
                double t = 0.0;
                if (nr > 0) {
#pragma unroll
                    for (int r = 0; r < kFitPer; ++r)
                        if (r < nr) t = fma(a[r][k], a[r][m], t);
                    t = slmc::warp_allsum(t);
                }
                if (lane == 0) part[m][warp] = t;
            }
            __syncthreads();
            if (warp >= k && warp < 7) {  // warp m finishes product m
                const double t = slmc::warp_allsum(lane < NW ? part[warp][lane] : 0.0);
                if (lane == 0) dot[warp] = t;
            }
            __syncthreads();
            if (warp == 0) {
                const double alpha = sR[k * 7 + k], sig = dot[k];
                double tau = 0.0, beta = alpha, scal = 0.0;
                if (sig != 0.0) {
                    const double nrm = sqrt(fma(alpha, alpha, sig));
                    beta = (alpha >= 0.0) ? -nrm : nrm;
                    tau = (beta - alpha) / beta;
                    scal = 1.0 / (alpha - beta);
                }
                __syncwarp();
                if (lane == 0) {
                    sR[k * 7 + k] = fabs(beta);
                    par[0] = tau;
                    par[1] = scal;
                }
                if (lane > k && lane < 7) {  // row k of R: R_km -= tau (R_km + v . a_m)
                    const double d = tau * fma(scal, dot[lane], sR[k * 7 + lane]);
                    const double v = sR[k * 7 + lane] - d;
                    sR[k * 7 + lane] = beta < 0.0 ? -v : v;
                    dot[lane] = d;
                }
            }
            __syncthreads();
            const double scal = par[1];
#pragma unroll
            for (int m = k + 1; m < 7; ++m) {
                const double d = dot[m] * scal;
#pragma unroll
                for (int r = 0; r < kFitPer; ++r)
                    if (r < nr) a[r][m] = fma(-d, a[r][k], a[r][m]);
            }
            __syncthreads();  // part and dot are rewritten by the next column
        }
    }
    if (tid < 49) R[tid] = sR[tid];
    if (tid == 0) R[56] += nconf;
}

// Merges partial states (same layout as R) into R. Each state's factor is first moved to the
// reference of the first non-empty state: its rows [1, (F - F_b)/sc, y - y_b] equal the rows
// [1, (F - F_c)/sc, y - y_c] minus row 0 times d, d = ((F_b - F_c)/sc, y_b - y_c), i.e. the
// columns change by a unit upper-triangular matrix, which touches only row 0 of R.
__global__ void k_fit_merge(const double* __restrict__ states, int nparts, double* __restrict__ R, double sc) {
    const int lane = threadIdx.x;
    int ref = -1;
    for (int p = 0; p < nparts; ++p)
        if (states[(size_t)p * SLMC_FIT_STATE_DOUBLES + 55] != 0.0) {
            ref = p;
            break;
        }
    const double* C = states + (size_t)(ref < 0 ? 0 : ref) * SLMC_FIT_STATE_DOUBLES;
    double Rrow[7];
    for (int k = 0; k < 7; ++k) Rrow[k] = 0.0;
    double count = 0.0;
    for (int p = 0; p < nparts; ++p) {
        const double* S = states + (size_t)p * SLMC_FIT_STATE_DOUBLES;
        if (S[55] == 0.0) continue;
        count += S[56];
        for (int k = 0; k < 7; ++k) {
            double a = (lane < 7) ? S[k * 7 + lane] : 0.0;
            if (k == 0 && lane >= 1 && lane < 7) {
                const double d = (lane < 6) ? (S[49 + lane - 1] - C[49 + lane - 1]) / sc : S[54] - C[54];
                a = fma(S[0], d, a);
            }
            givens_absorb(Rrow, a, lane);
        }
    }
    for (int k = 0; k < 7; ++k)
        if (lane < 7) R[k * 7 + lane] = Rrow[k];
    if (lane < 6) R[49 + lane] = (ref < 0) ? 0.0 : C[49 + lane];
    if (lane == 0) {
        R[55] = (ref < 0) ? 0.0 : 1.0;
        R[56] = count;
    }
    if (lane >= 7 && lane < 14) R[57 + lane - 7] = 0.0;
}

__global__ void k_fit_finish(const double* __restrict__ R, double dtau, double sc, double* __restrict__ J,
                             double* __restrict__ resid, unsigned int* __restrict__ err) {
    if (threadIdx.x != 0) return;
    double c[6];
    bool ok = true;
    for (int k = 5; k >= 0; --k) {
        double s = R[k * 7 + 6];
        for (int m = k + 1; m < 6; ++m) s -= R[k * 7 + m] * c[m];
        if (R[k * 7 + k] == 0.0) ok = false;
        c[k] = s / R[k * 7 + k];
    }
    double icpt = c[0] + R[54];
    for (int q = 0; q < 5; ++q) icpt -= c[q + 1] * R[49 + q] / sc;
    J[0] = -icpt / dtau;
    for (int q = 0; q < 5; ++q) J[q + 1] = -(c[q + 1] / sc) / dtau;
    if (resid) resid[0] = fabs(R[6 * 7 + 6]) / sqrt(fmax(R[56], 1.0));
    if (!ok) atomicOr(err, SLMC_EBIT_SINGULAR);
}

}  // namespace

namespace slmc {

// Multiplier of fast_div for dividends below n (0 where n d reaches 2^32: the kernel divides).
uint32_t div_magic(long long n, int d) {
    if (d < 2 || n * d >= (1ll << 32)) return 0u;
    return (uint32_t)(((1ull << 32) + d - 1) / (unsigned)d);
}

cudaError_t bose_log_weight(slmc_ctx* c, const double* x, int nf, const double* lndet, double* lnw, cudaStream_t s) {
    k_bose<<<nf, kThreads, 0, s>>>(x, c->N, c->L, c->p.dtau, c->p.lambda, c->p.omega0 * c->p.omega0, lndet, lnw);
    return cudaGetLastError();
}

cudaError_t eff_features(slmc_ctx* c, const double* x, int nf, const double* J, double* F, int ldF, double* lnw_eff,
                         cudaStream_t s) {
    const double a = c->p.lambda / (c->p.omega0 * c->p.omega0);
    k_features<<<nf, kThreads, 0, s>>>(x, c->p.Lx, c->p.Ly, c->L, div_magic(kThreads, c->L), div_magic(c->N, c->p.Lx),
                                       kThreads / c->L, a * a, c->p.dtau, J, F, ldF, lnw_eff);
    return cudaGetLastError();
}

cudaError_t eff_half_sweep(slmc_ctx* c, double* x, int nf, int chain0, const double* J, uint64_t sweep, int colour,
                           const int* colour_per_chain, int colour_xor, long long* n_acc, cudaStream_t s,
                           const unsigned long long* dctr, int nsweeps) {
    const double a = c->p.lambda / (c->p.omega0 * c->p.omega0);
    const int sites = c->N * (c->L / 2);
    dim3 grid((sites + kThreads - 1) / kThreads, nf);
    k_half_sweep<<<grid, kThreads, 0, s>>>(x, c->p.Lx, c->p.Ly, c->L, div_magic(sites, c->L / 2),
                                           div_magic(c->N, c->p.Lx), J, c->p.dtau, a * a, c->p.sweep_delta,
                                           (uint32_t)(c->p.seed & 0xffffffffu), (uint32_t)(c->p.seed >> 32),
                                           (uint32_t)sweep, colour, colour_per_chain, colour_xor, chain0,
                                           reinterpret_cast<unsigned long long*>(n_acc), dctr, nsweeps);
    return cudaGetLastError();
}

cudaError_t update_draws(slmc_ctx* c, int nf, int chain0, uint64_t u_off, int* first_colour, double* u_acc,
                         cudaStream_t s) {
    k_update_draws<<<(nf + 127) / 128, 128, 0, s>>>(nf, chain0, (uint32_t)u_off, c->dctr, (uint32_t)(c->p.seed & 0xffffffffu),
                                                    (uint32_t)(c->p.seed >> 32), first_colour, u_acc);
    return cudaGetLastError();
}

cudaError_t accept_update(slmc_ctx* c, int nf, double* x, const double* x_old, const double* lnw_new,
                          const double* lnweff_old, const double* lnweff_new, const double* u_acc, double* lnw,
                          int* accepted, long long* n_acc, cudaStream_t s) {
    k_accept<<<(nf + 127) / 128, 128, 0, s>>>(nf, lnw_new, lnweff_old, lnweff_new, u_acc, lnw, accepted,
                                              reinterpret_cast<unsigned long long*>(n_acc));
    const int NL = c->N * c->L;
    dim3 grid((NL + 255) / 256 < 64 ? (NL + 255) / 256 : 64, nf);
    k_restore<<<grid, 256, 0, s>>>(x, x_old, accepted, NL);
    return cudaGetLastError();
}

cudaError_t eff_wolff(slmc_ctx* c, double* x, int nf, int chain0, const double* J, uint64_t sweep, int k,
                      cudaStream_t s, const unsigned long long* dctr, int nsweeps) {
    k_wolff<<<nf, 256, 3 * c->N, s>>>(x, c->p.Lx, c->p.Ly, c->L, J, c->p.dtau, (uint32_t)(c->p.seed & 0xffffffffu),
                                      (uint32_t)(c->p.seed >> 32), (uint32_t)sweep, dctr, nsweeps, c->nwolff, k,
                                      chain0, c->wolff_sites);
    return cudaGetLastError();
}

// Whether the sweeps of n chains run in one launch, a chain per SM with its field in shared memory (up to 8192
// sites times slices, two CTAs per SM), or as a launch per half-sweep that spreads the chains over the GPU. With
// Wolff updates (a launch each otherwise) one launch is faster at any n: 1 chain of 8x8, L = 40, 20 sweeps 223 us
// against 386, of 8x8, L = 128, 515 against 684, 16 chains 536 against 785. Without them it is for up to 4096
// values (8x8, L = 40: 123 against 182 us for 1 chain, 126 against 226 for 16; 4x4, L = 240: 153 / 182), and above
// once there are enough chains for the half-sweeps to grow: 20 sweeps of 5120, 6144, 7168 and 8192 values take 195,
// 220, 255 and 280 us in one launch for 1 to 16 chains; launches per half-sweep 186 to 190 us for one
// chain, 208, 210, 216, 219 for 4, 226, 229, 235, 242 for 8, 249, 252, 255, 256 for 16 (and at 8192 values 338 for 32).
constexpr int kChainSites = 8192, kChainSitesAny = 4096;

bool eff_sweeps_fused(const slmc_ctx* c, int n) {
    const long long sites = c->N * (long long)c->L;
    if (sites > kChainSites) return false;
    int most = kChainSitesAny;  // and 1024 more for every doubling of n from 4 on
    for (int m = n; m >= 4; m >>= 1) most += 1024;
    return c->nwolff > 0 || sites <= most;
}

cudaError_t eff_chain_sweeps(slmc_ctx* c, double* x, int nf, int chain0, const double* J, uint64_t sweep0, int nsweeps,
                             int colour, const int* colour_per_chain, long long* n_acc, cudaStream_t s,
                             const unsigned long long* dctr, int ctr_mul) {
    const double a = c->p.lambda / (c->p.omega0 * c->p.omega0);
    const int sites = c->N * (c->L / 2), iters = (sites + 1023) / 1024;
    const int threads = std::max(64, ((sites + iters - 1) / iters + 31) / 32 * 32);
    const size_t smem = (size_t)c->N * (c->L + 1) * sizeof(double) + 3 * (size_t)c->N;
    cudaError_t e = slmc::allow_smem(k_chain_sweeps, smem);
    if (e != cudaSuccess) return e;
    k_chain_sweeps<<<nf, threads, smem, s>>>(
        x, c->p.Lx, c->p.Ly, c->L, div_magic(sites, c->L / 2), div_magic(c->N, c->p.Lx), J, c->p.dtau, a * a,
        c->p.sweep_delta, (uint32_t)(c->p.seed & 0xffffffffu), (uint32_t)(c->p.seed >> 32), (uint32_t)sweep0, nsweeps,
        colour, colour_per_chain, chain0, c->nwolff, reinterpret_cast<unsigned long long*>(n_acc), c->wolff_sites, dctr,
        ctr_mul);
    return cudaGetLastError();
}

int sweep_queue_grid() {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sweep_queue, kThreads, 3 * 1024) != cudaSuccess)
        return 0;
    return sms * (per_sm < 1 ? 1 : per_sm);
}

cudaError_t sweep_queue(const QueueClass* classes, int ncls, const int4* items, int nitems, unsigned int* done,
                        unsigned int* ctl, int max_N, uint32_t u, long long wait_cycles, int grid, cudaStream_t s) {
    k_sweep_queue<<<grid, kThreads, 3 * max_N, s>>>(classes, ncls, items, nitems, done, ctl, u, wait_cycles);
    return cudaGetLastError();
}

cudaError_t cdw_measure(slmc_ctx* c, const double* G, int nf, double* S, const int* only_if, double* obs,
                        cudaStream_t s) {
    k_cdw<<<nf, kThreads, 0, s>>>(G, c->p.Lx, c->p.Ly, S, only_if, obs);
    return cudaGetLastError();
}

__global__ void k_counter(unsigned long long* __restrict__ ctr, unsigned long long v, int add) {
    if (threadIdx.x == 0) *ctr = add ? *ctr + v : v;
}

cudaError_t counter_op(slmc_ctx* c, uint64_t v, bool add, cudaStream_t s) {
    k_counter<<<1, 32, 0, s>>>(c->dctr, (unsigned long long)v, add ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t fit_begin(slmc_ctx* c, double* R, cudaStream_t s) {
    (void)c;
    k_fit_begin<<<1, 64, 0, s>>>(R);
    return cudaGetLastError();
}

cudaError_t fit_accumulate(slmc_ctx* c, double* R, const double* feat, const double* lnw, int nconf, cudaStream_t s) {
    // a row per thread while they fit: warps without rows would only lengthen the FP64 queue
    const int threads = std::min(kFitThreads, std::max(kFitMinThreads, (nconf + 31) / 32 * 32));
    k_fit_accumulate<<<1, threads, 0, s>>>(R, feat, 8, lnw, nconf, (double)c->N * c->L);
    return cudaGetLastError();
}

cudaError_t fit_merge(slmc_ctx* c, const double* states, int nparts, cudaStream_t s) {
    k_fit_merge<<<1, 32, 0, s>>>(states, nparts, c->fitR, (double)c->N * c->L);
    return cudaGetLastError();
}

cudaError_t fit_finish(slmc_ctx* c, int nconf, double* J_out, double* resid, cudaStream_t s) {
    (void)nconf;
    k_fit_finish<<<1, 32, 0, s>>>(c->fitR, c->p.dtau, (double)c->N * c->L, J_out, resid, c->err);
    return cudaGetLastError();
}

}  // namespace slmc
