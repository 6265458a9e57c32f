// Set-up kernels: Grunwald weights (eq. (1.2)), FFT twiddles, the FFT symbol of the
// circulant embedding of the shifted-Grunwald Toeplitz matrix G (eq. (1.5)), the
// Strang symbols phi_k / psi_k (Sec. 3.1) and the right-hand side of eq. (1.10).
#include "fde_internal.h"
#include "bfp_device.cuh"
#include "fft_device.cuh"

namespace fde {

// g_0 = 1, g_{k+1} = (1 - (alpha+1)/(k+1)) g_k (eq. (1.2)).  One CTA of 256: thread t runs
// the recurrence over its own contiguous chunk of factors starting from 1, the chunk
// products are scanned across the threads (multiplicative prefix), and each thread rescales
// its chunk.  The result is the same product of the same factors as the sequential
// recurrence, associated differently (a few ulps apart).  (The chain of FP64 divisions is what
// takes time: 58 us at m = 4095 by one warp.)
__device__ __forceinline__ void grunwald_weights(double alpha, int count, double* __restrict__ g) {
    __shared__ double warp_prod[8];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int chunk = (count + 255) / 256;
    const int k0 = t * chunk;  // this thread produces g[k0+1 .. k0+chunk]
    double prod = 1.0;
    for (int k = k0; k < k0 + chunk && k + 1 < count; ++k) {
        prod *= (1.0 - (alpha + 1.0) / (double)(k + 1));
        g[k + 1] = prod;  // partial product, rescaled below
    }
    double pre = prod;  // inclusive scan of chunk products over the warp
    for (int off = 1; off < 32; off <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, pre, off);
        if (lane >= off) pre *= v;
    }
    if (lane == 31) warp_prod[warp] = pre;
    double excl = __shfl_up_sync(0xffffffffu, pre, 1);
    if (lane == 0) excl = 1.0;
    __syncthreads();
    for (int w = 0; w < warp; ++w) excl *= warp_prod[w];
    for (int k = k0; k < k0 + chunk && k + 1 < count; ++k) g[k + 1] *= excl;
    if (t == 0) g[0] = 1.0;
}

// Everything that depends on (alpha, m, s, scheme) alone, in one launch (seven small ones took
// as long as the symbol transform that follows): CTA 0 the Grunwald weights, the others one
// table entry a thread -- exp(-2 pi i k / L) in FP64 and FP32 for k < L, exp(-2 pi i k / s) for
// k < s, the block floating-point twiddles (k < L, then the first L/2 in bit-reversed
// order), and the Strang symbols
//   phi_k = sum_{r=-nu}^{mu-nu} a_{r+nu} exp(2 pi i r k / s), psi_k likewise with b, k = 0..s/2.
struct TableArgs {
    double alpha;
    int m, logL, s, mu, nu;
    double a[FDE_MAX_MU + 1], b[FDE_MAX_MU + 1];
    double* g;
    double2* twL;
    float2* twL32;
    double2* tws;
    float2* tws32;
    bfp::Tw* twq;
    double2* phi;
    double2* psi;
};
__global__ void __launch_bounds__(256) tables_kernel(const __grid_constant__ TableArgs A) {
    if (blockIdx.x == 0) {
        grunwald_weights(A.alpha, A.m + 2, A.g);
        return;
    }
    const int L = 1 << A.logL, s = A.s;
    int k = (blockIdx.x - 1) * blockDim.x + threadIdx.x;
    if (k < L) {
        double sn, cs;
        sincospi(-2.0 * (double)k / (double)L, &sn, &cs);
        A.twL[k] = make_double2(cs, sn);
        A.twL32[k] = make_float2((float)cs, (float)sn);
        return;
    }
    k -= L;
    if (k < s) {
        double sn, cs;
        sincospi(-2.0 * (double)k / (double)s, &sn, &cs);
        A.tws[k] = make_double2(cs, sn);
        A.tws32[k] = make_float2((float)cs, (float)sn);
        return;
    }
    k -= s;
    if (k < L + L / 2) {
        A.twq[k] = bfp::twiddle(k < L ? k : bitrev(k - L, A.logL - 1), A.logL);
        return;
    }
    k -= L + L / 2;
    if (k <= s / 2) {
        double pr = 0, pi = 0, qr = 0, qi = 0;
        for (int r = -A.nu; r <= A.mu - A.nu; ++r) {
            long rk = ((long)r * k) % s;
            double sn, cs;
            sincospi(2.0 * (double)rk / (double)s, &sn, &cs);
            pr += A.a[r + A.nu] * cs;
            pi += A.a[r + A.nu] * sn;
            qr += A.b[r + A.nu] * cs;
            qi += A.b[r + A.nu] * sn;
        }
        A.phi[k] = make_double2(pr, pi);
        A.psi[k] = make_double2(qr, qi);
    }
}

// Time-dependent coefficients: a thread per point checks every time level and forms the means
// over the unknown ones.
__global__ void __launch_bounds__(128)
timevar_check_kernel(int m, int s, const double* __restrict__ dpt, const double* __restrict__ dmt,
                     double* __restrict__ dp, double* __restrict__ dm, int* __restrict__ bad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    double sp = 0.0, sm = 0.0;
    bool ok = true;
    for (int n = 0; n <= s; ++n) {
        const double p = dpt[(size_t)n * m + i], q = dmt[(size_t)n * m + i];
        ok = ok && p >= 0.0 && q >= 0.0 && p + q > 0.0 && isfinite(p) && isfinite(q);
        if (n > 0) {
            sp += p;
            sm += q;
        }
    }
    dp[i] = sp / s;
    dm[i] = sm / s;
    ok = ok && isfinite(dp[i]) && isfinite(dm[i]) && dp[i] + dm[i] > 0.0;
    if (!ok) *bad = 1;
}

// First column of the L-periodic circulant C that embeds G (G[i][j] = g_{i-j+1}
// for j <= i+1): c[k] = g_{k+1} for 0 <= k < m, c[L-1] = g_0, zero elsewhere.
// lambda = FFT_L(c); (lambda + i conj(lambda)) = (lr + li)(1 + i), so with kap = lr + li one
// inverse FFT of kap FFT(z), rotated by 1 + i, returns (G z) + i (G^T z) for real z
// (C^T has eigenvalues conj(lambda) in the same Fourier basis).  kap is stored in the
// bit-reversed order in which the transform leaves it; |kap| <= sqrt 2 sum |g| < 5.7.
// sym32 keeps scale / L times the complex symbol in natural order, in FP32.
__global__ void __launch_bounds__(512)
toeplitz_symbol_kernel(const double* __restrict__ g, int m, int logL, double scale, const bfp::Tw* __restrict__ tw,
                       bfp::Q61* __restrict__ kap, float2* __restrict__ sym32) {
    extern __shared__ __align__(16) unsigned char sym_smem[];
    bfp::I2* buf = reinterpret_cast<bfp::I2*>(sym_smem);
    __shared__ uint32_t red[4];
    const int L = 1 << logL;
    constexpr int EMAX = 1024;  // |g_k| < 2
    if (threadIdx.x < 4) red[threadIdx.x] = 0u;
    __syncthreads();
    for (int k = threadIdx.x; k < L; k += blockDim.x) {
        const double v = k < m ? g[k + 1] : k == L - 1 ? g[0] : 0.0;
        buf[bfp::slot(k)] = bfp::I2{bfp::to_fixed(v, EMAX), 0};
    }
    __syncthreads();
    bfp::RowBits bits{red};
    int shifts = 0;
    bfp::transform(buf, logL, false, 0, tw, logL, false, bits, 0u, &shifts);
    for (int p = threadIdx.x; p < L; p += blockDim.x) {
        const bfp::I2 v = buf[bfp::slot(p)];
        const long long s = v.x + v.y;  // units of 2^(shifts - 56)
        kap[p] = bfp::q61((long long)((unsigned long long)s << (2 + shifts)));
        const float f = (float)(scalbn(bfp::to_double(s), shifts - (bfp::BITS - 1 + 1023 - EMAX)) * (scale / L));
        sym32[bitrev(p, logL)] = make_float2(f, f);
    }
}

// b_t = h sum_q B[t][start+q] f_{start+q} - A[t][0] u0 + h B[t][0] J u0, t = 1..s
// (eq. (1.10) with the known block u_0 moved to the right-hand side).
__global__ void rhs_kernel(int m, int s, int mu, double h, const int* __restrict__ start,
                           const double* __restrict__ A, const double* __restrict__ B,
                           const double* __restrict__ f, const double* __restrict__ u0,
                           const double* __restrict__ Ju0, double* __restrict__ b) {
    const int t = blockIdx.y + 1;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const int st = start[t];
    const double* a = A + (size_t)t * (mu + 1);
    const double* bb = B + (size_t)t * (mu + 1);
    double acc = 0.0;
    for (int q = 0; q <= mu; ++q) acc += bb[q] * f[(size_t)(st + q) * m + i];
    acc *= h;
    if (st == 0) acc += -a[0] * u0[i] + h * bb[0] * Ju0[i];
    b[(size_t)(t - 1) * m + i] = acc;
}

int launch_tables(const Problem& P, cudaStream_t st) {
    TableArgs A{P.alpha, P.m, P.logL, P.s, P.mu, P.nu, {}, {}, P.d_g, P.d_twL, P.d_twL32, P.d_tws, P.d_tws32,
                P.d_twq, P.d_phi, P.d_psi};
    for (int i = 0; i <= P.mu; ++i) {
        A.a[i] = P.h_a_main[i];
        A.b[i] = P.h_b_main[i];
    }
    const int items = P.L + P.s + P.L + P.L / 2 + P.s / 2 + 1;
    tables_kernel<<<1 + (items + 255) / 256, 256, 0, st>>>(A);
    FDE_LAUNCH_CHECK("tables_kernel");
    return FDE_OK;
}

int launch_timevar_check(const Problem& P, int* bad, cudaStream_t st) {
    timevar_check_kernel<<<(P.m + 127) / 128, 128, 0, st>>>(P.m, P.s, P.d_dplus_t, P.d_dminus_t, P.d_dplus,
                                                           P.d_dminus, bad);
    FDE_LAUNCH_CHECK("timevar_check_kernel");
    return FDE_OK;
}

int launch_toeplitz_symbol(const double* g, int m, int L, double scale, const bfp::Tw* twq, bfp::Q61* kap,
                           float2* sym32, cudaStream_t st) {
    const size_t smem = (size_t)L * sizeof(bfp::I2);
    FDE_TRY(allow_smem((const void*)toeplitz_symbol_kernel, 226 * 1024));
    const int threads = L / 8 > 512 ? 512 : L / 8 < 64 ? 64 : L / 8;
    toeplitz_symbol_kernel<<<1, threads, smem, st>>>(g, m, ilog2(L), scale, twq, kap, sym32);
    FDE_LAUNCH_CHECK("toeplitz_symbol_kernel");
    return FDE_OK;
}

int launch_rhs(const Problem& P, const double* Ju0, cudaStream_t st) {
    dim3 grid((P.m + 255) / 256, P.s);
    rhs_kernel<<<grid, 256, 0, st>>>(P.m, P.s, P.mu, P.h, P.d_start, P.d_a, P.d_b, P.d_f, P.d_u0, Ju0, P.d_b_rhs);
    FDE_LAUNCH_CHECK("rhs_kernel");
    return FDE_OK;
}

}  // namespace fde
