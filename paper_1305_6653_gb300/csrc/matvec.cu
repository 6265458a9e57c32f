// Space-time matvec y = M z, M = A_1 (x) I - h B_1 (x) J (eq. (1.10) with u_0
// eliminated), and the plain Toeplitz-like apply y = J z (eq. (1.4)).
//
// One CTA per time row t.  By linearity
//     y_t = sum_q A[t][c_q] z_{c_q}  -  h J ( sum_q B[t][c_q] z_{c_q} ),
// so each CTA forms both band combinations of the mu+1 neighbouring time columns
// (read straight from HBM; the neighbours are shared through L2), then applies J
// once: J v = dx^-alpha (D+ G v + D- G^T v) through the length-L circulant
// embedding of G (Sec. 2.1: Toeplitz matvec by FFT), with one forward FFT of v
// (real input: a half-length complex FFT and a split) and one inverse FFT whose
// real / imaginary parts, rotated, are G v and G^T v.
//
// The product runs its FFTs in block floating point on the integer units (bfp_fft.cuh):
// in FP64 they took about 330,000 FP64 instructions a row at L = 4096, which the two FP64
// lanes of an SM need 85 us for.  What stays in FP64 are the band sums and the output,
// about ten instructions a point.
#include "fde_internal.h"
#include "bfp_device.cuh"
#include "fft_device.cuh"

namespace fde {

template <typename T, int MODE>
__device__ __forceinline__ void matvec_body(int m, int logL, int mu, double h, const int* __restrict__ start,
                                            const double* __restrict__ A, const double* __restrict__ B,
                                            const double* __restrict__ dplus, const double* __restrict__ dminus,
                                            const cplx_t<T>* __restrict__ sym, const cplx_t<T>* __restrict__ tw,
                                            const double* __restrict__ z, double* __restrict__ y, int row,
                                            int dstride = 0) {
    // T = float: the band sums, the A-band part and the output stay FP64; only the Toeplitz
    // apply J w (both FFTs and the symbol product) runs in FP32 (the inexact inner product
    // of the flexible GMRES).
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = 1 << logL, N = L >> 1, logN = logL - 1;
    C* buf = reinterpret_cast<C*>(smem_raw);
    double* ubuf = reinterpret_cast<double*>(buf + L);  // row = reduced time row: unknown u_{row+1}

    double ca[FDE_MAX_MU + 1], cb[FDE_MAX_MU + 1];
    int st = 0;
    if (MODE == 0) {
        const int t = row + 1;
        st = start[t];
#pragma unroll
        for (int q = 0; q <= FDE_MAX_MU; ++q) {
            ca[q] = q <= mu ? A[(size_t)t * (mu + 1) + q] : 0.0;
            cb[q] = q <= mu ? B[(size_t)t * (mu + 1) + q] : 0.0;
        }
    }
    // The input v of the Toeplitz apply is real: its length-L FFT comes from the
    // length-N = L/2 FFT of zc[n] = v[2n] + i v[2n+1] (bit-reversed for the DIT).
    for (int n = threadIdx.x; n < N; n += blockDim.x) {
        double v2[2] = {0.0, 0.0};
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int i = 2 * n + e;
            if (i < m) {
                if (MODE == 0) {
                    double u = 0.0, w = 0.0;
#pragma unroll
                    for (int q = 0; q <= FDE_MAX_MU; ++q) {
                        const int col = st + q;  // full-system time index; column 0 (u_0) is eliminated
                        if (q <= mu && col >= 1) {
                            const double zz = z[(size_t)(col - 1) * m + i];
                            u += ca[q] * zz;
                            w += cb[q] * zz;
                        }
                    }
                    ubuf[i] = u;
                    v2[e] = w;
                } else {
                    v2[e] = z[(size_t)row * m + i];
                }
            }
        }
        buf[bitrev(n, logN)] = mk((T)v2[0], (T)v2[1]);
    }
    __syncthreads();
    fft_dit4<false>(buf, logN, tw, 2);  // tw holds W_L^k; stride 2 gives W_N^k
    // Split Zc into V (length L) and multiply by the symbol, in place: the thread of
    // pair (k, N-k) reads Zc[k], Zc[N-k] and writes V[k], V[k+N], V[N-k], V[2N-k] with
    //   E = (Zc[k] + conj Zc[N-k]) / 2,  O = (Zc[k] - conj Zc[N-k]) / 2i,
    //   V[k] = E + W_L^k O,  V[k+N] = E - W_L^k O.
    for (int k = threadIdx.x; k <= N / 2; k += blockDim.x) {
        const int kk = (N - k) & (N - 1);
        const C zk = buf[k], zn = buf[kk];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            if (e == 1 && kk == k) break;
            const int idx = e == 0 ? k : kk;
            const C za = e == 0 ? zk : zn, zb = e == 0 ? zn : zk;
            const T half = T(0.5);
            const C E = mk(half * (za.x + zb.x), half * (za.y - zb.y));
            const C O = mk(half * (za.y + zb.y), -half * (za.x - zb.x));
            const C wo = cmul(tw[idx], O);
            buf[idx] = cmul(cadd(E, wo), sym[idx]);
            buf[idx + N] = cmul(csub(E, wo), sym[idx + N]);
        }
    }
    __syncthreads();
    fft_dif4<true>(buf, logL, tw, 1);
    const double* dp = dplus + (size_t)row * dstride;  // MODE 1 with per-column coefficients
    const double* dm = dminus + (size_t)row * dstride;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const C wv = buf[bitrev(i, logL)];
        const double jz = dp[i] * (double)wv.x + dm[i] * (double)wv.y;
        if (MODE == 0)
            y[(size_t)row * m + i] = ubuf[i] - h * jz;
        else
            y[(size_t)row * m + i] = jz;
    }
}

// The FP32 product of the relaxed Arnoldi steps.
__global__ void __launch_bounds__(1024)
st_matvec32_kernel(int m, int logL, int mu, double h, const int* __restrict__ start, const double* __restrict__ A,
                   const double* __restrict__ B, const double* __restrict__ dplus, const double* __restrict__ dminus,
                   const float2* __restrict__ sym, const float2* __restrict__ tw, const double* __restrict__ z,
                   double* __restrict__ y, const int* __restrict__ live) {
    if (live && !*live) return;
    matvec_body<float, 0>(m, logL, mu, h, start, A, B, dplus, dminus, sym, tw, z, y, blockIdx.x);
}

// ---------------------------------------------------------------------------
// The full-precision product: block floating-point FFTs.
// ---------------------------------------------------------------------------
namespace {

// One time row.  MODE 0: y_t = sum a z - h J (sum b z); MODE 1: y = J z with coefficients
// dplus + row dstride.  tw: exp(-2 pi i k / L), k < L, followed by the L/2 of them that the
// split uses, in bit-reversed order; kap: the Toeplitz symbol in bit-reversed order, in
// units of 2^-58; fac = 4 dx^-alpha / L.
//
// m = 2047, s = 256: 56 us where the FP64 transforms took 190 (FP64 pipe 80 % busy); m = 1023,
// s = 64: 24 (50); m = 4095, s = 128: 62 (206); m = 96, s = 128: 13.7 (13.9).  Radix 8 in
// registers halves the trips through shared memory; what bounds the kernel now is latency (16
// warps an SM, a third of the issue slots used) and, at s = 256, two rows on 104 of 152 SMs.
// The error against the exact product is 2 to 17 times smaller than that of the FP64
// transforms (m = 63 .. 4095, white and smooth z).
template <int MODE>
__device__ __forceinline__ void bfp_row(int m, int logL, int mu, double h, const int* __restrict__ start,
                                        const double* __restrict__ A, const double* __restrict__ B,
                                        const double* __restrict__ dplus, const double* __restrict__ dminus,
                                        const bfp::Tw* __restrict__ tw, const bfp::Q61* __restrict__ kap, double fac,
                                        const double* __restrict__ z, double* __restrict__ y, int row, int dstride) {
    using bfp::I2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t red[4];
    const int L = 1 << logL, N = L >> 1, logN = logL - 1;
    const int tid = threadIdx.x, T = blockDim.x;
    I2* buf = reinterpret_cast<I2*>(smem_raw);
    double* ubuf = reinterpret_cast<double*>(buf + L);  // row = reduced time row: unknown u_{row+1}
    if (tid < 4) red[tid] = 0u;
    // the nonzero coefficients of the row's band in A and in B (half of them are zero, whatever
    // the family) and the time columns they apply to; column 0 (u_0) is eliminated
    __shared__ double coef[2][FDE_MAX_MU + 1];
    __shared__ int cols[2][FDE_MAX_MU + 1], taps[2];
    if (MODE == 0 && tid < 64) {
        const int which = tid >> 5, q = tid & 31, t = row + 1;
        const int st = start[t];
        const double c = q <= mu && st + q >= 1 ? (which ? B : A)[(size_t)t * (mu + 1) + q] : 0.0;
        const uint32_t on = __ballot_sync(0xffffffffu, c != 0.0);
        if (c != 0.0) {
            const int k = __popc(on & ((1u << q) - 1u));
            coef[which][k] = c;
            cols[which][k] = st + q - 1;
        }
        if (q == 0) taps[which] = __popc(on);
    }
    __syncthreads();
    // v as packed points v[2n] + i v[2n+1], still doubles; the row's largest exponent.  A
    // non-finite z in the band of the row makes the whole row NaN.
    uint32_t mx = 0;
    const int nh = N > 1 ? N / 2 : 1;
    for (int n = tid; n < nh; n += T) {
        double v2[2] = {0.0, 0.0};
        const int i0 = 2 * n, i1 = 2 * n + 1 < m ? 2 * n + 1 : i0;
        if (i0 < m) {
            if (MODE == 0) {
                double u0 = 0.0, u1 = 0.0;
                for (int k = 0; k < taps[0]; ++k) {
                    const double* zc = z + (size_t)cols[0][k] * m;
                    const double c = coef[0][k], z0 = zc[i0], z1 = zc[i1];
                    u0 += c * z0;
                    u1 += c * z1;
                    const uint32_t zh = max((uint32_t)__double2hiint(z0) & 0x7fffffffu,
                                            (uint32_t)__double2hiint(z1) & 0x7fffffffu);
                    if (zh >= 0x7ff00000u) mx = zh;
                }
                ubuf[i0] = u0;
                ubuf[i1] = i1 > i0 ? u1 : u0;
                for (int k = 0; k < taps[1]; ++k) {
                    const double* zc = z + (size_t)cols[1][k] * m;
                    const double c = coef[1][k];
                    v2[0] += c * zc[i0];
                    v2[1] += c * zc[i1];
                }
            } else {
                v2[0] = z[(size_t)row * m + i0];
                v2[1] = z[(size_t)row * m + i1];
            }
            if (i1 == i0) v2[1] = 0.0;
            mx = max(mx, max((uint32_t)__double2hiint(v2[0]) & 0x7fffffffu, (uint32_t)__double2hiint(v2[1]) & 0x7fffffffu));
        }
        buf[bfp::slot(n)] = I2{__double_as_longlong(v2[0]), __double_as_longlong(v2[1])};
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((tid & 31) == 0) atomicMax(red + 3, mx);
    __syncthreads();
    mx = red[3];
    if (mx >= 0x7ff00000u) {
        for (int i = tid; i < m; i += T) y[(size_t)row * m + i] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    const int emax = max(1, (int)(mx >> 20));
    for (int n = tid; n < N; n += T) {
        I2& b = buf[bfp::slot(n)];  // the thread's own points
        b = n < nh ? I2{bfp::to_fixed(__longlong_as_double(b.x), emax), bfp::to_fixed(__longlong_as_double(b.y), emax)}
                   : I2{0, 0};
    }
    __syncthreads();
    bfp::RowBits bits{red};
    int shifts = 0;
    uint32_t tops = bfp::transform(buf, logN, false, 0, tw, logL, false, bits, 0u, &shifts);

    // Split, symbol and the inverse's first level: position p of the half-length transform
    // holds k = rev(p), its partner N - k is at the mirrored place of p's binary octave
    // ([2b, 4b): p <-> 6b - 1 - p), and k, k + N go to positions 2p, 2p + 1.  Octave by
    // octave from the top (an octave's outputs lie above its inputs), the rest staged in
    // registers.
    {
        const int sh = bfp::shift_for(tops);
        shifts += sh;
        const bfp::Tw* twr = tw + L;
        const auto at = [&](int p) { return bfp::shr(buf[bfp::slot(p)], sh); };
        const auto pair = [&](int p, int q, I2 (&o)[4]) {
            bfp::split_pair(at(p), at(q), twr[p], kap[2 * p], kap[2 * p + 1], kap[2 * q], kap[2 * q + 1], o);
        };
        uint32_t t = 0;
        const auto put = [&](int p, I2 a, I2 b) {
            buf[bfp::slot(2 * p)] = I2{a.y, a.x};  // exchanged, for the inverse
            buf[bfp::slot(2 * p + 1)] = I2{b.y, b.x};
            t |= bfp::top(a) | bfp::top(b);
        };
        int nrem = nh;
        while (nrem > T) {
            const int b = nrem >> 1;
            for (int e = b + tid; e < nrem; e += T) {
                const int p = e + b, q = 6 * b - 1 - p;
                I2 o[4];
                pair(p, q, o);
                put(p, o[0], o[1]);
                put(q, o[2], o[3]);
            }
            __syncthreads();
            nrem = b;
        }
        I2 o[4];
        int p = 0, q = 0;
        if (tid < nrem) {
            if (tid == 0) {  // k = 0 and k = N / 2 are their own partners
                I2 o2[4];
                pair(0, 0, o2);
                o[0] = o2[0];
                o[1] = o2[1];
                if (N > 1) {
                    q = 1;
                    pair(1, 1, o2);
                    o[2] = o2[0];
                    o[3] = o2[1];
                }
            } else {
                const int b = 1 << (31 - __clz(tid));
                p = tid + b;
                q = 6 * b - 1 - p;
                pair(p, q, o);
            }
        }
        __syncthreads();
        if (tid < nrem) {
            put(p, o[0], o[1]);
            if (q > 0) put(q, o[2], o[3]);
        }
        tops = bits.sync_or(t);
    }

    bfp::transform(buf, logL, true, 1, tw, logL, true, bits, tops, &shifts);

    const double* dp = dplus + (size_t)row * dstride;  // MODE 1 with per-column coefficients
    const double* dm = dminus + (size_t)row * dstride;
    // The row's scale: its power of two goes into the integers' conversion, so that d+, d- of any
    // magnitude multiply numbers of the result's own; what is beyond 2^900 of it is left to the factor.
    int ef;
    const double f = bfp::mantissa(MODE == 0 ? h * fac : fac, &ef);
    const int whole = shifts - (bfp::BITS - 1 + 1023 - emax) + ef, e = min(max(whole, -900), 900);
    const double s1 = f * bfp::power_of_two(min(max(whole - e, -1000), 1000));
    for (int i = tid; i < m; i += T) {
        const I2 v = buf[bfp::slot(i)];  // (imaginary, real)
        const double jz = dp[i] * bfp::to_double(v.y - v.x, e) + dm[i] * bfp::to_double(v.x + v.y, e);
        y[(size_t)row * m + i] = MODE == 0 ? ubuf[i] - s1 * jz : s1 * jz;
    }
}

}  // namespace

// NT: the most threads a launch uses (the launch takes min(NT, L/8), at least 64); every
// loop is strided by blockDim.x, so all thread counts compute the same integers.  Register
// use is capped so that 512 / NT CTAs fit an SM when shared memory allows.
template <int MODE, int NT = 512>
__global__ void __launch_bounds__(NT, 512 / NT)
st_matvec_kernel(int m, int logL, int mu, double h, const int* __restrict__ start, const double* __restrict__ A,
                 const double* __restrict__ B, const double* __restrict__ dplus, const double* __restrict__ dminus,
                 const bfp::Tw* __restrict__ tw, const bfp::Q61* __restrict__ kap, double fac,
                 const double* __restrict__ z, double* __restrict__ y, int dstride, const int* __restrict__ live) {
    if (live && !*live) return;
    bfp_row<MODE>(m, logL, mu, h, start, A, B, dplus, dminus, tw, kap, fac, z, y, blockIdx.x, dstride);
}

// Time-dependent coefficients: y_n = sum_q a_{n,q} z_q - h sum_q b_{n,q} (J_q z_q) over the
// BVM band of row n (u_0 eliminated), with jz = [J_1 z_1; ..; J_s z_s] from the Toeplitz
// apply; one CTA per time row, threads along x.
__global__ void __launch_bounds__(256)
st_band_kernel(int m, int mu, double h, const int* __restrict__ start, const double* __restrict__ A,
               const double* __restrict__ B, const double* __restrict__ z, const double* __restrict__ jz,
               double* __restrict__ y) {
    const int row = blockIdx.x, t = row + 1;
    const int st = start[t];
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        double u = 0.0, w = 0.0;
        for (int q = 0; q <= mu; ++q) {
            const int col = st + q;  // full-system time index; column 0 (u_0) is eliminated
            if (col >= 1) {
                u += A[(size_t)t * (mu + 1) + q] * z[(size_t)(col - 1) * m + i];
                w += B[(size_t)t * (mu + 1) + q] * jz[(size_t)(col - 1) * m + i];
            }
        }
        y[(size_t)row * m + i] = u - h * w;
    }
}

// Batched M z over the active instances: grid (max s, active count).
// which = 0: z = Z_j, y = V_{j+1} (Arnoldi step); which = 1: z = x, y = work (residual).
__global__ void __launch_bounds__(256, 2)
st_matvec_batched(const InstDev* __restrict__ I, const int* __restrict__ act, int which, int j) {
    const InstDev& d = I[act[blockIdx.y]];
    if ((int)blockIdx.x >= d.s || !d.ctl[0]) return;
    const double* z = which == 0 ? d.Z + (size_t)j * d.n : d.x;
    double* y = which == 0 ? d.V + (size_t)(j + 1) * d.n : d.work;
    bfp_row<0>(d.m, d.logL, d.mu, d.h, d.start, d.A, d.B, d.dplus, d.dminus, d.twq, d.kap, d.jfac, z, y, blockIdx.x,
               0);
}

static int row_threads(int L, int most) {
    const int t = L / 8;
    return t > most ? most : t < 64 ? 64 : t;
}

int launch_matvec_batched(const InstDev* I, const int* act, int nact, int max_s, int max_L, int max_m, int which,
                          int j, cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    const size_t smem = (size_t)max_L * sizeof(bfp::I2) + (size_t)max_m * sizeof(double);
    FDE_TRY(allow_smem((const void*)st_matvec_batched, 226 * 1024));
    st_matvec_batched<<<dim3(max_s, nact), row_threads(max_L, 256), smem, st>>>(I, act, which, j);
    FDE_LAUNCH_CHECK("st_matvec_batched");
    return FDE_OK;
}

template <int MODE, int NT = 512>
static int launch_st(const Problem& P, const double* z, double* y, int ncols, cudaStream_t st,
                     const double* dplus = nullptr, const double* dminus = nullptr, int dstride = 0) {
    const size_t smem = (size_t)P.L * sizeof(bfp::I2) + (MODE == 0 ? (size_t)P.m * sizeof(double) : 0);
    auto kern = st_matvec_kernel<MODE, NT>;
    FDE_TRY(allow_smem((const void*)kern, 226 * 1024));
    kern<<<ncols, row_threads(P.L, NT), smem, st>>>(P.m, P.logL, P.mu, P.h, P.d_start, P.d_a, P.d_b,
                                                    dplus ? dplus : P.d_dplus, dminus ? dminus : P.d_dminus, P.d_twq,
                                                    P.d_kap, toeplitz_scale(P), z, y, dstride, P.live);
    FDE_LAUNCH_CHECK("st_matvec_kernel");
    return FDE_OK;
}

int launch_matvec32(const Problem& P, const double* z, double* y, cudaStream_t st) {
    if (P.timevar) return launch_matvec64(P, z, y, st);  // the time-level products stay FP64
    const size_t smem = (size_t)P.L * sizeof(float2) + (size_t)P.m * sizeof(double);
    const int threads = P.L / 2 > 1024 ? 1024 : P.L / 2 < 64 ? 64 : P.L / 2;
    FDE_TRY(allow_smem((const void*)st_matvec32_kernel, 227 * 1024));
    st_matvec32_kernel<<<P.s, threads, smem, st>>>(P.m, P.logL, P.mu, P.h, P.d_start, P.d_a, P.d_b, P.d_dplus,
                                                   P.d_dminus, P.d_sym32, P.d_twL32, z, y, P.live);
    FDE_LAUNCH_CHECK("st_matvec32_kernel");
    return FDE_OK;
}

// The tuned variants of the full-precision space-time product: at most 512, 256 or 128
// threads per time row (FDE_TUNE_MATVEC).
int launch_matvec64_variant(const Problem& P, const double* z, double* y, int variant, cudaStream_t st) {
    if (variant == 1) return launch_st<0, 256>(P, z, y, P.s, st);
    if (variant == 2) return launch_st<0, 128>(P, z, y, P.s, st);
    return launch_st<0, 512>(P, z, y, P.s, st);
}

namespace {
struct MatvecTuneCtx {
    const Problem* P;
    const double* z;
    double* y;
};
int matvec_trial(void* ctx, int v, cudaStream_t st) {
    const MatvecTuneCtx& c = *static_cast<const MatvecTuneCtx*>(ctx);
    return launch_matvec64_variant(*c.P, c.z, c.y, v, st);
}
}  // namespace

// Measure the variants for this shape (z = b, y = the work vector) unless the table
// already has it or a variant is forced.
int autotune_matvec(Problem& P) {
    if (P.timevar) return FDE_OK;
    bool need = false;
    tune_lookup(FDE_TUNE_MATVEC, P.mp, P.s, FDE_FP64, &need);
    if (!need) return FDE_OK;
    MatvecTuneCtx ctx{&P, P.d_b_rhs, P.d_work};
    int best = 0;
    float ms[TUNE_MAX_VARIANTS] = {};
    const int rc = tune_measure(FDE_TUNE_MATVEC, P.stream, matvec_trial, &ctx, &best, ms,
                                tune_default_variant(FDE_TUNE_MATVEC, FDE_FP64));
    if (rc) return rc;
    tune_store(FDE_TUNE_MATVEC, P.mp, P.s, FDE_FP64, best, ms);
    return FDE_OK;
}

int launch_matvec64(const Problem& P, const double* z, double* y, cudaStream_t st) {
    if (!P.timevar)
        return launch_matvec64_variant(P, z, y, tune_lookup(FDE_TUNE_MATVEC, P.mp, P.s, FDE_FP64, nullptr), st);
    // J_q z_q for q = 1..s with the coefficients of time level q, then the BVM band
    int rc = launch_st<1>(P, z, P.d_jz, P.s, st, P.d_dplus_t + P.m, P.d_dminus_t + P.m, P.m);
    if (rc) return rc;
    st_band_kernel<<<P.s, 256, 0, st>>>(P.m, P.mu, P.h, P.d_start, P.d_a, P.d_b, z, P.d_jz, y);
    FDE_LAUNCH_CHECK("st_band_kernel");
    return FDE_OK;
}

int launch_japply64(const Problem& P, const double* z, double* y, int ncols, cudaStream_t st) {
    return launch_st<1>(P, z, y, ncols, st);
}

int launch_japply64_d(const Problem& P, const double* z, double* y, int ncols, const double* dplus,
                      const double* dminus, int dstride, cudaStream_t st) {
    return launch_st<1>(P, z, y, ncols, st, dplus, dminus, dstride);
}

}  // namespace fde
