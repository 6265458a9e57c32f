// Strang blocks in FP64 (the plain method): blocked right-looking LU without pivoting and
// the block solves, on the same planes and tile inverses as lu.cu.
//
// GB300 has two FP64 lanes per SM: a warp-wide FP64 instruction occupies a scheduler for 64
// cycles whatever its lanes do.  So these kernels are about using all four schedulers with full
// warps and computing nothing that is padding: panels of 32 columns stop at m rounded up
// to 32 (the storage pads to 64, and a 64 x 64 tile of the trailing matrix of m = 63 was three
// quarters padding), the serial parts (diagonal block, tile inverses, triangular solves)
// split each row or column over several lanes, and reductions between lanes, which cost
// FP64 instructions of their own, are kept to two or three levels.
//
// GB300, us, against 64 x 64 tiles in 256 threads, a warp a tile inverse and a solver warp beside
// streaming warps: m = 63, s = 32 factorisation and inverses 231 (was 717), block solves 10.7 (34);
// m = 96, s = 128: 432 (1838) and 18.8 (79); m = 400, s = 64: 7060 (16000) and 240 (441); m = 2047,
// s = 64: 0.61 s (1.07 s) and 4919 (6823).  lu64_update runs at the FP64 rate; the diagonal block is a
// chain of 32 reciprocals (60 us, was 106).
#include "fde_internal.h"
#include "fft_device.cuh"

namespace fde {
namespace {

constexpr int NB = LU_NB;
constexpr int D64_THREADS = 256;

__device__ __forceinline__ double2 shfl2(double2 v, int src, int width = 32) {
    return make_double2(__shfl_sync(0xffffffffu, v.x, src, width), __shfl_sync(0xffffffffu, v.y, src, width));
}
// a - b c
__device__ __forceinline__ double2 cfms(double2 a, double2 b, double2 c) {
    a.x = fma(-b.x, c.x, fma(b.y, c.y, a.x));
    a.y = fma(-b.x, c.y, fma(-b.y, c.x, a.y));
    return a;
}
// a + b c
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {
    a.x = fma(b.x, c.x, fma(-b.y, c.y, a.x));
    a.y = fma(b.x, c.y, fma(b.y, c.x, a.y));
    return a;
}
// Sums x and y over W neighbouring lanes: even lanes return sum x, odd ones sum y.  The first
// exchange splits the pair, so a level costs one FP64 addition, not two.
template <int W>
__device__ __forceinline__ double pair_sum(double x, double y) {
    const bool odd = threadIdx.x & 1;
    double v = odd ? y : x;
    v += __shfl_xor_sync(0xffffffffu, odd ? x : y, 1);
#pragma unroll
    for (int off = 2; off < W; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// LU of the 32 x 32 diagonal block of every matrix: lane = row, warp w holds columns w, w + 8,
// .. in registers.  Per column every warp updates its own columns with the published
// multipliers (the pivot row's entry comes from a shuffle); the warp of the next column does that
// one first and publishes its multipliers, so that the division runs beside the updates.
__global__ void __launch_bounds__(D64_THREADS)
lu64_diag_kernel(int mp, int p, int steps, double* __restrict__ fac, double2* __restrict__ dinv, int* __restrict__ info) {
    __shared__ double2 D[NB][NB + 1];
    __shared__ double2 mult[2][NB];
    const int k = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, o = p * NB;
    double* re = fac + (size_t)k * 2 * mp * mp + (size_t)o * mp + o;
    double* im = re + (size_t)mp * mp;
    if (p + 1 == steps && o + NB + tid < mp) dinv[(size_t)k * mp + o + NB + tid] = make_double2(1.0, 0.0);  // padding
    for (int r = warp; r < NB; r += 8) D[r][lane] = make_double2(re[(size_t)r * mp + lane], im[(size_t)r * mp + lane]);
    __syncthreads();
    double2 a[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = D[lane][warp + 8 * i];
    // column c, held in v by this warp, is up to date: its multipliers
    const auto publish = [&](int c, double2& v) {
        const double2 piv = shfl2(v, c);
        const double den = piv.x * piv.x + piv.y * piv.y;
        const bool ok = den > 0.0 && isfinite(den);
        const double part = ((lane & 1) ? -piv.y : piv.x) / den;  // even lanes the real part, odd the imaginary
        double2 inv = make_double2(__shfl_sync(0xffffffffu, part, 0), __shfl_sync(0xffffffffu, part, 1));
        if (!ok) inv = make_double2(0.0, 0.0);
        if (lane == c) {
            if (!ok) atomicCAS(info + k, 0, o + c + 1);
            dinv[(size_t)k * mp + o + c] = inv;
        }
        const double2 l = cmul(v, inv);
        if (lane > c) v = l;
        mult[c & 1][lane] = v;
    };
    if (warp == 0) publish(0, a[0]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        for (int w = 0; w < 8; ++w) {
            const int c = 8 * i + w;
            __syncthreads();
            const double2 l = mult[c & 1][lane];
#pragma unroll
            for (int q = i; q < 4; ++q) {
                if (warp + 8 * q <= c) continue;  // at or left of c (q == i only)
                const double2 u = shfl2(a[q], c);
                if (lane > c) a[q] = cfms(a[q], l, u);
                // the next column goes out before the warp's others are updated
                if (q <= i + 1 && warp + 8 * q == c + 1) publish(c + 1, a[q]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) D[lane][warp + 8 * i] = a[i];
    __syncthreads();
    for (int r = warp; r < NB; r += 8) {
        re[(size_t)r * mp + lane] = D[r][lane].x;
        im[(size_t)r * mp + lane] = D[r][lane].y;
    }
}

// Panels: CTAs x < nch solve 32 rows of A21 against U11 (x U = a), the others 32 columns of
// A12 against L11 (L x = a).  Four lanes a row (column), lane q the entries q, q + 4, ..: a solved
// entry is broadcast among the four, each then updates its own.
constexpr int P64_THREADS = 128;
__global__ void __launch_bounds__(P64_THREADS)
lu64_panel_kernel(int mp, int p, int nch, double* __restrict__ fac, const double2* __restrict__ dinv) {
    __shared__ double2 D[NB][NB + 1];
    __shared__ double2 X[NB][NB + 1];  // [row or column][entry]
    __shared__ double2 di[NB];
    const int k = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, o = p * NB;
    double* re = fac + (size_t)k * 2 * mp * mp;
    double* im = re + (size_t)mp * mp;
    const bool rows = (int)blockIdx.x < nch;
    const int b0 = o + NB + ((int)blockIdx.x - (rows ? 0 : nch)) * NB;
    if (tid < NB) di[tid] = dinv[(size_t)k * mp + o + tid];
    for (int r = warp; r < NB; r += 4) {
        const size_t d = (size_t)(o + r) * mp + o + lane;
        D[r][lane] = make_double2(re[d], im[d]);
        if (rows) {
            const size_t g = (size_t)(b0 + r) * mp + o + lane;
            X[r][lane] = make_double2(re[g], im[g]);
        } else {
            const size_t g = (size_t)(o + r) * mp + b0 + lane;
            X[lane][r] = make_double2(re[g], im[g]);
        }
    }
    __syncthreads();
    const int q = tid >> 2, s = tid & 3;
    double2 x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = X[q][4 * u + s];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int c = 4 * u + t;
            if (rows && s == t) x[u] = cmul(x[u], di[c]);
            const double2 xc = shfl2(x[u], t, 4);
#pragma unroll
            for (int v = u; v < 8; ++v) {
                if (v == u && t == 3) continue;  // nothing right of c in this group
                const int cc = 4 * v + s;
                const double2 d = rows ? D[c][cc] : D[cc][c];
                if (v > u || s > t) x[v] = cfms(x[v], xc, d);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) X[q][4 * u + s] = x[u];
    __syncthreads();
    for (int r = warp; r < NB; r += 4) {
        const size_t g = rows ? (size_t)(b0 + r) * mp + o + lane : (size_t)(o + r) * mp + b0 + lane;
        const double2 v = rows ? X[r][lane] : X[lane][r];
        re[g] = v.x;
        im[g] = v.y;
    }
}

// C -= L21 U12 on a 32 x 32 tile, eight complex entries a thread (rows 8 i + warp.. of column
// lane): 4096 FP64 instructions a warp against 150 loads.
constexpr int U64_THREADS = 128;
__global__ void __launch_bounds__(U64_THREADS)
lu64_update_kernel(int mp, int p, int nt, double* __restrict__ fac) {
    __shared__ double2 Ls[NB][NB + 1], Us[NB][NB + 1];
    const int k = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int kb = p * NB, r0 = kb + NB + (blockIdx.x / nt) * NB, c0 = kb + NB + (blockIdx.x % nt) * NB;
    double* re = fac + (size_t)k * 2 * mp * mp;
    double* im = re + (size_t)mp * mp;
    double2 acc[8];
    for (int r = warp; r < NB; r += 4) {
        const size_t l = (size_t)(r0 + r) * mp + kb + lane, u = (size_t)(kb + r) * mp + c0 + lane;
        Ls[r][lane] = make_double2(re[l], im[l]);
        Us[r][lane] = make_double2(re[u], im[u]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const size_t g = (size_t)(r0 + 4 * i + warp) * mp + c0 + lane;
        acc[i] = make_double2(re[g], im[g]);
    }
    __syncthreads();
#pragma unroll 4
    for (int q = 0; q < NB; ++q) {
        const double2 u = Us[q][lane];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = cfms(acc[i], Ls[4 * i + warp][q], u);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const size_t g = (size_t)(r0 + 4 * i + warp) * mp + c0 + lane;
        re[g] = acc[i].x;
        im[g] = acc[i].y;
    }
}

// Block solves in place on rhat[k], one CTA per block: per 32-row tile x = D^-1 a (eight lanes a
// row), then the tile's strip times x from the rows that remain (four lanes a row, the loads of
// the first rows issued before the tile is solved).  Rows from nt 32 on are padding (zero).
constexpr int T64_THREADS = 256;
template <bool FWD>
__device__ __forceinline__ void trsv64_sweep(int mp, int nt, const double* __restrict__ re, const double* __restrict__ im,
                                             const double* __restrict__ tinv, double2* y, double2* xs) {
    const int tid = threadIdx.x, row = tid >> 3, g = tid & 7, sr = tid >> 2, s = tid & 3;
    double dr[4], di[4];
    const auto load_d = [&](int t) {
        const double2* p = reinterpret_cast<const double2*>(tinv + (size_t)t * 4096 + (FWD ? 0 : 2048) + row * NB + 4 * g);
        const double2 a = p[0], b = p[1], c = p[512], d = p[513];
        dr[0] = a.x; dr[1] = a.y; dr[2] = b.x; dr[3] = b.y;
        di[0] = c.x; di[1] = c.y; di[2] = d.x; di[3] = d.y;
    };
    double lr[8], li[8];
    const auto load_l = [&](int r, int c0) {
        const double2* p = reinterpret_cast<const double2*>(re + (size_t)r * mp + c0 + 8 * s);
        const double2* q = reinterpret_cast<const double2*>(im + (size_t)r * mp + c0 + 8 * s);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const double2 a = p[u], b = q[u];
            lr[2 * u] = a.x; lr[2 * u + 1] = a.y;
            li[2 * u] = b.x; li[2 * u + 1] = b.y;
        }
    };
    load_d(FWD ? 0 : nt - 1);
    for (int d = 0; d < nt; ++d) {
        const int t = FWD ? d : nt - 1 - d, r0 = NB * t;
        const int lo = FWD ? r0 + NB : 0, hi = FWD ? NB * nt : r0;
        if (lo + sr < hi) load_l(lo + sr, r0);
        double2 a = make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < 4; ++u) a = cfma(a, make_double2(dr[u], di[u]), y[r0 + 4 * g + u]);
        const double x = pair_sum<8>(a.x, a.y);
        if (g < 2) reinterpret_cast<double*>(xs + row)[g] = x;
        __syncthreads();
        if (g < 2) reinterpret_cast<double*>(y + r0 + row)[g] = x;
        if (d + 1 < nt) load_d(FWD ? t + 1 : t - 1);
        for (int r = lo + sr; r - sr < hi; r += T64_THREADS / 4) {
            if (r - (sr & 7) >= hi) continue;  // none of the warp's rows (hi is a multiple of 32)
            double2 a = make_double2(0.0, 0.0);
#pragma unroll
            for (int u = 0; u < 8; ++u) a = cfma(a, make_double2(lr[u], li[u]), xs[8 * s + u]);
            if (r + T64_THREADS / 4 < hi) load_l(r + T64_THREADS / 4, r0);
            const double v = pair_sum<4>(a.x, a.y);
            if (s < 2) reinterpret_cast<double*>(y + r)[s] -= v;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(T64_THREADS)
trsv64_kernel(int mp, int nt, const double* __restrict__ fac, const double* __restrict__ tinv,
              double2* __restrict__ rhat, const int* __restrict__ live) {
    if (live && !*live) return;
    extern __shared__ __align__(16) unsigned char t64_smem[];
    double2* y = reinterpret_cast<double2*>(t64_smem);
    __shared__ double2 xs[NB];
    const int k = blockIdx.x;
    const double* re = fac + (size_t)k * 2 * mp * mp;
    const double* im = re + (size_t)mp * mp;
    const double* ti = tinv + (size_t)k * (mp / NB) * 4096;
    double2* x = rhat + (size_t)k * mp;
    for (int i = threadIdx.x; i < NB * nt; i += T64_THREADS) y[i] = x[i];
    __syncthreads();
    trsv64_sweep<true>(mp, nt, re, im, ti, y, xs);
    trsv64_sweep<false>(mp, nt, re, im, ti, y, xs);
    for (int i = threadIdx.x; i < NB * nt; i += T64_THREADS) x[i] = y[i];
}

}  // namespace

int launch_lu64(Problem& P, cudaStream_t st) {
    double* fac = reinterpret_cast<double*>(P.d_fac);
    double2* dinv = reinterpret_cast<double2*>(P.d_dinv);
    const int mp = P.mp, nb = P.nblk, steps = (P.m + NB - 1) / NB;
    for (int p = 0; p < steps; ++p) {
        {
            StageTimer t(P, FDE_STAGE_LU_DIAG);
            lu64_diag_kernel<<<nb, D64_THREADS, 0, st>>>(mp, p, steps, fac, dinv, P.d_info);
            FDE_LAUNCH_CHECK("lu64_diag_kernel");
        }
        const int nt = steps - p - 1;
        if (nt == 0) break;
        {
            StageTimer t(P, FDE_STAGE_LU_PANEL);
            lu64_panel_kernel<<<dim3(2 * nt, nb), P64_THREADS, 0, st>>>(mp, p, nt, fac, dinv);
            FDE_LAUNCH_CHECK("lu64_panel_kernel");
        }
        StageTimer t(P, FDE_STAGE_LU_UPDATE);
        lu64_update_kernel<<<dim3(nt * nt, nb), U64_THREADS, 0, st>>>(mp, p, nt, fac);
        FDE_LAUNCH_CHECK("lu64_update_kernel");
    }
    return FDE_OK;
}

int launch_trsv64(const Problem& P, void* rhat, cudaStream_t st) {
    const int nt = (P.m + NB - 1) / NB;
    const size_t smem = (size_t)NB * nt * sizeof(double2);
    FDE_TRY(allow_smem((const void*)trsv64_kernel, smem));
    trsv64_kernel<<<P.nblk, T64_THREADS, smem, st>>>(
        P.mp, nt, (const double*)P.d_fac, (const double*)P.d_tinv, (double2*)rhat, P.live);
    FDE_LAUNCH_CHECK("trsv64_kernel");
    return FDE_OK;
}

}  // namespace fde
