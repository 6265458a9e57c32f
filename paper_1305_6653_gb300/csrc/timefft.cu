// FFT along time for every spatial index (Sec. 3.2: S^{-1} = (F^* (x) I)
// (Lambda_A (x) I - h Lambda_B (x) J)^{-1} (F (x) I)).
//
// Vectors are time-major [t][x] (x contiguous), so a CTA takes a tile of XW
// consecutive x and all s time levels.  Two real columns are packed into one complex FFT
// (z = r_a + i r_b) and separated with the Hermitian split, so XW / 2 complex length-s
// FFTs per tile.  XW is 16 (a time row of the tile is one 128-byte read) where that
// gives every SM a tile, and 8, 4 or 2 for shorter vectors, whose few tiles of 16 left most SMs idle
// (m = 96, s = 128, FP64: 6.7 us, 14.7 with 8 tiles of 16; the data comes from L2 then).
// Output / input of the frequency side: [k][mp] complex for k = 0..s/2 (the distinct frequencies of a real signal), padded to mp with zeros.
#include "fde_internal.h"
#include "fft_device.cuh"

namespace fde {

// In-place decimation-in-time FFT of NCOL columns of s = 2^logn points (input in bit-reversed
// order, column c from buf + c s); tw[k] = exp(-2 pi i k / s), k < s.  FP32 radix 4.  FP64
// radix 2: there a warp's FP64 instructions take 64 cycles each, and the shorter chain over
// twice as many warps is the faster one while an SM has few (m = 1023, s = 64: 8.0 us, radix 4
// 10.9).
template <int NCOL, bool INVERSE, typename C>
__device__ __forceinline__ void fft_columns(C* buf, int logn, const C* __restrict__ tw) {
    constexpr bool R4 = sizeof(C) == 8;
    const int N = 1 << logn;
    int st = 1;
    const int r2 = R4 ? (logn & 1) : logn;  // radix-2 stages
    for (; st <= r2; ++st) {
        const int half = 1 << (st - 1), tws = N >> st;
        for (int b = threadIdx.x; b < NCOL * N / 2; b += blockDim.x) {  // columns follow one another
            const int pos = b & (half - 1);
            const int i0 = ((b >> (st - 1)) << st) + pos;
            C w = tw[pos * tws];
            if (INVERSE) w.y = -w.y;
            const C a = buf[i0], t = cmul(w, buf[i0 + half]);
            buf[i0] = cadd(a, t);
            buf[i0 + half] = csub(a, t);
        }
        __syncthreads();
    }
    if constexpr (R4) {
        for (; st < logn; st += 2) {
            const int half = 1 << (st - 1), tws = N >> (st + 1);
            for (int b = threadIdx.x; b < NCOL * N / 4; b += blockDim.x) {
                const int pos = b & (half - 1);
                const int i0 = ((b >> (st - 1)) << (st + 1)) + pos;
                C w2 = tw[pos * tws], w1 = tw[2 * pos * tws], w3 = tw[3 * pos * tws];
                if (INVERSE) {
                    w1.y = -w1.y;
                    w2.y = -w2.y;
                    w3.y = -w3.y;
                }
                const C a = buf[i0], b1 = cmul(w1, buf[i0 + half]), c = cmul(w2, buf[i0 + 2 * half]),
                        d = cmul(w3, buf[i0 + 3 * half]);
                const C apb = cadd(a, b1), amb = csub(a, b1), cpd = cadd(c, d), cmd = csub(c, d);
                const C rot = INVERSE ? mk(-cmd.y, cmd.x) : mk(cmd.y, -cmd.x);
                buf[i0] = cadd(apb, cpd);
                buf[i0 + half] = cadd(amb, rot);
                buf[i0 + 2 * half] = csub(apb, cpd);
                buf[i0 + 3 * half] = csub(amb, rot);
            }
            __syncthreads();
        }
    }
}

template <typename T, int XW>
__device__ __forceinline__ void fwd_body(int m, int mp, int logs, const double* __restrict__ r,
                                         const cplx_t<T>* __restrict__ tw, cplx_t<T>* __restrict__ rhat, int bx) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int NCOL = XW / 2;
    C* buf = reinterpret_cast<C*>(smem_raw);  // NCOL columns of length s
    const int s = 1 << logs;
    const int x0 = bx * XW;
    for (int e = threadIdx.x; e < s * XW; e += blockDim.x) {
        const int t = e / XW;
        const int xx = e - t * XW;
        const int x = x0 + xx;
        const T v = x < m ? (T)r[(size_t)t * m + x] : T(0);
        T* dst = reinterpret_cast<T*>(&buf[(xx >> 1) * s + bitrev(t, logs)]);
        dst[xx & 1] = v;
    }
    __syncthreads();
    fft_columns<NCOL, false>(buf, logs, tw);
    const int nk = s / 2 + 1;
    for (int e = threadIdx.x; e < nk * NCOL; e += blockDim.x) {
        const int k = e / NCOL;
        const int c = e - k * NCOL;
        const C Z = buf[c * s + k];
        const C Zc = cconj(buf[c * s + ((s - k) & (s - 1))]);
        const T half = T(0.5);
        // Ra = (Z + conj Z_{s-k}) / 2,  Rb = (Z - conj Z_{s-k}) / (2i)
        C Ra = mk((Z.x + Zc.x) * half, (Z.y + Zc.y) * half);
        C Rb = mk((Z.y - Zc.y) * half, -(Z.x - Zc.x) * half);
        const int xa = x0 + 2 * c;
        if (xa < mp) rhat[(size_t)k * mp + xa] = Ra;
        if (xa + 1 < mp) rhat[(size_t)k * mp + xa + 1] = Rb;
    }
}

template <typename T, int XW>
__global__ void __launch_bounds__(256)
time_fft_fwd_kernel(int m, int mp, int logs, const double* __restrict__ r, const cplx_t<T>* __restrict__ tw,
                    cplx_t<T>* __restrict__ rhat) {
    fwd_body<T, XW>(m, mp, logs, r, tw, rhat, blockIdx.x);
}

template <typename T, int XW>
__device__ __forceinline__ void inv_body(int m, int mp, int logs, const cplx_t<T>* __restrict__ xhat,
                                         const cplx_t<T>* __restrict__ tw, double* __restrict__ z, int bx) {
    using C = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int NCOL = XW / 2;
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int s = 1 << logs;
    const int x0 = bx * XW;
    const int nk = s / 2 + 1;
    for (int e = threadIdx.x; e < nk * NCOL; e += blockDim.x) {
        const int k = e / NCOL;
        const int c = e - k * NCOL;
        const int xa = x0 + 2 * c;
        C Xa = xa < mp ? xhat[(size_t)k * mp + xa] : mk(T(0), T(0));
        C Xb = xa + 1 < mp ? xhat[(size_t)k * mp + xa + 1] : mk(T(0), T(0));
        if (k == 0 || k == s / 2) {  // real signal: DC and Nyquist terms are real
            Xa.y = T(0);
            Xb.y = T(0);
        }
        // Z_k = Xa_k + i Xb_k; for the mirrored frequency Z_{s-k} = conj(Xa_k) + i conj(Xb_k)
        buf[c * s + bitrev(k, logs)] = mk(Xa.x - Xb.y, Xa.y + Xb.x);
        if (k > 0 && k < s / 2) buf[c * s + bitrev(s - k, logs)] = mk(Xa.x + Xb.y, Xb.x - Xa.y);
    }
    __syncthreads();
    fft_columns<NCOL, true>(buf, logs, tw);
    const double inv = 1.0 / (double)s;
    for (int e = threadIdx.x; e < s * XW; e += blockDim.x) {
        const int t = e / XW;
        const int xx = e - t * XW;
        const int x = x0 + xx;
        if (x < m) {
            const T* src = reinterpret_cast<const T*>(&buf[(xx >> 1) * s + t]);
            z[(size_t)t * m + x] = (double)src[xx & 1] * inv;
        }
    }
}

template <typename T, int XW>
__global__ void __launch_bounds__(256)
time_fft_inv_kernel(int m, int mp, int logs, const cplx_t<T>* __restrict__ xhat, const cplx_t<T>* __restrict__ tw,
                    double* __restrict__ z) {
    inv_body<T, XW>(m, mp, logs, xhat, tw, z, blockIdx.x);
}

constexpr int XWB = 16;  // batches have instances enough to fill the SMs

// Batched over the active instances act[]: grid (max x-tiles, active count), FP32
// transforms (the batched path uses FP32/TF32/BF16 preconditioners).  The forward
// transform reads the Krylov vector V_j, the inverse one writes Z_j.
__global__ void __launch_bounds__(256)
time_fft_fwd_batched(const InstDev* __restrict__ I, const int* __restrict__ act, int j) {
    const InstDev& d = I[act[blockIdx.y]];
    if ((int)blockIdx.x * XWB >= d.mp || !d.ctl[0]) return;
    fwd_body<float, XWB>(d.m, d.mp, d.logs, d.V + (size_t)j * d.n, d.tws32, (float2*)d.rhat, blockIdx.x);
}

__global__ void __launch_bounds__(256)
time_fft_inv_batched(const InstDev* __restrict__ I, const int* __restrict__ act, int j) {
    const InstDev& d = I[act[blockIdx.y]];
    if ((int)blockIdx.x * XWB >= d.mp || !d.ctl[0]) return;
    inv_body<float, XWB>(d.m, d.mp, d.logs, (const float2*)d.rhat, d.tws32, d.Z + (size_t)j * d.n, blockIdx.x);
}

int launch_time_fft_batched(const InstDev* I, const int* act, int nact, int max_mp, int max_s, int j,
                            cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    const dim3 grid((max_mp + XWB - 1) / XWB, nact);
    const size_t smem = (size_t)(XWB / 2) * max_s * sizeof(float2);
    FDE_TRY(allow_smem((const void*)time_fft_fwd_batched, 227 * 1024));
    time_fft_fwd_batched<<<grid, 256, smem, st>>>(I, act, j);
    FDE_LAUNCH_CHECK("time_fft_fwd_batched");
    return FDE_OK;
}

int launch_time_ifft_batched(const InstDev* I, const int* act, int nact, int max_mp, int max_s, int j,
                             cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    const dim3 grid((max_mp + XWB - 1) / XWB, nact);
    const size_t smem = (size_t)(XWB / 2) * max_s * sizeof(float2);
    FDE_TRY(allow_smem((const void*)time_fft_inv_batched, 227 * 1024));
    time_fft_inv_batched<<<grid, 256, smem, st>>>(I, act, j);
    FDE_LAUNCH_CHECK("time_fft_inv_batched");
    return FDE_OK;
}

namespace {

// one thread a butterfly of a stage
int fft_threads(int n) { return n >= 256 ? 256 : n <= 64 ? 64 : 128; }

template <typename T, int XW>
int fwd_tiles(const Problem& P, const double* r, void* rhat, const cplx_t<T>* tw, cudaStream_t st) {
    const size_t smem = (size_t)(XW / 2) * P.s * sizeof(cplx_t<T>);
    const int threads = fft_threads(P.s * XW / (sizeof(T) == 8 ? 4 : 8));
    FDE_TRY(allow_smem((const void*)time_fft_fwd_kernel<T, XW>, smem));
    time_fft_fwd_kernel<T, XW><<<(P.mp + XW - 1) / XW, threads, smem, st>>>(P.m, P.mp, P.logs, r, tw,
                                                                            (cplx_t<T>*)rhat);
    FDE_LAUNCH_CHECK("time_fft_fwd_kernel");
    return FDE_OK;
}
template <typename T, int XW>
int inv_tiles(const Problem& P, const void* xhat, double* z, const cplx_t<T>* tw, cudaStream_t st) {
    const size_t smem = (size_t)(XW / 2) * P.s * sizeof(cplx_t<T>);
    const int threads = fft_threads(P.s * XW / (sizeof(T) == 8 ? 4 : 8));
    FDE_TRY(allow_smem((const void*)time_fft_inv_kernel<T, XW>, smem));
    time_fft_inv_kernel<T, XW><<<(P.mp + XW - 1) / XW, threads, smem, st>>>(P.m, P.mp, P.logs, (const cplx_t<T>*)xhat,
                                                                            tw, z);
    FDE_LAUNCH_CHECK("time_fft_inv_kernel");
    return FDE_OK;
}
// the widest tile that leaves no SM of 152 without one
int tile_width(int mp) { return mp / 16 >= 120 ? 16 : mp / 8 >= 120 ? 8 : mp / 4 >= 120 ? 4 : 2; }

template <typename T>
int fwd_any(const Problem& P, const double* r, void* rhat, const cplx_t<T>* tw, cudaStream_t st) {
    switch (tile_width(P.mp)) {
        case 16: return fwd_tiles<T, 16>(P, r, rhat, tw, st);
        case 8: return fwd_tiles<T, 8>(P, r, rhat, tw, st);
        case 4: return fwd_tiles<T, 4>(P, r, rhat, tw, st);
        default: return fwd_tiles<T, 2>(P, r, rhat, tw, st);
    }
}
template <typename T>
int inv_any(const Problem& P, const void* xhat, double* z, const cplx_t<T>* tw, cudaStream_t st) {
    switch (tile_width(P.mp)) {
        case 16: return inv_tiles<T, 16>(P, xhat, z, tw, st);
        case 8: return inv_tiles<T, 8>(P, xhat, z, tw, st);
        case 4: return inv_tiles<T, 4>(P, xhat, z, tw, st);
        default: return inv_tiles<T, 2>(P, xhat, z, tw, st);
    }
}

}  // namespace

int launch_time_fft_fwd(const Problem& P, const double* r, void* rhat, int prec, cudaStream_t st) {
    return prec == FDE_FP64 ? fwd_any<double>(P, r, rhat, P.d_tws, st) : fwd_any<float>(P, r, rhat, P.d_tws32, st);
}

int launch_time_fft_inv(const Problem& P, const void* xhat, double* z, int prec, cudaStream_t st) {
    return prec == FDE_FP64 ? inv_any<double>(P, xhat, z, P.d_tws, st) : inv_any<float>(P, xhat, z, P.d_tws32, st);
}

}  // namespace fde
