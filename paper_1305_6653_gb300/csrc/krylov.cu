// FP64 Krylov kernels of the flexible GMRES(restart) iteration (Sec. 3.2 cites
// Saad's GMRES; Sec. 4 runs GMRES(20)): classical Gram-Schmidt with one
// re-orthogonalisation (CGS2), the Givens least-squares update and the
// normalisation of the new basis vector as one kernel, and small vector kernels.
//
// Reductions are deterministic: partial sums are added in a fixed order.
#include <algorithm>

#include "fde_internal.h"

namespace fde {

constexpr int RED_CTAS = 304;  // 2 per SM on 152 SMs
constexpr int RED_THREADS = 256;
constexpr int KMAX = 64;       // max Krylov vectors per multi-dot

// Sum over a warp of C values a thread (C = 8 or 16), 15 / 16 additions a lane where C
// butterflies take 5 C: every step halves the number of values, a lane keeping one half and
// handing over the other.  Lane l ends with the sum of value l / (32 / C).
template <int C>
__device__ __forceinline__ double warp_sums(double (&a)[C]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16, h = C / 2; h >= 1; off >>= 1, h >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double keep = up ? a[i + h] : a[i], give = up ? a[i] : a[i + h];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
    }
#pragma unroll
    for (int off = 16 / C; off; off >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], off);
    return a[0];
}

// |w|^2 of a vector: CTA sums to partial, the last CTA to finish (atomic ticket after a
// fence; nothing waits) adds them.
__device__ __forceinline__ void to_host(double* host, double v);
__device__ __forceinline__ void norm_body(const double* w, long n, double* __restrict__ out,
                                          double* __restrict__ partial, unsigned int* __restrict__ counter, int bx,
                                          int nblocks, double* __restrict__ host = nullptr) {
    __shared__ double red[RED_THREADS / 32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v = 0.0;
    const long stride = (long)nblocks * blockDim.x;
    for (long x = (long)bx * blockDim.x + threadIdx.x; x < n; x += stride) v += w[x] * w[x];
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < RED_THREADS / 32; ++q) v += red[q];
        partial[bx] = v;
        __threadfence();
        last = (atomicAdd(counter, 1u) == (unsigned)nblocks - 1);
    }
    __syncthreads();
    if (last && warp == 0) {
        __threadfence();
        v = 0.0;
        for (int c = lane; c < nblocks; c += 32) v += __ldcg(partial + c);
        for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) {
            *out = v;
            *counter = 0u;
            if (host) to_host(host, v);
        }
    }
}

// Results the host waits for go to pinned memory, the sequence word last.
__device__ __forceinline__ void to_host(double* host, double v) {
    volatile double* h = host;
    h[0] = v;
    __threadfence_system();
    h[1] = 1.0;
}

// out[0] = |w|^2 (SUB: of w = b - ax, which is stored)
template <bool SUB>
__global__ void __launch_bounds__(RED_THREADS)
norm_kernel(const double* __restrict__ b, const double* __restrict__ ax, double* __restrict__ w, long n,
            double* __restrict__ out, double* __restrict__ partial, unsigned int* __restrict__ counter,
            double* __restrict__ host) {
    if (SUB) {
        const long stride = (long)gridDim.x * blockDim.x;
        for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) w[i] = b[i] - ax[i];
    }
    norm_body(w, n, out, partial, counter, blockIdx.x, gridDim.x, host);  // each thread the elements it stored
}

// ---------------------------------------------------------------------------
// One Gram-Schmidt step: w against V_0..V_{k-1} (k = j + 1), column j of the Hessenberg
// matrix with its Givens rotation, w / |w|.
//
//   h1 = V^T w;  w -= V h1, h2 = V^T w (with re-orthogonalisation);  w -= V h, |w|^2;
//   w /= |w|.
//
// All passes run in one cooperative launch of G CTAs that meet at a barrier after each
// pass; every CTA then adds the CTAs' partial sums itself.  GB300's two FP64 lanes an SM
// bound it at large n (4 k n multiply-adds; m = 2047, s = 256: 49 us at the mean k = 13.5
// were the lanes never idle), so what matters there is that nothing but those runs on them:
// the passes' reductions took 5 butterfly additions per value and warp, half as much again
// as the dots themselves.  At small n it is bound by latency: three barriers and three
// reductions instead of five launches, and V stays in registers (ONE).
// Mean step of a solve at m = 2047, s = 256 (26 steps): 144 -> 101 us; at m = 255, s = 64 (15
// steps): 49 -> 19 us.
// ---------------------------------------------------------------------------
constexpr int GS_CTAS = 152;                 // at most one CTA per SM; partial sums are [2][64][GS_CTAS]
constexpr int GS_WARPS = RED_THREADS / 32;   // most warps of a CTA
constexpr int GS_SMEM = 200 * 1024;          // for the staged V of the looping form
constexpr unsigned GS_SPINS = 1u << 24;      // polls before a wait gives up (seconds)

struct GsArgs {
    const double* V;
    double* w;
    long n;
    int k, ldh, reorth;
    double *H, *cs, *sn, *g, *scal;  // scal: [128] |w|^2, [129] estimate, [130] H(j+1,j) before rotation
    double* partial;
    unsigned int* bar;  // a counter per barrier, zero before the launch
    int* err;
    int* live;                    // Problem::d_live, or NULL (a batch: ctl)
    Problem::StepOutcome* host;   // where the host waits for the step, or NULL
};

// The CTAs of one Gram-Schmidt step meet.  CTA 0 clears the next counter before it arrives
// (nobody can be there yet), and counter 0 once everybody has left it.
__device__ __forceinline__ void gs_barrier(unsigned int* bar, int slot, int cta, int G, int* err) {
    __syncthreads();
    if (threadIdx.x == 0) {
        if (cta == 0) bar[slot + 1] = 0u;
        __threadfence();
        atomicAdd(bar + slot, 1u);
        unsigned seen, polls = 0;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar + slot) : "memory");
        } while (seen < (unsigned)G && ++polls < GS_SPINS);
        if (seen < (unsigned)G) *err = 1;
        if (cta == 0 && slot > 0) bar[0] = 0u;
    }
    __syncthreads();
}

// out[i] = sum over the CTAs of sum over the warps of red[warp][i], i < k
template <int KC, int NT>
__device__ __forceinline__ void gs_collect(const GsArgs& A, const double (*red)[KC], int k, int slot, int cta, int G,
                                           double* out) {
    constexpr int NW = NT / 32;
    __syncthreads();
    double* part = A.partial + (size_t)(slot & 1) * 64 * GS_CTAS;
    if ((int)threadIdx.x < k) {
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < NW; ++q) v += red[q][threadIdx.x];
        if (G > 1) part[(size_t)threadIdx.x * GS_CTAS + cta] = v;
        else out[threadIdx.x] = v;
    }
    if (G > 1) {
        gs_barrier(A.bar, slot, cta, G, A.err);
        // tpv threads a vector (as many as there are for k), so that the additions fill their warps
        int tpv = 32;
        while (tpv * k > NT) tpv >>= 1;
        const int i = threadIdx.x / tpv, c0 = threadIdx.x % tpv;
        double v = 0.0;
        if (i < k) {
#pragma unroll 4
            for (int c = c0; c < G; c += tpv) v += __ldcg(part + (size_t)i * GS_CTAS + c);
        }
        for (int off = tpv >> 1; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (i < k && c0 == 0) out[i] = v;
    }
    __syncthreads();
}

// red[warp][i] = the warp's sum of a(i), i < k: eights, of which those beyond k are skipped by
// a branch (as everywhere below: a predicated FP64 instruction costs what an executed one does)
template <int KC, typename F>
__device__ __forceinline__ void gs_warp_sums(double (*red)[KC], int k, F a) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    static_assert(KC % 8 == 0, "whole eights");
#pragma unroll
    for (int i0 = 0; i0 < KC; i0 += 8) {
        if (i0 < k) {
            double b[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) b[i] = a(i0 + i);
            const double v = warp_sums<8>(b);
            if ((lane & 3) == 0) red[warp][i0 + (lane >> 2)] = v;
        }
    }
}

// Column j of the rotated Hessenberg matrix, its rotation and the rotated right-hand side;
// |g_{j+1}| is the residual estimate.  H is column-major.  One thread.
struct GsColumn {
    double est, hnext, nrm;
};
__device__ __forceinline__ GsColumn gs_column(const GsArgs& A, const double* h1, const double* h2, const double* c0,
                                              const double* s0, double nrm) {
    const int j = A.k - 1;
    double* col = A.H + (size_t)j * A.ldh;
    double t = h1[0] + (h2 ? h2[0] : 0.0);
    for (int i = 0; i < j; ++i) {
        const double c = c0[i], s = s0[i], b = h1[i + 1] + (h2 ? h2[i + 1] : 0.0);
        col[i] = c * t + s * b;
        t = -s * t + c * b;
    }
    const double b = sqrt(nrm), r = hypot(t, b);
    const double c = r > 0.0 ? t / r : 1.0, s = r > 0.0 ? b / r : 0.0;
    A.cs[j] = c;
    A.sn[j] = s;
    col[j] = r;
    col[j + 1] = 0.0;
    const double gj = A.g[j];
    A.g[j + 1] = -s * gj;
    A.g[j] = c * gj;
    GsColumn out{fabs(s * gj), b, nrm};
    A.scal[128] = nrm;
    A.scal[129] = out.est;
    A.scal[130] = b;
    return out;
}

// The end of the cycle (the test the host makes too) and the outcome to the host.  One thread.
__device__ __forceinline__ void gs_outcome(const GsArgs& A, const GsColumn& col) {
    if (!isfinite(col.est) || !isfinite(col.nrm) || col.est <= A.scal[133] || fabs(col.hnext) <= 1e-300) *A.live = 0;
    volatile Problem::StepOutcome* h = A.host;
    h->nrm_sq = col.nrm;
    h->est = col.est;
    h->hnext = col.hnext;
    __threadfence_system();
    h->seq = (unsigned long long)A.k;
}

__device__ __forceinline__ void cp_async_elems(double* dst, const double* src, int bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (bytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// The end of a step: |w|^2 from the warps' sums, w's scale, and on CTA 0 the column.
template <int KC, int NT, typename Scale, typename Done>
__device__ __forceinline__ void gs_end(const GsArgs& A, double sq, double (*red)[KC], const double* h1,
                                       const double* h2, const double* gc, const double* gsn, int slot, int cta,
                                       int G, Scale scale, Done done) {
    __shared__ double nrm[1];
    for (int off = 16; off; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][0] = sq;
    gs_collect<KC, NT>(A, red, 1, slot, cta, G, nrm);
    const double len = sqrt(nrm[0]);
    scale(len > 0.0 ? 1.0 / len : 0.0);
    if (cta == 0 && threadIdx.x == 0) done(gs_column(A, h1, A.reorth ? h2 : nullptr, gc, gsn, nrm[0]));
}

// At most one element a thread (E neighbours): V and w stay in registers.
template <int KC, int E, int NT>
__global__ void __launch_bounds__(NT, 1) gs_one_kernel(const __grid_constant__ GsArgs A) {
    __shared__ double red[NT / 32][KC];
    __shared__ double h1[KC], h2[KC], gc[KC], gsn[KC];
    if (!*A.live) return;  // cleared by this launch only after every CTA has come to its last barrier
    const int tid = threadIdx.x, k = A.k, cta = blockIdx.x, G = gridDim.x;
    const long n = A.n, x = ((long)cta * NT + tid) * E;
    if (cta == 0 && tid < k - 1) {  // earlier rotations, for the column at the end
        gc[tid] = A.cs[tid];
        gsn[tid] = A.sn[tid];
    }
    double v[KC][E], w[E];
#pragma unroll
    for (int e = 0; e < E; ++e) w[e] = 0.0;
#pragma unroll
    for (int i = 0; i < KC; ++i)
#pragma unroll
        for (int e = 0; e < E; ++e) v[i][e] = 0.0;
    if (x < n) {
        if constexpr (E == 2) {
            const double2 t = *reinterpret_cast<const double2*>(A.w + x);
            w[0] = t.x;
            w[1] = t.y;
        } else {
            w[0] = A.w[x];
        }
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            if (i < k) {
                if constexpr (E == 2) {
                    const double2 t = *reinterpret_cast<const double2*>(A.V + (size_t)i * n + x);
                    v[i][0] = t.x;
                    v[i][1] = t.y;
                } else {
                    v[i][0] = A.V[(size_t)i * n + x];
                }
            }
        }
    }
    const auto dots = [&](int slot, double* out) {
        gs_warp_sums<KC>(red, k, [&](int i) {
            double a = v[i][0] * w[0];
#pragma unroll
            for (int e = 1; e < E; ++e) a += v[i][e] * w[e];
            return a;
        });
        gs_collect<KC, NT>(A, red, k, slot, cta, G, out);
    };
    const auto update = [&](const double* c) {
        double s0[E], s1[E];
#pragma unroll
        for (int e = 0; e < E; ++e) s0[e] = s1[e] = 0.0;
#pragma unroll
        for (int i0 = 0; i0 < KC; i0 += 4) {
            if (i0 < k) {
#pragma unroll
                for (int i = i0; i < i0 + 4; i += 2) {
                    const double c0 = i < k ? c[i] : 0.0, c1 = i + 1 < k ? c[i + 1] : 0.0;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        s0[e] += c0 * v[i][e];
                        s1[e] += c1 * v[i + 1][e];
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) w[e] -= s0[e] + s1[e];
    };
    dots(0, h1);
    update(h1);
    int slot = 1;
    if (A.reorth) {
        dots(1, h2);
        update(h2);
        slot = 2;
    }
    double sq = w[0] * w[0];
#pragma unroll
    for (int e = 1; e < E; ++e) sq += w[e] * w[e];
    gs_end<KC, NT>(A, sq, red, h1, h2, gc, gsn, slot, cta, G, [&](double inv) {
        if (x < n) {
#pragma unroll
            for (int e = 0; e < E; ++e) A.w[x + e] = w[e] * inv;
        }
    }, [&](const GsColumn& col) { gs_outcome(A, col); });
}

// Any number of elements a thread, E neighbours at a time (E = 2: n even).  A thread copies
// its own elements of V asynchronously into shared memory, one group ahead of the one it
// works on, so the FP64 lanes do not wait for the loads and the registers hold only the sums.
template <int KC, int E, typename Done>
__device__ __forceinline__ void gs_body(const GsArgs& A, int cta, int G, double* stage, Done done) {
    __shared__ double red[GS_WARPS][KC];
    __shared__ double h1[KC], h2[KC], gc[KC], gsn[KC];
    constexpr int ROW = RED_THREADS * E;
    const int tid = threadIdx.x, k = A.k, k4 = (k + 3) & ~3;
    const int stages = 2 * k4 * ROW * (int)sizeof(double) <= GS_SMEM ? 2 : 1;
    const long n = A.n, step = (long)G * ROW, x0 = ((long)cta * RED_THREADS + tid) * E;
    if (cta == 0 && tid < k - 1) {  // earlier rotations, for the column at the end
        gc[tid] = A.cs[tid];
        gsn[tid] = A.sn[tid];
    }
    // rows k .. k4 - 1 stay zero, so that the loops run in fours
    for (int s = 0; s < stages; ++s)
        for (int i = k; i < k4; ++i)
#pragma unroll
            for (int e = 0; e < E; ++e) stage[(s * k4 + i) * ROW + tid * E + e] = 0.0;
    const auto issue = [&](long x, int s) {
        if (x < n) {
            const double* src = A.V + x;
            double* dst = stage + s * k4 * ROW + tid * E;
#pragma unroll 4
            for (int i = 0; i < k; ++i) cp_async_elems(dst + i * ROW, src + (size_t)i * n, 8 * E);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const auto load_w = [&](long x, double (&t)[E]) {
        if (x >= n) return;
        if constexpr (E == 2) {
            const double2 u = *reinterpret_cast<const double2*>(A.w + x);
            t[0] = u.x;
            t[1] = u.y;
        } else {
            t[0] = A.w[x];
        }
    };
    const auto store_w = [&](long x, const double (&t)[E]) {
        if constexpr (E == 2) *reinterpret_cast<double2*>(A.w + x) = make_double2(t[0], t[1]);
        else A.w[x] = t[0];
    };
    const auto row = [&](const double* v, int i, double (&t)[E]) {
        if constexpr (E == 2) {
            const double2 u = *reinterpret_cast<const double2*>(v + i * ROW);
            t[0] = u.x;
            t[1] = u.y;
        } else {
            t[0] = v[i * ROW];
        }
    };
    // w -= V c where c is given (stored), then work(v, w) for every group of elements
    const auto pass = [&](const double* c, auto work) {
        double w[E], wn[E];
        int s = 0;
        issue(x0, 0);
        load_w(x0, wn);
        for (long x = x0; x < n; x += step) {
#pragma unroll
            for (int e = 0; e < E; ++e) w[e] = wn[e];
            if (stages == 2) {
                issue(x + step, s ^ 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            load_w(x + step, wn);
            const double* v = stage + s * k4 * ROW + tid * E;
            if (c) {
                double p[4][E];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int e = 0; e < E; ++e) p[u][e] = 0.0;
#pragma unroll 2
                for (int i = 0; i < k4; i += 4) {
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        double t[E];
                        row(v, i + u, t);
                        const double ci = c[i + u];
#pragma unroll
                        for (int e = 0; e < E; ++e) p[u][e] += ci * t[e];
                    }
                }
#pragma unroll
                for (int e = 0; e < E; ++e) w[e] -= (p[0][e] + p[1][e]) + (p[2][e] + p[3][e]);
                store_w(x, w);
            }
            work(v, w);
            if (stages == 2) s ^= 1;
            else issue(x + step, 0);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    };
    const auto dots = [&](const double* c, int slot, double* out) {
        double acc[KC];
#pragma unroll
        for (int i = 0; i < KC; ++i) acc[i] = 0.0;
        pass(c, [&](const double* v, const double (&w)[E]) {
#pragma unroll
            for (int i0 = 0; i0 < KC; i0 += 4) {
                if (i0 < k) {
#pragma unroll
                    for (int i = i0; i < i0 + 4; ++i) {
                        double t[E];
                        row(v, i, t);
#pragma unroll
                        for (int e = 0; e < E; ++e) acc[i] += t[e] * w[e];
                    }
                }
            }
        });
        gs_warp_sums<KC>(red, k, [&](int i) { return acc[i]; });
        gs_collect<KC, RED_THREADS>(A, red, k, slot, cta, G, out);
    };
    if (tid >= k && tid < KC) h1[tid] = h2[tid] = 0.0;  // the coefficients of the zero rows
    dots(nullptr, 0, h1);
    const double* c = h1;
    int slot = 1;
    if (A.reorth) {
        dots(h1, 1, h2);
        c = h2;
        slot = 2;
    }
    double sq = 0.0;
    pass(c, [&](const double*, const double (&w)[E]) {
#pragma unroll
        for (int e = 0; e < E; ++e) sq += w[e] * w[e];
    });
    gs_end<KC, RED_THREADS>(A, sq, red, h1, h2, gc, gsn, slot, cta, G, [&](double inv) {
        for (long x = x0; x < n; x += step) {
            double w[E];
            load_w(x, w);
#pragma unroll
            for (int e = 0; e < E; ++e) w[e] *= inv;
            store_w(x, w);
        }
    }, done);
}

template <int KC, int E>
__global__ void __launch_bounds__(RED_THREADS, 1) gs_kernel(const __grid_constant__ GsArgs A) {
    extern __shared__ __align__(16) unsigned char gs_smem[];
    if (!*A.live) return;  // as in gs_one_kernel
    gs_body<KC, E>(A, blockIdx.x, gridDim.x, reinterpret_cast<double*>(gs_smem),
                   [&](const GsColumn& col) { gs_outcome(A, col); });
}

// shared memory of the staged V for k vectors
static size_t gs_stage_bytes(int k, int E) {
    const size_t one = (size_t)((k + 3) & ~3) * RED_THREADS * E * sizeof(double);
    return 2 * one <= (size_t)GS_SMEM ? 2 * one : one;
}

// w += sign * sum_i coef[i] V_i
__global__ void update_kernel(const double* __restrict__ V, int k, const double* __restrict__ coef, double sign,
                              double* __restrict__ w, long n) {
    __shared__ double c[KMAX];
    for (int i = threadIdx.x; i < k; i += blockDim.x) c[i] = sign * coef[i];
    __syncthreads();
    const long stride = (long)gridDim.x * blockDim.x;
    for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) {
        double acc = w[x];
        for (int i = 0; i < k; ++i) acc += c[i] * V[(size_t)i * n + x];
        w[x] = acc;
    }
}

__global__ void cycle_start_kernel(const double* src, const double* __restrict__ nrm_sq, double* dst, long n,
                                   double* __restrict__ g, int restart, double threshold, double* __restrict__ thr,
                                   int* __restrict__ live) {
    const double nr = sqrt(*nrm_sq);
    const double inv = nr > 0.0 ? 1.0 / nr : 0.0;
    const long stride = (long)gridDim.x * blockDim.x;
    for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) dst[x] = src[x] * inv;
    if (blockIdx.x == 0) {
        for (int i = threadIdx.x; i <= restart; i += blockDim.x) g[i] = i == 0 ? nr : 0.0;
        if (threadIdx.x == 0) {
            *thr = threshold;
            *live = 1;
        }
    }
}

// y = R^{-1} g with R the k x k upper-triangular part of the rotated H: a warp, columns
// in registers' reach (R staged in shared memory: every step of the serial chain otherwise waited
// for a load from global memory, 56 us at k = 27).
__device__ __forceinline__ void lsq_body(const double* __restrict__ H, int ldh, int k, const double* __restrict__ g,
                                         double* __restrict__ y, double* R) {
    const int lane = threadIdx.x & 31;
    for (int c = 0; c < k; ++c)
        for (int i = lane; i <= c; i += 32) R[c * KMAX + i] = H[(size_t)c * ldh + i];
    double v0 = lane < k ? g[lane] : 0.0, v1 = lane + 32 < k ? g[lane + 32] : 0.0;
    __syncwarp();
    for (int c = k - 1; c >= 0; --c) {
        double yc = 0.0;
        if (lane == (c & 31)) yc = (c < 32 ? v0 : v1) / R[c * KMAX + c];
        yc = __shfl_sync(0xffffffffu, yc, c & 31);
        if (lane == (c & 31)) y[c] = yc;
        if (lane < c) v0 -= R[c * KMAX + lane] * yc;
        if (lane + 32 < c) v1 -= R[c * KMAX + lane + 32] * yc;
    }
}

__global__ void __launch_bounds__(32) lsq_solve_kernel(const double* __restrict__ H, int ldh, int k,
                                                       const double* __restrict__ g, double* __restrict__ y) {
    __shared__ double R[KMAX * KMAX];
    lsq_body(H, ldh, k, g, y, R);
}

// ---------------------------------------------------------------------------
// Batched variants over the active instances act[0..gridDim.y) of a batch.
// Each instance owns its vectors, scalars, partial sums and reduction ticket.
// ---------------------------------------------------------------------------
constexpr int RED_CTAS_B = 32;  // reduction CTAs per instance in a batch

// mode 3: |V_0|^2 -> scal[132];  mode 4: |b|^2 -> scal[131]
__global__ void __launch_bounds__(RED_THREADS)
norm_batched(const InstDev* __restrict__ I, const int* __restrict__ act, int mode) {
    const InstDev& d = I[act[blockIdx.y]];
    if (!d.ctl[0]) return;  // the instance has left the cycle: no CTA of it takes part
    norm_body(mode == 3 ? d.V : d.b, d.n, d.scal + (mode == 3 ? 132 : 131), d.partial, d.counter, blockIdx.x,
              gridDim.x);
}

// x += Z_{0..k-1} y with k = kvec[instance]
__global__ void update_batched(const InstDev* __restrict__ I, const int* __restrict__ act,
                               const int* __restrict__ kvec) {
    __shared__ double c[KMAX];
    const int inst = act[blockIdx.y];
    const InstDev& d = I[inst];
    if (!d.ctl[0]) return;
    const int k = kvec[inst];
    for (int i = threadIdx.x; i < k; i += blockDim.x) c[i] = d.y[i];
    __syncthreads();
    const long stride = (long)gridDim.x * blockDim.x;
    for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < d.n; x += stride) {
        double acc = d.x[x];
        for (int i = 0; i < k; ++i) acc += c[i] * d.Z[(size_t)i * d.n + x];
        d.x[x] = acc;
    }
}

// V_0 /= sqrt(scal[132]) and g = (sqrt(scal[132]), 0, ...)
__global__ void scale_batched(const InstDev* __restrict__ I, const int* __restrict__ act, int restart) {
    const InstDev& d = I[act[blockIdx.y]];
    if (!d.ctl[0]) return;
    const double nr = sqrt(d.scal[132]);
    const double inv = nr > 0.0 ? 1.0 / nr : 0.0;
    const long stride = (long)gridDim.x * blockDim.x;
    for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < d.n; x += stride) d.V[x] *= inv;
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i <= restart; i += blockDim.x) d.gv[i] = i == 0 ? nr : 0.0;
}

// Sums of x and y over the CTA before this thread; x and y become the sums over the CTA.
struct GsScan {
    int x;
    long y;
};
__device__ __forceinline__ GsScan gs_scan(int& x, long& y) {
    __shared__ int wx[GS_WARPS];
    __shared__ long wy[GS_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int ix = x;
    long iy = y;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int ux = __shfl_up_sync(0xffffffffu, ix, off);
        const long uy = __shfl_up_sync(0xffffffffu, iy, off);
        if (lane >= off) {
            ix += ux;
            iy += uy;
        }
    }
    __syncthreads();  // the words may still be read from the call before
    if (lane == 31) {
        wx[warp] = ix;
        wy[warp] = iy;
    }
    __syncthreads();
    GsScan before{ix - x, iy - y};
    x = 0;
    y = 0;
    for (int w = 0; w < GS_WARPS; ++w) {
        if (w < warp) {
            before.x += wx[w];
            before.y += wy[w];
        }
        x += wx[w];
        y += wy[w];
    }
    return before;
}

// The Gram-Schmidt step j of every live instance in one cooperative launch.  The CTAs are
// shared out in proportion to the instances' lengths, one at least; with more live instances
// than CTAs each CTA takes instances of its own, alone.  Every CTA works the shares out for
// itself, by a scan over the list in pieces of a CTA's threads, so the list may have any length.  (The
// order of an instance's partial sums follows from the lengths of those that are live with it: the
// same batch gives the same bits, another batch other last bits.  A fixed number of partial sums
// an instance, 32 as there once were, would leave most SMs idle once few instances are live.)  An
// instance takes part if it is live or has already finished this step (a CTA that
// starts late may see the flags its step has left: ctl[1] = j + 1 is written before ctl[0]).
// An instance leaves the cycle on the device: tolerance met (Givens estimate), maxit,
// breakdown, or a non-finite value.
template <int KC, int E>
__global__ void __launch_bounds__(RED_THREADS, 1)
gs_batched(const InstDev* __restrict__ I, const int* __restrict__ act, int nact, int j, int ldh, int reorth,
           double tol, int maxit, int* __restrict__ err) {
    extern __shared__ __align__(16) unsigned char gs_smem[];
    double* stage = reinterpret_cast<double*>(gs_smem);
    __shared__ int sh_inst, sh_cta, sh_G;
    __shared__ int mine[RED_THREADS];  // a piece's entries that this CTA takes alone
    // length of entry a of the list, 0 if it takes no part
    const auto length = [&](int a) -> long {
        if (a >= nact) return 0;
        const InstDev& d = I[act[a]];
        volatile int* c = d.ctl;
        bool on = c[0] != 0;
        __threadfence();
        if (!on) on = c[1] == j + 1;
        return on ? d.n : 0;
    };
    const auto step = [&](int a, int cta, int G) {
        const InstDev& d = I[act[a]];
        GsArgs A{d.V, d.V + (size_t)(j + 1) * d.n, d.n, j + 1, ldh, reorth, d.H, d.cs, d.sn, d.gv, d.scal,
                 d.partial, d.counter, err, nullptr, nullptr};
        gs_body<KC, E>(A, cta, G, stage, [&](const GsColumn& col) {
            volatile int* c = d.ctl;
            const int its = c[2] + 1;
            c[2] = its;
            c[1] = j + 1;
            const bool bad = !isfinite(col.est) || !isfinite(col.nrm);
            if (bad) c[3] = 1;
            __threadfence();
            if (bad || col.est <= tol * sqrt(d.scal[131]) || its >= maxit || fabs(col.hnext) <= 1e-300) c[0] = 0;
        });
    };
    const int B = gridDim.x, me = blockIdx.x;
    int live = 0;
    long total = 0;
    for (int a = threadIdx.x; a < nact; a += RED_THREADS) {
        const long n = length(a);
        live += n > 0;
        total += n;
    }
    gs_scan(live, total);
    if (threadIdx.x == 0) sh_inst = -1;
    int first = 0;  // live entries before the piece, and their length
    long cum = 0;
    if (live > 0 && live <= B) {
        for (int a0 = 0; a0 < nact; a0 += RED_THREADS) {
            const int a = a0 + threadIdx.x;
            const long n = length(a);
            int px = n > 0;
            long py = n;
            const GsScan before = gs_scan(px, py);
            if (n > 0) {  // CTAs [at, end)
                const long i = first + before.x, c = cum + before.y;
                const int at = (int)(i + (B - live) * c / total), end = (int)(i + 1 + (B - live) * (c + n) / total);
                if (me >= at && me < end) {
                    sh_inst = a;
                    sh_cta = me - at;
                    sh_G = end - at;
                }
            }
            __syncthreads();
            if (sh_inst >= 0) break;
            first += px;
            cum += py;
        }
        if (sh_inst >= 0) step(sh_inst, sh_cta, sh_G);
    } else if (live > B) {
        for (int a0 = 0; a0 < nact; a0 += RED_THREADS) {
            const int a = a0 + threadIdx.x;
            const long n = length(a);
            int px = n > 0;
            long py = n;
            const GsScan before = gs_scan(px, py);
            const int i = first + before.x;
            // entries i = me, me + B, ..: numbered within the piece
            const int skip = (me - first % B + B) % B;  // live entries of the piece before the first of them
            if (n > 0 && i % B == me) mine[(before.x - skip) / B] = a;
            __syncthreads();
            for (int q = 0; q * B + skip < px; ++q) {
                step(mine[q], 0, 1);
                __syncthreads();
            }
            first += px;
        }
    }
}

// V_0 = b - work (work = M x)
__global__ void residual_batched(const InstDev* __restrict__ I, const int* __restrict__ act) {
    const InstDev& d = I[act[blockIdx.y]];
    if (!d.ctl[0]) return;
    const long stride = (long)gridDim.x * blockDim.x;
    for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < d.n; x += stride) d.V[x] = d.b[x] - d.work[x];
}

__global__ void ctl_set_batched(const InstDev* __restrict__ I, const int* __restrict__ act, int nact, int live,
                                int reset) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= nact) return;
    int* c = I[act[a]].ctl;
    c[0] = live;
    if (reset) c[1] = 0;
    if (reset > 1) {
        c[2] = 0;
        c[3] = 0;
    }
}

__global__ void __launch_bounds__(32) lsq_batched(const InstDev* __restrict__ I, const int* __restrict__ act,
                                                  const int* __restrict__ kvec, int ldh) {
    __shared__ double R[KMAX * KMAX];
    const int inst = act[blockIdx.x];
    const InstDev& d = I[inst];
    if (!d.ctl[0]) return;
    lsq_body(d.H, ldh, kvec[inst], d.gv, d.y, R);
}

// out[5*i + q] = scal[128 + q] of instance i (q = 0..2), out[5*i+3] = scal[132], out[5*i+4] = scal[131]
__global__ void gather_scalars(const InstDev* __restrict__ I, int ninst, double* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ninst) return;
    const double* sc = I[i].scal;
    for (int q = 0; q < 3; ++q) out[5 * i + q] = sc[128 + q];
    out[5 * i + 3] = sc[132];
    out[5 * i + 4] = sc[131];
}

static int grid_for(long n);

int launch_norm_batched(const InstDev* I, const int* act, int nact, int mode, cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    norm_batched<<<dim3(RED_CTAS_B, nact), RED_THREADS, 0, st>>>(I, act, mode);
    FDE_LAUNCH_CHECK("norm_batched");
    return FDE_OK;
}

int launch_update_batched(const InstDev* I, const int* act, int nact, const int* kvec, long max_n, cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    int g = (int)((max_n + 255) / 256);
    if (g > 64) g = 64;
    update_batched<<<dim3(g, nact), 256, 0, st>>>(I, act, kvec);
    FDE_LAUNCH_CHECK("update_batched");
    return FDE_OK;
}

int launch_scale_batched(const InstDev* I, const int* act, int nact, int restart, long max_n, cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    int g = (int)((max_n + 255) / 256);
    if (g > 64) g = 64;
    scale_batched<<<dim3(g, nact), 256, 0, st>>>(I, act, restart);
    FDE_LAUNCH_CHECK("scale_batched");
    return FDE_OK;
}

// CTAs of a cooperative Gram-Schmidt launch: one per SM of the current device
static int gs_ctas(int* out) {
    int dev = 0, sms = 0;
    FDE_CUDA_TRY(cudaGetDevice(&dev));
    FDE_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    *out = std::min(sms, GS_CTAS);
    return FDE_OK;
}

int launch_gs_batched(const InstDev* I, const int* act, int nact, int j, int ldh, int reorth, double tol, int maxit,
                      int* err, cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    const int k = j + 1;
    if (k > KMAX) return set_error(FDE_ERR_ARG, "too many Krylov vectors for one Gram-Schmidt step");
    int ctas = 0, rc = gs_ctas(&ctas);
    if (rc) return rc;
    const void* kern = k <= 8    ? (const void*)gs_batched<8, 2>
                       : k <= 16 ? (const void*)gs_batched<16, 2>
                       : k <= 24 ? (const void*)gs_batched<24, 2>
                       : k <= 32 ? (const void*)gs_batched<32, 1>
                                 : (const void*)gs_batched<64, 1>;
    const size_t smem = gs_stage_bytes(k, k <= 24 ? 2 : 1);
    FDE_TRY(allow_smem((const void*)kern, smem));
    void* args[] = {&I, &act, &nact, &j, &ldh, &reorth, &tol, &maxit, &err};
    FDE_CUDA_TRY(cudaLaunchCooperativeKernel(kern, dim3(ctas), dim3(RED_THREADS), args, smem, st));
    FDE_LAUNCH_CHECK("gs_batched");
    return FDE_OK;
}

int launch_residual_batched(const InstDev* I, const int* act, int nact, long max_n, cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    int g = (int)((max_n + 255) / 256);
    if (g > 64) g = 64;
    residual_batched<<<dim3(g, nact), 256, 0, st>>>(I, act);
    FDE_LAUNCH_CHECK("residual_batched");
    return FDE_OK;
}

int launch_ctl_set_batched(const InstDev* I, const int* act, int nact, int live, int reset, cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    ctl_set_batched<<<(nact + 63) / 64, 64, 0, st>>>(I, act, nact, live, reset);
    FDE_LAUNCH_CHECK("ctl_set_batched");
    return FDE_OK;
}

int launch_lsq_batched(const InstDev* I, const int* act, int nact, const int* kvec, int ldh, cudaStream_t st) {
    if (nact <= 0) return FDE_OK;
    lsq_batched<<<nact, 32, 0, st>>>(I, act, kvec, ldh);
    FDE_LAUNCH_CHECK("lsq_batched");
    return FDE_OK;
}

int launch_gather_scalars(const InstDev* I, int ninst, double* out, cudaStream_t st) {
    gather_scalars<<<(ninst + 63) / 64, 64, 0, st>>>(I, ninst, out);
    FDE_LAUNCH_CHECK("gather_scalars");
    return FDE_OK;
}

static int grid_for(long n) {
    long g = (n + 255) / 256;
    if (g > 4 * 152) g = 4 * 152;
    if (g < 1) g = 1;
    return (int)g;
}

// The form for n elements and k <= KC vectors: one element a thread in CTAs of 64, 128 or 256
// threads (the fewest that need no more CTAs than SMs, so that all SMs share the FP64 work),
// then the loop over pairs.  At n = 16,320 a step of k <= 8 takes 15.7 us with 128 threads a CTA and
// 16.5 with 256 on half as many SMs.
struct GsForm {
    const void* kern;
    int grid, threads;
    size_t smem;
};
template <int KC, int E>
static GsForm gs_form(long n, int k, int ctas) {
    const auto fits = [&](int per) { return (n + per - 1) / per <= ctas; };
    const auto grid = [&](int per) { return (int)((n + per - 1) / per); };
    if constexpr (KC <= 32) {
        if (fits(64)) return {(const void*)gs_one_kernel<KC, 1, 64>, grid(64), 64, 0};
        if (fits(128)) return {(const void*)gs_one_kernel<KC, 1, 128>, grid(128), 128, 0};
        if (fits(256)) return {(const void*)gs_one_kernel<KC, 1, 256>, grid(256), 256, 0};
    }
    // n = s m is even (s is a power of two), as the pairs of E = 2 need it
    return {(const void*)gs_kernel<KC, E>, std::min(grid(RED_THREADS * E), ctas), RED_THREADS, gs_stage_bytes(k, E)};
}

int launch_gram_schmidt(Problem& P, int j, int ldh, int reorth, cudaStream_t st) {
    const int k = j + 1;
    if (k > KMAX) return set_error(FDE_ERR_ARG, "too many Krylov vectors for one Gram-Schmidt step");
    int ctas = 0, rc = gs_ctas(&ctas);
    if (rc) return rc;
    const GsForm f = k <= 8    ? gs_form<8, 2>(P.n, k, ctas)
                     : k <= 16 ? gs_form<16, 2>(P.n, k, ctas)
                     : k <= 24 ? gs_form<24, 2>(P.n, k, ctas)
                     : k <= 32 ? gs_form<32, 1>(P.n, k, ctas)
                               : gs_form<64, 1>(P.n, k, ctas);
    if (f.smem) FDE_TRY(allow_smem((const void*)f.kern, f.smem));
    GsArgs A{P.d_V, P.d_V + (size_t)k * P.n, P.n, k, ldh, reorth, P.d_H, P.d_cs, P.d_sn, P.d_gv, P.d_scal,
             P.d_partial, P.d_counter, P.d_err, P.d_live, P.h_step + j % Problem::STEP_RING};
    void* args[] = {&A};
    FDE_CUDA_TRY(cudaLaunchCooperativeKernel(f.kern, dim3(f.grid), dim3(f.threads), args, f.smem, st));
    FDE_LAUNCH_CHECK("gs_kernel");
    return FDE_OK;
}

int launch_update(const double* V, int k, const double* coef, double sign, double* w, long n, cudaStream_t st) {
    if (k <= 0) return FDE_OK;
    update_kernel<<<grid_for(n), 256, 0, st>>>(V, k, coef, sign, w, n);
    FDE_LAUNCH_CHECK("update_kernel");
    return FDE_OK;
}

static int norm_grid(long n) { return (int)std::max<long>(1, std::min<long>(RED_CTAS, (n + 1023) / 1024)); }

int launch_norm(const double* w, long n, double* out, double* partial, unsigned int* counter, double* host,
                cudaStream_t st) {
    norm_kernel<false><<<norm_grid(n), RED_THREADS, 0, st>>>(nullptr, nullptr, const_cast<double*>(w), n, out, partial,
                                                             counter, host);
    FDE_LAUNCH_CHECK("norm_kernel");
    return FDE_OK;
}

int launch_residual_norm(const double* b, const double* ax, double* r, long n, double* out, double* partial,
                         unsigned int* counter, double* host, cudaStream_t st) {
    norm_kernel<true><<<norm_grid(n), RED_THREADS, 0, st>>>(b, ax, r, n, out, partial, counter, host);
    FDE_LAUNCH_CHECK("norm_kernel(residual)");
    return FDE_OK;
}

int launch_cycle_start(Problem& P, const double* r, const double* nrm_sq, int restart, double threshold,
                       cudaStream_t st) {
    cycle_start_kernel<<<grid_for(P.n), 256, 0, st>>>(r, nrm_sq, P.d_V, P.n, P.d_gv, restart, threshold,
                                                      P.d_scal + 133, P.d_live);
    FDE_LAUNCH_CHECK("cycle_start_kernel");
    return FDE_OK;
}

int launch_lsq_solve(const double* H, int ldh, int k, const double* g, double* y, cudaStream_t st) {
    lsq_solve_kernel<<<1, 32, 0, st>>>(H, ldh, k, g, y);
    FDE_LAUNCH_CHECK("lsq_solve_kernel");
    return FDE_OK;
}

}  // namespace fde
