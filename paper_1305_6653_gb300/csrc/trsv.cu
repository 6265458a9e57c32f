// Block solves of one problem's FP32 factors: forward (unit lower L) then backward (U)
// substitution for one Strang block per CTA, in place on rhat[k], over 32-row tiles.  Step d of a
// sweep resolves tile T(d) (T(d) = d forward, nt-1-d backward) as the product x = D^-1 a with the
// inverted diagonal tile, and subtracts the 32-column strip of L (U) below (above) it, times the
// 32 new values, from the remaining right-hand side.
//
// Two roles:
//   * CW consumer warps stream the strips of both sweeps in units of 32 x 32 (Re and Im).  The
//     warp of a row tile is fixed, so a tile's updates are ordered without any barrier; a unit
//     only needs x_d (mbarrier x[d]).  Each warp fills its own ring of stages by tensor-map copies,
//     across steps and sweeps (the factors do not depend on the solution): one thread that
//     filled a common ring took 0.29 us a unit.  Two lanes a row, 16 columns each, x_d in registers:
//     one exchange a row, where eight lanes a row spent more instructions on their shuffles than
//     on the products;
//   * four solver warps, four lanes a row.  Before solving tile d they apply strip d-1 to it
//     themselves (look-ahead), so they need the consumers' strip d-2 on tile d (b[d]) only.
//     Their diagonal and look-ahead tiles arrive by cp.async NBUF steps ahead.
// The units land swizzled, so that eight rows' 16-byte chunks of one column group fall into
// different banks.
//
// Bound by the consumers' products (about 0.1 us a unit with 14 warps on an SM; the copies alone run at
// 6.6 TB/s) and, for small blocks, by the chain of steps (0.5 us each).  us a launch, before
// (strips in registers, eight lanes a row, one solver warp) and now: m = 255, 33 blocks 20 -> 16; m = 511,
// 65 blocks 50 -> 43; m = 700, 65 blocks 87 -> 73; m = 1023, 33 blocks 151 -> 123; m = 4095, 65 blocks
// 1959 -> 1667 (5.2 TB/s).  A bfloat16 copy is better read the old way (block_trsv_bf16_kernel in lu.cu;
// m = 4095: 1150 against 1290 us), since its units cost the same products for half the bytes.
//
// Every wait is bounded: the first one to run out records an error and marks the CTA, whose other
// waits then return at once; a warp lets its copies land before it ends.
#include <cuda.h>  // CUtensorMap (the encoder is fetched from the driver at run time)

#include "fde_internal.h"
#include "fft_device.cuh"
#include "tc_ptx.cuh"
#include "trsv.cuh"

namespace fde {
namespace {

constexpr int NBUF = 4;         // solver tile buffers
constexpr int SW = 128;         // solver threads
constexpr int MAX_NT = 128;     // 32-row tiles of the largest block
constexpr int RING = 114688;    // bytes of all stages
constexpr int BAR_SOLVER = 6;   // named barrier of the solver warps
constexpr int LD = TRSV_LD;     // row pitch of the solver tiles
constexpr int TS = 32 * LD;

constexpr int UNIT = 8192;       // 32 x 32 of Re and of Im
constexpr int STAGES = RING / UNIT;

struct Ctl {
    uint64_t full[STAGES];
    uint64_t x[2][MAX_NT], b[2][MAX_NT];  // per sweep and step: x_d is there; tile d has strips <= d-2
    int dead;
};
static_assert(sizeof(Ctl) <= 5120, "");

// Bounded (a try sleeps for at most a millisecond); gives up early where another wait of the CTA has
// run out.
__device__ __forceinline__ bool wait(Ctl& c, uint64_t* bar, uint32_t parity, int* err) {
    const uint32_t a = tc::smem_u32(bar);
    for (int i = 0; i < 100000; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred P;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, P;\n\t}"
            : "=r"(ok)
            : "r"(a), "r"(parity), "r"(1000000)
            : "memory");
        if (ok) return true;
        if (*(volatile int*)&c.dead) return false;
    }
    *(volatile int*)&c.dead = 1;
    atomicCAS(err, 0, 3);
    return false;
}
__device__ __forceinline__ void arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(tc::smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(tc::smem_u32(bar))
        : "memory");
}

// The units of warp w in order: step d of a sweep, tile u >= d + 2 (counted in the sweep's direction)
// with u mod CW = w.
template <int CW> struct UnitIter {
    int nt, w, sweep = 0, d = 0, u;
    __device__ __forceinline__ UnitIter(int nt_, int w_) : nt(nt_), w(w_) {
        first();
        settle();
    }
    __device__ __forceinline__ void first() { u = d + 2 + (w - (d + 2) % CW + CW) % CW; }
    __device__ __forceinline__ void settle() {
        while (u >= nt && sweep < 2) {
            if (++d + 2 >= nt) {
                d = 0;
                ++sweep;
            }
            first();
        }
    }
    __device__ __forceinline__ bool valid() const { return sweep < 2; }
    __device__ __forceinline__ void next() {
        u += CW;
        if (u >= nt) settle();
    }
    __device__ __forceinline__ int col() const { return sweep ? nt - 1 - d : d; }
    __device__ __forceinline__ int row() const { return 32 * (sweep ? nt - 1 - u : u); }
};

// Columns 16 half .. of rows rr and rr + 16 of a unit times x, in four chains.  Explicit fused
// multiply-adds: the same rounding in every launch shape.
__device__ __forceinline__ void madd(float vr, float vi, float2 x, float2& s) {
    s.x = fmaf(-vi, x.y, fmaf(vr, x.x, s.x));
    s.y = fmaf(vi, x.x, fmaf(vr, x.y, s.y));
}
__device__ __forceinline__ void unit_product(const unsigned char* re, int rr, int half, const float2 (&x)[16], float2& a,
                                             float2& b) {
    const unsigned char* im = re + UNIT / 2;
    a = b = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int o = rr * 128 + (((4 * half + i) ^ (rr & 7)) << 4);  // the same chunk 16 rows on
        const float4 ar = *reinterpret_cast<const float4*>(re + o), ai = *reinterpret_cast<const float4*>(im + o);
        const float4 br = *reinterpret_cast<const float4*>(re + o + 2048);
        const float4 bi = *reinterpret_cast<const float4*>(im + o + 2048);
        madd(ar.x, ai.x, x[4 * i], a);
        madd(br.x, bi.x, x[4 * i], b);
        madd(ar.y, ai.y, x[4 * i + 1], a);
        madd(br.y, bi.y, x[4 * i + 1], b);
        madd(ar.z, ai.z, x[4 * i + 2], a);
        madd(br.z, bi.z, x[4 * i + 2], b);
        madd(ar.w, ai.w, x[4 * i + 3], a);
        madd(br.w, bi.w, x[4 * i + 3], b);
    }
}

template <int LAY, int CW>
__device__ __forceinline__ void consumer(int mp, int nt, int k, const CUtensorMap* map, float2* y, unsigned char* ring,
                                         Ctl& c, int* err, int w, int lane) {
    constexpr int K = STAGES / CW;  // stages of the warp
    ring += w * K * UNIT;
    uint64_t* full = c.full + w * K;
    const int half = lane >> 4, rr = lane & 15;
    UnitIter<CW> ld(nt, w), it(nt, w);
    int nld = 0, n = 0, xsw = -1, xd = -1;
    const auto load = [&] {
        if (!ld.valid()) return;
        if (lane == 0) {
            const int s = nld % K, col = ld.col(), row = ld.row();
            tc::mbar_arrive_expect_tx(full + s, (uint32_t)UNIT);
            tma_load_3d(ring + s * UNIT, map, LAY == LAY_PLANES ? 32 * col : 0,
                        LAY == LAY_PLANES ? row : col * mp + row, 2 * k, full + s);
        }
        ++nld;
        ld.next();
    };
    for (int i = 0; i < K; ++i) load();
    float2 x[16];
    for (; it.valid(); it.next(), ++n) {
        if (it.d != xd || it.sweep != xsw) {
            xd = it.d;
            xsw = it.sweep;
            if (!wait(c, &c.x[xsw][xd], 0, err)) break;
            const float4* p = reinterpret_cast<const float4*>(y + 32 * it.col() + 16 * half);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 v = p[i];
                x[2 * i] = make_float2(v.x, v.y);
                x[2 * i + 1] = make_float2(v.z, v.w);
            }
        }
        const int s = n % K;
        if (!wait(c, full + s, (uint32_t)((n / K) & 1), err)) break;
        float2 a, b;
        unit_product(ring + s * UNIT, rr, half, x, a, b);
        // the halves of a row: each lane ends with row `lane`
        float vx = half ? b.x : a.x, vy = half ? b.y : a.y;
        vx += __shfl_xor_sync(0xffffffffu, half ? a.x : b.x, 16);
        vy += __shfl_xor_sync(0xffffffffu, half ? a.y : b.y, 16);
        float2& t = y[it.row() + lane];
        t = make_float2(t.x - vx, t.y - vy);
        // every lane's reads of the stage have arrived (the sums depend on them): copy the next unit
        asm volatile("" ::"f"(vx), "f"(vy) : "memory");
        __syncwarp();
        load();
        if (it.u == xd + 2 && lane == 0) arrive(&c.b[xsw][it.u]);
    }
    for (; n < nld; ++n) tc::mbar_wait(full + n % K, (uint32_t)((n / K) & 1));  // only after a wait has run out
}

// Eight columns of one row times x: two chains a part, then the four lanes of the row.
__device__ __forceinline__ void madd8(const float (&vr)[8], const float (&vi)[8], const float2* x, float& sx, float& sy) {
    float ax = 0, ay = 0, bx = 0, by = 0;
#pragma unroll
    for (int c = 0; c < 8; c += 2) {
        const float4 v = *reinterpret_cast<const float4*>(x + c);
        ax = fmaf(-vi[c], v.y, fmaf(vr[c], v.x, ax));
        ay = fmaf(vi[c], v.x, fmaf(vr[c], v.y, ay));
        bx = fmaf(-vi[c + 1], v.w, fmaf(vr[c + 1], v.z, bx));
        by = fmaf(vi[c + 1], v.z, fmaf(vr[c + 1], v.w, by));
    }
    sx = ax + bx;
    sy = ay + by;
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
        sx += __shfl_xor_sync(0xffffffffu, sx, off);
        sy += __shfl_xor_sync(0xffffffffu, sy, off);
    }
}
__device__ __forceinline__ void tile_row8(const float* p, float (&v)[8]) {
    const float4 a = reinterpret_cast<const float4*>(p)[0], b = reinterpret_cast<const float4*>(p)[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

template <int LAY>
__device__ __forceinline__ void solver(int mp, int nt, int sweep, const float* re, const float* im, const float* tinv,
                                       float2* y, float* tiles, float2* av, Ctl& c, int* err) {
    const int tid = threadIdx.x, row = tid >> 2, q = tid & 3;
    const auto tile_of = [&](int d) { return sweep ? nt - 1 - d : d; };
    const auto issue = [&](int d) {
        if (d < nt) {
            float* b = tiles + (d & (NBUF - 1)) * 4 * TS;  // [D re, D im, L re, L im]
            const int j = tile_of(d);
            const float* ti = tinv + (size_t)j * 4096 + (sweep ? 2048 : 0);
            tile_async<float, SW>(b, ti, 32, tid);
            tile_async<float, SW>(b + TS, ti + 1024, 32, tid);
            if (d >= 1) {
                const size_t o = fac_at<LAY>(mp, 32 * j, 32 * tile_of(d - 1));
                tile_async<float, SW>(b + 2 * TS, re + o, LAY == LAY_PLANES ? mp : 32, tid);
                tile_async<float, SW>(b + 3 * TS, im + o, LAY == LAY_PLANES ? mp : 32, tid);
            }
        }
        cp_async_commit();
    };
    for (int d = 0; d < NBUF; ++d) issue(d);
    cp_async_wait<NBUF - 1>();
    named_sync(BAR_SOLVER, SW);
    for (int d = 0; d < nt; ++d) {
        const int r0 = 32 * tile_of(d);
        const float* buf = tiles + (d & (NBUF - 1)) * 4 * TS;
        const float* D = buf + row * LD + 8 * q;
        float vr[8], vi[8], dr[8], di[8], sx, sy;
        tile_row8(D, dr);
        tile_row8(D + TS, di);
        if (d >= 1) {  // look-ahead: strip d-1 on tile d's rows
            tile_row8(D + 2 * TS, vr);
            tile_row8(D + 3 * TS, vi);
            madd8(vr, vi, y + 32 * tile_of(d - 1) + 8 * q, sx, sy);
        }
        if (d >= 2) wait(c, &c.b[sweep][d], 0, err);
        float2 a = y[r0 + row];
        if (d >= 1) {
            a.x -= sx;
            a.y -= sy;
        }
        if (q == 0) av[row] = a;
        named_sync(BAR_SOLVER, SW);
        madd8(dr, di, av + 8 * q, sx, sy);
        if (q == 0) y[r0 + row] = make_float2(sx, sy);
        __syncwarp();
        if ((tid & 31) == 0) arrive(&c.x[sweep][d]);
        cp_async_wait<NBUF - 2>();    // the next step's tiles
        named_sync(BAR_SOLVER, SW);   // x_d and those tiles are everyone's, this step's buffer is free
        issue(d + NBUF);
    }
    cp_async_wait<0>();
}

template <int LAY, int CW>
__global__ void __launch_bounds__(SW + 32 * CW)
block_trsv_kernel(int mp, int nt, const float* __restrict__ fac, const float* __restrict__ tinv,
                  float2* __restrict__ rhat, int* __restrict__ err,
                  const __grid_constant__ CUtensorMap fmap, const int* __restrict__ live) {
    if (live && !*live) return;
    extern __shared__ __align__(1024) unsigned char trsv_smem[];
    __shared__ __align__(8) Ctl c;
    __shared__ __align__(16) float2 av[32];
    // the swizzle patterns repeat every 1024 bytes of the shared window
    unsigned char* ring = trsv_smem + ((1024u - (tc::smem_u32(trsv_smem) & 1023u)) & 1023u);
    float2* y = reinterpret_cast<float2*>(ring + RING);  // 32 nt
    float* tiles = reinterpret_cast<float*>(y + mp);
    const int k = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const auto* re = fac + (size_t)k * 2 * mp * mp;
    const auto* im = re + (size_t)mp * mp;
    float2* x = rhat + (size_t)k * mp;
    for (int i = threadIdx.x; i < STAGES; i += blockDim.x) tc::mbar_init(&c.full[i], 1);
    for (int i = threadIdx.x; i < nt; i += blockDim.x)
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&c.x[s][i], SW / 32);
            tc::mbar_init(&c.b[s][i], 1);
        }
    if (threadIdx.x == 0) c.dead = 0;
    tc::fence_barrier_init();
    for (int i = threadIdx.x; i < 32 * nt; i += blockDim.x) y[i] = x[i];
    __syncthreads();
    if (warp < SW / 32) {
        const float* ti = tinv + (size_t)k * (mp / 32) * 4096;
        for (int sweep = 0; sweep < 2; ++sweep) solver<LAY>(mp, nt, sweep, re, im, ti, y, tiles, av, c, err);
    } else {
        consumer<LAY, CW>(mp, nt, k, &fmap, y, ring, c, err, warp - SW / 32, lane);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 32 * nt; i += blockDim.x) x[i] = y[i];
}

// The factor as a 3-D array of boxes of 32 x 32 of both planes: planes [2 nblk][m_p rows][m_p columns],
// strips [2 nblk][(m_p / 32) m_p rows][32 columns].
template <int LAY>
int tensor_map(const Problem& P, const void* fac, CUtensorMap* map) {
    using Fn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                            const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                            CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const Fn encode = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        return e == cudaSuccess && q == cudaDriverEntryPointSuccess ? reinterpret_cast<Fn>(fn) : nullptr;
    }();
    if (!encode) return set_error(FDE_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
    const cuuint64_t esz = sizeof(float), cols = LAY == LAY_PLANES ? P.mp : 32;
    const cuuint64_t dims[3] = {cols, (cuuint64_t)P.mp * P.mp / cols, (cuuint64_t)2 * P.nblk};
    const cuuint64_t strides[2] = {cols * esz, (cuuint64_t)P.mp * P.mp * esz};
    const cuuint32_t box[3] = {32, 32, 2};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(fac), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(FDE_ERR_CUDA, "cuTensorMapEncodeTiled failed for the factors");
    return FDE_OK;
}

template <int LAY, int CW>
int launch_shape(const Problem& P, void* rhat, const void* fac, cudaStream_t st) {
    CUtensorMap map;
    FDE_TRY(tensor_map<LAY>(P, fac, &map));
    const size_t smem = 1024 + RING + (size_t)P.mp * sizeof(float2) + (size_t)NBUF * 4 * TS * sizeof(float);
    const auto kern = block_trsv_kernel<LAY, CW>;
    FDE_TRY(allow_smem((const void*)kern, smem));
    kern<<<P.nblk, SW + 32 * CW, smem, st>>>(P.mp, (P.m + 31) / 32, (const float*)fac, (const float*)P.d_tinv,
                                                  (float2*)rhat, P.d_err, map, P.live);
    FDE_LAUNCH_CHECK("block_trsv_kernel");
    return FDE_OK;
}

template <int LAY>
int launch_layout(const Problem& P, void* rhat, const void* fac, int variant, cudaStream_t st) {
    switch (variant) {  // consumer warps (FDE_TUNE_TRSV)
        case 0: return launch_shape<LAY, 7>(P, rhat, fac, st);
        case 2: return launch_shape<LAY, 12>(P, rhat, fac, st);
        case 3: return launch_shape<LAY, 10>(P, rhat, fac, st);
        default: return launch_shape<LAY, 14>(P, rhat, fac, st);
    }
}

// The tuning key of the block solves: the storage of the factors they read (FP64,
// FP32, or FDE_BF16 for the bfloat16 strip copy).
int trsv_key(const Problem& P) {
    if (P.precision == FDE_FP64) return FDE_FP64;
    return P.strips_ok && P.d_strips && P.strips_bf16 ? FDE_BF16 : FDE_FP32;
}

int launch_variant(const Problem& P, void* rhat, int variant, cudaStream_t st) {
    if (P.precision == FDE_FP64) return launch_trsv64(P, rhat, st);
    // the strip-major copy of the factor (FP32 or bfloat16), where the tensor-core LU wrote one
    if (!(P.strips_ok && P.d_strips)) return launch_layout<LAY_PLANES>(P, rhat, P.d_fac, variant, st);
    if (P.strips_bf16) return launch_trsv_bf16(P, rhat, variant, st);
    return launch_layout<LAY_STRIPS>(P, rhat, P.d_strips, variant, st);
}

struct TuneCtx {
    const Problem* P;
    void* rhat;
};
int trial(void* ctx, int v, cudaStream_t st) {
    const TuneCtx& c = *static_cast<const TuneCtx*>(ctx);
    return launch_variant(*c.P, c.rhat, v, st);
}

}  // namespace

int launch_block_trsv(const Problem& P, void* rhat, cudaStream_t st) {
    return launch_variant(P, rhat, tune_lookup(FDE_TUNE_TRSV, P.mp, P.nblk, trsv_key(P), nullptr), st);
}

// Measure the block-solve shapes for this problem's factors, on its frequency-side
// vector (zeroed first: the solves run in place and their timing does not depend on
// the data), unless the table already has the shape or a variant is forced.
int autotune_trsv(Problem& P) {
    const int prec = trsv_key(P);
    bool need = false;
    tune_lookup(FDE_TUNE_TRSV, P.mp, P.nblk, prec, &need);
    if (!need) return FDE_OK;
    if (prec == FDE_FP64) {  // one form for every variant: nothing to time
        tune_store(FDE_TUNE_TRSV, P.mp, P.nblk, prec, 0, nullptr);
        return FDE_OK;
    }
    FDE_CUDA_TRY(cudaMemsetAsync(P.d_rhat, 0, (size_t)P.nblk * P.mp * 2 * sizeof(float), P.stream));
    TuneCtx ctx{&P, P.d_rhat};
    int best = 0;
    float ms[TUNE_MAX_VARIANTS] = {};
    const int rc = tune_measure(FDE_TUNE_TRSV, P.stream, trial, &ctx, &best, ms,
                                tune_default_variant(FDE_TUNE_TRSV, prec), prec == FDE_BF16 ? 3 : 0);
    if (rc) return rc;
    tune_store(FDE_TUNE_TRSV, P.mp, P.nblk, prec, best, ms);
    return FDE_OK;
}

}  // namespace fde
