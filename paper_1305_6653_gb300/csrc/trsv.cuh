// The factors' layouts and the small copies that the block solves share (trsv.cu: one problem,
// lu.cu: batches).
#pragma once
#include <cstdint>

namespace fde {

template <typename T> struct vec4;
template <> struct vec4<float> { using type = float4; };

// Streaming loads (the factor planes are read once per solve).
__device__ __forceinline__ float4 ld4(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void named_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void named_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// 32 x 32 FP32 tile with row pitch `pitch` (elements) -> shared rows of TRSV_LD elements (16 bytes of
// padding: 16-byte aligned cp.async destinations), by NTH threads.
constexpr int TRSV_LD = 36;
template <typename T, int NTH = 32>
__device__ __forceinline__ void tile_async(T* dst, const T* src, size_t pitch, int tid) {
    static_assert(sizeof(T) == 4, "");
    for (int e = tid; e < 32 * 8; e += NTH) {
        const int r = e >> 3, ch = e & 7;
        cp_async16(dst + r * TRSV_LD + ch * 4, src + (size_t)r * pitch + ch * 4);
    }
}

// Factor planes as the block solves read them (LAY): 0 row-major in the compute type
// (element (r, c) at r m_p + c); 1 strip-major in the compute type (32-column strips
// one after the other, each strip's rows contiguous: (c / 32) 32 m_p + 32 r + c mod 32),
// so every strip of a sweep is one sequential stream; 2 strip-major in bfloat16 (FP32
// compute).  The tensor-core LU writes the final factor row-major and, where it can,
// in one of the strip-major forms as well.
constexpr int LAY_PLANES = 0, LAY_STRIPS = 1, LAY_STRIPS_BF16 = 2;
template <int LAY>
__device__ __forceinline__ size_t fac_at(int mp, int r, int c) {
    return LAY != LAY_PLANES ? (size_t)(c >> 5) * 32 * mp + (size_t)r * 32 + (c & 31) : (size_t)r * mp + c;
}
// Element type of the factor as stored for layout LAY, and its streaming loads: four
// consecutive entries of one row, widened to the compute type (a bfloat16 is the top
// half of the float it came from, so the widening is exact).
template <typename T, int LAY> struct fac_store {
    using elem = T;
    using raw = typename vec4<T>::type;
    static __device__ __forceinline__ raw load(const elem* p) { return ld4(p); }
    static __device__ __forceinline__ raw widen(const raw& v) { return v; }
};
template <> struct fac_store<float, LAY_STRIPS_BF16> {
    using elem = unsigned short;
    using raw = uint2;
    static __device__ __forceinline__ raw load(const elem* p) { return __ldcs(reinterpret_cast<const uint2*>(p)); }
    static __device__ __forceinline__ float4 widen(const raw& v) {
        return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                           __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
    }
};
// 32 x 32 bfloat16 tile of a strip (rows of 64 bytes, contiguous) -> shared rows of
// TRSV_LDH elements (80 bytes: 16-byte aligned cp.async destinations).
constexpr int TRSV_LDH = 40;
template <int NTH = 32>
__device__ __forceinline__ void tile_async_bf16(unsigned short* dst, const unsigned short* src, int tid) {
    for (int e = tid; e < 32 * 4; e += NTH) {
        const int r = e >> 2, ch = e & 3;
        cp_async16(dst + r * TRSV_LDH + ch * 8, src + r * 32 + ch * 8);
    }
}

__device__ __forceinline__ void widen8(const uint4& v, float* f) {
    f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xffff0000u);
    f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xffff0000u);
    f[4] = __uint_as_float(v.z << 16); f[5] = __uint_as_float(v.z & 0xffff0000u);
    f[6] = __uint_as_float(v.w << 16); f[7] = __uint_as_float(v.w & 0xffff0000u);
}
}  // namespace fde
