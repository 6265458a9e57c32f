// CTA-wide passes of the block floating-point FFT (bfp_fft.cuh) over a row in shared memory.
#pragma once

#include "bfp_fft.cuh"

namespace fde {
namespace bfp {

// Upper bits of a row's components, OR-ed over the CTA at the barrier that ends a pass
// (three words in turn: the next one is cleared before the barrier that publishes this one).
struct RowBits {
    uint32_t* red;
    int c = 0;
    __device__ __forceinline__ uint32_t sync_or(uint32_t t) {
        t = __reduce_or_sync(0xffffffffu, t);
        if ((threadIdx.x & 31) == 0) atomicOr(red + c, t);
        const int nx = c == 2 ? 0 : c + 1;
        if (threadIdx.x == 0) red[nx] = 0u;
        __syncthreads();
        t = red[c];
        c = nx;
        return t;
    }
};

// One transform of 2^lev points (forward or inverse, see task), of which levels lh0.. are
// done in the inverse.  tw: the twiddles of 2^logL points.  tops: the upper bits of the
// input; returns those of the result, and counts the scaling in *shifts.  half: only the
// lower half of the inverse's result is wanted.
__device__ __forceinline__ uint32_t transform(I2* buf, int lev, bool inv, int lh0, const Tw* __restrict__ tw, int logL,
                                              bool half, RowBits& bits, uint32_t tops, int* shifts) {
    const int N = 1 << lev;
    int lh = lh0, prev = 0;
    for (int r = inv ? lev - lh0 : lev; r > 0;) {
        const int k = inv ? radix_inv(r) : radix_fwd(r);
        const int sh = shift_for(tops);
        *shifts += sh;
        if (!inv) lh = r - k;
        // forward: the previous pass worked on blocks of 2^(r + prev) points
        const int ts = inv ? logL - lh - k : logL - r - prev;
        const int keep = (1 << k) >> (half && inv && r == k ? 1 : 0);
        uint32_t t = 0;
        if (k == 3)
            for (int g = threadIdx.x; g < N / 8; g += blockDim.x) t |= task<8>(buf, g, lh, inv, tw, ts, prev, sh, keep);
        else if (k == 2)
            for (int g = threadIdx.x; g < N / 4; g += blockDim.x) t |= task<4>(buf, g, lh, inv, tw, ts, prev, sh, keep);
        else
            for (int g = threadIdx.x; g < N / 2; g += blockDim.x) t |= task<2>(buf, g, lh, inv, tw, ts, prev, sh, keep);
        tops = bits.sync_or(t);
        prev = k;
        lh += k;
        r -= k;
    }
    return tops;
}

}  // namespace bfp
}  // namespace fde
