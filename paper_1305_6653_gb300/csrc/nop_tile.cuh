// Places of a convolution tile's positions.  A tile takes consecutive positions of the
// flattened batch, so that it is full whatever the number of modes m: position t of the tile is
// point (x0 + t) mod m of sample b0 + (x0 + t) / m, where (b0, x0) is its first one.  Every
// sample's piece of the tile is staged with a halo of h zeros or neighbours on either side.
// Offsets into the batch are 64-bit: batch x channels x modes may pass 2^31.
//
// The helpers are also compiled for the host, where the tests of the arithmetic run.
#pragma once

#include <stddef.h>

#ifdef __CUDACC__
#define NOP_FN __host__ __device__ __forceinline__
#else
#define NOP_FN inline
#endif

namespace fde {

// First position n (flattened) of a tile.
struct CvTile {
    long b0;
    int x0;
};
NOP_FN CvTile cv_tile(long n, int m) {
    // (a 64-bit division takes as long as a small layer's products)
    const long b = (n >> 32) == 0 ? (long)((unsigned)n / (unsigned)m) : n / m;
    return CvTile{b, (int)(n - b * m)};
}
// Point x of the sample d after the tile's first one; x < 0: a zero beyond the sample's ends.
struct CvPoint {
    int d, x;
};
// the tile's position t
NOP_FN CvPoint cv_position(int x0, int m, int t) {
    const int d = (x0 + t) / m;
    return CvPoint{d, x0 + t - d * m};
}
// slot t of a staged row
NOP_FN CvPoint cv_slot(int x0, int m, int h, int t) {
    const int head = m - x0 + 2 * h;  // slots of the first sample's piece
    CvPoint p{0, x0 - h + t};
    if (t >= head) {
        const int u = t - head, w = m + 2 * h;
        p.d = 1 + u / w;
        p.x = u - (p.d - 1) * w - h;
    }
    if (p.x >= m) p.x = -1;
    return p;
}
// slot that the first tap of the tile's position t reads in a staged row (the halo's h points
// before its own)
NOP_FN int cv_place(int t, int x0, int m, int h) { return t + (x0 + t) / m * 2 * h; }
// length of a staged row of `count` positions
NOP_FN int cv_length(int count, int x0, int m, int h) { return count + ((x0 + count - 1) / m + 1) * 2 * h; }
// offset of a point (channel 0) from the tile's first sample, `sample` entries each
NOP_FN size_t cv_offset(CvPoint p, size_t sample) { return (size_t)p.d * sample + p.x; }

}  // namespace fde
