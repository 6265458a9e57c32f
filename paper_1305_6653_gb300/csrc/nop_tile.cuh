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
    const long b = n / m;
    return CvTile{b, (int)(n - b * m)};
}
// slot that the first tap of the tile's position t reads in a staged row (the halo's h points before its own)
NOP_FN int cv_place(int t, int x0, int m, int h) { return t + (x0 + t) / m * 2 * h; }
// length of a staged row of `count` positions
NOP_FN int cv_length(int count, int x0, int m, int h) { return count + ((x0 + count - 1) / m + 1) * 2 * h; }
// offset of slot t's point for channel 0 in a batch of Q channels, or -1 for a zero
NOP_FN ptrdiff_t cv_source(CvTile tile, int Q, int m, int h, int t) {
    const int head = m - tile.x0 + 2 * h;  // slots of the first sample's piece
    long b = tile.b0;
    int x = tile.x0 - h + t;
    if (t >= head) {
        const int u = t - head, w = m + 2 * h;
        b += 1 + u / w;
        x = u - u / w * w - h;
    }
    return x >= 0 && x < m ? (ptrdiff_t)b * Q * m + x : -1;
}
// offset of the tile's position t for channel p of a batch of P channels
NOP_FN size_t cv_offset(CvTile tile, int P, int p, int m, int t) {
    const int d = (tile.x0 + t) / m;
    return ((size_t)(tile.b0 + d) * P + p) * m + (tile.x0 + t - d * m);
}

}  // namespace fde
