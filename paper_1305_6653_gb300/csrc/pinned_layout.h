// What a problem keeps in pinned host memory, and the sizes that blocks of it come in.  Plain
// C++: also compiled for the host alone, where the tests of the layout run.
#pragma once

#include <cstddef>

namespace fde {

// Offsets in doubles: scalars [0, 8), step outcomes [8, 24), check flag [24], status words of the
// blocks and of the bounded waits from `info` on, then the upload: A and B bands, d+, d-, zeroed
// scalars and counters, and (as ints) the band's row starts.
struct PinnedLayout {
    static constexpr size_t SCALARS = 0, OUTCOMES = 8, FLAG = 24, INFO = 32;
    static constexpr size_t NSCAL = 256, NCNT = 2;  // doubles of the device's scalars and counters
    size_t a, b, dplus, dminus, scal, cnt, start;
    size_t bytes, up_bytes;  // the whole block, the upload (from a to its end)

    PinnedLayout(int m, int s, int mu) {
        const size_t nblk = (size_t)s / 2 + 1, rows = (size_t)s + 1, band = rows * (mu + 1);
        a = INFO + ((nblk + 1) * sizeof(int) + sizeof(double) - 1) / sizeof(double);
        b = a + band;
        dplus = b + band;
        dminus = dplus + m;
        scal = dminus + m;
        cnt = scal + NSCAL;
        start = cnt + NCNT;
        bytes = start * sizeof(double) + rows * sizeof(int);
        up_bytes = bytes - a * sizeof(double);
    }
};

// Blocks come in powers of two from 4 KB to 256 KB and are cached by that size; what is larger is
// allocated as it is asked for.
constexpr size_t PINNED_LEAST = 4096;
constexpr int PINNED_CLASSES = 7;
inline int pinned_class(size_t bytes) {  // PINNED_CLASSES: larger than every class
    int c = 0;
    while (c < PINNED_CLASSES && (PINNED_LEAST << c) < bytes) ++c;
    return c;
}

}  // namespace fde
