"""Places of a convolution tile's positions (the network's kernels stage through them), compiled
for the host: every slot against the layout written out, also where batch x channels x modes
passes 2^31 and 2^32."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

SRC = r'''
#include "nop_tile.cuh"
using namespace fde;
extern "C" int places(long n0, int count, int Q, int m, int h, long* src, int* place, long* off) {
    const CvTile tile = cv_tile(n0, m);
    const int len = cv_length(count, tile.x0, m, h);
    const size_t sample = (size_t)Q * m, base = tile.b0 * sample;
    for (int t = 0; t < len; ++t) {
        const CvPoint p = cv_slot(tile.x0, m, h, t);
        src[t] = p.x < 0 ? -1 : (long)(base + cv_offset(p, sample));
    }
    for (int t = 0; t < count; ++t) place[t] = cv_place(t, tile.x0, m, h);
    for (int t = 0; t < count; ++t) off[t] = (long)(base + cv_offset(cv_position(tile.x0, m, t), sample) + (size_t)(Q - 1) * m);
    return len;
}
'''


@pytest.fixture(scope="module")
def places(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs a host C++ compiler")
    d = tmp_path_factory.mktemp("nop_tile")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1305_6653_gb300", "csrc")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", inc, str(d / "t.cpp"), "-o", str(d / "t.so")],
                   check=True)
    return ctypes.CDLL(str(d / "t.so")).places


@pytest.mark.parametrize("B,Q,m,h", [(5, 8, 1, 3), (9, 3, 5, 1), (7, 12, 16, 2), (4, 2, 130, 3), (512, 1030, 4095, 2),
                                     (2048, 1030, 2047, 1), (3_000_000, 7, 1000, 3)])
@pytest.mark.parametrize("tile", [16, 64])
def test_every_slot(places, B, Q, m, h, tile):
    N = B * m
    src, place, off = np.zeros(2048, np.int64), np.zeros(64, np.int32), np.zeros(64, np.int64)
    P = lambda x: x.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    starts = range(0, N, tile) if N < 2000 else [0, tile, N // 3 // tile * tile, (N - 1) // tile * tile]
    for n0 in starts:
        count = min(tile, N - n0)
        length = places(ctypes.c_long(n0), count, Q, m, h, P(src), P(place), P(off))
        want, at, pos = [], [], []
        for n in range(n0, n0 + count):  # a piece per sample, its halo before and after it
            b, x = divmod(n, m)
            if n == n0 or x == 0:
                want += [b * Q * m + x - d if x - d >= 0 else -1 for d in range(h, 0, -1)]
            at.append(len(want) - h)  # the first tap
            want.append(b * Q * m + x)
            pos.append((b * Q + Q - 1) * m + x)
            if n == n0 + count - 1 or x == m - 1:
                want += [b * Q * m + x + d if x + d < m else -1 for d in range(1, h + 1)]
        assert length == len(want)
        assert src[:length].tolist() == want and place[:count].tolist() == at and off[:count].tolist() == pos
