"""The pinned block of a problem, compiled for the host: its parts follow one another without
overlap, it holds what the problem needs, and a block is not much larger than that."""
import ctypes
import os
import shutil
import subprocess

import pytest

SRC = r'''
#include "pinned_layout.h"
using namespace fde;
extern "C" void layout(int m, int s, int mu, size_t* o) {
    const PinnedLayout p(m, s, mu);
    const size_t v[] = {p.INFO, p.a, p.b, p.dplus, p.dminus, p.scal, p.cnt, p.start, p.bytes, p.up_bytes};
    for (size_t x : v) *o++ = x;
    const int c = pinned_class(p.bytes);
    *o++ = c;
    *o = c < PINNED_CLASSES ? PINNED_LEAST << c : 0;
}
extern "C" int size_class(size_t bytes) { return pinned_class(bytes); }
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs a host C++ compiler")
    d = tmp_path_factory.mktemp("pinned")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1305_6653_gb300", "csrc")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", inc, str(d / "t.cpp"), "-o", str(d / "t.so")],
                   check=True)
    return ctypes.CDLL(str(d / "t.so"))


@pytest.mark.parametrize("m,s,mu,block", [(1, 2, 1, 4096), (7, 16, 3, 4096), (63, 32, 3, 8192), (255, 64, 5, 16384),
                                          (2047, 256, 5, 65536), (4095, 1024, 6, 262144)])
def test_blocks_grow_with_the_problem(lib, m, s, mu, block):
    o = (ctypes.c_size_t * 12)()
    lib.layout(m, s, mu, o)
    info, a, b, dplus, dminus, scal, cnt, start, total, up, c, size = list(o)
    assert 8 * (a - info) >= 4 * (s // 2 + 2)  # a pivot word per block and the bounded waits' word
    band = (s + 1) * (mu + 1)
    assert (b - a, dplus - b, dminus - dplus, scal - dminus, start - cnt) == (band, band, m, m, 2)
    assert cnt - scal >= 134 and total == 8 * start + 4 * (s + 1) and up == total - 8 * a
    assert size == block and total <= size and (size == 4096 or size < 2 * total)


def test_sizes_beyond_the_classes_are_not_pooled(lib):
    lib.size_class.argtypes = [ctypes.c_size_t]
    assert [lib.size_class(v) for v in (1, 4096, 4097, 262144, 262145, 1 << 40)] == [0, 0, 1, 6, 7, 7]
