"""The 64-bit products of the block floating-point FFT, compiled for the host: every result
is the exact product rounded to a unit, up to the largest magnitudes a pass can meet."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

SRC = r'''
#include "bfp_fft.cuh"
using namespace fde::bfp;
extern "C" void mul(int n, const long long* z, const int* k, int lg, long long* out, long long* w, long long* r) {
    for (int i = 0; i < n; ++i) {
        const Tw t = twiddle(k[i], lg);
        w[2 * i] = ((long long)t.ch << 31) + t.cl;
        w[2 * i + 1] = ((long long)t.dh << 31) + t.dl;
        const I2 p = cmul(I2{z[2 * i], z[2 * i + 1]}, t);
        out[2 * i] = p.x;
        out[2 * i + 1] = p.y;
        r[i] = rmul(z[2 * i], Q61{t.ch, t.cl});
    }
}
'''


def circle(k, L):
    """(cos, sin) of 2 pi k / L with the angle reduced to the first eighth of the circle in
    integers, so that the doubles carry no rounding of the angle's turns."""
    q, r = divmod(8 * k, L)
    r = L - r if q & 1 else r
    a = 2 * np.pi * (r / (8 * L))
    c, s = np.cos(a), np.sin(a)
    return [(c, s), (s, c), (-s, c), (-c, s), (-c, -s), (-s, -c), (s, -c), (c, -s)][q]


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host C++ compiler")
@pytest.mark.parametrize("lg", [1, 3, 13])
def test_products_are_exact_to_the_rounding(tmp_path, lg):
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1305_6653_gb300", "csrc")
    (tmp_path / "mul.cpp").write_text(SRC)
    so = str(tmp_path / "mul.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-shared", "-fPIC", "-I", inc,
                    str(tmp_path / "mul.cpp"), "-o", so], check=True)
    rng = np.random.default_rng(lg)
    n = 2000
    k = rng.integers(0, 1 << lg, n).astype(np.int32)
    # moduli up to the 2^61.5 of a radix-8 pass, with every low bit set or clear as well
    r = np.concatenate([rng.uniform(0, 2 ** 61.5, n - 500), np.full(500, 2 ** 61.4999)])
    a = rng.uniform(0, 2 * np.pi, n)
    z = np.stack([r * np.cos(a), r * np.sin(a)], axis=1).astype(np.int64)
    z[: n // 4] |= 0x7fffffff
    z[n // 4: n // 2] &= ~0x7fffffff
    z = np.ascontiguousarray(z)
    out, w, s = np.zeros((n, 2), np.int64), np.zeros((n, 2), np.int64), np.zeros(n, np.int64)
    P = lambda x: x.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    ctypes.CDLL(so).mul(n, P(z), P(k), lg, P(out), P(w), P(s))
    one = 1 << 61
    for (x, y), (c, d), (p, q), t, kk in zip(z.tolist(), w.tolist(), out.tolist(), s.tolist(), k.tolist()):
        # a unit: half of it the final rounding, the rest the floors of the low products
        assert abs((x * c - y * d) - p * one) <= one and abs((x * d + y * c) - q * one) <= one
        assert abs(x * c - t * one) <= one
        u = circle(kk, 1 << lg)
        assert abs(c - u[0] * one) <= 2 ** 10 and abs(d + u[1] * one) <= 2 ** 10  # the double's own rounding
