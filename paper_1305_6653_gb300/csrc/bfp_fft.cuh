// Block floating-point FFT on the integer units.
//
// GB300 retires two FP64 multiply-adds per clock and SM, against 64 integer ones, so an
// FP64 FFT is bound by the FP64 pipe however it is staged.  Here a transform runs on
// 64-bit fixed-point numbers with one exponent per row (block floating point): the sums
// of a butterfly are exact 64-bit additions, a twiddle product takes sixteen 32 x 32-bit
// multiply-adds, and before every pass the row is shifted so that its largest component
// stays below 2^58 (a radix-8 pass grows a component by at most 8 sqrt 2, so nothing
// overflows).  The rounding of a pass is a few units of the last place.  While a row fills its
// 58 bits, as in the forward transform, that is below 2^-55 of the row's largest entry, where an
// FP64 pass rounds to 2^-53 of every entry.  Rows are shifted down only: the symbol shrinks the
// spectrum of a smooth row (by 2^-14 at m = 255 to 2^-22 at m = 4095), and the inverse's units are then
// of the forward spectrum's largest entry, not of what is left of it.  The symbol's own rounding,
// in units of 2^-58 against its largest value below 5.7, has the same effect there; an FP64 symbol from
// an FP64 transform has errors of 2^-53 of its largest value.  Measured totals: matvec.cu.
//
// The helpers are also compiled for the host, where the tests of the arithmetic run.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define BFP_FN __host__ __device__ __forceinline__
#else
#define BFP_FN inline
#endif

namespace fde {
namespace bfp {

struct alignas(16) I2 {
    long long x, y;
};
// exp(-2 pi i k / L) in units of 2^-61: cos = ch 2^31 + cl, sin = dh 2^31 + dl (cl, dl
// the low 31 bits, so that every partial product is one signed 32 x 32 -> 64 multiply)
struct alignas(16) Tw {
    int ch, cl, dh, dl;
};
// A real factor in units of 2^-61, split the same way
struct alignas(8) Q61 {
    int h, l;
};

constexpr int BITS = 58;  // components are below 2^BITS when a pass begins

BFP_FN Q61 q61(long long v) { return Q61{(int)(v >> 31), (int)(v & 0x7fffffff)}; }
BFP_FN I2 add(I2 a, I2 b) { return I2{a.x + b.x, a.y + b.y}; }
BFP_FN I2 sub(I2 a, I2 b) { return I2{a.x - b.x, a.y - b.y}; }
// a b + c: one 32 x 32 -> 64 multiply-add (written out, since the compiler does not always
// see that the factors fit in 32 bits)
BFP_FN long long mad(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (long long)a * b + c;
#endif
}
BFP_FN int high31(long long v) { return (int)(v >> 31); }
BFP_FN int low31(long long v) { return (int)((uint32_t)v & 0x7fffffffu); }
// z w, rounded: with a = ah 2^31 + al the product a c / 2^61 is
// 2 ah ch + (ah cl + al ch + al cl / 2^31) / 2^30.  |z| < 2^61.6, so that the middle sum
// stays below 2^63 (|ah| + |bh| <= sqrt 2 |z| / 2^31, |ch| + |dh| <= sqrt 2 2^30).
BFP_FN I2 cmul(I2 z, Tw w) {
    const int ah = high31(z.x), al = low31(z.x), bh = high31(z.y), bl = low31(z.y);
    // half a unit of the result; the low products of the imaginary part add up (below 2^63)
    // and are taken from -2^62 on, two units of the result that the high products give back
    constexpr long long RN = 1ll << 60, OFF = 1ll << 62;
    const long long rl = mad(-bl, w.dl, mad(al, w.cl, RN));
    const long long il = mad(al, w.dl, mad(bl, w.cl, RN - OFF));
    const long long rh = mad(-bh, w.dh, mad(ah, w.ch, 0));
    const long long rm = mad(-bl, w.dh, mad(-bh, w.dl, mad(al, w.ch, mad(ah, w.cl, rl >> 31))));
    const long long ih = mad(ah, w.dh, mad(bh, w.ch, 1));
    const long long im = mad(al, w.dh, mad(ah, w.dl, mad(bl, w.ch, mad(bh, w.cl, il >> 31))));
    return I2{rh * 2 + (rm >> 30), ih * 2 + (im >> 30)};
}
// x q, rounded, for a real factor |q| <= 1 and |x| < 2^62
BFP_FN long long rmul(long long x, Q61 q) {
    const int h = high31(x), l = low31(x);
    const long long m = mad(l, q.h, mad(h, q.l, mad(l, q.l, 1ll << 60) >> 31));
    return mad(h, q.h, 0) * 2 + (m >> 30);
}

// shift right by s >= 0 with rounding
BFP_FN long long shr(long long v, int s) { return s > 0 ? (v + (1ll << (s - 1))) >> s : v; }
BFP_FN I2 shr(I2 v, int s) { return I2{shr(v.x, s), shr(v.y, s)}; }
// the bits of |v|'s upper word, to be OR-ed over a row
BFP_FN uint32_t top(I2 v) { return (uint32_t)((v.x ^ (v.x >> 63)) >> 32) | (uint32_t)((v.y ^ (v.y >> 63)) >> 32); }
BFP_FN int lead(uint32_t v) {  // leading zeros
#ifdef __CUDA_ARCH__
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}
BFP_FN int lead(unsigned long long v) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
// how far a row with these upper bits has to be shifted before the next pass
BFP_FN int shift_for(uint32_t tops) {
    const int s = 64 - lead(tops) - BITS;
    return s > 0 ? s : 0;
}

BFP_FN unsigned long long bits_of(double v) {
    unsigned long long u;
#ifdef __CUDA_ARCH__
    u = (unsigned long long)__double_as_longlong(v);
#else
    __builtin_memcpy(&u, &v, 8);
#endif
    return u;
}
BFP_FN double double_of(unsigned long long u) {
    double v;
#ifdef __CUDA_ARCH__
    v = __longlong_as_double((long long)u);
#else
    __builtin_memcpy(&v, &u, 8);
#endif
    return v;
}
// v 2^(BITS - 1 + 1023 - emax) rounded, for |v| < 2^(emax - 1022), emax >= 1 the row's
// largest exponent field; integer operations only (FP64 conversions are as slow as FP64)
BFP_FN long long to_fixed(double v, int emax) {
    const unsigned long long u = bits_of(v);
    const int e = (int)(u >> 52) & 0x7ff;
    const int s = emax - (e ? e : 1);  // right shift of the significand, which starts at bit BITS - 1
    unsigned long long sig = (u & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
    sig <<= BITS - 53;
    long long r = s > 62 ? 0 : (long long)(s > 0 ? (sig + (1ull << (s - 1))) >> s : sig);
    return (long long)u < 0 ? -r : r;
}
// the double nearest to v 2^e (v an integer, |e| <= 900); integer operations only
BFP_FN double to_double(long long v, int e = 0) {
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int n = lead(a);
    if (n == 64) return 0.0;
    const unsigned long long m = a << n;  // leading bit at 63
    // significand without its leading bit, plus the rounding bit (ties upward; a carry
    // runs into the exponent, as it should)
    const unsigned long long b = ((unsigned long long)(1023 + 63 - n - 1 + e) << 52) + (m >> 11) + ((m >> 10) & 1);
    return double_of(b | (v < 0 ? 0x8000000000000000ull : 0ull));
}
BFP_FN double power_of_two(int e) { return double_of((unsigned long long)(1023 + e) << 52); }  // |e| <= 1000
// f = mantissa 2^exponent with 1 <= mantissa < 2; what is no positive normal number keeps exponent 0
BFP_FN double mantissa(double f, int* exponent) {
    const unsigned long long u = bits_of(f);
    const int x = (int)(u >> 52);
    *exponent = x > 0 && x < 0x7ff ? x - 1023 : 0;
    return x > 0 && x < 0x7ff ? double_of((u & 0xfffffffffffffull) | 0x3ff0000000000000ull) : f;
}

// sqrt(1/2) in units of 2^-61
constexpr long long HALF_SQRT = 0x16A09E667F3BCC91ll;

// -i v, v exp(-i pi / 4), v exp(-3 i pi / 4)
BFP_FN I2 rot(I2 v) { return I2{v.y, -v.x}; }
BFP_FN I2 w8(I2 v) {
    const Q61 r = q61(HALF_SQRT);
    return I2{rmul(v.x + v.y, r), rmul(v.y - v.x, r)};
}
BFP_FN I2 w83(I2 v) {
    const Q61 r = q61(HALF_SQRT);
    return I2{rmul(v.y - v.x, r), rmul(-v.x - v.y, r)};
}

BFP_FN void dft4(I2 a0, I2 a1, I2 a2, I2 a3, I2& y0, I2& y1, I2& y2, I2& y3) {
    const I2 s02 = add(a0, a2), d02 = sub(a0, a2), s13 = add(a1, a3), r = rot(sub(a1, a3));
    y0 = add(s02, s13);
    y1 = add(d02, r);
    y2 = sub(s02, s13);
    y3 = sub(d02, r);
}

// y_q = sum_j a_j exp(-2 pi i j q / R), R = 2, 4, 8
template <int R>
BFP_FN void dft(const I2 (&a)[R], I2 (&y)[R]) {
    if constexpr (R == 2) {
        y[0] = add(a[0], a[1]);
        y[1] = sub(a[0], a[1]);
    } else if constexpr (R == 4) {
        dft4(a[0], a[1], a[2], a[3], y[0], y[1], y[2], y[3]);
    } else {
        I2 b[4], c[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            b[j] = add(a[j], a[j + 4]);
            c[j] = sub(a[j], a[j + 4]);
        }
        c[1] = w8(c[1]);
        c[2] = rot(c[2]);
        c[3] = w83(c[3]);
        dft4(b[0], b[1], b[2], b[3], y[0], y[2], y[4], y[6]);
        dft4(c[0], c[1], c[2], c[3], y[1], y[3], y[5], y[7]);
    }
}

template <int R> BFP_FN constexpr int rev(int j) {  // bit reversal of log2(R) bits
    return R == 8 ? ((j & 1) << 2) | (j & 2) | (j >> 2) : R == 4 ? ((j & 1) << 1) | (j >> 1) : j;
}

// Shared-memory slot of element p: the low three bits are exchanged with the next three,
// so that the strided accesses of the short passes spread over the banks.
BFP_FN int slot(int p) { return p ^ ((p >> 3) & 7); }

// One butterfly of a pass, task g: the R points i0 + j 2^lh of a block of R 2^lh, in place.
// Both directions are the same code, since a row runs each pass once or twice and waits for
// its instructions: with a function a direction the warps of st_matvec_kernel were stalled on
// instruction fetch three times as often (1.6 against 0.56 of 8 stalls an instruction).
//   forward (decimation in frequency, natural order in, bit-reversed out): the twiddles of
//     the previous pass, radix 2^prev (0: none before), are applied on load:
//     W^(q P) to point P of the block, q the bit-reversed index of the block within it;
//   inverse (decimation in time, bit-reversed in, natural out): W^(pos j) on load.  It runs
//     on points whose two components are exchanged, which turns the inverse transform into
//     the forward one.
// tw[k << ts] is the twiddle table in units of the pass.  keep: outputs stored (R, or R / 2 in
// a last pass of which only the lower half is wanted).  Returns the upper bits it stored.
template <int R>
BFP_FN uint32_t task(I2* buf, int g, int lh, bool inv, const Tw* tw, int ts, int prev, int sh, int keep) {
    constexpr int LR = R == 8 ? 3 : R == 4 ? 2 : 1;
    const int pos = g & ((1 << lh) - 1), blk = g >> lh, i0 = (blk << (lh + LR)) + pos;
    const int q = inv || prev == 0 ? 0 : prev == 3 ? rev<8>(blk & 7) : prev == 2 ? rev<4>(blk & 3) : blk & 1;
    I2 a[R], y[R];
#pragma unroll
    for (int j = 0; j < R; ++j) a[j] = shr(buf[slot(i0 + ((inv ? rev<R>(j) : j) << lh))], sh);
    if (inv ? lh > 0 : q > 0) {
        const int base = (q * pos) << ts, step = inv ? pos << ts : (q << lh) << ts;
        if (!inv) a[0] = cmul(a[0], tw[base]);
#pragma unroll
        for (int j = 1; j < R; ++j) a[j] = cmul(a[j], tw[base + j * step]);
    }
    dft<R>(a, y);
    uint32_t t = 0;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        if (k < keep) {
            buf[slot(i0 + ((inv ? k : rev<R>(k)) << lh))] = y[k];
            t |= top(y[k]);
        }
    }
    return t;
}

// Radix (as a power of two) of the next forward pass when r levels remain, and of the next
// inverse pass: eights and fours, the short ones last forward and first inverse, where the
// strides are short (a two only for a transform of two points).
BFP_FN int radix_fwd(int r) { return r >= 3 && r != 4 ? 3 : r >= 2 ? 2 : 1; }
BFP_FN int radix_inv(int r) { return r % 3 == 0 ? 3 : r == 1 ? 1 : 2; }

// The two frequencies k and N - k of a length-2N real transform from the length-N
// transform Z of its packed points (z[n] = v[2n] + i v[2n+1]), times the real symbol kap,
// and the first level of the length-2N inverse: with E = Z_k + conj Z_{N-k},
// O = -i (Z_k - conj Z_{N-k}), V_k = (E + W^k O) / 2, V_{k+N} = (E - W^k O) / 2,
// V_{N-k} = conj V_{k+N}, V_{2N-k} = conj V_k (the halves stay in the caller's scale).
// out[0], out[1]: kap_k V_k +- kap_{k+N} V_{k+N}; out[2], out[3] the same for N - k.
BFP_FN I2 scale2(I2 v, Q61 q) { return I2{rmul(v.x, q), rmul(v.y, q)}; }
BFP_FN void split_pair(I2 za, I2 zb, Tw w, Q61 ka, Q61 kaN, Q61 kb, Q61 kbN, I2 (&out)[4]) {
    const I2 E{za.x + zb.x, za.y - zb.y};
    const I2 O{za.y + zb.y, zb.x - za.x};
    const I2 wo = cmul(O, w);
    const I2 v = add(E, wo), vN = sub(E, wo);
    const I2 a = scale2(v, ka), aN = scale2(vN, kaN);
    const I2 b = scale2(I2{vN.x, -vN.y}, kb), bN = scale2(I2{v.x, -v.y}, kbN);
    out[0] = add(a, aN);
    out[1] = sub(a, aN);
    out[2] = add(b, bN);
    out[3] = sub(b, bN);
}

// exp(-2 pi i k / 2^lgL) in units of 2^-61, by the Taylor series of sine and cosine in
// 64-bit fixed point on [0, pi/4] and the symmetries of the circle.
BFP_FN unsigned long long mulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
BFP_FN Tw twiddle(int k, int lgL) {
    // eighth of the circle and the fraction f (units of 2^-64) within it
    const unsigned long long turn = (unsigned long long)k << (64 - lgL);
    const int oct = (int)(turn >> 61);
    unsigned long long f = turn << 3;
    const bool full = (oct & 1) && f == 0;  // reflected: exactly pi/4
    if (oct & 1) f = 0ull - f;
    // x = (pi / 4) f, z = x^2, both in units of 2^-64
    const unsigned long long P = 0xC90FDAA22168C235ull;  // pi / 4
    const unsigned long long x = full ? P : mulhi(f, P);
    const unsigned long long z = mulhi(x, x);
    // sin x = x (1 - z/6 (1 - z/20 (1 - ..))), cos x = 1 - z/2 (1 - z/12 (1 - ..)); the inner
    // factors lie in (0, 1] and are held as t = 1 - factor in units of 2^-64
    unsigned long long ts = 0, tc = 0;
#pragma unroll 1
    for (int j = 11; j >= 1; --j) {
        ts = mulhi(z, ts ? 0ull - ts : ~0ull) / (unsigned)(2 * j * (2 * j + 1));
        tc = mulhi(z, tc ? 0ull - tc : ~0ull) / (unsigned)(2 * j * (2 * j - 1));
    }
    long long s = (long long)((x - mulhi(x, ts) + 4) >> 3);
    long long c = (1ll << 61) - (long long)((tc + 4) >> 3);
    // angle = oct pi/4 + (oct even: x, oct odd: pi/4 - x)
    const bool swap = ((oct + 1) & 2) != 0;  // octants 1, 2, 5, 6
    const long long cs = swap ? s : c, sn = swap ? c : s;
    const long long re = (oct >= 2 && oct <= 5) ? -cs : cs;
    const long long im = oct >= 4 ? sn : -sn;  // exp(-i angle)
    const Q61 qc = q61(re), qs = q61(im);
    return Tw{qc.h, qc.l, qs.h, qs.l};
}

}  // namespace bfp
}  // namespace fde
