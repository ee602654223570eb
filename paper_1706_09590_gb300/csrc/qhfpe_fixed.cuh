// Block fixed-point transforms for the FP64 form.
//
// GB300 issues two FP64 instructions per clock and SM, and 64 integer ones (measured: DFMA 1.7, 32-bit
// IMAD / shift / add 57 to 62, 32 x 32 + 64 multiply-add 25 to 30 per clock and SM; a DFMA costs the same
// with one active lane as with 32).  A length-128 FFT along p needs about 20 FP64 instructions per
// point, so the FP64 pipe bounded the whole FP64 stage.  Here the butterflies of a transform run on
// 64-bit integers: the inputs of one butterfly share a binary exponent (that of their largest component),
// sums are exact, and twiddle products keep the upper 64 of 128 bits.  An FFT mixes all points of a row, so
// its rounding error is relative to the row's norm in either arithmetic; with 58 to 60 bits below the
// largest input and a binary point that follows the growth of the sums, that error is smaller than the FP64
// butterflies' (forward 4e-17 to 1.3e-16 against 8e-17 to 2.1e-16 of the norm, tests/test_fixed_fft_fp64.py).
//
// Magnitudes (complex): a radix-16 pass takes inputs below 2^60 and scales by 1/4 between its two layers
// of length-4 transforms (outputs below 2^62); a radix-8 pass takes inputs below 2^59; a twiddle product
// takes inputs below 2^62 and scales by 1/4 or 1/8.  Every intermediate stays below 2^63.
// Common exponents of transforms go past those of doubles; conversions near the ends of the range of doubles are
// to_fixed_any and from_fixed_any.  A row with an infinity or a NaN (exponent EXP_BAD) gives NaN.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define QH_HD __host__ __device__ __forceinline__
#else
#define QH_HD inline
#endif

namespace qhfx {

struct I2 {  // complex fixed-point value
    long long x, y;
};

// common exponents of a transform: from here on an infinity or a NaN among its inputs
constexpr int EXP_BAD = 16000;
// ... of a row of zeros, and the exponent of a table row of zeros: sums with one of those are below EXP_ZERO (others are
// above -1300), and the values zero
constexpr int EXP_NONE = -6000, EXP_NO_TABLE = -4096, EXP_ZERO = -1500;
// exponents of doubles outside of these (values below 2^-895, from 2^927) take the functions for any value; between
// them rates from 2^-60 to 2^90 leave normal numbers
constexpr int EXP_SMALL = 128, EXP_BIG = 1950;
QH_HD bool exp_far(int M) { return (unsigned)(M - EXP_SMALL) >= (unsigned)(EXP_BIG - EXP_SMALL) && M >= EXP_ZERO; }
QH_HD bool exp_plain(int E) { return (unsigned)(E - EXP_SMALL) < (unsigned)(EXP_BIG - EXP_SMALL); }

QH_HD unsigned long long dbits(double v)
{
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long u;
    memcpy(&u, &v, 8);
    return u;
#endif
}
QH_HD double bitsd(unsigned long long u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double v;
    memcpy(&v, &u, 8);
    return v;
#endif
}
// shifts by any s >= 0 (64 and more: all bits go, as in PTX)
QH_HD unsigned long long shr_u(unsigned long long m, int s)
{
#ifdef __CUDA_ARCH__
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(s));
    return m;
#else
    return s > 63 ? 0 : m >> s;
#endif
}
QH_HD long long shr_s(long long m, int s)
{
#ifdef __CUDA_ARCH__
    asm("shr.s64 %0, %0, %1;" : "+l"(m) : "r"(s));
    return m;
#else
    return m >> (s > 63 ? 63 : s);
#endif
}

// v / 2^s rounded (half up), |v| <= 2^62, any s >= 0: sums over cells must not collect a floor's bias
QH_HD long long shr_round(long long v, int s)
{
    s = s > 62 ? 62 : s;
    return (v + (long long)((1ull << s) >> 1)) >> s;
}

// biased exponent of a double
QH_HD int exponent_of(double v) { return (int)(dbits(v) >> 52) & 2047; }
// common exponents are at least this, so that zeros (and inputs below 2^-1022) are shifted out
constexpr int EXP_MIN = 64;

// v as a multiple of 2^(E - 1022 - B), where E >= its exponent and EXP_MIN: below 2^B, truncated toward zero.
template <int B> QH_HD long long to_fixed(double v, int E)
{
    const unsigned long long u = dbits(v);
    const int ex = (int)(u >> 52) & 2047;
    const unsigned long long m = shr_u(((u & 0xfffffffffffffull) | 0x10000000000000ull) << (B - 53), E - ex);
    const long long s = (long long)u >> 63;
    return ((long long)m ^ s) - s;
}

// ... for any E from max(its exponent, 1) on, subnormal values too
template <int B> QH_HD long long to_fixed_any(double v, int E)
{
    const unsigned long long u = dbits(v);
    const int ex = (int)(u >> 52) & 2047;
    const unsigned long long m = shr_u(((u & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0)) << (B - 53), E - (ex ? ex : 1));
    const long long s = (long long)u >> 63;
    return ((long long)m ^ s) - s;
}

QH_HD int clz64(unsigned long long u)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)u);
#else
    return u ? __builtin_clzll(u) : 64;
#endif
}

// v * 2^K rounded to a double (half away from zero), where the result is zero or a normal number.  Integer operations: the conversion instruction takes two and more slots of the FP64
// pipe (stage on 96 x 128, depth 8: 0.73 ms with it).
QH_HD double from_fixed(long long v, int K)
{
    const long long s = v >> 63;
    unsigned long long m = (unsigned long long)((v ^ s) - s);
    const int n = clz64(m);
    m <<= n & 63;
    unsigned long long r = (m >> 11) + ((m >> 10) & 1);
    r += (unsigned long long)(unsigned)(K - n + 63 + 1022) << 52;  // the leading bit carries into the exponent
    r |= (unsigned long long)s & 0x8000000000000000ull;
    return bitsd(v ? r : 0);
}

// v * 2^K over the whole range of doubles: subnormal results and infinities too
QH_HD double from_fixed_any(long long v, int K)
{
    const unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
    const int e = K + 63 - clz64(m) + 1022;
    if (v == 0 || (unsigned)e <= 2045u) return from_fixed(v, K);
    K = K < -2044 ? -2044 : (K > 2044 ? 2044 : K);
    const int h = K >> 1;  // in two steps, the first of them exact
    return (double)v * bitsd((unsigned long long)(h + 1023) << 52) * bitsd((unsigned long long)(K - h + 1023) << 52);
}

// The two halves of a 64-bit factor, the low one signed: c = h * 2^32 + l
struct Half {
    int h, l;
};
QH_HD Half halves(long long c)
{
#ifdef __CUDA_ARCH__
    int lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(c));
    return Half{hi + (int)((unsigned)lo >> 31), lo};
#else
    return Half{(int)((c + 0x80000000ll) >> 32), (int)(unsigned)(unsigned long long)c};
#endif
}
// c + a b, one instruction (written out: as C, two to three times the instructions came out -- a twiddle
// product took 65 of them instead of 29, a real product 17 instead of 7)
QH_HD long long madw(int a, int b, long long c)
{
#ifdef __CUDA_ARCH__
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return c + (long long)a * b;
#endif
}

// (a ca + b cb) / 2^64, rounded; the product of the two low halves (below half a unit) is left out
QH_HD long long mul_add(Half a, Half ca, Half b, Half cb)
{
    long long cross = madw(a.h, ca.l, 0x80000000ll);
    cross = madw(a.l, ca.h, cross);
    cross = madw(b.h, cb.l, cross);
    cross = madw(b.l, cb.h, cross);
    return madw(b.h, cb.h, madw(a.h, ca.h, cross >> 32));
}
QH_HD long long mul_hi(Half a, Half k)  // a k / 2^64, rounded
{
    const long long cross = madw(a.l, k.h, madw(a.h, k.l, 0x80000000ll));
    return madw(a.h, k.h, cross >> 32);
}
QH_HD long long mul_hi(long long v, long long c) { return mul_hi(halves(v), halves(c)); }

// a (c + i s) over 2^64
QH_HD I2 rot_p(I2 a, long long c, long long s)
{
    const Half x = halves(a.x), y = halves(a.y), C = halves(c), S = halves(s);
    return I2{mul_add(x, C, y, Half{-S.h, -S.l}), mul_add(x, S, y, C)};
}
template <int SG> QH_HD I2 rot(I2 a, long long c, long long s) { return rot_p(a, c, SG * s); }

template <int SH> QH_HD I2 shr(I2 a)  // a / 2^SH, rounded
{
    constexpr long long h = 1ll << (SH - 1);
    return I2{(a.x + h) >> SH, (a.y + h) >> SH};
}

// Normalisation of a run of values by the bits that any of them has: their magnitude words ORed, and the
// left shift (negative: right) that brings them below 2^top
QH_HD unsigned magnitude(I2 a)
{
    const int x = (int)(a.x >> 32), y = (int)(a.y >> 32);
    return (unsigned)((x ^ (x >> 31)) | (y ^ (y >> 31)));
}
template <int TOP> QH_HD int norm_shift(unsigned o)
{
#ifdef __CUDA_ARCH__
    const int n = __clz((int)o);
#else
    const int n = o ? __builtin_clz(o) : 32;
#endif
    return n + TOP - 64;
}
QH_HD I2 shift(I2 a, int n)
{
    return n >= 0 ? I2{(long long)((unsigned long long)a.x << n), (long long)((unsigned long long)a.y << n)}
                  : I2{a.x >> -n, a.y >> -n};
}

QH_HD I2 add(I2 a, I2 b) { return I2{a.x + b.x, a.y + b.y}; }
QH_HD I2 sub(I2 a, I2 b) { return I2{a.x - b.x, a.y - b.y}; }
template <int SG> QH_HD I2 mul_si(I2 a) { return SG > 0 ? I2{-a.y, a.x} : I2{a.y, -a.x}; }
template <int SG> QH_HD I2 add_si(I2 a, I2 b) { return SG > 0 ? I2{a.x - b.y, a.y + b.x} : I2{a.x + b.y, a.y - b.x}; }
template <int SG> QH_HD I2 sub_si(I2 a, I2 b) { return add_si<-SG>(a, b); }

// round(cos(pi/8) 2^62), round(sin(pi/8) 2^62), round(2^61.5), round(2^62.5)
constexpr long long C1 = 0x3b20d79e651a8c51ll, S1 = 0x187de2a6aea962d2ll, H62 = 0x2d413cccfe779921ll,
                    H63 = 0x5a827999fcef3242ll;

template <int SG> QH_HD void dft4(I2 &x0, I2 &x1, I2 &x2, I2 &x3)
{
    const I2 t0 = add(x0, x2), t1 = sub(x0, x2), t2 = add(x1, x3), d = sub(x1, x3);
    x0 = add(t0, t2);
    x2 = sub(t0, t2);
    x1 = add_si<SG>(t1, d);
    x3 = sub_si<SG>(t1, d);
}
// length 8: inputs below 2^59, outputs below 2^62 (no scaling)
template <int SG> QH_HD void dft8(I2 *x)
{
    I2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    I2 o0 = x[1], o1 = x[3], o2 = x[5], o3 = x[7];
    dft4<SG>(e0, e1, e2, e3);
    dft4<SG>(o0, o1, o2, o3);
    // o1 (1 + SG i) / sqrt 2 and o3 (-1 + SG i) / sqrt 2: the product with 2^62.5 leaves half of it
    const I2 a = add_si<SG>(o1, o1), b = sub_si<SG>(o3, o3);
    const I2 w1 = {2 * mul_hi(a.x, H63), 2 * mul_hi(a.y, H63)};
    const I2 w3 = {-2 * mul_hi(b.x, H63), -2 * mul_hi(b.y, H63)};
    x[0] = add(e0, o0);
    x[4] = sub(e0, o0);
    x[1] = add(e1, w1);
    x[5] = sub(e1, w1);
    x[2] = add_si<SG>(e2, o2);
    x[6] = sub_si<SG>(e2, o2);
    x[3] = add(e3, w3);
    x[7] = sub(e3, w3);
}
// length 16 as 4 x 4: inputs below 2^60, outputs (over 4) below 2^62
template <int SG> QH_HD void dft16(I2 *x)
{
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) dft4<SG>(x[n2], x[4 + n2], x[8 + n2], x[12 + n2]);  // y[n2][k1] at x[4 k1 + n2]
    // w16^(n2 k1), over 4
    x[0] = shr<2>(x[0]);
    x[1] = shr<2>(x[1]);
    x[2] = shr<2>(x[2]);
    x[3] = shr<2>(x[3]);
    x[4] = shr<2>(x[4]);
    x[8] = shr<2>(x[8]);
    x[12] = shr<2>(x[12]);
    const auto h45 = [](I2 a, int sx, int sy) {  // (a.x sx - a.y sy) h ... for the multiples of 45 degrees
        return I2{mul_hi(a.x * sx - a.y * sy, H62), mul_hi(a.x * sy + a.y * sx, H62)};
    };
    x[5] = rot<SG>(x[5], C1, S1);        // n2 = 1, k1 = 1
    x[9] = h45(x[9], 1, SG);             // n2 = 1, k1 = 2
    x[13] = rot<SG>(x[13], S1, C1);      // n2 = 1, k1 = 3
    x[6] = h45(x[6], 1, SG);             // n2 = 2, k1 = 1
    x[10] = shr<2>(mul_si<SG>(x[10]));   // n2 = 2, k1 = 2
    x[14] = h45(x[14], -1, SG);          // n2 = 2, k1 = 3
    x[7] = rot<SG>(x[7], S1, C1);        // n2 = 3, k1 = 1
    x[11] = h45(x[11], -1, SG);          // n2 = 3, k1 = 2
    x[15] = rot<SG>(x[15], -C1, -S1);    // n2 = 3, k1 = 3
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) dft4<SG>(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);  // -> X[k1 + 4 k2] at x[4 k1 + k2]
    I2 t[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) t[k1 + 4 * k2] = x[4 * k1 + k2];
#pragma unroll
    for (int k = 0; k < 16; ++k) x[k] = t[k];
}
template <int R, int SG> QH_HD void dft_small(I2 *x)
{
    if constexpr (R == 2) {
        const I2 t = x[0];
        x[0] = add(t, x[1]);
        x[1] = sub(t, x[1]);
    } else if constexpr (R == 4) dft4<SG>(x[0], x[1], x[2], x[3]);
    else if constexpr (R == 8) dft8<SG>(x);
    else dft16<SG>(x);
}

// ---- the radix-R0 butterflies of a transform of length R0 * 16 and its inverse ----------------------------
// Forward: radix R0 with twiddles, then radix 16.  Inverse, of values with exchanged parts (which makes it a
// forward one): radix 16, then radix R0 after the twiddles.  w: e^{2 pi i t / np} times 2^62; j: the
// butterfly (points j, j + 16, ...).
template <int R0> struct Scale {
    static constexpr int bits = R0 == 8 ? 58 : (R0 == 2 ? 60 : 59);  // forward input components below 2^bits
    static constexpr int down = R0 == 16 ? 2 : 0;                    // dft_small<R0> leaves the sum over 2^down
    static constexpr int inv = R0 == 8 ? 3 : 2;                      // inverse twiddle products leave 2^-inv
    // an input v 2^(E - 1022 - bits) leaves the first forward pass as v 2^(E + K_fwd), the second as
    // v 2^(E + K_fwd + 2); the inverse multiplies the unit by 2^(2 + inv + down)
    static constexpr int K_fwd = -1022 - bits + down + 2;
};
template <int R> QH_HD int common_exponent(const double *re, const double *im)
{
    int E = EXP_MIN;
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int a = exponent_of(re[t]), b = exponent_of(im[t]);
        E = E > a ? E : a;
        E = E > b ? E : b;
    }
    return E;
}
// values of exponents e[] brought to the largest one
template <int R> QH_HD int align(I2 *x, const int *e)
{
    int E = e[0];
#pragma unroll
    for (int t = 1; t < R; ++t) E = E > e[t] ? E : e[t];
#pragma unroll
    for (int t = 0; t < R; ++t) x[t] = I2{shr_s(x[t].x, E - e[t]), shr_s(x[t].y, E - e[t])};
    return E;
}
template <int R0> QH_HD void forward_butterfly(I2 *x, const I2 *w, int j)
{
    dft_small<R0, +1>(x);
    x[0] = shr<2>(x[0]);
#pragma unroll
    for (int u = 1; u < R0; ++u) x[u] = rot_p(x[u], w[j * u].x, w[j * u].y);
}
template <int R0> QH_HD void inverse_butterfly(I2 *x, const I2 *w, int j)
{
    constexpr int SH = Scale<R0>::inv;
    x[0] = shr<SH>(x[0]);
#pragma unroll
    for (int u = 1; u < R0; ++u) x[u] = rot_p(x[u], w[j * u].x >> (SH - 2), w[j * u].y >> (SH - 2));
    dft_small<R0, +1>(x);
}

}  // namespace qhfx
