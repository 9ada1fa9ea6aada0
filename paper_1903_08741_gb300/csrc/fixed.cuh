// 64-bit fixed-point arithmetic of the field generator: complex products, FFT
// butterflies and standard normals in integers.
//
// Why integers: GB300 issues 2 FP64 operations per SM and clock, a radix-2 FP64
// butterfly with its twiddle takes 8 of them (4 clocks a lane), and the normals
// and transforms of a field batch were bound by that pipe alone.  The same
// butterfly in 64-bit integers is 12 32-bit multiplies with a 64-bit sum and
// about 30 additions and shifts, on pipes 16 to 32 times as wide.
//
// Precision: every value of a transform of white Gaussian noise has a known
// standard deviation, so one scale for all of them wastes no bits.  It is kept
// at 2^55 (overflow is at 2^61, more than 22 standard deviations away), so a
// rounding is 2^-56.8 of the value's deviation, where FP64's is about 2^-54.
#pragma once
#include <stdint.h>
#include <math.h>

namespace rich_fx {

#ifdef __CUDACC__
#define FX __host__ __device__ __forceinline__
#else
#define FX inline
#endif

constexpr int FX_BITS = 55;                 // a standard normal is 2^55

struct fx2 { long long re, im; };
// Q62 factors in balanced halves: w = h 2^32 + l with l signed.  All four
// partial products are then signed 32 x 32, and the one left out, l l', has
// mean zero and at most one unit of the result.
struct wq { int h, l; };
struct cw { wq re, im; };

FX wq split(long long a) {
    wq r;
    r.l = (int)(unsigned)(unsigned long long)a;
    r.h = (int)((a - r.l) >> 32);
    return r;
}
// of a table's value: the low half is not -2^31, so that it can be negated
FX wq split_w(long long a) {
    const wq r = split(a);
    return r.l == INT32_MIN ? split(a + 1) : r;
}
FX wq neg(wq w) { return wq{-w.h, -w.l}; }

FX long long wide(int a, int b) { return (long long)a * b; }

// x w, w in Q62: |x| <= 2^62, |w| <= 1
FX long long rmul(long long x, wq w) {
    const wq s = split(x);
    const long long mid = wide(s.h, w.l) + wide(s.l, w.h);
    return (wide(s.h, w.h) << 2) + ((mid + (1ll << 29)) >> 30);
}
FX long long rmul(long long x, long long w) { return rmul(x, split(w)); }

// x w 2^-sh, sh = 0, 1, 2: |x| < 2^61 in either part, |w| <= 1
FX fx2 cmul(fx2 x, cw w, int sh) {
    const wq a = split(x.re), b = split(x.im), v = neg(w.im);
    const long long mr = wide(a.h, w.re.l) + wide(a.l, w.re.h) + wide(b.h, v.l) + wide(b.l, v.h);
    const long long mi = wide(a.h, w.im.l) + wide(a.l, w.im.h) + wide(b.h, w.re.l) + wide(b.l, w.re.h);
    const long long hr = wide(a.h, w.re.h) + wide(b.h, v.h);
    const long long hi = wide(a.h, w.im.h) + wide(b.h, w.re.h);
    const long long rnd = 1ll << (29 + sh);
    return fx2{(hr << (2 - sh)) + ((mr + rnd) >> (30 + sh)), (hi << (2 - sh)) + ((mi + rnd) >> (30 + sh))};
}

FX long long rshift(long long x, int sh) { return sh ? (x + (1ll << (sh - 1))) >> sh : x; }

FX fx2 operator+(fx2 a, fx2 b) { return fx2{a.re + b.re, a.im + b.im}; }
FX fx2 operator-(fx2 a, fx2 b) { return fx2{a.re - b.re, a.im - b.im}; }

constexpr long long HALF_SQRT2 = 0x2D413CCCFE779921ll;      // sqrt(1/2) 2^62

// times exp(-2 pi i k / 8) (INV: its conjugate), k = 1, 2, 3
template <int K, bool INV>
FX fx2 rot8(fx2 x) {
    if (INV) { const long long t = x.re; x.re = x.im; x.im = t; }     // conjugate rotation: swap in and out
    fx2 y;
    if (K == 2) y = fx2{x.im, -x.re};
    else {
        const long long s = rmul(x.re + x.im, HALF_SQRT2), d = rmul(x.im - x.re, HALF_SQRT2);
        y = K == 1 ? fx2{s, d} : fx2{d, -s};
    }
    if (INV) { const long long t = y.re; y.re = y.im; y.im = t; }
    return y;
}

// R-point transform in registers.  Forward: natural order in, bit-reversed out
// (decimation in frequency); inverse (unnormalised): bit-reversed in, natural out.
template <int R>
FX void dft_fwd(fx2 (&a)[R]) {
    if (R == 8) {
        for (int j = 0; j < 4; ++j) { const fx2 u = a[j] + a[(j + 4) % R], v = a[j] - a[(j + 4) % R]; a[j] = u; a[(j + 4) % R] = v; }
        a[5 % R] = rot8<1, false>(a[5 % R]); a[6 % R] = rot8<2, false>(a[6 % R]); a[7 % R] = rot8<3, false>(a[7 % R]);
    }
    if (R >= 4) {
        for (int b = 0; b < R; b += 4) {
            for (int j = b; j < b + 2; ++j) { const fx2 u = a[j] + a[(j + 2) % R], v = a[j] - a[(j + 2) % R]; a[j] = u; a[(j + 2) % R] = v; }
            a[(b + 3) % R] = rot8<2, false>(a[(b + 3) % R]);
        }
    }
    for (int b = 0; b < R; b += 2) { const fx2 u = a[b] + a[b + 1], v = a[b] - a[b + 1]; a[b] = u; a[b + 1] = v; }
}
template <int R>
FX void dft_inv(fx2 (&a)[R]) {
    for (int b = 0; b < R; b += 2) { const fx2 u = a[b] + a[b + 1], v = a[b] - a[b + 1]; a[b] = u; a[b + 1] = v; }
    if (R >= 4) {
        for (int b = 0; b < R; b += 4) {
            a[(b + 3) % R] = rot8<2, true>(a[(b + 3) % R]);
            for (int j = b; j < b + 2; ++j) { const fx2 u = a[j] + a[(j + 2) % R], v = a[j] - a[(j + 2) % R]; a[j] = u; a[(j + 2) % R] = v; }
        }
    }
    if (R == 8) {
        a[5 % R] = rot8<1, true>(a[5 % R]); a[6 % R] = rot8<2, true>(a[6 % R]); a[7 % R] = rot8<3, true>(a[7 % R]);
        for (int j = 0; j < 4; ++j) { const fx2 u = a[j] + a[(j + 4) % R], v = a[j] - a[(j + 4) % R]; a[j] = u; a[(j + 4) % R] = v; }
    }
}

template <int R> FX int revr(int q) {
    return R == 8 ? ((q & 1) << 2) | (q & 2) | (q >> 2) : R == 4 ? ((q & 1) << 1) | (q >> 1) : q;
}

// Radices of an n = 2^logn transform, in the forward order: eights, the rest
// fours (a two only for n = 2).  A pass that takes the transform from b0 to b1
// of its logn bits multiplies the deviation by 2^((b1 - b0)/2); the shift b1/2
// - b0/2 (integer halves) brings it back.
FX int pass_bits(int logn, int b0) {
    const int left = logn - b0;
    return left == 4 || left == 2 ? 2 : left == 1 ? 1 : 3;
}

// tables of the normals: logarithms over 256 intervals of [1, 2), points of the
// unit circle at 256ths of a turn
struct LogEntry { long long l57; int inv; int pad; };
constexpr long long LN2_57 = 0x162E42FEFA39EF3ll >> 0;      // ln 2 in Q57
struct NormTab { LogEntry lg[256]; cw cs[256]; };

FX int clz64(unsigned long long x) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}

// fl((m + 1/2) 2^-53) 2^54 for the 53 bits m of two words, the uniform in (0, 1]
// rounded to FP64 as the definition of the noise has it (ties to even)
FX unsigned long long uniform54(uint32_t hi, uint32_t lo) {
    const unsigned long long m = (((unsigned long long)hi << 32) | lo) >> 11;
    return (m >> 52) ? 2 * (m + (m & 1)) : 2 * m + 1;
}

// log(1 + r) in Q70 for r in Q70, |r| <= 2^-8: r - r^2 P(r), Taylor to r^8
// (remainder 2^-67 of r); the factors of r^3 and on in 32 bits
FX long long log1p70(long long r) {
    const long long r62 = r >> 8;
    const int r31 = (int)(r >> 39);
    int t = (int)(0x80000000u / 7) - (int)(wide(0x10000000, r31) >> 31);
    t = (int)(0x80000000u / 6) - (int)(wide(t, r31) >> 31);
    t = (int)(0x80000000u / 5) - (int)(wide(t, r31) >> 31);
    long long p = (1ll << 60) - rmul(r62, (long long)t << 31);
    p = (1ll << 62) / 3 - rmul(r62, p);
    p = (1ll << 61) - rmul(r62, p);
    return r - rmul(rmul(r, p), r62);
}

// Two independent standard normals (Box-Muller) in Q55 from four Philox words:
// sqrt(-2 ln a) (cos, sin)(2 pi b).  ln a by intervals (Tang, ACM TOMS 16, 1990):
// a = 2^-e f, f inv = 1 + r exact; the square root from a 22-bit reciprocal root
// and its third-order correction; the angle as a table point and a remainder
// below pi/256.  Absolute error about 2^-58 (FP64's functions: 2^-53).
FX void normal_pair(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const NormTab* tab, long long& y0,
                    long long& y1) {
    // -ln a = U 2^-F
    const unsigned long long na = uniform54(c0, c1);
    const int s = clz64(na) - 10;                     // (-1 for a = 1)
    const unsigned long long M = s < 0 ? na >> 1 : na << s;
    const int i = (int)(M >> 45) & 255;
    const LogEntry e = tab->lg[i];
    const long long lg = log1p70((long long)(M * (unsigned long long)e.inv) << 5);
    const bool near1 = s == 0 && i == 255;            // there the table's part cancels
    const unsigned long long U = near1 ? -lg : (1 + s) * LN2_57 - e.l57 - ((lg + 4096) >> 13);
    if (U == 0 || s < 0) { y0 = y1 = 0; return; }
    // sqrt(2 U 2^-F) = q 2^t, q in Q62
    const int z = clz64(U);
    int ex = 1 - (near1 ? 70 : 57) - z;
    unsigned long long V = U << z;
    if (ex & 1) { V >>= 1; ++ex; }
    const float fv = (float)(uint32_t)(V >> 32) * 2.3283064365386963e-10f;
#ifdef __CUDA_ARCH__
    const float fy = rsqrtf(fv);
#else
    const float fy = 1.0f / sqrtf(fv);
#endif
    const uint32_t Y = (uint32_t)(fy * 1073741824.0f);
    const unsigned long long q0 = (V >> 32) * Y + (((V & 0xFFFFFFFFull) * Y) >> 32);
    const long long d = (1ll << 62) - (long long)((((q0 >> 32) * Y) << 2) + (((q0 & 0xFFFFFFFFull) * Y) >> 30));
    const long long dh = d >> 16;
    const long long q = (long long)q0 + rmul((long long)q0, (d >> 1) + ((3 * dh * dh) >> 33));
    const int t = 32 + (ex >> 1);
    // the angle: phi of a turn = k / 256 + x / (2 pi)
    const unsigned long long phi = uniform54(c2, c3) << 10;
    const int k = (int)((phi + (1ull << 55)) >> 56) & 255;
    const cw w = tab->cs[k];
    const long long dl = (long long)(phi - ((unsigned long long)k << 56));
    const long long x = rmul((long long)((unsigned long long)dl << 7), 0x3243F6A8885A308Dll);     // pi/4; x in Q68
    const long long x2 = rmul(x, x >> 6);                                                           // Q68
    const int x31 = (int)(x2 >> 37), x43 = (int)(x2 >> 25);
    const int s37 = (int)((1ll << 37) / 120) - (int)(wide(x31, (int)((1ll << 37) / 5040)) >> 31);
    const int c35 = (int)((1ll << 35) / 24) - (int)(wide(x31, (int)((1ll << 35) / 720)) >> 31);
    const long long S = (1ll << 62) / 6 - (wide(x43, s37) >> 18);
    const long long C = (1ll << 61) - (wide(x43, c35) >> 16);
    const long long sn = x - rmul(x, rmul(x2, S) >> 6);                                             // sin x, Q68
    const long long cm = rmul(x2, C);                                                               // 1 - cos x, Q68
    const long long ck = (((long long)w.re.h) << 32) + w.re.l, sk = (((long long)w.im.h) << 32) + w.im.l;
    const long long cb = ck - rshift(rmul(cm, w.re) + rmul(sn, w.im), 6);
    const long long sb = sk + rshift(rmul(sn, w.re) - rmul(cm, w.im), 6);
    const wq qs = split(q);
    const int sh = 62 - FX_BITS - t;                  // at least 3: |y| < 2^4
    y0 = sh > 62 ? 0 : rshift(rmul(cb, qs), sh);
    y1 = sh > 62 ? 0 : rshift(rmul(sb, qs), sh);
}

// the tables, from the host's long double functions
inline long long to_q(long double v, int bits) { return (long long)llrintl(ldexpl(v, bits)); }
inline cw circle_point(long long k, long long n) {
    const long double t = 2.0L * 3.14159265358979323846264338327950288L * (long double)k / (long double)n;
    return cw{split_w(to_q(cosl(t), 62)), split_w(to_q(sinl(t), 62))};
}
inline void make_norm_tab(NormTab& t) {
    for (int i = 0; i < 256; ++i) {
        const int inv = i == 255 ? 2048 : (int)lrint(4096.0 / (1.0 + (i + 0.5) / 256.0));
        t.lg[i] = LogEntry{inv == 2048 ? LN2_57 : to_q(-logl((long double)inv / 4096.0L), 57), inv, 0};
        t.cs[i] = circle_point(i, 256);
    }
}

}  // namespace rich_fx
