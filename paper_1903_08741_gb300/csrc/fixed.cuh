// 64-bit fixed-point arithmetic: the field generator's complex products, FFT
// butterflies and standard normals, and the closures' elementary functions.
//
// Why integers: GB300 issues 2 FP64 operations per SM and clock, a radix-2 FP64
// butterfly with its twiddle takes 8 of them (4 clocks a lane), and the normals
// and transforms of a field batch were bound by that pipe alone.  The same
// butterfly in 64-bit integers is 12 32-bit multiplies with a 64-bit sum and
// about 30 additions and shifts, on pipes 16 to 32 times as wide.
//
// Precision: every value of a transform of white Gaussian noise has a known
// standard deviation, so one scale for all of them wastes no bits.  It starts at
// 2^55 and, as the shifts are whole bits, is up to 2^55.5 between the passes of a
// row and 2^56 between those of a column (behind rows of an odd power of two);
// inside a pass, before its shift, it is up to 2^57 and 2^57.5.  Overflow is at
// 2^61: 16 and 11 standard deviations (probabilities of 1e-57 and 1e-29 a value).
// A rounding is 2^-56.8 of the scale, where FP64's is about 2^-54 of the value.
#pragma once
#include <stdint.h>
#include <math.h>
#include <string.h>

namespace rich_fx {

#ifdef __CUDACC__
#define FX __host__ __device__ __forceinline__
#define FXD __device__ __forceinline__       // reads the tables of device memory
#else
#define FX inline
#define FXD inline
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
struct PhiEntry { long long phi, c[4]; int b[4], e, pad; };    // Phi_k = phi 2^-62 2^e
constexpr int PHI_SIDE = 256;
struct NormTab { LogEntry lg[256]; cw cs[256]; PhiEntry phi[2 * PHI_SIDE + 1]; };

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
// (remainder 2^-67 of r); the factors of r^3 and on from 32-bit halves (2^-63)
FX long long log1p70(long long r) {
    const long long r62 = r >> 8;
    const int r39 = (int)(r >> 31);
    int t = (int)(0x80000000u / 7) - (int)(wide(0x10000000, r39) >> 39);
    t = (int)(0x80000000u / 6) - (int)(wide(t, r39) >> 39);
    t = (int)(0x80000000u / 5) - (int)(wide(t, r39) >> 39);
    t = 0x20000000 - (int)(wide(t, r39) >> 39);
    const long long p = (1ll << 61) - rmul(r62, (1ll << 62) / 3 - (wide(t, r39) >> 8));
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

// ---------------------------------------------------------------- exp and log
// The closures' elementary functions without the FP64 pipe (CUDA's exp holds it
// for 16 multiply-adds, this one for none and about 70 integer instructions on
// pipes 16 times as wide).  Tables and remainders after Tang (ACM TOMS 15, 1989
// and 16, 1990); working precision 2^-60.
#ifdef __CUDACC__
#define FX_TABLE static __device__ const
#else
#define FX_TABLE static const
#endif
#include "fixed_tables.cuh"

constexpr unsigned long long LN2_128 = 0x58B90BFBE8E7BCull;  // ln 2 / 128: Q62 and the next 32 bits
constexpr unsigned int LN2_128_LO = 0xD5E4F1D9u;

// 2^(k/128) e^r = v 2^n: v in Q62, 1 <= v < 2 (up to rounding); r in Q62, |r| < 2^-7.9
FXD unsigned long long exp_core(int k, long long r, int& n) {
    const int r31 = (int)(r >> 31);
    const int c24 = (int)((1ll << 31) / 24) + (int)(wide(r31, (int)((1ll << 31) / 120)) >> 31);
    long long p = (1ll << 62) / 6 + wide(r31, c24);
    p = (1ll << 61) + rmul(r, p);
    p = r + rmul(rmul(r, r), p);
    const long long t = EXP_TAB[k & 127];
    n = k >> 7;
    const unsigned long long v = (unsigned long long)(t + rmul(t, p));
    if (v >> 62) return v;
    --n;                                                     // 2^0 e^r with r < 0
    return v << 1;
}

FX double bits_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d; memcpy(&d, &b, 8); return d;
#endif
}
// v 2^n (v in Q62) rounded to FP64; the result is normal
FX double fx_to_double(unsigned long long v, int n) {
    const unsigned long long m = (v + 512) >> 10;            // 2^52 <= m <= 2^53
    return bits_double(m + ((unsigned long long)(n + 1022) << 52));
}
FX unsigned long long double_bits(double x) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long b; memcpy(&b, &x, 8); return b;
#endif
}

// exp(x) to 0.54 units in the last place for |x| < 512 (any other x: the library's)
FXD double fx_exp(double x) {
    const unsigned long long b = double_bits(x);
    const int e = (int)(b >> 52 & 0x7FF) - 1023;
    if (e >= 9 || e < -60) return exp(x);                    // large, NaN; tiny, zero
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    int k = 0;
    if (e >= -8) {                                           // round(|x| 128 / ln 2)
        const unsigned long long q = (m >> 21) * 0xB8AA3B29ull;
        k = (int)((q + (1ull << (54 - e))) >> (55 - e));
    }
    long long r = e >= -10 ? (long long)(m << (e + 10)) : (long long)(m >> -(e + 10));   // |x| in Q62 mod 4
    r -= (long long)((unsigned long long)k * LN2_128 + (((unsigned long long)k * LN2_128_LO) >> 32));
    if (b >> 63) { k = -k; r = -r; }
    int n;
    const unsigned long long v = exp_core(k, r, n);
    return fx_to_double(v, n);
}

// a / b, correctly rounded, where both are positive and normal and the quotient is
// well inside the normal range (all else: the FP64 division, which holds its pipe
// for about 9 multiply-adds, two to four of them a cell and Picard iteration).  A
// 23-bit reciprocal of b and its third-order correction give the quotient to within
// a unit of its last place, and the exact remainder against half of b decides that
// unit (no quotient of two 53-bit numbers lies midway).  Against the FP64 division,
// same bits: 608 samples on 128^2, two steps, in mixed precision 290 -> 276 ms, in
// FP64 542 -> 532 (runs 4 % apart), 64 samples on 32^2, ten steps, 98.9 -> 98.1.
FX double fx_div(double a, double b) {
    const unsigned long long ba = double_bits(a), bb = double_bits(b), one = 1ull << 52;
    const int ea = (int)(ba >> 52), eb = (int)(bb >> 52), ex = ea - eb + 1023;
    if ((unsigned)(ea - 1) >= 2046u || (unsigned)(eb - 1) >= 2046u || ex < 8 || ex > 2038) return a / b;
    const unsigned long long ma = (ba & (one - 1)) | one, mb = (bb & (one - 1)) | one, B = mb << 11;   // (B in Q63)
    const unsigned int fb = 0x3F800000u | ((unsigned int)(B >> 40) & 0x7FFFFFu);
#ifdef __CUDA_ARCH__
    const unsigned int fy = __float_as_uint(__frcp_rn(__uint_as_float(fb)));
#else
    float f; memcpy(&f, &fb, 4); f = 1.0f / f;
    unsigned int fy; memcpy(&fy, &f, 4);
#endif
    const uint32_t Y = fy == 0x3F800000u ? 0x7FFFFFFFu : ((fy & 0x7FFFFFu) | 0x800000u) << 7;     // 1/b in Q31
    // d = 1 - b Y in Q62, |d| < 2^-21
    const long long d = (long long)((1ull << 62) - ((B >> 32) * Y + (((B & 0xFFFFFFFFull) * Y) >> 32)));
    const long long dh = d >> 16;
    const long long c = d + ((dh * dh) >> 30);
    const long long y = ((long long)Y << 31) + rmul(c, (long long)Y << 31);
    const long long q = rmul((long long)ma << 9, y);         // ma / mb in Q61, good to 2^-58
    // 53 bits of it, exactly s fraction bits, and their remainder, modulo 2^64
    const int s = ma < mb ? 53 : 52;
    unsigned long long m = (unsigned long long)((q + (1ll << (60 - s))) >> (61 - s));
    const long long rem = (long long)((ma << s) - m * mb);
    m += (unsigned long long)((long long)(2 * rem > (long long)mb) - (long long)(2 * rem < -(long long)mb));
    return bits_double(m + ((unsigned long long)(ex - 1 + 52 - s) << 52));
}

// e^(y 2^-F), |y 2^-F| < 512, as v 2^n
template <int F>
FXD unsigned long long exp_fixed(long long y, int& n) {
    const int k = (int)((wide((int)(y >> (F - 22)), 1549082005) + (1ll << 44)) >> 45);     // 128 / ln 2 in Q23
    const unsigned long long c = (unsigned long long)(long long)k * LN2_128 +
                                 (unsigned long long)(((long long)k * (long long)LN2_128_LO) >> 32);
    return exp_core(k, (long long)(((unsigned long long)y << (62 - F)) - c), n);
}
template <int F>
FXD double exp_fixed(long long y) {
    int n;
    const unsigned long long v = exp_fixed<F>(y, n);
    return fx_to_double(v, n);
}

// ln(M 2^(e-59)) in Q57, 2^59 <= M < 2^60, |e| < 90
FXD long long log_fixed(unsigned long long M, int e) {
    const int i = (int)(M >> 51) & 255;
    const long long r = (long long)(M * (unsigned long long)LOG_INV[i]) >> 1;
    return e * LN2_57 + LOG_TAB[i] + ((log1p70(r) + 4096) >> 13);
}

// van Genuchten saturation at -p = ap/a, in logarithms: with L = ln ap,
// s = (1 + ap^n)^-m = e^t.  False where a value leaves the fixed-point ranges
// (2^-59 <= ap < 2^59, 2^-6 <= n < 16, 2^-20 <= m < 1, 2^-369 < ap^n < 2^58).
struct VgLog { long long t, g, l1; };       // t in Q57; g = (n - 1) L in Q53; l1 = ln(1 + ap^n) in Q57
FXD bool vg_log(double ap, double n, double m, VgLog& o) {
    const unsigned long long ba = double_bits(ap), bn = double_bits(n), bm = double_bits(m), one = 1ull << 52;
    const int ea = (int)(ba >> 52) - 1023, en = (int)(bn >> 52) - 1023, em = (int)(bm >> 52) - 1023;   // (negative: > 1024)
    if (ea < -59 || ea > 58 || en < -6 || en > 3 || em < -20 || em > -1) return false;
    const long long L = log_fixed(((ba & (one - 1)) | one) << 7, ea);
    const long long y = rmul(L, (long long)(((bn & (one - 1)) | one) << (en + 6)));          // n L in Q53
    if (y >= 256ll << 53 || y <= -(256ll << 53)) return false;
    int ne;
    const unsigned long long v = exp_fixed<53>(y, ne);                                       // ap^n
    if (ne > 57) return false;
    const unsigned long long W = ne >= 0 ? v + (1ull << (62 - ne)) : (1ull << 62) + (ne > -63 ? v >> -ne : 0);
    const int z = clz64(W);
    o.l1 = log_fixed((W << z) >> 4, (ne > 0 ? ne : 0) + 1 - z);
    const unsigned long long mm = (bm & (one - 1)) | one;
    o.t = -rmul(o.l1, (long long)(em >= -10 ? mm << (em + 10) : mm >> -(em + 10)));
    o.g = y - (L >> 4);
    return true;
}
// s
FXD double vg_s(const VgLog& o) { return exp_fixed<57>(o.t); }
// the relative conductivity sqrt(s) (1 - s ap^n / ap)^2 and ds/dp / (m n a) =
// s ap^n / (ap (1 + ap^n))
FXD void vg_k(const VgLog& o, double& krw, double& d) {
    const long long q = o.g + (o.t >> 4);
    const double b = 1.0 - exp_fixed<53>(q);
    krw = exp_fixed<57>(o.t >> 1) * b * b;
    d = exp_fixed<53>(q - (o.l1 >> 4));
}

// The normal distribution function about z_k = k/64, |z_k| <= 4: Phi(z_k + d) =
// Phi_k (1 + s), s the Taylor series of degree 8 (remainder 2^-63), its n-th
// coefficient phi_k He_{n-1}(z_k) (-1)^(n-1) / (n! Phi_k) in units of 2^-7n; those
// from the fifth on in 32 bits (all Q62).  erfc held the FP64 pipe for 78
// operations a value, most of the last transform kernel's time.
FX double normal_cdf(double z, const PhiEntry* tab) {
    const unsigned long long bits = double_bits(z), one = 1ull << 52;
    const int e = (int)(bits >> 52 & 0x7FF) - 1023;
    if (e > 1) return 0.5 * erfc(-z / sqrt(2.0));            // |z| >= 4, NaN
    const unsigned long long m = (bits & (one - 1)) | one;
    long long q = e >= -7 ? (long long)(m << (e + 7)) : e >= -60 ? (long long)(m >> -(e + 7)) : 0;   // |z| in Q59
    if (bits >> 63) q = -q;
    const int k = (int)((q + (1ll << 52)) >> 53);
    const long long d = (q - ((long long)k << 53)) << 10;    // 2^7 (z - z_k) in Q62
    const PhiEntry t = tab[k + PHI_SIDE];
    const int d31 = (int)((d - (d >> 62)) >> 31);            // (1 as the largest number below)
    int b = t.b[3];
    b = t.b[2] + (int)(wide(b, d31) >> 31);
    b = t.b[1] + (int)(wide(b, d31) >> 31);
    b = t.b[0] + (int)(wide(b, d31) >> 31);
    long long s = t.c[3] + (wide(b, d31) >> 31);
    s = t.c[2] + rmul(s, d);
    s = t.c[1] + rmul(s, d);
    s = t.c[0] + rmul(s, d);
    s = rmul(s, d);
    unsigned long long v = (unsigned long long)(t.phi + rmul(t.phi, s));
    int n = t.e;
    if (v >> 63) { v >>= 1; ++n; }
    else if (!(v >> 62)) { v <<= 1; --n; }
    return fx_to_double(v, n);
}

// the tables, from the host's long double functions
inline long long to_q(long double v, int bits) { return (long long)llrintl(ldexpl(v, bits)); }
inline cw circle_point(long long k, long long n) {
    const long double t = 2.0L * 3.14159265358979323846264338327950288L * (long double)k / (long double)n;
    return cw{split_w(to_q(cosl(t), 62)), split_w(to_q(sinl(t), 62))};
}
inline void make_phi(PhiEntry& o, int k) {
    const long double z = k / 64.0L, P = 0.5L * erfcl(-z * sqrtl(0.5L));
    const long double l = expl(-0.5L * z * z) / (sqrtl(2.0L * 3.14159265358979323846264338327950288L) * P);
    long double h0 = 1.0L, h1 = z, c = l;                    // He_{n-1}, He_n; l 2^-7n (-1)^(n-1) / n!
    int e;
    o.phi = to_q(frexpl(P, &e), 63);
    o.e = e - 1;
    o.pad = 0;
    for (int n = 1; n <= 8; ++n) {
        c = n == 1 ? l / 128.0L : -c / (128.0L * n);
        if (n <= 4) o.c[n - 1] = to_q(c * h0, 62);
        else o.b[n - 5] = (int)to_q(c * h0, 62);
        const long double h2 = z * h1 - n * h0;
        h0 = h1; h1 = h2;
    }
}
inline void make_norm_tab(NormTab& t) {
    for (int k = -PHI_SIDE; k <= PHI_SIDE; ++k) make_phi(t.phi[k + PHI_SIDE], k);
    for (int i = 0; i < 256; ++i) {
        const int inv = i == 255 ? 2048 : (int)lrint(4096.0 / (1.0 + (i + 0.5) / 256.0));
        t.lg[i] = LogEntry{inv == 2048 ? LN2_57 : to_q(-logl((long double)inv / 4096.0L), 57), inv, 0};
        t.cs[i] = circle_point(i, 256);
    }
}

}  // namespace rich_fx
