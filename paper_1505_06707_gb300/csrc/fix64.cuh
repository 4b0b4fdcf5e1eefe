// Complex128 FFTs in 64-bit fixed point.
//
// GB300 runs 2 FP64 instructions per clock and SM, but 64 32 x 32 -> 64 bit
// multiply-adds (mad.wide) or 64-bit additions (probe/alu_peak.cu: DFMA 1.98,
// mad.wide 62.7, add.s64 63.7 per clock and SM, the two in turn 63.6).  A
// complex product of 64-bit fixed-point numbers takes 12 mad.wide, 0.19 clocks
// of an SM against 2 clocks for the 4 FP64 instructions (0.51 with the halves'
// splitting and carries, fx_mul), and a complex sum and difference 0.06 against
// 2.  So the complex128 FFTs run on integers: a line's samples are X 2^e with
// one exponent e per line and X a 64-bit integer.
//
// Range.  Every operator between two conversions is unitary (FFT passes with
// their power-of-2 shares of 1/N, phase factors), so the Euclidean norm of a
// line is kept, and it bounds every component.  Lines enter with
// norm < FX_NORM = 2^60.8; a radix-16 butterfly, unscaled, grows that to
// 2^62.8 < 2^63 at most, and the products after it, or before the next one,
// take the unitary scaling back (FxPass, fx_center).
//
// Accuracy.  Products round to 1/2 unit in the last place.  With the norm
// between 2^59.6 and 2^60.8 units, k roundings of n complex samples leave
// about 0.3 sqrt(2 n k) units: 2e-16 of the norm for a forward and inverse
// FFT of n = 16384 (k = 14), less for shorter lines; the FP64 passes, whose
// roundings are relative to each sample, leave 2e-16 to 4e-16.
//
// A factor w with |w| <= 1 (up to 1.9 where the comments say so) is stored as
// W = w 2^62 split into signed 32-bit halves, W = h 2^32 + l: int4 (re.h, re.l,
// im.h, im.l), l > -2^31.
#pragma once
#include "device_common.cuh"

namespace soft {

using fx2 = longlong2;

constexpr float FX_NORM2 = 2.1815e17f;        // 2^57.6: FX_NORM^2 in units of 2^32
constexpr float FX_NORM2_LOW = 4.7416e16f;    // 2^55.4: below it one more bit fits

// a b and a b + c, 32 x 32 -> 64 bit (in PTX: the compiler folds a sign
// extension of a high word into a 64-bit shift and then multiplies 64 x 64)
__device__ __forceinline__ long long fx_mw(int a, int b) {
    long long r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ int fx_hi(long long v) {
    int l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(v));
    return h;
}
constexpr long long FX_RND = 0x80000000LL;

// signed halves of v 2^K
template <int K>
__device__ __forceinline__ void fx_halves(long long v, int& h, int& l) {
    v = (long long)((unsigned long long)v << K);
    l = (int)v;
    h = fx_hi(v) + (int)((unsigned)l >> 31);
}

// v w 2^(K-2) (CONJ: v conj(w)).  Range: the middle sum is at most
// (|v| 2^K + |w| 2^62)/sqrt(2) in size (|v|, |w|: moduli of the complex values),
// and must stay below 2^63: |v| 2^K <= 2^62.8 for |w| <= 1.01 (lines with norms
// of FX_NORM in units of 1/4), 2^62.3 for |w| <= 1.43, 2^61.5 for |w| <= 1.9.
// The product of the low halves (below 1/4 unit) is dropped.  The high word of the middle
// sum is added by a multiplication by 1, which needs no sign extension into a
// register pair: 27 instructions, 0.51 clocks of an SM (0.57 with the
// extension and the halves' carry as 64-bit additions), bound by the wide
// multiplies' operand reads.
__device__ __forceinline__ long long fx_addhi(long long m, long long c) { return fx_mad(fx_hi(m), 1, c); }
template <int K, bool CONJ = false>
__device__ __forceinline__ fx2 fx_mul(fx2 v, int4 w) {
    int ah, al, bh, bl;
    fx_halves<K>(v.x, ah, al);
    fx_halves<K>(v.y, bh, bl);
    const long long p = fx_mad(ah, w.y, fx_mad(al, w.x, FX_RND));     // re re
    const long long r = fx_mad(bh, w.y, fx_mad(bl, w.x, FX_RND));     // im re
    const int nz = -w.z;
    fx2 o;
    if constexpr (!CONJ) {
        const long long q = fx_mad(bh, w.w, fx_mw(bl, w.z));          // im im
        const long long m = p - q, n = fx_mad(ah, w.w, fx_mad(al, w.z, r));
        o.x = fx_addhi(m, fx_mad(bh, nz, fx_mw(ah, w.x)));
        o.y = fx_addhi(n, fx_mad(ah, w.z, fx_mw(bh, w.x)));
    } else {
        const long long q = fx_mad(ah, w.w, fx_mw(al, w.z));          // re im
        const long long m = fx_mad(bh, w.w, fx_mad(bl, w.z, p)), n = r - q;
        o.x = fx_addhi(m, fx_mad(bh, w.z, fx_mw(ah, w.x)));
        o.y = fx_addhi(n, fx_mad(ah, nz, fx_mw(bh, w.x)));
    }
    return o;
}

// factor -> sample units 2^62, product of two factors as a factor (to 2^-61)
__device__ __forceinline__ fx2 fx_lift(int4 w) {
    return make_longlong2((long long)w.x * 4294967296LL + w.y, (long long)w.z * 4294967296LL + w.w);
}
template <int K>
__device__ __forceinline__ int4 fx_factor(fx2 v) {     // the factor v 2^K / 2^62
    int4 w;
    fx_halves<K>(v.x, w.x, w.y);
    fx_halves<K>(v.y, w.z, w.w);
    w.y = max(w.y, -0x7fffffff);
    w.w = max(w.w, -0x7fffffff);
    return w;
}
__device__ __forceinline__ int4 fx_mulw(int4 a, int4 b) { return fx_factor<2>(fx_mul<0>(fx_lift(a), b)); }

// a b 2^-63 of signed 64-bit fixed-point numbers with 63 fraction bits
__device__ __forceinline__ long long fx_mulq63(long long a, long long b) { return __mul64hi(a, b) << 1; }
// e^{i ph} as a factor, in integer arithmetic but for the reduction of ph:
// the phase in turns (a product to 106 bits, so that the reduction adds no
// error to ph's own), 1/32-turn sectors from a table, and Taylor series for
// the rest |r| <= pi/32 (the first terms left out are below 2^-67).  The
// library's sincos spends about 70 FP64 instructions, 64 clocks each for a
// warp's scheduler; this spends 9.
static __constant__ long long FX_SECT[9] = {     // cos(pi k/16) 2^62, k = 0 .. 8
    4611686018427387904LL, 4523073764714963030LL, 4260642322793532497LL, 3834476785802888710LL,
    3260954456333195553LL, 2562115475870945497LL, 1764815834521887442LL, 899695310372275547LL, 0LL};
__device__ __forceinline__ long long fx_sect_cos(int k) {      // cos(2 pi k/32), k mod 32
    k &= 31;
    const int q = k >> 3, j = k & 7;
    const long long v = FX_SECT[(q & 1) ? 8 - j : j];
    return (q == 1 || q == 2) ? -v : v;
}
__device__ __forceinline__ int4 fx_cexp(double ph) {
    constexpr double C_HI = 0.15915494309189535, C_LO = -9.839338337591243e-18;     // 1/(2 pi)
    const double th = ph * C_HI;
    const double tl = fma(ph, C_HI, -th) + ph * C_LO;
    const double f = th - rint(th);                                       // exact
    const unsigned long long t = (unsigned long long)((__double2ll_rn(f * 0x1p62) << 2)) +
                                 (unsigned long long)__double2ll_rn(tl * 0x1p64);     // turns 2^-64
    const int k = (int)((t + (1ULL << 58)) >> 59);                        // nearest sector
    const long long d = (long long)(t - ((unsigned long long)k << 59));   // |d| <= 2^58 (1/64 turn)
    // r = 2 pi d/2^64 with 63 fraction bits: d pi = d (3 + 0.14159...)
    const long long r = d * 3 + fx_mulq63(d, 1305961721744163946LL);
    const long long r2 = fx_mulq63(r, r);
    // 1/n! with 63 fraction bits
    constexpr long long c2 = 1LL << 62, c4 = 384307168202282325LL, c6 = 12810238940076078LL, c8 = 228754266787073LL,
                        c10 = 2541714075412LL, s3 = 1537228672809129301LL, s5 = 76861433640456465LL,
                        s7 = 1830034134296583LL, s9 = 25417140754119LL, s11 = 231064915947LL;
    const long long cm = fx_mulq63(r2, c2 - fx_mulq63(r2, c4 - fx_mulq63(r2, c6 - fx_mulq63(r2, c8 - fx_mulq63(r2, c10)))));
    const long long sm = fx_mulq63(r2, s3 - fx_mulq63(r2, s5 - fx_mulq63(r2, s7 - fx_mulq63(r2, s9 - fx_mulq63(r2, s11)))));
    const long long sn = (r - fx_mulq63(r, sm)) >> 1;                     // sin r, units 2^-62
    const long long cs = (1LL << 62) - (cm >> 1);                         // cos r
    const int4 w = fx_factor<0>(make_longlong2(fx_sect_cos(k), fx_sect_cos(k - 8)));
    return fx_factor<2>(fx_mul<0>(make_longlong2(cs, sn), w));
}

// v / 2^S rounded
template <int S>
__device__ __forceinline__ long long fx_shr(long long v) {
    if constexpr (S == 0) return v;
    else return (v + (1LL << (S - 1))) >> S;
}
template <int S>
__device__ __forceinline__ fx2 fx_shr(fx2 v) { return make_longlong2(fx_shr<S>(v.x), fx_shr<S>(v.y)); }
// v 2^k, rounded for k < 0 (|k| < 63)
__device__ __forceinline__ long long fx_scale(long long v, int k) {
    if (k >= 0) return (long long)((unsigned long long)v << k);
    return ((v >> (-k - 1)) + 1) >> 1;
}
__device__ __forceinline__ fx2 fx_scale(fx2 v, int k) { return make_longlong2(fx_scale(v.x, k), fx_scale(v.y, k)); }

// ------------------------------------------------- butterfly rotations
// multiplication by exp(SIGN 2 pi i t16/16) at full scale: u c = u + u (c - 1)
// with the constants cos(pi/8) - 1, sin(pi/8) and 1/sqrt(2) - 1 in units 2^-64
constexpr long long FX_C1 = -1404174782535421627LL, FX_S1 = 7059263338087549767LL, FX_R1 = -5402926248376769404LL;
__host__ __device__ constexpr int fx_ch(long long c) { return (int)((c + FX_RND) >> 32); }
__host__ __device__ constexpr int fx_cl(long long c) { return (int)(c - (long long)fx_ch(c) * 4294967296LL); }

__device__ __forceinline__ long long fx_rsqrt2(long long u) {          // u / sqrt(2)
    int h, l;
    fx_halves<0>(u, h, l);
    const long long m = fx_mad(h, fx_cl(FX_R1), fx_mad(l, fx_ch(FX_R1), FX_RND));
    return fx_addhi(m, fx_mad(h, fx_ch(FX_R1), u));
}
template <int SG>                                                     // SG = +-1: e^{SG i pi/8}
__device__ __forceinline__ fx2 fx_rot8(fx2 a) {
    int xh, xl, yh, yl;
    fx_halves<0>(a.x, xh, xl);
    fx_halves<0>(a.y, yh, yl);
    constexpr int ch = fx_ch(FX_C1), cl = fx_cl(FX_C1), sh = SG * fx_ch(FX_S1), sl = SG * fx_cl(FX_S1);
    const long long m = fx_mad(xh, cl, fx_mad(xl, ch, fx_mad(yh, -sl, fx_mad(yl, -sh, FX_RND))));
    const long long n = fx_mad(yh, cl, fx_mad(yl, ch, fx_mad(xh, sl, fx_mad(xl, sh, FX_RND))));
    return make_longlong2(fx_addhi(m, fx_mad(xh, ch, fx_mad(yh, -sh, a.x))),
                          fx_addhi(n, fx_mad(yh, ch, fx_mad(xh, sh, a.y))));
}
template <int Q>                                                      // multiplication by i^Q
__device__ __forceinline__ fx2 fx_quarter(fx2 a) {
    if constexpr ((Q & 3) == 0) return a;
    else if constexpr ((Q & 3) == 1) return make_longlong2(-a.y, a.x);
    else if constexpr ((Q & 3) == 2) return make_longlong2(-a.x, -a.y);
    else return make_longlong2(a.y, -a.x);
}
template <int R, int SIGN, int t>
__device__ __forceinline__ fx2 fx_twc(fx2 a) {
    constexpr int t16 = ((SIGN * t * 16 / R) % 16 + 16) & 15;
    if constexpr ((t16 & 3) == 0) {
        return fx_quarter<t16 / 4>(a);
    } else if constexpr ((t16 & 3) == 2) {           // (1 + i)/sqrt(2), times i^(t16/4)
        return fx_quarter<t16 / 4>(make_longlong2(fx_rsqrt2(a.x - a.y), fx_rsqrt2(a.x + a.y)));
    } else if constexpr ((t16 & 3) == 1) {
        return fx_quarter<t16 / 4>(fx_rot8<1>(a));
    } else {
        return fx_quarter<t16 / 4 + 1>(fx_rot8<-1>(a));
    }
}

// ------------------------------------------------- conversions
// X as a double, round to nearest: integer instructions only (3.0 per clock
// and SM; the conversion instruction runs on the FP64 pipe at 1.9)
__device__ __forceinline__ double fx_to_double(long long x) {
    const int s = fx_hi(x) >> 31;
    unsigned long long m = (unsigned long long)((x ^ (long long)s) - (long long)s);
    const int lz = __clzll((long long)m);
    m <<= lz & 63;
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1);
    int hi = (int)(r >> 32) + ((1085 - lz) << 20);
    hi = x == 0 ? 0 : hi;
    return __hiloint2double(hi | (s & 0x80000000), (int)r);
}
__device__ __forceinline__ double2 fx_to_double(fx2 v) { return make_double2(fx_to_double(v.x), fx_to_double(v.y)); }

// round(d 2^-e) for a normal or zero d with |d| 2^-e < 2^62 (smaller d round to 0)
__device__ __forceinline__ long long fx_from_double(double d, int e) {
    const int hi = __double2hiint(d);
    const unsigned lo = (unsigned)__double2loint(d);
    const int E = (hi >> 20) & 0x7ff;
    // mantissa with its leading bit at 62, value m 2^(E - 1085)
    const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 42) | ((unsigned long long)lo << 10);
    const int sh = min(1085 + e - E, 64);            // >= 1
    const long long r = (long long)(((m >> (sh - 1)) + 1) >> 1);
    return hi < 0 ? -r : r;
}
__device__ __forceinline__ fx2 fx_from_double(double2 d, int e) {
    return make_longlong2(fx_from_double(d.x, e), fx_from_double(d.y, e));
}
// the larger exponent-and-leading-mantissa word of the two components
__device__ __forceinline__ unsigned fx_mag(double2 d) {
    return max((unsigned)__double2hiint(d.x) & 0x7fffffffu, (unsigned)__double2hiint(d.y) & 0x7fffffffu);
}
// d 2^e, exact unless the result is subnormal (then rounded) or overflows
__device__ __forceinline__ double fx_ldexp(double d, int e) {
    if (e > 1000) { d *= 0x1p1000; e = min(e - 1000, 1000); }
    if (e < -1000) { d *= 0x1p-900; e += 900; if (e < -1000) { d *= 0x1p-900; e = max(e + 900, -1000); } }
    return d * __hiloint2double((e + 1023) << 20, 0);
}
// X 2^e; small: -900 < e < 900 (no subnormal, no overflow)
__device__ __forceinline__ double fx_out(long long x, int e, bool small) {
    const double d = fx_to_double(x);
    if (small) return __hiloint2double(__double2hiint(d) + (x == 0 ? 0 : e << 20), __double2loint(d));
    return fx_ldexp(d, e);
}
// |v|^2 in units of 2^64 (FP32: the norm only steers the scaling)
__device__ __forceinline__ float fx_abs2(fx2 v) {
    const float a = (float)fx_hi(v.x), b = (float)fx_hi(v.y);
    return a * a + b * b;
}
// larger |high word| of the two components (one less for negative ones)
__device__ __forceinline__ unsigned fx_hmag(fx2 v) {
    const int a = fx_hi(v.x), b = fx_hi(v.y);
    return (unsigned)max(a ^ (a >> 31), b ^ (b >> 31));
}
// shift that brings a line with sum of fx_abs2 = t2 below FX_NORM, by as
// little as possible; truncation of the n samples' high words included
__device__ __forceinline__ int fx_norm_shift(float t2, int n) {
    const float s = sqrtf(t2) + sqrtf(2.0f * (float)n);
    const float t = s * s;
    if (t <= FX_NORM2 && t > FX_NORM2_LOW) return 0;
    // t 4^k in (2^55.6, 2^57.6]
    return (int)floorf(0.5f * (57.6f - __log2f(t)) - 1e-4f);
}
}  // namespace soft
