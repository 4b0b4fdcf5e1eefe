// The complex128 resident 1D step: the scheme of soft1d.cuh with the FFTs,
// the phase factors, the strip Crank-Nicolson and the state in 64-bit fixed
// point (fix64.cuh).
//
// A step in FP64 (N = 16384) spent 64 clocks of its SM per point, 87 % of
// them in the FP64 pipe, most of it FFT butterflies.  In fixed point all of it
// runs on the integer pipes, but for plans with the flag `gen` below.
//
// Exponent.  The state is X 2^e.  Each step sums |X|^2 (FP32, of the high
// words) as the rows are written and shifts the state as the next forward
// pass loads it, so that its norm stays in (2^59.6, 2^60.8]; the shift is 0
// in almost every step.  Potential factors enter scaled by 2^-p, p = 0
// (|e^{-iU tau}| <= 1.01, which the products' range allows) or 1 (<= 2).  A
// plan with a larger or non-finite factor, or none above 1/8 (a user potential
// with a large gain or a loss at every point; fx_gen_factors in plan.cu), or
// with strip multipliers above 1 (backward steps) has the flag `gen` in its
// tables: its factors and strip solve are applied in FP64 and the state is
// converted anew in every step, so that a sample keeps its relative precision
// however the factors spread.
//
// Strip solve (strip_cn_fx): every product rounds to half a unit and the
// multipliers are at most 1, so the two sweeps leave at most 2^lg units where
// they grow the rows by 2^lg; a block shifted by lg + 2 bits first (`coarse`,
// a packet inside the strip) loses those bits of its samples' 59.
//
// Code size.  A step runs once through straight-line code, and with 4 to 16
// warps per SM the instruction fetch bounds it when that code leaves the
// instruction cache: fully unrolled and templated per pass (225 to 340 KB), the
// step of N = 1024 took 46k clocks at 10 or more clocks per instruction.  So
// the passes of one radix are one runtime loop, the potential factors and the
// strip solve are loops over the state in shared memory, and rare paths are
// out of line.
// Included by soft1d.cuh (after the pass geometry it uses).
#pragma once
#include "fix64.cuh"

namespace soft {

// Twiddle tables (factor format): passes of a stride of at most FXFULL_MAXS
// hold every W^{M off} in shared memory; a radix-16 first pass of a larger
// stride (N >= 4096) holds M = 1 .. 8 there and reads the other seven from
// global memory, where they follow the table (N = 16384's full table would
// take 245 KB; N = 4096 keeps two CTAs per SM: 1216 instances x 16 steps
// 4.29 -> 3.24 ms).  The last pass, of stride 1, has none.
template <int LOGN, int LOGRM, int P>
struct FxGeom {
    using G = PassGeom<LOGN, LOGRM, P>;
    static constexpr bool FULL = G::S > 1 && G::S <= FXFULL_MAXS;
    static constexpr int ROWS = G::S == 1 ? 0 : (FULL || G::LOGR < 4) ? (1 << G::LOGR) - 1 : 8;
    static constexpr int TOFF = FxGeom<LOGN, LOGRM, P - 1>::TOFF +
                                FxGeom<LOGN, LOGRM, P - 1>::ROWS * PassGeom<LOGN, LOGRM, P - 1>::S;
};
template <int LOGN, int LOGRM>
struct FxGeom<LOGN, LOGRM, -1> { static constexpr bool FULL = false; static constexpr int ROWS = 0, TOFF = 0; };
template <int LOGN, int LOGRM>
struct TwCountT<TwFix, LOGN, LOGRM> {
    static constexpr int NP = LOGN / LOGRM + ((LOGN % LOGRM) ? 1 : 0);
    static constexpr int value = FxGeom<LOGN, LOGRM, NP - 1>::TOFF +
                                 FxGeom<LOGN, LOGRM, NP - 1>::ROWS * PassGeom<LOGN, LOGRM, NP - 1>::S;
};

// Scaling.  Every pass of radix 2^r is made unitary: its twiddles carry
// 2^(-r/2) as the product's 2^(K-2) and, for odd r, a factor sqrt(2) in the
// table (moduli up to 1.42 fit the halves).  Forward passes multiply after
// the butterfly, inverse passes before it, so an inverse pass leaves its
// outputs 2^(r/2) too large and the next one, or the potential factors, take
// that in their product: no separate shift.  An element without a twiddle is
// scaled by fx_unit.
template <int r> struct FxPass {
    static constexpr int K = r >= 3 ? 0 : 1;              // 2^(K-2) sqrt(2)^(r odd) = 2^(-r/2)
};
template <int r>
__device__ __forceinline__ long long fx_unit(long long v) {      // v 2^(-r/2)
    if constexpr (r & 1) v = fx_rsqrt2(v);
    return fx_shr<r / 2>(v);
}
template <int r>
__device__ __forceinline__ fx2 fx_unit(fx2 v) { return make_longlong2(fx_unit<r>(v.x), fx_unit<r>(v.y)); }

// Addresses of a butterfly: element m at sb ^ x(m), x(m) = swz(m s) =
// XOR of c[j] = swz(2^j s) over the set bits j of m.
template <int LOGR>
struct FxAddr {
    int sb, c[LOGR];
    __device__ __forceinline__ FxAddr(int base, int logs) : sb(swz<fx2>(base)) {
#pragma unroll
        for (int j = 0; j < LOGR; ++j) c[j] = swz<fx2>(1 << (logs + j));
    }
    __device__ __forceinline__ int operator()(int m) const {
        int x = sb;
#pragma unroll
        for (int j = 0; j < LOGR; ++j)
            if ((m >> j) & 1) x ^= c[j];
        return x;
    }
};

template <int LOGN, int LOGE, int LOGRM>
struct Fx1D {
    using K = Cfg1D<double, LOGN, LOGE, LOGRM>;
    static constexpr int N = K::N, T = K::T, E = K::E, NPASS = K::NPASS;
    static constexpr int RR = 1 << LOGRM;
    static_assert(E % RR == 0, "whole butterflies per thread");
    // the first pass's twiddles above 8 are read from ext (stride > FXFULL_MAXS)
    static constexpr bool PART = LOGRM == 4 && (N >> LOGRM) > FXFULL_MAXS;
    static constexpr int TWN = TwCountT<TwFix, LOGN, LOGRM>::value;

    __device__ __forceinline__ static int4 tw(const int4* t, const int4* __restrict__ ext, int s, int m, bool part) {
        if (PART && m > 8 && part) return __ldg(&ext[(m - 9) * s]);
        return t[(m - 1) * s];
    }
    // W: the table in shared memory, Wg in global memory (used by PART only)
    template <class B>
    __device__ __forceinline__ static void fwd_all(fx2* S, const int4* W, const int4* __restrict__ Wg, int tid, B bar) {
        const int4* Wp = W;
#pragma unroll 1
        for (int P = 0; P < NPASS - 1; ++P) {
            const int logs = LOGN - LOGRM * (P + 1), s = 1 << logs;
            const bool part = PART && P == 0;
#pragma unroll 1
            for (int u = 0; u < E / RR; ++u) {
                const int b = tid + u * T, off = b & (s - 1);
                const FxAddr<LOGRM> at(((b >> logs) << (logs + LOGRM)) + off, logs);
                fx2 v[RR];
#pragma unroll
                for (int j = 0; j < RR; ++j) v[j] = S[at(j)];
                dft_reg<fx2, RR, -1>(v);
                S[at.sb] = fx_unit<LOGRM>(v[0]);
                const int4* t = Wp + off;
#pragma unroll
                for (int m = 1; m < RR; ++m)
                    S[at(m)] = fx_mul<FxPass<LOGRM>::K>(v[bitrev_c(m, LOGRM)], tw(t, Wg + TWN + off, s, m, part));
            }
            Wp += (part ? 8 : RR - 1) << logs;
            bar.sync();
        }
    }
    template <class B>
    __device__ __forceinline__ static void inv_all(fx2* S, const int4* W, const int4* __restrict__ Wg, int tid, B bar) {
        const int4* Wp = W + TWN;
#pragma unroll 1
        for (int P = NPASS - 2; P >= 0; --P) {
            const int logs = LOGN - LOGRM * (P + 1), s = 1 << logs;
            const bool part = PART && P == 0;
            Wp -= (part ? 8 : RR - 1) << logs;
#pragma unroll 1
            for (int u = 0; u < E / RR; ++u) {
                const int b = tid + u * T, off = b & (s - 1);
                const FxAddr<LOGRM> at(((b >> logs) << (logs + LOGRM)) + off, logs);
                const int4* t = Wp + off;
                fx2 v[RR];
                v[0] = fx_unit<LOGRM>(S[at.sb]);
#pragma unroll
                for (int m = 1; m < RR; ++m) v[m] = fx_mul<FxPass<LOGRM>::K, true>(S[at(m)], tw(t, Wg + TWN + off, s, m, part));
                dft_reg<fx2, RR, +1>(v);
#pragma unroll
                for (int m = 0; m < RR; ++m) S[at(m)] = v[bitrev_c(m, LOGRM)];
            }
            bar.sync();
        }
    }
    // last forward pass, k-space factor, first inverse pass (soft1d.cuh,
    // kcenter).  SURF: acc[r] += (spectrum x weight row r)/4
    template <bool SURF>
    __device__ __forceinline__ static void center(fx2* S, const int4* __restrict__ tab, int tid,
                                                  const int4* __restrict__ sw, fx2* acc) {
        using Gp = PassGeom<LOGN, LOGRM, NPASS - 1>;
        constexpr int LOGR = Gp::LOGR, R = 1 << LOGR, NU = E / R;
        constexpr FxCenter FC = fx_center(LOGR, LOGRM);
        static_assert(Gp::S == 1 && FC.K >= 0, "the last pass has stride 1");
        constexpr bool PF = R <= 4 && NU > 1;        // next butterfly's factors in flight
        int4 tn[PF ? R : 1];
        if constexpr (PF) {
#pragma unroll
            for (int m = 0; m < R; ++m) tn[m] = __ldg(&tab[m * (N / R) + tid]);
        }
#pragma unroll 1
        for (int u = 0; u < NU; ++u) {
            int4 tc[R];
            if constexpr (PF) {
#pragma unroll
                for (int m = 0; m < R; ++m) tc[m] = tn[m];
                if (u + 1 < NU) {
#pragma unroll
                    for (int m = 0; m < R; ++m) tn[m] = __ldg(&tab[m * (N / R) + tid + (u + 1) * T]);
                }
            } else if constexpr (R <= 8) {
#pragma unroll
                for (int m = 0; m < R; ++m) tc[m] = __ldg(&tab[m * (N / R) + tid + u * T]);
            }
            const int sb = swz<fx2>((tid + u * T) * R);
            fx2 v[R], w[R];
#pragma unroll
            for (int j = 0; j < R; ++j) v[j] = S[sb ^ swz<fx2>(j)];
            dft_reg<fx2, R, -1>(v);
            if constexpr (SURF) {
#pragma unroll
                for (int m = 0; m < R; ++m) {
                    const int q = m * (N / R) + tid + u * T;
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        acc[r] = cadd(acc[r], fx_mul<0>(v[bitrev_c(m, LOGR)], __ldg(&sw[r * N + q])));
                }
            }
#pragma unroll
            for (int m = 0; m < R; ++m) {
                if constexpr (R > 8) tc[m] = __ldg(&tab[m * (N / R) + tid + u * T]);
                w[m] = fx_mul<FC.K>(v[bitrev_c(m, LOGR)], tc[m]);
            }
            dft_reg<fx2, R, +1>(w);
#pragma unroll
            for (int m = 0; m < R; ++m) {
                const fx2 o = w[bitrev_c(m, LOGR)];
                S[sb ^ swz<fx2>(m)] = make_longlong2(o.x << FC.cs, o.y << FC.cs);
            }
        }
    }
};

// ---- field factors exp(-i alpha x), alpha = tau E(t + tau/2)/2, at: [j] j T h
// and [E + j] their squares, j < E; [2E], [2E + 1] the clamped values beyond
// +R0, -R0; [2E + 2 + k] and [2E + 10 + k], k < 8, the strip rows just inside
// -R0 and +R0; [2E + 18 + a] x0 + 32 a h and [2E + 34 + b] b h: the factor at
// grid index tid + j T, tid = 32 a + b, is [2E + 18 + a] [2E + 34 + b] [j]
template <int LOGN, int LOGE, int LOGRM>
__device__ __noinline__ void field_setup_fx(int4* fr, double al, const Inst1D& I, int tid) {
    using K = Cfg1D<double, LOGN, LOGE, LOGRM>;
    constexpr int E = K::E, NA = (K::T + 31) / 32;
    const double h = I.h;
    for (int i = tid; i < E + 17 + NA + 32; i += K::T) {
        double x;
        int at;
        if (i < E) { x = (double)(i * K::T) * h; at = i; }
        else if (i == E) { x = I.R0; at = 2 * E; }
        else if (i < E + 17) {
            const int k = i - E - 1;
            x = I.x0 + (double)(k < 8 ? I.iL + k : I.iR - 16 + k) * h;
            at = 2 * E + 2 + k;
        } else if (i < E + 17 + NA) { x = I.x0 + (double)(32 * (i - E - 17)) * h; at = 2 * E + 18 + i - E - 17; }
        else { x = (double)(i - E - 17 - NA) * h; at = 2 * E + 34 + i - E - 17 - NA; }
        const int4 w = fx_cexp(-al * x);
        fr[at] = w;
        if (i < E) fr[E + i] = fx_mulw(w, w);
        if (i == E) fr[2 * E + 1] = make_int4(w.x, w.y, -w.z, -w.w);
    }
}
static __device__ __noinline__ int4 field_direct_fx(double al, double x0, double h, int n) {
    return fx_cexp(-al * (x0 + (double)n * h));
}
// half field factor on strip row n: clamped beyond +-R0
template <int E>
__device__ __forceinline__ int4 strip_field_fx(const int4* fr, double al, const Inst1D& I, int n) {
    const int a = n - I.iL, b = n - I.iR;
    const int at = b >= 0 ? 2 * E : a < 0 ? 2 * E + 1 : a < 8 ? 2 * E + 2 + a : b >= -8 ? 2 * E + 18 + b : -1;
    if (at < 0) return field_direct_fx(al, I.x0, I.h, n);
    return fr[at];
}

// potential table: N factors scaled by 2^-p, then the entry (p, gen, 0, 0),
// then (gen only) the N factors as double2
template <int LOGN>
struct FxV {
    const int4* t;
    int p;
    bool gen;
    __device__ __forceinline__ explicit FxV(const void* tab, int n) : t(reinterpret_cast<const int4*>(tab)) {
        const int4 m = __ldg(&t[n]);
        p = m.x;
        gen = m.y != 0;
    }
    __device__ __forceinline__ const double2* d(int n) const { return reinterpret_cast<const double2*>(t + n + 1); }
};

__device__ __forceinline__ fx2 fx_bits(double2 d) {
    return make_longlong2(__double_as_longlong(d.x), __double_as_longlong(d.y));
}
__device__ __forceinline__ double2 fx_asd(fx2 v) {
    return make_double2(__longlong_as_double(v.x), __longlong_as_double(v.y));
}

// The potential factor of the next step on the thread's own rows, after the
// last inverse pass: e^{-iU tau} off the strip block, e^{-iU tau/2} on it (the
// table also takes the pass's scaling).  t2: the sum of fx_abs2 over the rows
// off the block; mr: the largest |high word| on the block.
template <int LOGN, int LOGE, int LOGRM>
__device__ __forceinline__ void potential_fx(fx2* S, const FxV<LOGN>& TV, const int4* fr, const Inst1D& I, int tid,
                                             float& t2, unsigned& mr) {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    constexpr int N = F::N, E = F::E, T = F::T, Q = E < 4 ? E : 4;
    const int nb = I.nb, blk0 = I.blk0, iL = I.iL, iR = I.iR;
    const bool fld = I.has_field;
    t2 = 0.0f;
    mr = 0;
    int4 ft = make_int4(0, 0, 0, 0), ft2 = ft;
    if (fld) {
        ft = fx_mulw(fr[2 * E + 18 + (tid >> 5)], fr[2 * E + 34 + (tid & 31)]);
        ft2 = fx_mulw(ft, ft);
    }
#pragma unroll 1
    for (int j0 = 0; j0 < E; j0 += Q) {
        int4 tv[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) tv[q] = __ldg(&TV.t[tid + (j0 + q) * T]);
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int n = tid + (j0 + q) * T;
            const bool inb = ((n - blk0) & (N - 1)) < nb;
            fx2& r = S[swz<fx2>(n)];
            fx2 x = fx_mul<FxPass<LOGRM>::K>(r, tv[q]);
            if (fld) {
                int4 f = fx_mulw(inb ? ft : ft2, fr[j0 + q + (inb ? 0 : E)]);
                if (inb && (n >= iR || n < iL)) f = fr[2 * E + (n < iL)];
                x = fx_mul<2>(x, f);
            }
            r = x;
            if (inb) mr = max(mr, fx_hmag(x));
            else t2 += fx_abs2(x);
        }
    }
}
// gen: the same in FP64, rows left as doubles in units 2^e
template <int LOGN, int LOGE, int LOGRM>
__device__ __noinline__ void potential_gen(fx2* S, const double2* __restrict__ tvd, const int4* fr, const Inst1D& I,
                                           int tid) {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    constexpr int N = F::N, E = F::E, T = F::T;
    int4 ft = make_int4(0, 0, 0, 0), ft2 = ft;
    if (I.has_field) {
        ft = fx_mulw(fr[2 * E + 18 + (tid >> 5)], fr[2 * E + 34 + (tid & 31)]);
        ft2 = fx_mulw(ft, ft);
    }
#pragma unroll 1
    for (int j = 0; j < E; ++j) {
        const int n = tid + j * T;
        const bool inb = ((n - I.blk0) & (N - 1)) < I.nb;
        fx2& r = S[swz<fx2>(n)];
        fx2 x = fx_unit<LOGRM>(r);
        if (I.has_field) {
            int4 f = fx_mulw(inb ? ft : ft2, fr[j + (inb ? 0 : E)]);
            if (inb && (n >= I.iR || n < I.iL)) f = fr[2 * E + (n < I.iL)];
            x = fx_mul<2>(x, f);
        }
        r = fx_bits(cmul(fx_to_double(x), __ldg(&tvd[n])));
    }
}
// the thread's own rows times 2^k (rows of the strip block) and 2^(k - kx)
template <int LOGN, int LOGE, int LOGRM>
__device__ __noinline__ void rescale_fx(fx2* S, int k, int kx, int nb, int blk0, int tid) {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    const int ko = max(k - kx, -62);
#pragma unroll 1
    for (int j = 0; j < F::E; ++j) {
        const int n = tid + j * F::T;
        fx2& r = S[swz<fx2>(n)];
        r = fx_scale(r, ((n - blk0) & (F::N - 1)) < nb ? k : ko);
    }
}

// largest value over the group's threads (red: one word per warp, free
// before the call; a barrier must follow before its next use)
template <int T, class B>
__device__ __forceinline__ unsigned fx_group_max(unsigned v, unsigned* red, int tid, B bar) {
    v = __reduce_max_sync(0xffffffffu, v);
    if ((tid & 31) == 0) red[tid >> 5] = v;
    bar.sync();
    unsigned m = red[0];
#pragma unroll
    for (int w = 1; w < T / 32; ++w) m = max(m, red[w]);
    return m;
}

// The state as doubles in units 2^e -> fixed point: the largest component
// between 2^59 and 2^60, e changed to match (not for zeros).  Returns the
// thread's sum of fx_abs2; bad: a non-finite sample.
template <int LOGN, int LOGE, int LOGRM, class B>
__device__ __noinline__ float fx_normalise(fx2* S, int& e, unsigned* red, int tid, B bar, bool& bad) {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    constexpr int E = F::E, T = F::T;
    unsigned m = 0;
#pragma unroll 1
    for (int j = 0; j < E; ++j) m = max(m, fx_mag(fx_asd(S[swz<fx2>(tid + j * T)])));
    m = fx_group_max<T>(m, red, tid, bar);
    bool zero = false;
    int off = 0;
    if (m < (128u << 20)) {                       // tiny (or zero): scale up first
        unsigned q = 0;
#pragma unroll 1
        for (int j = 0; j < E; ++j) {
            fx2& r = S[swz<fx2>(tid + j * T)];
            const double2 d = cscale(fx_asd(r), 0x1p800);
            r = fx_bits(d);
            q = max(q, fx_mag(d));
        }
        off = -800;
        bar.sync();
        m = fx_group_max<T>(q, red, tid, bar);
        zero = m < (128u << 20);
        if (zero) m = 1023u << 20;
    }
    bad = (m >> 20) == 0x7ff;
    const int ed = (int)(m >> 20) - 1022 - 60;
    float t2 = 0.0f;
#pragma unroll 1
    for (int j = 0; j < E; ++j) {
        fx2& r = S[swz<fx2>(tid + j * T)];
        const fx2 v = fx_from_double(fx_asd(r), ed);
        r = v;
        t2 += fx_abs2(v);
    }
    if (!zero) e += ed + off;
    return t2;
}

// Strip Crank-Nicolson tables of complex128 plans (host: plan.cu,
// strip_tables_fx), T threads of ch rows: entry 0 is the header (lg, rounds of
// the forward and backward scans, spans), then factors in chunk order as in
// strip_cn: mf of rows t ch + c, c <= ch, at c T + t, and g; then for the
// forward and for the backward scan the products [5][T] of the 2^r chunk
// totals that end (start) at t, the exclusive product of t's warp [T] and the
// warp totals [T/32]; last (gen) mf and g as double2.
template <int T>
struct FxCn {
    const int4* m;          // mf
    const int4* g;
    const int4* scan[2];    // forward, backward
    int lg, rounds[2], span[2];
    const double2* cd;      // mf, g in FP64
    __device__ __forceinline__ FxCn(const void* cn, int nb) {
        const int4* p = reinterpret_cast<const int4*>(cn);
        lg = 0; rounds[0] = rounds[1] = span[0] = span[1] = 0;
        if (nb <= 0) return;
        const int ch = (nb + T - 1) / T;
        const int4 h = __ldg(p);
        lg = h.x; rounds[0] = h.y; rounds[1] = h.z; span[0] = h.w & 0xffff; span[1] = h.w >> 16;
        m = p + 1;
        g = m + (ch + 1) * T;
        scan[0] = g + ch * T;
        scan[1] = scan[0] + 6 * T + T / 32;
        cd = reinterpret_cast<const double2*>(scan[1] + 6 * T + T / 32);
    }
};

// carry that enters this thread's chunk: the chunks' constant parts Y under
// the affine maps whose products the tables hold.  scratch: T/32 values.
template <int T, bool REV, class B>
__device__ __forceinline__ fx2 fx_carry(fx2 Y, const int4* __restrict__ tab, int rounds, int span, fx2* scratch,
                                        int tid, B bar) {
    const int lane = tid & 31, warp = tid >> 5;
    auto shift = [&](fx2 v, int d) {
        return REV ? make_longlong2(__shfl_down_sync(0xffffffffu, v.x, d), __shfl_down_sync(0xffffffffu, v.y, d))
                   : make_longlong2(__shfl_up_sync(0xffffffffu, v.x, d), __shfl_up_sync(0xffffffffu, v.y, d));
    };
#pragma unroll
    for (int r = 0; r < 5; ++r) {
        if (r < rounds) {
            const fx2 o = shift(Y, 1 << r);
            const bool has = REV ? lane + (1 << r) < 32 : lane >= (1 << r);
            if (has) Y = cadd(Y, fx_mul<2>(o, __ldg(&tab[r * T + tid])));
        }
    }
    fx2 ex = shift(Y, 1);
    if (lane == (REV ? 31 : 0)) ex = make_longlong2(0, 0);
    if constexpr (T > 32) {
        constexpr int NW = T / 32;
        if (lane == (REV ? 0 : 31)) scratch[warp] = Y;
        bar.sync();
        if (REV ? warp + 1 < NW : warp > 0) {
            fx2 c = make_longlong2(0, 0);
            if constexpr (!REV) {
#pragma unroll 1
                for (int w = max(0, warp - span); w < warp; ++w)
                    c = cadd(fx_mul<2>(c, __ldg(&tab[6 * T + w])), scratch[w]);
            } else {
#pragma unroll 1
                for (int w = min(NW - 1, warp + span); w > warp; --w)
                    c = cadd(fx_mul<2>(c, __ldg(&tab[6 * T + w])), scratch[w]);
            }
            ex = cadd(ex, fx_mul<2>(c, __ldg(&tab[5 * T + tid])));
        }
    }
    return ex;
}

// Strip Crank-Nicolson (strip_cn in soft1d.cuh) in fixed point, followed by
// post(v, c, n) on row c of the thread, grid index n (|v| < 2^60.5): the second
// half potential and field factor.  Every multiplier and chunk product
// has modulus <= 1 and the sweeps grow the rows by at most 2^lg (host check;
// other plans take strip_cn_gen), so rows below 2^(59 - lg) cannot overflow;
// coarse: rows beyond that (a packet inside the strip) are shifted right by
// lg + 2 first.  Each sweep runs twice, with carry 0 for the scan and with the
// carry: the FP64 form's 46 FP64 instructions per row and 80 per scan (64
// clocks each for a warp's scheduler) become 8 complex products of 12 wide
// multiplies per row and 6 per scan.  The forward sweep leaves y in place of
// the rows r; r_c = y_c - mf_c y_{c-1}, the same integer product, returns them
// exactly.  kx: the block is left in units 2^kx times as large; returns the
// thread's sum of fx_abs2 in those units.
template <int LOGN, int LOGE, int LOGRM, class B, class Post>
__device__ __forceinline__ float strip_cn_fx(fx2* S, const FxCn<Fx1D<LOGN, LOGE, LOGRM>::T>& cn, int nb, int blk0,
                                             int tid, fx2* scan, B bar, bool coarse, int& kx, Post post) {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    constexpr int N = F::N, T = F::T;
    constexpr int U = 2;
    const int ch = (nb + T - 1) / T;             // host guarantees ch <= CMAX
    const int i0 = tid * ch;
    const int nv = max(0, min(ch, nb - i0));     // rows of this thread
    const int sh = coarse ? cn.lg + 2 : 0;
    const int4* __restrict__ cm = cn.m + tid;
    const int4* __restrict__ cg = cn.g + tid;
    auto row = [&](int c) -> fx2& { return S[swz<fx2>((blk0 + i0 + c) & (N - 1))]; };
    if (sh) {
#pragma unroll 1
        for (int c = 0; c < nv; ++c) row(c) = fx_scale(row(c), -sh);
    }
    fx2 l = make_longlong2(0, 0);
#pragma unroll U
    for (int c = 0; c < nv; ++c) l = cadd(fx_mul<2>(l, __ldg(&cm[c * T])), row(c));
    const fx2 c0 = fx_carry<T, false>(l, cn.scan[0], cn.rounds[0], cn.span[0], scan, tid, bar);
    l = c0;
#pragma unroll U
    for (int c = 0; c < nv; ++c) {
        l = cadd(fx_mul<2>(l, __ldg(&cm[c * T])), row(c));
        row(c) = l;
    }
    l = make_longlong2(0, 0);
#pragma unroll U
    for (int c = nv - 1; c >= 0; --c)
        l = cadd(fx_mul<2>(l, __ldg(&cm[(c + 1) * T])), fx_mul<2>(row(c), __ldg(&cg[c * T])));
    l = fx_carry<T, true>(l, cn.scan[1], cn.rounds[1], cn.span[1], scan + 32, tid, bar);
    unsigned mv = 0;
    int4 mu = nv > 0 ? __ldg(&cm[nv * T]) : make_int4(0, 0, 0, 0);
    fx2 y = nv > 0 ? row(nv - 1) : l;
#pragma unroll U
    for (int c = nv - 1; c >= 0; --c) {
        l = cadd(fx_mul<2>(l, mu), fx_mul<2>(y, __ldg(&cg[c * T])));
        mu = __ldg(&cm[c * T]);
        const fx2 yp = c > 0 ? row(c - 1) : c0;
        const fx2 v = csub(cadd(l, l), csub(y, fx_mul<2>(yp, mu)));
        row(c) = v;
        mv = max(mv, fx_hmag(v));
        y = yp;
    }
    const bool half = bar.any(mv >= (1u << 28));
    float t2 = 0.0f;
#pragma unroll U
    for (int c = 0; c < nv; ++c) {
        fx2& r = row(c);
        const fx2 v = post(half ? fx_shr<1>(r) : r, c, (blk0 + i0 + c) & (N - 1));
        r = v;
        t2 += fx_abs2(v);
    }
    kx = sh + (half ? 1 : 0);
    return t2;
}

// The same on rows held as doubles, in FP64 (the chunk products formed in the kernel): plans with the
// `gen` flag.  cn: mf and g in chunk order.
template <int LOGN, int LOGE, int LOGRM, class B, class Post>
__device__ __forceinline__ void strip_cn_gen(fx2* S, const double2* __restrict__ cn, int nb, int blk0, int tid,
                                             double2* scan, B bar, Post post) {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    using C = double2;
    constexpr int N = F::N, T = F::T, CMAX = F::K::CMAX;
    const int ch = (nb + T - 1) / T, P1 = (ch + 1) * T, i0 = tid * ch;
    const int nv = min(ch, nb - i0);
    auto row = [&](int c) -> fx2& { return S[swz<fx2>((blk0 + i0 + c) & (N - 1))]; };
    C y[CMAX];
    C Mp = cmk<C>(1, 0), yl = cmk<C>(0, 0);
    for (int c = 0; c < nv; ++c) {
        const C m = __ldg(&cn[c * T + tid]);
        yl = cfma(m, yl, fx_asd(row(c)));
        Mp = cmul(m, Mp);
    }
    yl = affine_carry<C, T, false>(Mp, yl, scan, tid, bar);
#pragma unroll
    for (int c = 0; c < CMAX; ++c)
        if (c < nv) {
            yl = cfma(__ldg(&cn[c * T + tid]), yl, fx_asd(row(c)));
            y[c] = cmul(__ldg(&cn[P1 + c * T + tid]), yl);
        }
    Mp = cmk<C>(1, 0);
    yl = cmk<C>(0, 0);
#pragma unroll
    for (int c = CMAX - 1; c >= 0; --c)
        if (c < nv) {
            const C m = __ldg(&cn[(c + 1) * T + tid]);
            yl = cfma(m, yl, y[c]);
            Mp = cmul(m, Mp);
        }
    yl = affine_carry<C, T, true>(Mp, yl, scan, tid, bar);
#pragma unroll
    for (int c = CMAX - 1; c >= 0; --c)
        if (c < nv) {
            yl = cfma(__ldg(&cn[(c + 1) * T + tid]), yl, y[c]);
            fx2& r = row(c);
            const C rc = fx_asd(r);
            r = fx_bits(post(cmk<C>(2 * yl.x - rc.x, 2 * yl.y - rc.y), c, (blk0 + i0 + c) & (N - 1)));
        }
}
// with the second half potential and field factor of the 1D step
template <int LOGN, int LOGE, int LOGRM, class B>
__device__ __noinline__ void strip_gen_1d(fx2* S, const double2* __restrict__ cn, const double2* __restrict__ tvs,
                                          const int4* fr, double al, const Inst1D& I, int tid, double2* scan, B bar) {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    strip_cn_gen<LOGN, LOGE, LOGRM>(S, cn, I.nb, I.blk0, tid, scan, bar, [&](double2 v, int c, int n) {
        v = cmul(v, __ldg(&tvs[c * F::T + tid]));
        if (I.has_field) v = cmul(v, cscale(fx_to_double(fx_lift(strip_field_fx<F::E>(fr, al, I, n))), 0x1p-62));
        return v;
    });
}

// Sum of the four accumulators over the group, times 2^e scale[r]; thread
// r < 4 writes row r.  The warp sums are exact: 64-bit integers, eight values
// halved at each of the first three exchanges.
template <int T, class B>
__device__ __forceinline__ void surf_reduce_fx(fx2 (&acc)[4], double2* scratch, int tid, B bar,
                                               const double* __restrict__ scale, int e, double2* __restrict__ out) {
    static_assert(T / 32 <= 16, "scratch of 64 complex");
    long long a[8];
#pragma unroll
    for (int r = 0; r < 4; ++r) { a[2 * r] = fx_shr<3>(acc[r].x); a[2 * r + 1] = fx_shr<3>(acc[r].y); }
#pragma unroll
    for (int h = 4; h > 0; h >>= 1) {
        const bool up = (tid & (4 * h)) != 0;      // lanes with the bit keep the upper half
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const long long send = up ? a[i] : a[i + h], keep = up ? a[i + h] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * h);
        }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    double* sc = reinterpret_cast<double*>(scratch);
    if ((tid & 3) == 0) sc[8 * (tid >> 5) + ((tid & 31) >> 2)] = fx_to_double(a[0]);
    bar.sync();
    if (tid < 4) {
        double2 t = make_double2(0, 0);
        for (int w = 0; w < (T + 31) / 32; ++w) t = cadd(t, scratch[4 * w + tid]);
        const double s = __ldg(&scale[tid]);
        out[tid] = make_double2(fx_ldexp(t.x * s, e + 3), fx_ldexp(t.y * s, e + 3));
    }
}

// soft1d_run for complex128.  SURF: sw holds eight weight rows in factor
// format followed by their eight scales (double).
template <int LOGN, int LOGE, int LOGRM, class B, bool SURF>
__device__ __forceinline__ void soft1d_run_fx(const Inst1D& I, void* __restrict__ psi_base, int64_t nsteps,
                                              const double* __restrict__ ftab_base, int64_t ftab_stride,
                                              int* __restrict__ status, fx2* Ss, double2* scan, const int4* Ws,
                                              int tid, B bar, const void* __restrict__ sw_v,
                                              double2* __restrict__ samples) {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    using K = typename F::K;
    constexpr int N = F::N, T = F::T, E = F::E, NW = K::NW;
    static_assert(K::NPASS >= 2, "at least two FFT passes");
    int4* fr = reinterpret_cast<int4*>(scan + 64);                   // 2 E + FX_FR factors
    float* part = reinterpret_cast<float*>(fr + 2 * E + FX_FR);          // one per warp
    unsigned* red = reinterpret_cast<unsigned*>(part + 16);          // one per warp
    fx2* __restrict__ g_psi = reinterpret_cast<fx2*>(psi_base) + I.off;
    fx2* S = K::GM ? g_psi : Ss;
    const int nb = I.nb, blk0 = I.blk0;
    const int4* __restrict__ Wg = reinterpret_cast<const int4*>(I.W);
    if (nsteps <= 0) return;
    const FxV<LOGN> TV(I.TV, N), TVs(nb > 0 ? I.TVs : I.TV, nb > 0 ? ((nb + T - 1) / T) * T : N);

    if constexpr (K::GM) {            // the buffer itself, permuted into the swizzled order
        for (int j = 0; j < E; ++j) {
            const int n = tid + j * T, p = swz<fx2>(n);
            if (n < p) { const fx2 a = S[n]; S[n] = S[p]; S[p] = a; }
        }
    } else {
#pragma unroll
        for (int j = 0; j < E; ++j) S[swz<fx2>(tid + j * T)] = g_psi[tid + j * T];
    }
    bar.sync();
    const double* __restrict__ ftab = I.has_field ? ftab_base + (int64_t)I.fcls * ftab_stride : nullptr;

    const FxCn<T> cn(I.cn, nb);
    const unsigned thr = 1u << (27 - cn.lg);     // rows of the block that need the coarse strip solve

    int e = 0;
    bool bad = false, coarse = false;
    double al = 0;
    float t2 = fx_normalise<LOGN, LOGE, LOGRM>(S, e, red, tid, bar, bad);
    int64_t step = -1;
    for (; step < nsteps && !bad; ++step) {
        int kx = 0;
        // ---- Crank-Nicolson on the strip block, then the second e^{-iU tau/2}
        if (step >= 0) {
            if (TV.gen) {
                if (nb > 0) {
                    strip_gen_1d<LOGN, LOGE, LOGRM, B>(S, cn.cd, TVs.d(((nb + T - 1) / T) * T), fr, al, I, tid, scan,
                                                       bar);
                    bar.sync();
                }
                t2 = fx_normalise<LOGN, LOGE, LOGRM>(S, e, red, tid, bar, bad);
                if (bad) break;
            } else {
                e += TV.p;
                if (nb > 0) {
                    const float ts = strip_cn_fx<LOGN, LOGE, LOGRM>(
                        S, cn, nb, blk0, tid, reinterpret_cast<fx2*>(scan), bar, coarse, kx,
                        [&](fx2 v, int c, int n) {
                            v = fx_mul<2>(v, __ldg(&TVs.t[c * T + tid]));
                            if (I.has_field) v = fx_mul<2>(v, strip_field_fx<E>(fr, al, I, n));
                            return v;
                        });
                    kx += TVs.p;
                    t2 = kx ? ts + t2 * exp2f(-2.0f * (float)kx) : ts + t2;
                    e += kx;
                }
            }
        }
        for (int o = 16; o > 0; o >>= 1) t2 += __shfl_xor_sync(0xffffffffu, t2, o);
        if ((tid & 31) == 0) part[tid >> 5] = t2;
        bar.sync();
        t2 = part[0];
#pragma unroll
        for (int w = 1; w < NW; ++w) t2 += part[w];
        const int k = fx_norm_shift(t2, N);
        e = max(e - k, -(1 << 24));     // (a zero state is shifted in every step; below 2^-1074 all is zero)
        if (k != 0 || kx != 0) rescale_fx<LOGN, LOGE, LOGRM>(S, k, kx, nb, blk0, tid);
        // ---- kinetic: forward FFT, e^{-iK tau} (e^{-iK tau/2} in the first
        //      and last pass of the call), inverse FFT, potential of the next step
        const bool more = step + 1 < nsteps;
        F::fwd_all(S, Ws, Wg, tid, bar);
        const int4* __restrict__ tk = reinterpret_cast<const int4*>((step >= 0 && more) ? I.TK : I.TKh);
        if constexpr (SURF) {
            fx2 acc[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[r] = make_longlong2(0, 0);
            const int4* sw = reinterpret_cast<const int4*>(sw_v);
            const double* scale = reinterpret_cast<const double*>(sw + 8 * N);
            F::template center<true>(S, tk, tid, sw + (step >= 0 ? 4 * N : 0), acc);
            // acc: 1/4, and the unitary scaling of the passes before (the host
            // puts its odd half bit into the scales)
            surf_reduce_fx<T>(acc, scan, tid, bar, scale + (step >= 0 ? 4 : 0), e + 2 + LOGRM * (K::NPASS - 1) / 2,
                              samples + 4 * (step + 1));
        } else {
            F::template center<false>(S, tk, tid, nullptr, nullptr);
        }
        if (more && I.has_field) {
            al = 0.5 * I.tau * I.E0 * __ldg(&ftab[step + 1]);
            bad = !isfinite(al);
            field_setup_fx<LOGN, LOGE, LOGRM>(fr, al, I, tid);
        }
        bar.sync();
        F::inv_all(S, Ws, Wg, tid, bar);
        unsigned mr = 0;
        if (more) {
            if (TV.gen) potential_gen<LOGN, LOGE, LOGRM>(S, TV.d(N), fr, I, tid);
            else potential_fx<LOGN, LOGE, LOGRM>(S, TV, fr, I, tid, t2, mr);
        }
        coarse = bar.any(mr >= thr);
    }

    const double qnan = __longlong_as_double(0x7ff8000000000000LL);
    if (SURF && bad)
        for (int64_t i = 4 * (step + 1) + tid; i < 4 * (nsteps + 1); i += T) samples[i] = make_double2(qnan, qnan);
    const bool small = e > -900 && e < 900;
    double2* __restrict__ out = reinterpret_cast<double2*>(g_psi);
    double2 first = make_double2(0, 0);
#pragma unroll 1
    for (int j = 0; j < E; ++j) {             // (the last inverse pass's scaling is still to apply)
        const int n = tid + j * T, p = swz<fx2>(n);
        if (bad) {
            out[n] = make_double2(qnan, qnan);
            if (j == 0) first = make_double2(qnan, qnan);
            continue;
        }
        const fx2 a = fx_unit<LOGRM>(S[p]);
        if constexpr (K::GM) {
            if (n > p) continue;                      // stored by the owner of the smaller index
            const fx2 b = fx_unit<LOGRM>(S[n]);
            out[n] = make_double2(fx_out(a.x, e, small), fx_out(a.y, e, small));
            out[p] = make_double2(fx_out(b.x, e, small), fx_out(b.y, e, small));
        } else {
            out[n] = make_double2(fx_out(a.x, e, small), fx_out(a.y, e, small));
        }
        if (j == 0) first = out[n];
    }
    if (tid == 0 && status && !(isfinite(first.x) && isfinite(first.y))) atomicOr(status, 1);
}

}  // namespace soft
