// Host side of the fixed-point factors (fix64.cuh): values in units 2^-62 and
// their signed 32-bit halves; e^{2 pi i t} to about 2^-61 from an integer
// phase t in turns 2^-64 (no rounding of the cosine and sine to doubles: a
// twiddle's modulus error would return in every pass of every step).
#pragma once
#include <cmath>
#include <cstdint>

namespace soft {

// W = h 2^32 + l, l > -2^31
inline void fx_halves_host(int64_t W, int32_t* hl) {
    int32_t l = (int32_t)(uint32_t)(uint64_t)W;
    if (l == INT32_MIN) l += 1;              // 2^-62 of the factor
    hl[0] = (int32_t)((W - l) >> 32);
    hl[1] = l;
}
inline int64_t fx_q63(int64_t a, int64_t b) { return (int64_t)(((__int128)a * b + (1LL << 62)) >> 63); }

// cos and sin of 2 pi t 2^-64, units 2^-62 (sectors of 1/32 turn and Taylor
// series, as fx_cexp on the device)
inline void fx_cis_host(uint64_t t, int64_t* c, int64_t* s) {
    static const int64_t sect[9] = {4611686018427387904LL, 4523073764714963030LL, 4260642322793532497LL,
                                    3834476785802888710LL, 3260954456333195553LL, 2562115475870945497LL,
                                    1764815834521887442LL, 899695310372275547LL, 0LL};
    auto cs = [&](int k) {
        k &= 31;
        const int q = k >> 3, j = k & 7;
        const int64_t v = sect[(q & 1) ? 8 - j : j];
        return (q == 1 || q == 2) ? -v : v;
    };
    const int k = (int)((t + (1ULL << 58)) >> 59);
    const int64_t d = (int64_t)(t - ((uint64_t)k << 59));
    const int64_t r = d * 3 + fx_q63(d, 1305961721744163946LL), r2 = fx_q63(r, r);       // 2 pi d, 63 fraction bits
    const int64_t cm = fx_q63(r2, (1LL << 62) - fx_q63(r2, 384307168202282325LL - fx_q63(r2, 12810238940076078LL -
                       fx_q63(r2, 228754266787073LL - fx_q63(r2, 2541714075412LL)))));
    const int64_t sm = fx_q63(r2, 1537228672809129301LL - fx_q63(r2, 76861433640456465LL - fx_q63(r2,
                       1830034134296583LL - fx_q63(r2, 25417140754119LL - fx_q63(r2, 231064915947LL)))));
    const int64_t sn = r - fx_q63(r, sm);                                                 // 63 fraction bits
    const __int128 C = ((__int128)1 << 63) - cm;
    const int64_t wc = cs(k), ws = cs(k - 8);
    *c = (int64_t)((C * wc - (__int128)sn * ws + (1LL << 62)) >> 63);
    *s = (int64_t)((C * ws + (__int128)sn * wc + (1LL << 62)) >> 63);
}

// the phase ph (radians) in turns 2^-64: ph/(2 pi) to 106 bits, mod 1.  Beyond
// 2^50 (a wall of 10^17, say) the second part of the product would leave the
// range of its integer; such a phase is reduced by the library.
inline uint64_t fx_turns_host(double ph) {
    if (std::fabs(ph) > 0x1p50) ph = std::atan2(std::sin(ph), std::cos(ph));
    const double chi = 0.15915494309189535, clo = -9.839338337591243e-18;
    const double th = ph * chi, tl = std::fma(ph, chi, -th) + ph * clo;
    const double f = th - std::rint(th);
    return ((uint64_t)std::llrint(f * 0x1p62) << 2) + (uint64_t)std::llrint(tl * 0x1p64);
}

// sqrt(2) W
inline int64_t fx_sqrt2_host(int64_t W) {
    return (int64_t)(((__int128)W * 6521908912666391106LL + (1LL << 61)) >> 62);
}

}  // namespace soft
