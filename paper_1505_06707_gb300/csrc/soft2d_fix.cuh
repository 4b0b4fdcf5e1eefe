// Complex128 line passes of the 2D and 3D steps (soft2d.cuh) in 64-bit fixed
// point (fix64.cuh): a line is read as doubles, given one exponent from its
// norm, and transformed, multiplied and strip-solved as in the 1D step
// (soft1d_fix.cuh); it is written as doubles again.
//
// The FP64 passes were bound by the FP64 pipe: 143 clocks of an SM per point
// and step (2048^2).  The state's 160 bytes of traffic per point and step in
// 2D take 8 clocks at the measured copy rate.
//
// Scaling: the kinetic tables carry 2^(-1/2) where a pass's radix has an odd
// log2, so that the last inverse pass leaves a line 2^(LOGRM/2) (an integer
// division) too large; the next product, or the store, takes that in.
#pragma once
#include "soft2d.cuh"

namespace soft {

// potential factors of a grid: (p, gen) as in FxV, the FP64 factors (gen)
struct FxMeta { int p, gen; const double2* d; };

// Exponent of a line from the thread's samples d (tid + j T): d 2^-ed has a
// norm just below FX_NORM.  Returns the line's exponent e (ed but for tiny
// lines, which are scaled up first); bad: a non-finite sample.
template <int E, int T, class B>
__device__ __forceinline__ int fx_line_exp(double2 (&d)[E], float* part, unsigned* red, int tid, B bar, int& ed,
                                           bool& bad) {
    unsigned m = 0;
#pragma unroll
    for (int j = 0; j < E; ++j) m = max(m, fx_mag(d[j]));
    m = fx_group_max<T>(m, red, tid, bar);
    int off = 0;
    if (m < (128u << 20)) {                       // tiny (or zero)
        unsigned q = 0;
#pragma unroll
        for (int j = 0; j < E; ++j) { d[j] = cscale(d[j], 0x1p800); q = max(q, fx_mag(d[j])); }
        off = -800;
        bar.sync();
        m = fx_group_max<T>(q, red, tid, bar);
        if (m < (128u << 20)) m = 1023u << 20;    // zero
    }
    const int Em = (int)(m >> 20);
    bad = Em == 0x7ff;
    // squares in FP32, of the high words rebuilt as floats below 1 (a
    // conversion would run on the FP64 pipe)
    float t2 = 0.0f;
    auto rel = [&](double v) {
        const int b = (__double2hiint(v) & 0x7fffffff) - ((Em - 126) << 20);
        return __int_as_float(max(b, 0) << 3);
    };
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const float a = rel(d[j].x), b = rel(d[j].y);
        t2 += a * a + b * b;
    }
    for (int o = 16; o > 0; o >>= 1) t2 += __shfl_xor_sync(0xffffffffu, t2, o);
    if ((tid & 31) == 0) part[tid >> 5] = t2;
    bar.sync();
    t2 = part[0];
#pragma unroll
    for (int w = 1; w < T / 32; ++w) t2 += part[w];
    ed = Em - 1022 + (t2 > 0.0f ? (int)ceilf(0.5f * __log2f(t2) + 1e-3f - 60.8f) : 0);
    return ed + off;
}

template <int LOGN, int LOGE, int LOGRM>
struct LineFx {
    using F = Fx1D<LOGN, LOGE, LOGRM>;
    static constexpr int N = F::N, T = F::T, E = F::E;
    static constexpr int SH = LOGRM / 2;                       // left over by the last inverse pass
    static constexpr int TWN = TwCountT<TwFix, LOGN, LOGRM>::value;
    static constexpr int VCAP = T * F::K::CMAX;                // strip rows a line takes
    static constexpr size_t SCR = sizeof(fx2) * 64 + 128;      // scan scratch, sums, maxima
    static constexpr size_t SMEM_ROW = sizeof(fx2) * (N + TWN) + SCR;
    static constexpr int MINB = F::K::MINB;
};

// gen plans, row pass: V/2, CN_x in FP64 on the line as doubles
template <int LOGN, int LOGE, int LOGRM, class B>
__device__ __noinline__ void row_gen(fx2* S, int e, const double2* __restrict__ tv, const double2* __restrict__ cn,
                                     int nb, int blk0, int tid, double2* scan, B bar) {
    using L = LineFx<LOGN, LOGE, LOGRM>;
    const bool small = e > -900 && e < 900;
#pragma unroll 1
    for (int j = 0; j < L::E; ++j) {
        const int n = tid + j * L::T;
        fx2& r = S[swz<fx2>(n)];
        const fx2 x = fx_shr<L::SH>(r);
        r = fx_bits(cmul(make_double2(fx_out(x.x, e, small), fx_out(x.y, e, small)), __ldg(&tv[n])));
    }
    bar.sync();
    if (nb > 0) {
        strip_cn_gen<LOGN, LOGE, LOGRM>(S, cn, nb, blk0, tid, scan, bar, [](double2 v, int, int) { return v; });
        bar.sync();
    }
}
// gen plans, column pass: CN on the block with V/2, V/2 off the block (off_v)
template <int LOGN, int LOGE, int LOGRM, class B>
__device__ __noinline__ void col_gen(fx2* S, const double2* __restrict__ tv, int64_t ld, bool off_v,
                                     const double2* __restrict__ cn, int nb, int blk0, int tid, double2* scan, B bar) {
    using L = LineFx<LOGN, LOGE, LOGRM>;
    if (off_v) {
#pragma unroll 1
        for (int j = 0; j < L::E; ++j) {
            const int n = tid + j * L::T;
            if (((n - blk0) & (L::N - 1)) < nb) continue;
            fx2& r = S[swz<fx2>(n)];
            r = fx_bits(cmul(fx_asd(r), __ldg(&tv[n * ld])));
        }
        bar.sync();
    }
    if (nb > 0) {
        strip_cn_gen<LOGN, LOGE, LOGRM>(S, cn, nb, blk0, tid, scan, bar,
                                        [&](double2 v, int, int n) { return cmul(v, __ldg(&tv[n * ld])); });
        bar.sync();
    }
}

// One CTA per row, as row_pass_kernel (soft2d.cuh).
template <int LOGN, int LOGE, int LOGRM, int MODE>
__global__ void __launch_bounds__(LineFx<LOGN, LOGE, LOGRM>::T, LineFx<LOGN, LOGE, LOGRM>::MINB)
row_fx_kernel(Geo2D g, void* __restrict__ psi_v, const void* __restrict__ tkx_v)
{
    using L = LineFx<LOGN, LOGE, LOGRM>;
    using F = typename L::F;
    constexpr int N = L::N, T = L::T, E = L::E, SH = L::SH;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* S = reinterpret_cast<fx2*>(smem_raw);
    int4* Ws = reinterpret_cast<int4*>(S + N);
    fx2* scan = reinterpret_cast<fx2*>(Ws + L::TWN);
    float* part = reinterpret_cast<float*>(scan + 64);
    unsigned* red = reinterpret_cast<unsigned*>(part + 16);
    const int tid = threadIdx.x;
    const BarCTA bar;
    const int64_t y = blockIdx.x;
    double2* __restrict__ row = reinterpret_cast<double2*>(psi_v) + y * N;
    const int4* __restrict__ tv = reinterpret_cast<const int4*>(g.TVh) + y * N;
    double2 d[E];
#pragma unroll
    for (int j = 0; j < E; ++j) d[j] = row[tid + j * T];
    const int4* __restrict__ W = reinterpret_cast<const int4*>(g.Wx);
    for (int i = tid; i < L::TWN; i += T) cp_async<16>(&Ws[i], &W[i]);
    cp_async_commit();
    int ed;
    bool bad;
    int e = fx_line_exp<E, T>(d, part, red, tid, bar, ed, bad);
    if (bad) {                                   // a non-finite sample spreads over the line
        const double q = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll 1
        for (int j = 0; j < E; ++j) row[tid + j * T] = make_double2(q, q);
        cp_async_wait<0>();
        return;
    }
#pragma unroll
    for (int j = 0; j < E; ++j) S[swz<fx2>(tid + j * T)] = fx_from_double(d[j], ed);
    cp_async_wait<0>();
    __syncthreads();
    F::fwd_all(S, Ws, W, tid, bar);
    F::template center<false>(S, reinterpret_cast<const int4*>(tkx_v), tid, nullptr, nullptr);
    __syncthreads();
    F::inv_all(S, Ws, W, tid, bar);
    const int nb = MODE == ROW_KVC ? g.nbx : 0, blk0 = g.blk0x;
    // rows outside the y- and z-strip blocks take the second V/2 here
    const int ry = (int)(y % g.ny1), rz = (int)(y / g.ny1);
    const bool v2 = MODE == ROW_KVC && g.v2 && ((ry - g.blk0y) & (g.ny1 - 1)) >= g.nby &&
                    ((rz - g.blk0z1) & (g.nz1 - 1)) >= g.nbz1;
    int kx = 0;
    if constexpr (MODE == ROW_KVC) {
        const FxMeta M = *reinterpret_cast<const FxMeta*>(g.vmeta);
        const FxCn<T> cn(g.cnx, nb);
        if (M.gen) {
            const double2* __restrict__ td = M.d + y * N;
            row_gen<LOGN, LOGE, LOGRM>(S, e, td, cn.cd, nb, blk0, tid, reinterpret_cast<double2*>(scan), bar);
#pragma unroll 1
            for (int j = 0; j < E; ++j) {
                const int n = tid + j * T;
                const double2 v = fx_asd(S[swz<fx2>(n)]);
                row[n] = v2 ? cmul(v, __ldg(&td[n])) : v;
            }
            return;
        }
        unsigned mr = 0;
        constexpr int Q = E < 4 ? E : 4;
#pragma unroll 1
        for (int j0 = 0; j0 < E; j0 += Q) {
            int4 t[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) t[q] = __ldg(&tv[tid + (j0 + q) * T]);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int n = tid + (j0 + q) * T;
                fx2& r = S[swz<fx2>(n)];
                const fx2 x = fx_mul<2 - SH>(r, t[q]);
                r = x;
                if (((n - blk0) & (N - 1)) < nb) mr = max(mr, fx_hmag(x));
            }
        }
        e += M.p;
        if (nb > 0) {
            const bool coarse = bar.any(mr >= (1u << (27 - cn.lg)));
            strip_cn_fx<LOGN, LOGE, LOGRM>(S, cn, nb, blk0, tid, scan, bar, coarse, kx,
                                           [](fx2 v, int, int) { return v; });
            __syncthreads();
        }
        if (v2) e += M.p;
    }
    const bool small = e > -900 && e + kx < 900;
#pragma unroll 1
    for (int j0 = 0; j0 < E; j0 += 2) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int n = tid + (j0 + q) * T;
            fx2 x = S[swz<fx2>(n)];
            if constexpr (MODE == ROW_K) x = fx_shr<SH>(x);
            else if (v2) x = fx_mul<2>(x, __ldg(&tv[n]));
            const int en = e + (((n - blk0) & (N - 1)) < nb ? kx : 0);
            row[n] = make_double2(fx_out(x.x, en, small), fx_out(x.y, en, small));
        }
    }
}

// TW lines per CTA, as col_pass_kernel (soft2d.cuh); each line's T threads
// have their own barrier.
template <int LOGN, int LOGE, int LOGRM, int TW>
struct ColFx : LineFx<LOGN, LOGE, LOGRM> {
    using L = LineFx<LOGN, LOGE, LOGRM>;
    static constexpr int THREADS = TW * L::T;
    static constexpr int MINB = THREADS >= 512 ? 1 : 512 / THREADS;      // <= 128 registers
    static constexpr int PITCH = L::N + 4;          // the TW columns of a row in different banks
    static constexpr size_t OFF_W = sizeof(fx2) * (size_t)TW * PITCH;
    static constexpr size_t OFF_SCR = OFF_W + sizeof(int4) * L::TWN;
    static constexpr size_t OFF_E = OFF_SCR + TW * L::SCR;              // exponents of the columns
    static constexpr size_t OFF_V = OFF_E + 16 * ((TW * 4 + 15) / 16);
    static constexpr size_t SMEM_K = OFF_V;
    static constexpr size_t SMEM_CVK = OFF_V + sizeof(int4) * (size_t)TW * L::VCAP;
};

template <int LOGN, int LOGE, int LOGRM, int TW, int MODE>
__global__ void __launch_bounds__(ColFx<LOGN, LOGE, LOGRM, TW>::THREADS, ColFx<LOGN, LOGE, LOGRM, TW>::MINB)
col_fx_kernel(LineGeo lg, void* __restrict__ psi_v, const void* __restrict__ tky_v)
{
    using CC = ColFx<LOGN, LOGE, LOGRM, TW>;
    using F = typename CC::F;
    constexpr int N = CC::N, T = CC::T, E = CC::E, PITCH = CC::PITCH;
    constexpr int BADE = 0x7fffffff;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* S = reinterpret_cast<fx2*>(smem_raw);
    int4* Ws = reinterpret_cast<int4*>(smem_raw + CC::OFF_W);
    int* ecol = reinterpret_cast<int*>(smem_raw + CC::OFF_E);
    int4* Tvs = reinterpret_cast<int4*>(smem_raw + CC::OFF_V);           // [TW][VCAP]
    const int64_t ld = lg.ld;
    const int64_t gpp = ld / TW;                    // CTAs per plane
    const int64_t poff = (int64_t)(blockIdx.x / gpp) * lg.plane;
    const int64_t c0 = (int64_t)(blockIdx.x % gpp) * TW;
    double2* __restrict__ psi = reinterpret_cast<double2*>(psi_v) + poff + c0;
    const int4* __restrict__ tv = reinterpret_cast<const int4*>(lg.tv) + poff + c0;
    const int4* __restrict__ W = reinterpret_cast<const int4*>(lg.W);
#pragma unroll 8
    for (int it = 0; it < E; ++it) {                // row by row: the TW columns of a row are adjacent
        const int idx = threadIdx.x + it * TW * T, yy = idx / TW, j = idx % TW;
        cp_async<16>(&S[j * PITCH + swz<fx2>(yy)], &psi[(int64_t)yy * ld + j]);
    }
    cp_async_commit();
    const int nb = MODE == COL_K ? 0 : lg.nb, blk0 = lg.blk0;
    for (int i = threadIdx.x; i < CC::TWN; i += TW * T) cp_async<16>(&Ws[i], &W[i]);
    FxMeta M{0, 0, nullptr};
    if constexpr (MODE != COL_K) {
        M = *reinterpret_cast<const FxMeta*>(lg.vmeta);
        if (!M.gen)
            for (int idx = threadIdx.x; idx < nb * TW; idx += TW * T) {
                const int i = idx / TW, j = idx % TW;
                cp_async<16>(&Tvs[j * CC::VCAP + i], &tv[(int64_t)((blk0 + i) & (N - 1)) * ld + j]);
            }
    }
    cp_async_commit();
    cp_async_wait<1>();
    __syncthreads();                                // the tile
    const int col = threadIdx.x / T, tid = threadIdx.x % T;
    const BarGroup bar{1 + col, T};
    fx2* Sc = S + col * PITCH;
    fx2* scan = reinterpret_cast<fx2*>(smem_raw + CC::OFF_SCR + col * CC::SCR);
    float* part = reinterpret_cast<float*>(scan + 64);
    unsigned* red = reinterpret_cast<unsigned*>(part + 16);
    bool off_v = MODE == COL_CVK;                   // V/2 off the strip block here
    if (MODE == COL_CVK && lg.sel_div > 0) {
        const int q = (int)((c0 / lg.sel_div) % lg.sel_n);
        off_v = ((q - lg.sel_blk0) & (lg.sel_n - 1)) < lg.sel_nb;
    }
    const FxCn<T> cn(lg.cn, nb);
    if constexpr (MODE != COL_K) {
        if (M.gen)
            col_gen<LOGN, LOGE, LOGRM>(Sc, M.d + poff + c0 + col, ld, off_v, cn.cd, nb, blk0, tid,
                                       reinterpret_cast<double2*>(scan), bar);
    }
    double2 d[E];
#pragma unroll
    for (int j = 0; j < E; ++j) d[j] = fx_asd(Sc[swz<fx2>(tid + j * T)]);
    int ed;
    bool bad;
    int e = fx_line_exp<E, T>(d, part, red, tid, bar, ed, bad);
    cp_async_wait<0>();
    __syncthreads();                                // twiddles and V/2 factors, copied by all columns' threads
    if (!bad) {
        const bool strip = MODE != COL_K && !M.gen && (nb > 0 || off_v);
        float t2 = 0.0f;
        unsigned mr = 0;
#pragma unroll
        for (int j = 0; j < E; ++j) {
            const int n = tid + j * T;
            fx2 x = fx_from_double(d[j], ed);
            if (strip) {
                if (((n - blk0) & (N - 1)) < nb) {
                    mr = max(mr, fx_hmag(x));
                } else {
                    if (off_v) x = fx_mul<2>(x, __ldg(&tv[(int64_t)n * ld + col]));
                    t2 += fx_abs2(x);
                }
            }
            Sc[swz<fx2>(n)] = x;
        }
        const bool coarse = bar.any(strip && mr >= (1u << (27 - cn.lg)));
        if (strip) {
            // units: 2^e times 2^po off the block, times 2^(kx + p) on it
            const int po = off_v ? M.p : 0;
            int kx = 0;
            if (nb > 0) {
                const int4* tvc = Tvs + col * CC::VCAP;
                const float ts = strip_cn_fx<LOGN, LOGE, LOGRM>(
                    Sc, cn, nb, blk0, tid, scan, bar, coarse, kx,
                    [&](fx2 v, int, int n) { return fx_mul<2>(v, tvc[(n - blk0) & (N - 1)]); });
                kx += M.p - po;
                t2 = kx ? ts + t2 * exp2f(-2.0f * (float)kx) : ts + t2;
            }
            e += po + kx;
            for (int o = 16; o > 0; o >>= 1) t2 += __shfl_xor_sync(0xffffffffu, t2, o);
            if ((tid & 31) == 0) part[tid >> 5] = t2;
            bar.sync();
            t2 = part[0];
#pragma unroll
            for (int w = 1; w < T / 32; ++w) t2 += part[w];
            const int k = fx_norm_shift(t2, N);
            e -= k;
            if (k != 0 || kx != 0) rescale_fx<LOGN, LOGE, LOGRM>(Sc, k, kx, nb, blk0, tid);
        }
    }
    bar.sync();
    F::fwd_all(Sc, Ws, W, tid, bar);
    F::template center<false>(Sc, reinterpret_cast<const int4*>(tky_v), tid, nullptr, nullptr);
    bar.sync();
    F::inv_all(Sc, Ws, W, tid, bar);
    if (tid == 0) ecol[col] = bad ? BADE : e;
    __syncthreads();
#pragma unroll 2
    for (int it = 0; it < E; ++it) {
        const int idx = threadIdx.x + it * TW * T, yy = idx / TW, j = idx % TW;
        const int ej = ecol[j];
        const fx2 x = fx_shr<CC::SH>(S[j * PITCH + swz<fx2>(yy)]);
        const bool small = ej > -900 && ej < 900;
        double2 o = make_double2(fx_out(x.x, ej, small), fx_out(x.y, ej, small));
        if (ej == BADE) o.x = o.y = __longlong_as_double(0x7ff8000000000000LL);
        psi[(int64_t)yy * ld + j] = o;
    }
}

// ---------------------------------------------------------------- launchers
template <int LOGN, int LOGE, int LOGRM>
int launch_row_fx(int mode, const Geo2D& g, void* psi, int nrows, const void* tkx, cudaStream_t st) {
    using L = LineFx<LOGN, LOGE, LOGRM>;
    void (*k)(Geo2D, void*, const void*) = nullptr;
    switch (mode) {
    case ROW_K: k = row_fx_kernel<LOGN, LOGE, LOGRM, ROW_K>; break;
    case ROW_KVC: k = row_fx_kernel<LOGN, LOGE, LOGRM, ROW_KVC>; break;
    default: return SOFT_ERR_INVALID_ARG;
    }
    if (L::SMEM_ROW > 48 * 1024 &&
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::SMEM_ROW) != cudaSuccess)
        return SOFT_ERR_CUDA;
    if (nrows <= 0 || !psi) return SOFT_OK;
    k<<<nrows, L::T, L::SMEM_ROW, st>>>(g, psi, tkx);
    return cudaGetLastError() == cudaSuccess ? SOFT_OK : SOFT_ERR_CUDA;
}

template <int LOGN, int LOGE, int LOGRM, int TW>
int launch_col_fx(int mode, const LineGeo& g, int planes, void* psi, const void* tky, cudaStream_t st) {
    using CC = ColFx<LOGN, LOGE, LOGRM, TW>;
    const size_t smem = mode == COL_K ? CC::SMEM_K : CC::SMEM_CVK;
    void (*k)(LineGeo, void*, const void*) = nullptr;
    switch (mode) {
    case COL_K: k = col_fx_kernel<LOGN, LOGE, LOGRM, TW, COL_K>; break;
    case COL_CVK: k = col_fx_kernel<LOGN, LOGE, LOGRM, TW, COL_CVK>; break;
    case COL_CBK: k = col_fx_kernel<LOGN, LOGE, LOGRM, TW, COL_CBK>; break;
    default: return SOFT_ERR_INVALID_ARG;
    }
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return SOFT_ERR_CUDA;
    if (!psi) return SOFT_OK;             // attribute set only
    if (g.ld % TW || planes < 1) return SOFT_ERR_INVALID_ARG;
    if (mode != COL_K && (g.nb + CC::T - 1) / CC::T > CC::F::K::CMAX) return SOFT_ERR_UNSUPPORTED;
    const int64_t grid = g.ld / TW * planes;
    if (grid > 0x7fffffff) return SOFT_ERR_TOO_LARGE;
    k<<<(unsigned)grid, CC::THREADS, smem, st>>>(g, psi, tky);
    return cudaGetLastError() == cudaSuccess ? SOFT_OK : SOFT_ERR_CUDA;
}

}  // namespace soft
