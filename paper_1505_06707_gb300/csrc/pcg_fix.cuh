// The FP64 passes of the stationary solver (pcg.cuh: A and the
// preconditioners on a 2D grid) with their FFTs, the kinetic factor and the
// band products in 64-bit fixed point (fix64.cuh): a line is read, given one
// exponent from its norm, transformed and converted back.  The potential and
// strip terms of A, the division by lambda - E, and the dot products stay in
// FP64, as does every vector in memory.
//
// One A and one banded P^-1 at 1024^2 took 341 clocks of an SM per point, 87 %
// of them in the FP64 pipe: 4 FFT pairs (240 FP64 instructions) and 4 band
// products of ten complex terms (160).
//
// Scaling.  Forward and inverse FFTs are unitary (1/sqrt N each, so the band
// rows come without it).  The band rows enter as X 2^-pb, pb from a bound of
// their operator norm, so that no line's norm grows.  The kinetic factor is
// applied in FP64 and the line given a new exponent after it (center_k): with
// k^2/2 2^-pk <= 1 as a fixed-point factor the inverse FFT's rounding is
// relative to max(k^2/2) |p| instead of |K p|, in the modes of small k too,
// where P^-1 amplifies it (COCG with absorbing potentials took up to 9
// iterations more, of 45, at low energies; A of a smooth vector, N = 1024: off
// by 9.7e-15 of |p|, 2.7e-15 so, 3.5e-14 in FP64).  It costs 2 FP64
// instructions per point (A and P^-1 at 1024^2: 335 -> 341 us).
#pragma once
#include "pcg.cuh"
#include "soft2d_fix.cuh"

namespace soft {

// per-line scratch behind the buffers: sums and maxima of fx_line_exp
struct PcgScr {
    float* part;
    unsigned* red;
    __device__ __forceinline__ explicit PcgScr(void* p) : part(reinterpret_cast<float*>(p)),
                                                         red(reinterpret_cast<unsigned*>(part + 16)) {}
};

template <int LOGN, int LR = 3>                  // radix 2^LR, a butterfly per thread
struct PcgFx : LineFx<LOGN, LR, LR> {
    using L = LineFx<LOGN, LR, LR>;
    using F = typename L::F;
    static constexpr int N = L::N, T = L::T, E = L::E;
    static constexpr int NP = F::NPASS, R = PassGeom<LOGN, LR, NP - 1>::LOGR;    // bits of the last pass
    static constexpr int PITCH = N + 4;
    static constexpr size_t SMEM_A = sizeof(fx2) * (N + L::TWN) + L::SCR;
    static constexpr size_t SMEM_P = sizeof(fx2) * (2 * N + L::TWN) + L::SCR;
    template <int TW> static constexpr size_t smem_col(int bufs) {
        return sizeof(fx2) * ((size_t)bufs * TW * PITCH + L::TWN) + TW * L::SCR + 64;
    }
    static constexpr int MINB = L::MINB;
    // last forward pass (stride 1, no twiddles), unitary
    __device__ __forceinline__ static void fwd_last(fx2* S, int tid) {
        constexpr int RR = 1 << R;
#pragma unroll 1
        for (int u = 0; u < E / RR; ++u) {
            const int sb = swz<fx2>((tid + u * T) * RR);
            fx2 v[RR];
#pragma unroll
            for (int j = 0; j < RR; ++j) v[j] = S[sb ^ swz<fx2>(j)];
            dft_reg<fx2, RR, -1>(v);
#pragma unroll
            for (int m = 0; m < RR; ++m) S[sb ^ swz<fx2>(m)] = fx_unit<R>(v[bitrev_c(m, R)]);
        }
    }
    // last forward pass, k^2/2 in FP64 (kt, the centre's transposed order), a
    // new exponent, first inverse pass.  Returns the exponent relative to the
    // line's before: of the normalisation, and of the scaling that the two
    // passes and the last inverse pass (2^-1) leave over, which is a power of 2.
    template <class B>
    __device__ __forceinline__ static int center_k(fx2* S, const double* __restrict__ kt, PcgScr sc, int tid, B bar,
                                                   bool& bad) {
        constexpr int RR = 1 << R, cs = (LR - R) / 2;
        double2 d[E];
#pragma unroll
        for (int u = 0; u < E / RR; ++u) {
            const int sb = swz<fx2>((tid + u * T) * RR);
            fx2 v[RR];
#pragma unroll
            for (int j = 0; j < RR; ++j) v[j] = S[sb ^ swz<fx2>(j)];
            dft_reg<fx2, RR, -1>(v);
#pragma unroll
            for (int m = 0; m < RR; ++m)
                d[u * RR + m] = cscale(fx_to_double(v[bitrev_c(m, R)]), __ldg(&kt[m * (N / RR) + tid + u * T]));
        }
        int ed;
        const int e = fx_line_exp<E, T>(d, sc.part, sc.red, tid, bar, ed, bad);
#pragma unroll
        for (int u = 0; u < E / RR; ++u) {
            const int sb = swz<fx2>((tid + u * T) * RR);
            fx2 w[RR];
#pragma unroll
            for (int m = 0; m < RR; ++m) w[m] = fx_from_double(d[u * RR + m], ed);
            dft_reg<fx2, RR, +1>(w);
#pragma unroll
            for (int m = 0; m < RR; ++m) {
                const fx2 o = w[bitrev_c(m, R)];
                S[sb ^ swz<fx2>(m)] = make_longlong2(o.x << cs, o.y << cs);
            }
        }
        return e - R - cs;
    }
    // first inverse pass, left as large as a pass of LR bits leaves it (the
    // tables before it carry the half bits)
    __device__ __forceinline__ static void inv_first(fx2* S, int tid) {
        constexpr int RR = 1 << R, cs = (LR - R) / 2;
#pragma unroll 1
        for (int u = 0; u < E / RR; ++u) {
            const int sb = swz<fx2>((tid + u * T) * RR);
            fx2 v[RR];
#pragma unroll
            for (int j = 0; j < RR; ++j) v[j] = S[sb ^ swz<fx2>(j)];
            dft_reg<fx2, RR, +1>(v);
#pragma unroll
            for (int m = 0; m < RR; ++m) {
                const fx2 o = v[bitrev_c(m, R)];
                S[sb ^ swz<fx2>(m)] = make_longlong2(o.x << cs, o.y << cs);
            }
        }
    }
};

__device__ __forceinline__ double2 fx_nan2() {
    const double q = __longlong_as_double(0x7ff8000000000000LL);
    return make_double2(q, q);
}
__device__ __forceinline__ fx2 fx_conj(fx2 v) { return make_longlong2(v.x, -v.y); }
__device__ __forceinline__ double2 fx_value(fx2 v, int e) {
    const bool small = e > -900 && e < 900;
    return make_double2(fx_out(v.x, e, small), fx_out(v.y, e, small));
}

// four band rows at once (band_rows in pcg.cuh): out[j] = sum tab in
template <int NJ, class In>
__device__ __forceinline__ void band_rows_fx(int nu0, int step, int n, const int* __restrict__ bs,
                                             const int* __restrict__ bw, const int4* __restrict__ tab, In in,
                                             fx2 (&out)[NJ]) {
    int s0[NJ], wm = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        s0[j] = __ldg(&bs[nu0 + j * step]);
        wm = max(wm, __ldg(&bw[nu0 + j * step]));
        out[j] = make_longlong2(0, 0);
    }
#pragma unroll 1
    for (int u = 0; u < wm; ++u) {
#pragma unroll
        for (int j = 0; j < NJ; ++j)
            out[j] = cadd(out[j], fx_mul<2>(in(min(s0[j] + u, n - 1)), __ldg(&tab[u * n + nu0 + j * step])));
    }
}

// w = F_x^-1 Kx F_x p + C_x p + (U - E) p, one CTA per (row, energy)
template <typename IO, int LOGN>
__global__ void __launch_bounds__(PcgFx<LOGN>::T, PcgFx<LOGN>::MINB)
a_row_fx_kernel(PcgGeo g, const void* __restrict__ p_v, void* __restrict__ w_v, const double* __restrict__ E,
                const int* __restrict__ active)
{
    using Q = PcgFx<LOGN>;
    using F = typename Q::F;
    constexpr int N = Q::N, T = Q::T, NE = Q::E;
    const int y = blockIdx.x, e = blockIdx.y;
    if (active && !active[e]) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* S = reinterpret_cast<fx2*>(smem_raw);
    int4* Ws = reinterpret_cast<int4*>(S + N);
    const PcgScr sc(Ws + Q::TWN);
    const int tid = threadIdx.x;
    const BarCTA bar;
    const int64_t base = (int64_t)e * g.N + (int64_t)y * N;
    const IO* __restrict__ p = reinterpret_cast<const IO*>(p_v) + base;
    IO* __restrict__ w = reinterpret_cast<IO*>(w_v) + base;
    const int4* __restrict__ W = reinterpret_cast<const int4*>(g.fWx);
    double2 d[NE];
#pragma unroll
    for (int j = 0; j < NE; ++j) d[j] = cto<double2>(p[tid + j * T]);
    for (int i = tid; i < Q::TWN; i += T) cp_async<16>(&Ws[i], &W[i]);
    cp_async_commit();
    int ed;
    bool bad;
    int el = fx_line_exp<NE, T>(d, sc.part, sc.red, tid, bar, ed, bad);
#pragma unroll
    for (int j = 0; j < NE; ++j) S[swz<fx2>(tid + j * T)] = fx_from_double(d[j], ed);
    cp_async_wait<0>();
    __syncthreads();
    F::fwd_all(S, Ws, W, tid, bar);
    bool bad2;
    el += Q::center_k(S, reinterpret_cast<const double*>(g.fKx), sc, tid, bar, bad2);
    bad = bad || bad2;
    __syncthreads();
    F::inv_all(S, Ws, W, tid, bar);
    const double2* __restrict__ U = reinterpret_cast<const double2*>(g.U) + (int64_t)y * N;
    const double2* __restrict__ Cx = reinterpret_cast<const double2*>(g.Cx);
    const double En = E[e];
#pragma unroll 2
    for (int j = 0; j < NE; ++j) {
        const int n = tid + j * T;
        const double2 pv = cto<double2>(p[n]);
        double2 u = __ldg(&U[n]);
        u.x -= En;
        double2 v = bad ? fx_nan2() : fx_value(S[swz<fx2>(n)], el);
        v = cfma(u, pv, v);
        if (((n - g.blk0x) & (N - 1)) < g.nbx) {
            v = cfma(__ldg(&Cx[n]), cto<double2>(p[(n + N - 1) & (N - 1)]), v);
            v = cfma(__ldg(&Cx[N + n]), pv, v);
            v = cfma(__ldg(&Cx[2 * N + n]), cto<double2>(p[(n + 1) & (N - 1)]), v);
        }
        w[n] = cto<IO>(v);
    }
}

// the tile of TW columns as doubles in shared memory, loaded row by row
template <typename IO, int LOGN, int TW, bool CONJ>
__device__ __forceinline__ void col_tile(fx2* S, const IO* __restrict__ p, int nx) {
    using Q = PcgFx<LOGN>;
#pragma unroll
    for (int it = 0; it < Q::E; ++it) {
        const int idx = threadIdx.x + it * TW * Q::T, yy = idx / TW, j = idx % TW;
        double2 v = cto<double2>(p[(int64_t)yy * nx + j]);
        if (CONJ) v.y = -v.y;
        S[j * Q::PITCH + swz<fx2>(yy)] = fx_bits(v);
    }
}
// a column of doubles in shared memory -> fixed point in place; returns its exponent
template <int LOGN, class B>
__device__ __forceinline__ int col_exp(fx2* Sc, bool swizzled, PcgScr sc, int tid, B bar, bool& bad) {
    using Q = PcgFx<LOGN>;
    double2 d[Q::E];
#pragma unroll
    for (int j = 0; j < Q::E; ++j) {
        const int n = tid + j * Q::T;
        d[j] = fx_asd(Sc[swizzled ? swz<fx2>(n) : n]);
    }
    int ed;
    const int e = fx_line_exp<Q::E, Q::T>(d, sc.part, sc.red, tid, bar, ed, bad);
#pragma unroll
    for (int j = 0; j < Q::E; ++j) {
        const int n = tid + j * Q::T;
        Sc[swizzled ? swz<fx2>(n) : n] = fx_from_double(d[j], ed);
    }
    return e;
}

// w += F_y^-1 Ky F_y p + C_y p, TW columns per CTA; partials of p^T w as
// a_col_kernel
template <typename IO, int LOGN, int TW>
__global__ void __launch_bounds__(TW * PcgFx<LOGN>::T, (TW * PcgFx<LOGN>::T >= 512 ? 1 : 512 / (TW * PcgFx<LOGN>::T)))
a_col_fx_kernel(PcgGeo g, const void* __restrict__ p_v, void* __restrict__ w_v, const int* __restrict__ active,
                double2* __restrict__ part, int pstride)
{
    using Q = PcgFx<LOGN>;
    using F = typename Q::F;
    constexpr int N = Q::N, T = Q::T, PITCH = Q::PITCH;
    const int e = blockIdx.y;
    if (active && !active[e]) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* S = reinterpret_cast<fx2*>(smem_raw);
    int4* Ws = reinterpret_cast<int4*>(S + TW * PITCH);
    unsigned char* scr = reinterpret_cast<unsigned char*>(Ws + Q::TWN);
    int* ecol = reinterpret_cast<int*>(scr + TW * Q::SCR);
    __shared__ double2 red[32];
    constexpr int BADE = 0x7fffffff;
    const int c0 = blockIdx.x * TW, nx = g.nx;
    const int64_t eb = (int64_t)e * g.N + c0;
    const IO* __restrict__ p = reinterpret_cast<const IO*>(p_v) + eb;
    IO* __restrict__ w = reinterpret_cast<IO*>(w_v) + eb;
    const int4* __restrict__ W = reinterpret_cast<const int4*>(g.fWy);
    for (int i = threadIdx.x; i < Q::TWN; i += TW * T) cp_async<16>(&Ws[i], &W[i]);
    cp_async_commit();
    col_tile<IO, LOGN, TW, false>(S, p, nx);
    cp_async_wait<0>();
    __syncthreads();
    const int col = threadIdx.x / T, tid = threadIdx.x % T;
    const BarGroup bar{1 + col, T};
    fx2* Sc = S + col * PITCH;
    const PcgScr sc(scr + col * Q::SCR);
    bool bad, bad2;
    int el = col_exp<LOGN>(Sc, true, sc, tid, bar, bad);
    bar.sync();
    F::fwd_all(Sc, Ws, W, tid, bar);
    el += Q::center_k(Sc, reinterpret_cast<const double*>(g.fKy), sc, tid, bar, bad2);
    bad = bad || bad2;
    bar.sync();
    F::inv_all(Sc, Ws, W, tid, bar);
    if (tid == 0) ecol[col] = bad ? BADE : el;
    __syncthreads();
    const double2* __restrict__ Cy = reinterpret_cast<const double2*>(g.Cy);
    IO acc = cmk<IO>(0, 0);
#pragma unroll 2
    for (int it = 0; it < Q::E; ++it) {
        const int idx = threadIdx.x + it * TW * T, yy = idx / TW, j = idx % TW;
        const int64_t a = (int64_t)yy * nx + j;
        const int ej = ecol[j];
        double2 v = ej == BADE ? fx_nan2() : fx_value(S[j * PITCH + swz<fx2>(yy)], ej);
        const IO pv = p[a];
        if (((yy - g.blk0y) & (N - 1)) < g.nby) {
            v = cfma(__ldg(&Cy[yy]), cto<double2>(p[(int64_t)((yy + N - 1) & (N - 1)) * nx + j]), v);
            v = cfma(__ldg(&Cy[N + yy]), cto<double2>(pv), v);
            v = cfma(__ldg(&Cy[2 * N + yy]), cto<double2>(p[(int64_t)((yy + 1) & (N - 1)) * nx + j]), v);
        }
        const IO wv = cto<IO>(cadd(cto<double2>(w[a]), v));
        w[a] = wv;
        acc.x += pv.x * wv.x - pv.y * wv.y;      // bilinear p^T w
        acc.y += pv.x * wv.y + pv.y * wv.x;
    }
    const double2 t = block_sum2(cto<double2>(acc), red);
    if (threadIdx.x == 0) {
        part[(int64_t)e * pstride + blockIdx.x] = t;
        for (int k = blockIdx.x + gridDim.x; k < pstride; k += gridDim.x)
            part[(int64_t)e * pstride + k] = make_double2(0.0, 0.0);
    }
}

// row pass 1 of the preconditioner: t = X_x F_x r, natural nu order
template <int LOGN>
__global__ void __launch_bounds__(PcgFx<LOGN>::T, PcgFx<LOGN>::MINB)
pc_row1_fx_kernel(PcgGeo g, const void* __restrict__ r_v, void* __restrict__ t_v, const int* __restrict__ active)
{
    using Q = PcgFx<LOGN>;
    using F = typename Q::F;
    constexpr int N = Q::N, T = Q::T, NE = Q::E;
    const int y = blockIdx.x, e = blockIdx.y;
    if (active && !active[e]) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* S = reinterpret_cast<fx2*>(smem_raw);
    fx2* Fn = S + N;                             // F_x r in natural index order
    int4* Ws = reinterpret_cast<int4*>(Fn + N);
    const PcgScr sc(Ws + Q::TWN);
    const int tid = threadIdx.x;
    const BarCTA bar;
    const int64_t base = (int64_t)e * g.N + (int64_t)y * N;
    const double2* __restrict__ r = reinterpret_cast<const double2*>(r_v) + base;
    double2* __restrict__ t = reinterpret_cast<double2*>(t_v) + base;
    const int4* __restrict__ W = reinterpret_cast<const int4*>(g.fWx);
    double2 d[NE];
#pragma unroll
    for (int j = 0; j < NE; ++j) d[j] = cconj(r[tid + j * T]);
    for (int i = tid; i < Q::TWN; i += T) cp_async<16>(&Ws[i], &W[i]);
    cp_async_commit();
    int ed;
    bool bad;
    const int el = fx_line_exp<NE, T>(d, sc.part, sc.red, tid, bar, ed, bad) + g.pfx;
#pragma unroll
    for (int j = 0; j < NE; ++j) S[swz<fx2>(tid + j * T)] = fx_from_double(d[j], ed);
    cp_async_wait<0>();
    __syncthreads();
    F::fwd_all(S, Ws, W, tid, bar);
    Q::fwd_last(S, tid);
    __syncthreads();
#pragma unroll 2
    for (int j = 0; j < NE; ++j) {
        const int m = tid + j * T;
        Fn[m] = fx_conj(S[swz<fx2>(__ldg(&g.posx[m]))]);
    }
    __syncthreads();
    const int4* __restrict__ xf = reinterpret_cast<const int4*>(g.xfx);
#pragma unroll 1
    for (int j0 = 0; j0 < NE; j0 += BAND_NJ) {
        fx2 o[BAND_NJ];
        band_rows_fx<BAND_NJ>(tid + j0 * T, T, N, g.bsx, g.bwx, xf, [&](int m) { return Fn[m]; }, o);
#pragma unroll
        for (int j = 0; j < BAND_NJ; ++j) t[tid + (j0 + j) * T] = bad ? fx_nan2() : fx_value(o[j], el);
    }
}

// column pass: F_y, X_y, / (lambda_x + lambda_y - E), X_y^T, F_y^-1 (in place on t)
template <int LOGN, int TW>
__global__ void __launch_bounds__(TW * PcgFx<LOGN>::T, (TW * PcgFx<LOGN>::T >= 512 ? 1 : 512 / (TW * PcgFx<LOGN>::T)))
pc_col_fx_kernel(PcgGeo g, void* __restrict__ t_v, const double* __restrict__ E, const int* __restrict__ active)
{
    using Q = PcgFx<LOGN>;
    using F = typename Q::F;
    constexpr int N = Q::N, T = Q::T, NE = Q::E, PITCH = Q::PITCH;
    constexpr int BADE = 0x7fffffff;
    const int e = blockIdx.y;
    if (active && !active[e]) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* S = reinterpret_cast<fx2*>(smem_raw);
    fx2* S2 = S + TW * PITCH;
    int4* Ws = reinterpret_cast<int4*>(S2 + TW * PITCH);
    unsigned char* scr = reinterpret_cast<unsigned char*>(Ws + Q::TWN);
    int* ecol = reinterpret_cast<int*>(scr + TW * Q::SCR);
    const int c0 = blockIdx.x * TW, nx = g.nx;
    double2* __restrict__ t = reinterpret_cast<double2*>(t_v) + (int64_t)e * g.N + c0;
    const int4* __restrict__ W = reinterpret_cast<const int4*>(g.fWy);
    for (int i = threadIdx.x; i < Q::TWN; i += TW * T) cp_async<16>(&Ws[i], &W[i]);
    cp_async_commit();
    col_tile<double2, LOGN, TW, true>(S, t, nx);
    cp_async_wait<0>();
    __syncthreads();
    const int col = threadIdx.x / T, tid = threadIdx.x % T;
    const BarGroup bar{1 + col, T};
    const PcgScr sc(scr + col * Q::SCR);
    fx2* Sc = S + col * PITCH;
    fx2* S2c = S2 + col * PITCH;
    bool bad, bad2;
    int el = col_exp<LOGN>(Sc, true, sc, tid, bar, bad) + g.pfy;
    bar.sync();
    F::fwd_all(Sc, Ws, W, tid, bar);
    Q::fwd_last(Sc, tid);
    bar.sync();
#pragma unroll 2
    for (int j = 0; j < NE; ++j) {                 // F_y t in natural index order
        const int m = tid + j * T;
        S2c[m] = fx_conj(Sc[swz<fx2>(__ldg(&g.posy[m]))]);
    }
    bar.sync();
    const double2 lx = reinterpret_cast<const double2*>(g.lamx)[c0 + col];
    const double En = E[e];
    const int4* __restrict__ xf = reinterpret_cast<const int4*>(g.xfy);
    const int4* __restrict__ xb = reinterpret_cast<const int4*>(g.xby);
    const double2* __restrict__ ly = reinterpret_cast<const double2*>(g.lamy);
#pragma unroll 1
    for (int j0 = 0; j0 < NE; j0 += BAND_NJ) {    // X_y, then the eigenvalue denominator
        fx2 o[BAND_NJ];
        band_rows_fx<BAND_NJ>(tid + j0 * T, T, N, g.bsy, g.bwy, xf, [&](int m) { return S2c[m]; }, o);
#pragma unroll
        for (int j = 0; j < BAND_NJ; ++j) {
            const int mu = tid + (j0 + j) * T;
            const double2 lm = __ldg(&ly[mu]);
            const double2 den = make_double2(lx.x + lm.x - En, lx.y + lm.y);
            const double dn = den.x * den.x + den.y * den.y;
            Sc[mu] = fx_bits(cscale(cmulc(fx_value(o[j], el), den), 1.0 / dn));    // c / den, natural order
        }
    }
    // (own rows: tid + j T)
    el = col_exp<LOGN>(Sc, false, sc, tid, bar, bad2) + g.pby;
    bad = bad || bad2;
    bar.sync();
#pragma unroll 1
    for (int j0 = 0; j0 < NE; j0 += BAND_NJ) {    // X_y^T into FFT positions (conjugated)
        fx2 o[BAND_NJ];
        band_rows_fx<BAND_NJ>(tid + j0 * T, T, N, g.bsy, g.bwy, xb, [&](int nu) { return Sc[nu]; }, o);
#pragma unroll
        for (int j = 0; j < BAND_NJ; ++j) S2c[swz<fx2>(__ldg(&g.posy[tid + (j0 + j) * T]))] = fx_conj(o[j]);
    }
    bar.sync();
    Q::inv_first(S2c, tid);
    bar.sync();
    F::inv_all(S2c, Ws, W, tid, bar);
    if (tid == 0) ecol[col] = bad ? BADE : el - 1;      // the last pass leaves a factor 2
    __syncthreads();
#pragma unroll 2
    for (int it = 0; it < NE; ++it) {
        const int idx = threadIdx.x + it * TW * T, yy = idx / TW, j = idx % TW;
        const int ej = ecol[j];
        t[(int64_t)yy * nx + j] = ej == BADE ? fx_nan2() : cconj(fx_value(S2[j * PITCH + swz<fx2>(yy)], ej));
    }
}

// row pass 2: z = F_x^-1 X_x^T t; with r, the partial of r^T z per CTA in part
template <int LOGN>
__global__ void __launch_bounds__(PcgFx<LOGN>::T, PcgFx<LOGN>::MINB)
pc_row2_fx_kernel(PcgGeo g, const void* __restrict__ t_v, void* __restrict__ z_v, const void* __restrict__ r_v,
                  const int* __restrict__ active, double2* __restrict__ part)
{
    using Q = PcgFx<LOGN>;
    using F = typename Q::F;
    constexpr int N = Q::N, T = Q::T, NE = Q::E;
    const int y = blockIdx.x, e = blockIdx.y;
    if (active && !active[e]) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fx2* S = reinterpret_cast<fx2*>(smem_raw);
    fx2* Tn = S + N;
    int4* Ws = reinterpret_cast<int4*>(Tn + N);
    const PcgScr sc(Ws + Q::TWN);
    __shared__ double2 red[32];
    const int tid = threadIdx.x;
    const BarCTA bar;
    const int64_t base = (int64_t)e * g.N + (int64_t)y * N;
    const double2* __restrict__ t = reinterpret_cast<const double2*>(t_v) + base;
    double2* __restrict__ z = reinterpret_cast<double2*>(z_v) + base;
    const int4* __restrict__ W = reinterpret_cast<const int4*>(g.fWx);
    double2 d[NE];
#pragma unroll
    for (int j = 0; j < NE; ++j) d[j] = t[tid + j * T];
    for (int i = tid; i < Q::TWN; i += T) cp_async<16>(&Ws[i], &W[i]);
    cp_async_commit();
    int ed;
    bool bad;
    const int el = fx_line_exp<NE, T>(d, sc.part, sc.red, tid, bar, ed, bad) + g.pbx - 1;   // (as pc_col_fx_kernel)
#pragma unroll
    for (int j = 0; j < NE; ++j) Tn[tid + j * T] = fx_from_double(d[j], ed);
    cp_async_wait<0>();
    __syncthreads();
    const int4* __restrict__ xb = reinterpret_cast<const int4*>(g.xbx);
#pragma unroll 1
    for (int j0 = 0; j0 < NE; j0 += BAND_NJ) {
        fx2 o[BAND_NJ];
        band_rows_fx<BAND_NJ>(tid + j0 * T, T, N, g.bsx, g.bwx, xb, [&](int nu) { return Tn[nu]; }, o);
#pragma unroll
        for (int j = 0; j < BAND_NJ; ++j) S[swz<fx2>(__ldg(&g.posx[tid + (j0 + j) * T]))] = fx_conj(o[j]);
    }
    __syncthreads();
    Q::inv_first(S, tid);
    __syncthreads();
    F::inv_all(S, Ws, W, tid, bar);
    double2 acc = make_double2(0.0, 0.0);
    const double2* r = r_v ? reinterpret_cast<const double2*>(r_v) + base : nullptr;
#pragma unroll 2
    for (int j = 0; j < NE; ++j) {
        const int n = tid + j * T;
        const double2 zv = bad ? fx_nan2() : cconj(fx_value(S[swz<fx2>(n)], el));
        z[n] = zv;
        if (r) {
            const double2 rv = r[n];
            acc.x += rv.x * zv.x - rv.y * zv.y;
            acc.y += rv.x * zv.y + rv.y * zv.x;
        }
    }
    if (part) {
        const double2 s = block_sum2(acc, red);
        if (threadIdx.x == 0) part[(int64_t)e * gridDim.x + blockIdx.x] = s;
    }
}

}  // namespace soft
