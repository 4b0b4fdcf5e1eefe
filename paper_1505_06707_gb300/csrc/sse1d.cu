// Stationary ECS equation on a 1D grid (Sec. III): A psi = f with
//   A = F^-1 K F + C + U - E            (the matrix under Eq. linsys)
// by complex-symmetric CG with the FFT preconditioner of Eq. PreconFFT or
// the banded ECS preconditioner of Eq. PreconFFT_ECS,
//   P^-1 = F^-1 X^T (Lambda - E)^-1 X F.
//
// One CTA owns one energy for the whole solve: the FFT work buffer and the
// vectors x, r, p, z of that energy stay in shared memory (6 N complex128,
// 192 KB at N = 2048), so an iteration touches global memory only for the
// tables, which every CTA shares through L2.  The scalars of the iteration
// are block sums, which every thread forms alike and so takes the same
// branch; the loop ends at convergence, breakdown or maxit.
//
// FFTs and the band products run in 64-bit fixed point (pcg_fix.cuh); the
// vectors, k^2/2, the potential and strip terms, 1/(lambda - E) and the sums
// are FP64.  In FP64 throughout, an iteration took about 170 clocks of an SM
// per point, most of it in the FP64 pipe (2 instructions per clock and SM); 38
// FP64 instructions per point are left.  30 energies at N = 1024, tolerance
// 1e-12: 4.83 -> 2.17 ms, and 1.76 ms with radix 4 instead of radix 8.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "band.h"
#include "pcg_fix.cuh"
#include "plan_internal.h"

namespace soft {

struct Sse1DGeo {
    const int4* W;                     // pass twiddles
    const double* K;                   // k^2/2 in the order of the fused centre
    const double2* U;                  // U(z(x_j)), natural order
    const double2* C;                  // C[j][j-1], C[j][j], C[j][j+1] (3N)
    int nb, blk0;                      // rows of the cyclic block where C is non-zero
    const int* pos;                    // FFT output position of natural index m
    const int* bs;                     // band start of row nu
    const int* bw;                     // band width of row nu
    const int4* xf;                    // band rows of X 2^-pf (u-major, e^{i k x0} folded in)
    const int4* xb;                    // band rows of X^T 2^-pb (u-major, e^{-i k x0} folded in)
    const double2* lam;                // eigenvalues lambda_nu
    int pf, pb;
};

namespace {

__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    const double d = b.x * b.x + b.y * b.y;
    return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}

// an energy has an SM to itself and mostly waits for its own barriers, so more
// threads (N/4) of smaller butterflies are faster
constexpr int SSE1_LOGRM = 2;

// One energy's CTA: S (the FFT buffer, swizzled), T1, x, r, p, z of N complex
// each, the twiddles, scratch and two sets of warp sums
template <int LOGN>
struct Sse1 {
    using Q = PcgFx<LOGN, SSE1_LOGRM>;
    using F = typename Q::F;
    static constexpr int N = Q::N, T = Q::T, E = Q::E, NW = T / 32;
    static constexpr size_t SMEM = sizeof(fx2) * (6 * N + Q::TWN) + Q::SCR + sizeof(double2) * 2 * NW;
    static_assert(SMEM <= 227 * 1024, "shared memory");
    const Sse1DGeo& g;
    fx2 *S, *T1;
    double2 *x, *r, *p, *z;
    int4* Ws;
    PcgScr sc;
    double2* red;
    const int tid;
    const BarCTA bar;
    int par = 0;
    double2 ri[E];                     // 1/(lambda_nu - E) on the thread's rows nu = tid + j T

    __device__ __forceinline__ Sse1(const Sse1DGeo& g_, unsigned char* sm, double En, bool pc)
        : g(g_), S(reinterpret_cast<fx2*>(sm)), T1(S + N), x(reinterpret_cast<double2*>(T1 + N)), r(x + N), p(r + N),
          z(p + N), Ws(reinterpret_cast<int4*>(z + N)), sc(Ws + Q::TWN),
          red(reinterpret_cast<double2*>(reinterpret_cast<unsigned char*>(Ws + Q::TWN) + Q::SCR)), tid(threadIdx.x), bar() {
        for (int i = tid; i < Q::TWN; i += T) cp_async<16>(&Ws[i], &g.W[i]);
        cp_async_commit();
#pragma unroll
        for (int j = 0; j < E; ++j) {
            if (!pc) { ri[j] = make_double2(0.0, 0.0); continue; }
            double2 den = __ldg(&g.lam[tid + j * T]);
            den.x -= En;
            ri[j] = cscale(cconj(den), 1.0 / (den.x * den.x + den.y * den.y));
        }
        cp_async_wait<0>();
        __syncthreads();
    }

    // sum of v over the CTA in every thread; consecutive sums use the two sets in turn
    __device__ __forceinline__ double2 bsum(double2 v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        }
        if constexpr (NW == 1) return v;
        double2* s = red + par * NW;
        par ^= 1;
        if ((tid & 31) == 0) s[tid >> 5] = v;
        __syncthreads();
        v = s[tid & (NW - 1)];
#pragma unroll
        for (int o = NW / 2; o > 0; o >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        }
        return v;
    }

    // z = A p on the thread's own rows; returns the thread's part of p^T z
    __device__ __forceinline__ double2 apply_A(double En) {
        double2 d[E];
#pragma unroll
        for (int j = 0; j < E; ++j) d[j] = p[tid + j * T];
        int ed;
        bool bad;
        int el = fx_line_exp<E, T>(d, sc.part, sc.red, tid, bar, ed, bad);
#pragma unroll
        for (int j = 0; j < E; ++j) S[swz<fx2>(tid + j * T)] = fx_from_double(d[j], ed);
        __syncthreads();
        F::fwd_all(S, Ws, g.W, tid, bar);
        bool bad2;
        el += Q::center_k(S, g.K, sc, tid, bar, bad2);
        bad = bad || bad2;
        __syncthreads();
        F::inv_all(S, Ws, g.W, tid, bar);
        double2 acc = make_double2(0.0, 0.0);
#pragma unroll 2
        for (int j = 0; j < E; ++j) {
            const int n = tid + j * T;
            const double2 pv = p[n];
            double2 u = __ldg(&g.U[n]);
            u.x -= En;
            double2 v = bad ? fx_nan2() : fx_value(S[swz<fx2>(n)], el);
            v = cfma(u, pv, v);
            if (((n - g.blk0) & (N - 1)) < g.nb) {
                v = cfma(__ldg(&g.C[n]), p[(n + N - 1) & (N - 1)], v);
                v = cfma(__ldg(&g.C[N + n]), pv, v);
                v = cfma(__ldg(&g.C[2 * N + n]), p[(n + 1) & (N - 1)], v);
            }
            z[n] = v;
            acc = cfma(pv, v, acc);
        }
        return acc;
    }

    // z = P^-1 r on the thread's own rows; returns the thread's part of r^T z.
    // The paper's F has e^{+ikx}: conj(FFT(conj(.))).
    __device__ __forceinline__ double2 apply_P() {
        double2 d[E];
#pragma unroll
        for (int j = 0; j < E; ++j) d[j] = cconj(r[tid + j * T]);
        int ed;
        bool bad, bad2;
        int el = fx_line_exp<E, T>(d, sc.part, sc.red, tid, bar, ed, bad) + g.pf;
#pragma unroll
        for (int j = 0; j < E; ++j) S[swz<fx2>(tid + j * T)] = fx_from_double(d[j], ed);
        __syncthreads();
        F::fwd_all(S, Ws, g.W, tid, bar);
        Q::fwd_last(S, tid);
        __syncthreads();
#pragma unroll 2
        for (int j = 0; j < E; ++j) {                  // F r in natural index order
            const int m = tid + j * T;
            T1[m] = fx_conj(S[swz<fx2>(__ldg(&g.pos[m]))]);
        }
        __syncthreads();
#pragma unroll
        for (int j0 = 0; j0 < E; j0 += BAND_NJ) {      // X F r, then / (lambda - E)
            fx2 o[BAND_NJ];
            band_rows_fx<BAND_NJ>(tid + j0 * T, T, N, g.bs, g.bw, g.xf, [&](int m) { return T1[m]; }, o);
#pragma unroll
            for (int j = 0; j < BAND_NJ; ++j) d[j0 + j] = cmul(fx_value(o[j], el), ri[j0 + j]);
        }
        el = fx_line_exp<E, T>(d, sc.part, sc.red, tid, bar, ed, bad2) + g.pb - 1;    // (-1: as pc_col_fx_kernel)
        bad = bad || bad2;
        fx2* zf = reinterpret_cast<fx2*>(z);
#pragma unroll
        for (int j = 0; j < E; ++j) zf[tid + j * T] = fx_from_double(d[j], ed);
        __syncthreads();
#pragma unroll 1
        for (int j0 = 0; j0 < E; j0 += BAND_NJ) {      // X^T into the FFT positions (conjugated)
            fx2 o[BAND_NJ];
            band_rows_fx<BAND_NJ>(tid + j0 * T, T, N, g.bs, g.bw, g.xb, [&](int nu) { return zf[nu]; }, o);
#pragma unroll
            for (int j = 0; j < BAND_NJ; ++j) S[swz<fx2>(__ldg(&g.pos[tid + (j0 + j) * T]))] = fx_conj(o[j]);
        }
        __syncthreads();
        Q::inv_first(S, tid);
        __syncthreads();
        F::inv_all(S, Ws, g.W, tid, bar);
        double2 acc = make_double2(0.0, 0.0);
#pragma unroll 2
        for (int j = 0; j < E; ++j) {
            const int n = tid + j * T;
            const double2 zv = bad ? fx_nan2() : cconj(fx_value(S[swz<fx2>(n)], el));
            z[n] = zv;
            acc = cfma(r[n], zv, acc);
        }
        return acc;
    }
};

// COCG (Sec. III after Eq. linsys: the bilinear r^T z replaces the inner
// product), x0 = 0, stop when ||r||_2/||f||_2 < tol; energy blockIdx.x
template <int LOGN>
__global__ void __launch_bounds__(Sse1<LOGN>::T, 1)
sse1d_cocg_kernel(Sse1DGeo g, const double2* __restrict__ f, double2* __restrict__ xout,
                  const double* __restrict__ Es, double tol, int maxit, int* __restrict__ iters,
                  double* __restrict__ relres, int* __restrict__ status)
{
    using Q = Sse1<LOGN>;
    constexpr int N = Q::N, T = Q::T, E_ = Q::E;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int e = blockIdx.x, tid = threadIdx.x;
    const double En = Es[e];
    Q q(g, smem_raw, En, true);
    double2 *x = q.x, *r = q.r, *p = q.p, *z = q.z;
    double ff = 0.0;
    for (int j = 0; j < E_; ++j) {
        const int n = tid + j * T;
        const double2 fv = f[n];
        r[n] = fv;
        x[n] = make_double2(0.0, 0.0);
        p[n] = make_double2(0.0, 0.0);
        ff += fv.x * fv.x + fv.y * fv.y;
    }
    ff = q.bsum(make_double2(ff, 0.0)).x;
    int st = SOFT_ERR_NOT_CONVERGED, it = 0;
    double rel = 1.0;
    if (!(ff > 0.0) || !isfinite(ff)) {
        st = ff == 0.0 ? SOFT_OK : SOFT_ERR_NONFINITE;
        rel = 0.0;
    } else {
        double2 rho = make_double2(0.0, 0.0);
#pragma unroll 1
        for (;;) {
            const double2 rn = q.bsum(q.apply_P());                   // r^T z
            double2 be = make_double2(0.0, 0.0);
            if (it > 0) {
                if (!(rho.x * rho.x + rho.y * rho.y > 0.0)) { st = SOFT_ERR_BREAKDOWN; break; }
                be = cdiv(rn, rho);
            }
            rho = rn;
            if (it >= maxit) break;
#pragma unroll 2
            for (int j = 0; j < E_; ++j) {
                const int n = tid + j * T;
                p[n] = cfma(be, p[n], z[n]);
            }
            __syncthreads();
            const double2 pw = q.bsum(q.apply_A(En));                 // z = w = A p
            if (!(pw.x * pw.x + pw.y * pw.y > 0.0)) { st = SOFT_ERR_BREAKDOWN; break; }
            const double2 al = cdiv(rho, pw), nal = make_double2(-al.x, -al.y);
            double rr = 0.0;
#pragma unroll 2
            for (int j = 0; j < E_; ++j) {
                const int n = tid + j * T;
                x[n] = cfma(al, p[n], x[n]);
                const double2 rv = cfma(nal, z[n], r[n]);
                r[n] = rv;
                rr += rv.x * rv.x + rv.y * rv.y;
            }
            rr = q.bsum(make_double2(rr, 0.0)).x;
            ++it;
            rel = sqrt(rr / ff);
            if (!isfinite(rel)) { st = SOFT_ERR_NONFINITE; break; }
            if (rel < tol) { st = SOFT_OK; break; }
        }
    }
    for (int j = 0; j < E_; ++j) {
        const int n = tid + j * T;
        xout[(int64_t)e * N + n] = x[n];
    }
    if (tid == 0) {
        iters[e] = it;
        relres[e] = rel;
        status[e] = st;
    }
}

// one application: what = 0: y = A x; 1: y = P^-1 x
template <int LOGN>
__global__ void __launch_bounds__(Sse1<LOGN>::T, 1)
sse1d_apply_kernel(Sse1DGeo g, const double2* __restrict__ in, double2* __restrict__ out, double En, int what)
{
    using Q = Sse1<LOGN>;
    constexpr int T = Q::T, E_ = Q::E;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x;
    Q q(g, smem_raw, En, what != 0);
    double2* a = what == 0 ? q.p : q.r;
    for (int j = 0; j < E_; ++j) a[tid + j * T] = in[tid + j * T];
    __syncthreads();
    if (what == 0) q.apply_A(En);
    else q.apply_P();
    for (int j = 0; j < E_; ++j) out[tid + j * T] = q.z[tid + j * T];
}

template <int LOGN>
int launch_t(const Sse1DGeo& g, int mode, const double2* in, double2* out, const double* dE, double En, int nE,
             double tol, int maxit, int* iters, double* relres, int* status, cudaStream_t st) {
    using Q = Sse1<LOGN>;
    const int smem = (int)Q::SMEM;
    if (mode == 0) {
        auto k = sse1d_cocg_kernel<LOGN>;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
            return SOFT_ERR_CUDA;
        if (nE > 0) k<<<nE, Q::T, smem, st>>>(g, in, out, dE, tol, maxit, iters, relres, status);
    } else {
        auto k = sse1d_apply_kernel<LOGN>;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
            return SOFT_ERR_CUDA;
        k<<<1, Q::T, smem, st>>>(g, in, out, En, mode - 1);
    }
    return cudaGetLastError() == cudaSuccess ? SOFT_OK : SOFT_ERR_CUDA;
}

int launch(int logn, const Sse1DGeo& g, int mode, const double2* in, double2* out, const double* dE, double En,
           int nE, double tol, int maxit, int* iters, double* relres, int* status, cudaStream_t st) {
    switch (logn) {
    case 8: return launch_t<8>(g, mode, in, out, dE, En, nE, tol, maxit, iters, relres, status, st);
    case 9: return launch_t<9>(g, mode, in, out, dE, En, nE, tol, maxit, iters, relres, status, st);
    case 10: return launch_t<10>(g, mode, in, out, dE, En, nE, tol, maxit, iters, relres, status, st);
    case 11: return launch_t<11>(g, mode, in, out, dE, En, nE, tol, maxit, iters, relres, status, st);
    }
    return SOFT_ERR_UNSUPPORTED;
}

}  // namespace

// Per-plan tables of the 1D solver, built on first use.
struct Sse1D {
    int logn = 0, n = 0;
    void *W = nullptr, *K = nullptr, *U = nullptr, *C = nullptr, *pos = nullptr;
    void* pc[2][5] = {};               // per preconditioner: bs, bw, xf, xb, lam
    double* dE = nullptr;
    int* iters = nullptr;
    double* relres = nullptr;
    int* status = nullptr;
    int cap = 0;
    Sse1DGeo geo[2] = {};
    ~Sse1D() {
        cudaFree(W); cudaFree(K); cudaFree(U); cudaFree(C); cudaFree(pos);
        for (auto& t : pc)
            for (void* b : t) cudaFree(b);
        cudaFree(dE); cudaFree(iters); cudaFree(relres); cudaFree(status);
    }
};

void sse1d_free(Sse1D* s) { delete s; }

static int upload_int(void** dst, const std::vector<int>& v) {
    return upload(dst, v.data(), v.size() * sizeof(int));
}

static int build(soft_plan* P) {
    if (P->s1) return SOFT_OK;
    const Tables1D& TB = *P->tabs[0];
    std::unique_ptr<Sse1D> S(new Sse1D());
    S->n = TB.ax.n;
    S->logn = TB.logn;
    if (S->logn < 8 || S->logn > 11) return SOFT_ERR_UNSUPPORTED;
    const Axis1D& A = TB.ax;
    const int n = S->n;
    int rc;
    if ((rc = upload_i32(&S->W, pass_twiddles_fx(S->logn, SSE1_LOGRM, FXFULL_MAXS)))) return rc;
    if ((rc = upload_ksq(&S->K, A, S->logn, SSE1_LOGRM))) return rc;
    const std::vector<int> perm = dif_output_order(S->logn, SSE1_LOGRM);
    std::vector<int> pos(n);
    for (int q = 0; q < n; ++q) pos[perm[q]] = q;
    if ((rc = upload_int(&S->pos, pos))) return rc;
    if ((rc = upload_c(&S->U, TB.U0, SOFT_C128))) return rc;
    std::vector<cd> c = A.Cs;
    c.insert(c.end(), A.Cd.begin(), A.Cd.end());
    c.insert(c.end(), A.Cu.begin(), A.Cu.end());
    if ((rc = upload_c(&S->C, c, SOFT_C128))) return rc;
    for (int type = 0; type < 2; ++type) {
        BandAxis B;
        double chk = 0;
        if ((rc = build_band_axis(A, P->opt.band_width, type == 0, B, &chk))) return rc;
        void** t = S->pc[type];
        if ((rc = upload_int(&t[0], B.start))) return rc;
        if ((rc = upload_int(&t[1], B.width))) return rc;
        Sse1DGeo& g = S->geo[type];
        if ((rc = upload_band_fx(&t[2], B, B.xf, S->logn, SSE1_LOGRM, false, &g.pf))) return rc;
        if ((rc = upload_band_fx(&t[3], B, B.xb, S->logn, SSE1_LOGRM, true, &g.pb))) return rc;
        if ((rc = upload_c(&t[4], B.lam, SOFT_C128))) return rc;
        g.W = (const int4*)S->W; g.K = (const double*)S->K; g.U = (const double2*)S->U;
        g.C = (const double2*)S->C; g.nb = TB.nb; g.blk0 = TB.blk0; g.pos = (const int*)S->pos;
        g.bs = (const int*)t[0]; g.bw = (const int*)t[1]; g.xf = (const int4*)t[2];
        g.xb = (const int4*)t[3]; g.lam = (const double2*)t[4];
    }
    P->s1 = S.release();
    return SOFT_OK;
}

static bool usable(const soft_plan* P) {
    return P && P->kind == 1 && P->single && P->tabs.size() == 1;
}

int sse1d_refill_potential(soft_plan* P) {
    if (!P->s1) return SOFT_OK;
    return refill_c(P->s1->U, P->tabs[0]->U0, SOFT_C128);
}

int sse1d_solve(soft_plan* P, const double* E, int nE, const void* rhs, void* psi_out, double tol, int maxit,
                int precond, int* iters_out, double* relres_out, cudaStream_t st) {
    if (!usable(P)) return SOFT_ERR_INVALID_ARG;
    if (precond != 0 && precond != 1) return SOFT_ERR_UNSUPPORTED;
    if (P->prec != SOFT_C128) return SOFT_ERR_UNSUPPORTED;
    int rc = build(P);
    if (rc) return rc;
    Sse1D* S = P->s1;
    if (S->cap < nE) {
        cudaFree(S->dE); cudaFree(S->iters); cudaFree(S->relres); cudaFree(S->status);
        S->dE = nullptr; S->iters = nullptr; S->relres = nullptr; S->status = nullptr; S->cap = 0;
        if ((rc = cuda_status(cudaMalloc((void**)&S->dE, sizeof(double) * nE)))) return rc;
        if ((rc = cuda_status(cudaMalloc((void**)&S->iters, sizeof(int) * nE)))) return rc;
        if ((rc = cuda_status(cudaMalloc((void**)&S->relres, sizeof(double) * nE)))) return rc;
        if ((rc = cuda_status(cudaMalloc((void**)&S->status, sizeof(int) * nE)))) return rc;
        S->cap = nE;
    }
    // pageable source: staged before cudaMemcpyAsync returns
    if ((rc = cuda_status(cudaMemcpyAsync(S->dE, E, sizeof(double) * nE, cudaMemcpyHostToDevice, st)))) return rc;
    if ((rc = launch(S->logn, S->geo[precond], 0, (const double2*)rhs, (double2*)psi_out, S->dE, 0.0, nE, tol,
                     maxit, S->iters, S->relres, S->status, st)))
        return rc;
    P->last_launches = 1;
    std::vector<int> it(nE), stt(nE);
    std::vector<double> rr(nE);
    if ((rc = cuda_status(cudaMemcpyAsync(it.data(), S->iters, sizeof(int) * nE, cudaMemcpyDeviceToHost, st)))) return rc;
    if ((rc = cuda_status(cudaMemcpyAsync(rr.data(), S->relres, sizeof(double) * nE, cudaMemcpyDeviceToHost, st)))) return rc;
    if ((rc = cuda_status(cudaMemcpyAsync(stt.data(), S->status, sizeof(int) * nE, cudaMemcpyDeviceToHost, st)))) return rc;
    if ((rc = cuda_status(cudaStreamSynchronize(st)))) return rc;
    if (iters_out) std::memcpy(iters_out, it.data(), sizeof(int) * nE);
    if (relres_out) std::memcpy(relres_out, rr.data(), sizeof(double) * nE);
    int out = SOFT_OK;
    for (int e = 0; e < nE; ++e) {
        if (stt[e] == SOFT_ERR_BREAKDOWN || stt[e] == SOFT_ERR_NONFINITE) return stt[e];
        if (stt[e] != SOFT_OK) out = SOFT_ERR_NOT_CONVERGED;
    }
    return out;
}

int sse1d_apply(soft_plan* P, double E, int what, int precond, const void* x, void* y, cudaStream_t st) {
    if (!usable(P)) return SOFT_ERR_INVALID_ARG;
    if (what == 1 && precond != 0 && precond != 1) return SOFT_ERR_UNSUPPORTED;
    if (P->prec != SOFT_C128) return SOFT_ERR_UNSUPPORTED;
    int rc = build(P);
    if (rc) return rc;
    Sse1D* S = P->s1;
    P->last_launches = 1;
    return launch(S->logn, S->geo[what == 1 ? precond : 0], what == 0 ? 1 : 2, (const double2*)x, (double2*)y,
                  nullptr, E, 1, 0.0, 0, nullptr, nullptr, nullptr, st);
}

}  // namespace soft
