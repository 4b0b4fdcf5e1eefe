// C ABI of the library: plan construction (host FP64 tables, uploaded once)
// and the 1D step / observables entry points.  The 2D and stationary entry
// points live in plan2d.cu.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <thread>
#include <tuple>

#include "fix64_host.h"
#include "nn.h"
#include "plan_internal.h"

using namespace soft;

namespace soft {

int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return SOFT_OK;
    if (e == cudaErrorMemoryAllocation) return SOFT_ERR_OOM;
    return SOFT_ERR_CUDA;
}

int upload(void** dst, const void* src, size_t bytes) {
    if (bytes == 0) { *dst = nullptr; return SOFT_OK; }
    cudaError_t e = cudaMalloc(dst, bytes);
    if (e != cudaSuccess) { *dst = nullptr; return cuda_status(e); }
    e = cudaMemcpy(*dst, src, bytes, cudaMemcpyHostToDevice);
    return cuda_status(e);
}

// phase table: double2 for complex128 plans; (hi, lo) float4 for complex64 plans
int upload_tab(void** dst, const std::vector<cd>& v, int prec) {
    if (prec == SOFT_C128) return upload_c(dst, v, prec);
    std::vector<float> buf(4 * v.size());
    for (size_t i = 0; i < v.size(); ++i) {
        const float hr = (float)v[i].real(), hi = (float)v[i].imag();
        buf[4 * i] = hr;
        buf[4 * i + 1] = hi;
        buf[4 * i + 2] = (float)(v[i].real() - (double)hr);
        buf[4 * i + 3] = (float)(v[i].imag() - (double)hi);
    }
    return upload(dst, buf.data(), buf.size() * sizeof(float));
}

// potential factor table: the factor itself (double2) for complex128 plans;
// its difference from 1 (float2) for complex64 plans
int upload_vtab(void** dst, const std::vector<cd>& v, int prec) {
    if (prec == SOFT_C128) return upload_c(dst, v, prec);
    std::vector<float> buf(2 * v.size());
    for (size_t i = 0; i < v.size(); ++i) {
        buf[2 * i] = (float)(v[i].real() - 1.0);
        buf[2 * i + 1] = (float)v[i].imag();
    }
    return upload(dst, buf.data(), buf.size() * sizeof(float));
}

// round a complex FP64 vector to the plan precision and upload it
int upload_c(void** dst, const std::vector<cd>& v, int prec) {
    if (prec == SOFT_C128) {
        std::vector<double> buf(2 * v.size());
        for (size_t i = 0; i < v.size(); ++i) { buf[2 * i] = v[i].real(); buf[2 * i + 1] = v[i].imag(); }
        return upload(dst, buf.data(), buf.size() * sizeof(double));
    }
    std::vector<float> buf(2 * v.size());
    for (size_t i = 0; i < v.size(); ++i) {
        buf[2 * i] = (float)v[i].real();
        buf[2 * i + 1] = (float)v[i].imag();
    }
    return upload(dst, buf.data(), buf.size() * sizeof(float));
}

// FFT twiddle table (unit-modulus values): complex128 as is; complex64 with
// each value rounded to the FP32 pair, within one ulp of (cos, sin) per
// component, whose modulus is closest to 1.  The forward and inverse passes
// use the same table (conjugated), so their phase roundings cancel and what
// repeats every step is the modulus error; choosing the pair this way cuts
// the complex64 drift per step by about 40 %.
int upload_tw(void** dst, const std::vector<cd>& v, int prec) {
    if (prec == SOFT_C128) return upload_c(dst, v, prec);
    std::vector<float> buf(2 * v.size());
    for (size_t i = 0; i < v.size(); ++i) {
        const double c = v[i].real(), s = v[i].imag();
        const float c0 = (float)c, s0 = (float)s;
        float bc = c0, bs = s0;
        double be = 1e300, bd = 1e300;
        for (int dc = -1; dc <= 1; ++dc)
            for (int ds = -1; ds <= 1; ++ds) {
                const float cc = dc ? std::nextafter(c0, dc > 0 ? 2.0f : -2.0f) : c0;
                const float ss = ds ? std::nextafter(s0, ds > 0 ? 2.0f : -2.0f) : s0;
                const double e = std::fabs((double)cc * cc + (double)ss * ss - 1.0);
                const double d = std::fabs(cc - c) + std::fabs(ss - s);
                if (e < be || (e == be && d < bd)) { be = e; bd = d; bc = cc; bs = ss; }
            }
        buf[2 * i] = bc;
        buf[2 * i + 1] = bs;
    }
    return upload(dst, buf.data(), buf.size() * sizeof(float));
}

// Twiddle bases of the 1D step kernel: complex128 as is; complex64 as
// compensated float4 (hi.re, hi.im, lo.re, lo.im), hi + lo = the FP64 value
// to ~2^-48 (the kernel applies them by compensated multiplies, see
// soft1d.cuh)
int upload_tw_comp(void** dst, const std::vector<cd>& v, int prec) {
    return upload_tab(dst, v, prec);
}

static double modulus(cd v) { return std::sqrt(std::norm(v)); }      // (std::abs guards against overflow, slowly)
static void fx_fill(int32_t* out, const std::vector<cd>& v, double scale) {
    for (size_t i = 0; i < v.size(); ++i) {
        fx_halves_host(std::llrint(v[i].real() * scale * 0x1p62), out + 4 * i);
        fx_halves_host(std::llrint(v[i].imag() * scale * 0x1p62), out + 4 * i + 2);
    }
}
int upload_fx(void** dst, const std::vector<cd>& v) {
    std::vector<int32_t> buf(4 * v.size());
    fx_fill(buf.data(), v, 1.0);
    return upload(dst, buf.data(), buf.size() * sizeof(int32_t));
}

int upload_fx_phases(void** dst, const std::vector<double>& ph, int half) {
    std::vector<int32_t> buf(4 * ph.size());
    auto sc = [&](int64_t w) { return half == 0 ? w : half > 0 ? fx_sqrt2_host(w) : (fx_sqrt2_host(w) + 1) >> 1; };
    host_parallel((int64_t)ph.size(), [&](int64_t b, int64_t e) {
        for (int64_t i = b; i < e; ++i) {
            int64_t c, s;
            fx_cis_host(fx_turns_host(ph[i]), &c, &s);
            fx_halves_host(sc(c), &buf[4 * i]);
            fx_halves_host(sc(s), &buf[4 * i + 2]);
        }
    });
    return upload(dst, buf.data(), buf.size() * sizeof(int32_t));
}

// the factor e^{lv} 2^-p, times sqrt(2) if s2
static void fx_put_factor(int32_t* out, cd lv, int p, bool s2) {
    int64_t c, s;
    fx_cis_host(fx_turns_host(lv.imag()), &c, &s);
    const int64_t mod = std::llrint(std::exp(lv.real()) * (p ? 0x1p60 : 0x1p61));
    c = (int64_t)(((__int128)c * mod + (1LL << 60)) >> 61);
    s = (int64_t)(((__int128)s * mod + (1LL << 60)) >> 61);
    fx_halves_host(s2 ? fx_sqrt2_host(c) : c, out);
    fx_halves_host(s2 ? fx_sqrt2_host(s) : s, out + 2);
}
// largest real part of the logarithms, the same with those of the nb rows from
// blk0 on doubled (factors that enter twice per step), and whether all are finite
struct LogRange { double gain, keep; bool finite; };
static LogRange log_range(const std::vector<cd>& lv, int64_t blk0 = 0, int64_t nb = 0) {
    const int64_t n = (int64_t)lv.size();
    LogRange R{-HUGE_VAL, -HUGE_VAL, true};
    std::mutex mx;
    host_parallel(n, [&](int64_t b, int64_t e) {
        LogRange r{-HUGE_VAL, -HUGE_VAL, true};
        for (int64_t i = b; i < e; ++i) {
            const double x = lv[i].real();
            const int64_t j = i < blk0 ? i - blk0 + n : i - blk0;
            r.finite = r.finite && std::isfinite(x) && std::isfinite(lv[i].imag());
            r.gain = std::max(r.gain, x);
            r.keep = std::max(r.keep, j < nb ? 2.0 * x : x);
        }
        std::lock_guard<std::mutex> l(mx);
        R.finite = R.finite && r.finite;
        R.gain = std::max(R.gain, r.gain);
        R.keep = std::max(R.keep, r.keep);
    }, 1 << 17);
    return R;
}
// Factors e^{lv} that are applied in FP64: a gain above 2, a non-finite one, or
// a loss to less than 1/8 at every point.  Products round to 2^-62 of the line's
// norm before them, 2^-55 in all at 16384 samples, so a loss that spares no
// point would take its bits from the result (a uniform e^-14 per step: 1.2e-10
// off after 3 steps at 16384 samples; e^-60: nothing left).  Where some points
// keep a factor near 1, the FFTs' rounding (2e-16 of the norm, at every point)
// passes there, in FP64 too.
static bool fx_gen_factors(const LogRange& r) {
    return !r.finite || std::exp(r.gain) > 2.0 || std::exp(r.keep) < 0.125;
}
// potential table of the fixed-point step (soft1d_fix.cuh, FxV) from the
// factors' logarithms: the factors times 2^-p, p = 0 (|v| <= 1.01) or 1 (<= 2),
// and sqrt(2) if s2 (the last inverse pass's share), then the entry
// (p, gen, 0, 0) and, for plans with gen, the factors as double2 instead
static std::vector<int32_t> fxv_table(const std::vector<cd>& lv, bool gen, bool s2) {
    const size_t n = lv.size();
    std::vector<int32_t> buf(8 * n + 4, 0);
    const int p = !gen && std::exp(log_range(lv).gain) > 1.01 ? 1 : 0;
    host_parallel((int64_t)n, [&](int64_t b, int64_t e) {
        for (int64_t i = b; i < e; ++i) {
            if (gen) {
                const cd v = std::exp(lv[i]);
                std::memcpy(buf.data() + 4 * n + 4 + 4 * i, &v, 16);
            } else {
                fx_put_factor(&buf[4 * i], lv[i], p, s2);
            }
        }
    });
    buf[4 * n] = p;
    buf[4 * n + 1] = gen;
    return buf;
}

// Chunked strip solve for thr threads of ch = ceil(nb/thr) rows (thread t: rows
// t ch + c): multipliers mf and g in chunk order (c thr + t), and for the
// forward and backward scans over the chunks the products of the chunk totals
// (soft1d_fix.cuh, FxCn) with the numbers of warp-scan rounds and of warps
// that still reach, where products below tiny count as zero.
struct StripScan {
    std::vector<cd> m, g, scan[2];
    int rounds[2], span[2];
};
static StripScan strip_scan(const std::vector<cd>& mf, const std::vector<cd>& g, int nb, int thr, double tiny) {
    const int ch = (nb + thr - 1) / thr, nw = thr / 32;
    StripScan Q;
    Q.m.assign((size_t)(ch + 1) * thr, 0.0);
    Q.g.assign((size_t)ch * thr, 0.0);
    std::vector<cd> &m = Q.m, &gg = Q.g;
    for (int t = 0; t < thr; ++t)
        for (int c = 0; c <= ch; ++c) {
            const int i = t * ch + c;
            if (i < nb) m[(size_t)c * thr + t] = mf[i];
            if (c < ch && i < nb) gg[(size_t)c * thr + t] = g[i];
        }
    for (int d = 0; d < 2; ++d) {
        std::vector<cd> tot(thr, 0.0);           // (0: chunks without rows, which carry nothing)
        for (int t = 0; t < thr; ++t) {
            if (t * ch < nb) tot[t] = 1.0;
            for (int c = 0; c < ch && t * ch + c < nb; ++c) tot[t] *= m[(size_t)(c + d) * thr + t];
        }
        std::vector<cd>& s = Q.scan[d];
        s.assign((size_t)6 * thr + nw, 1.0);
        std::vector<cd> prod = tot;              // of the 2^r totals ending (starting) at t
        Q.rounds[d] = 0;
        for (int r = 0; r < 5; ++r) {
            const int D = 1 << r;
            double big = 0.0;
            for (int t = 0; t < thr; ++t) {
                s[(size_t)r * thr + t] = prod[t];
                const int l = t & 31;
                if (d ? l + D < 32 : l >= D) big = std::max(big, modulus(prod[t]));
            }
            if (!(big <= tiny)) Q.rounds[d] = r + 1;
            std::vector<cd> nx = prod;
            for (int t = 0; t < thr; ++t) {
                const int o = d ? t + D : t - D;
                if (o >= 0 && o < thr) nx[t] = prod[t] * prod[o];
            }
            prod = nx;
        }
        for (int w = 0; w < nw; ++w) {
            cd p = 1.0;
            for (int l = 0; l < 32; ++l) {
                const int t = 32 * w + (d ? 31 - l : l);
                s[(size_t)5 * thr + t] = p;
                p *= tot[t];
            }
            s[(size_t)6 * thr + w] = p;
        }
        Q.span[d] = nw;                            // warps whose totals still reach
        for (int k = 1; k < nw; ++k) {
            double big = 0.0;
            for (int w = 0; w + k <= nw; ++w) {
                cd p = 1.0;
                for (int q = 0; q < k; ++q) p *= s[(size_t)6 * thr + w + q];
                big = std::max(big, modulus(p));
            }
            if (big <= tiny) { Q.span[d] = k; break; }
        }
    }
    return Q;
}
// the tables of a complex64 strip solve (soft1d.cuh, strip_cn); cnr: rounds of
// the forward and backward scans (4 bits each), their spans (8 bits each), also
// the first two entries
std::vector<cd> strip_tables_c(const std::vector<cd>& mf, const std::vector<cd>& g, int nb, int thr, int* cnr) {
    const StripScan Q = strip_scan(mf, g, nb, thr, 0x1p-40);
    *cnr = Q.rounds[0] | Q.rounds[1] << 4 | Q.span[0] << 8 | Q.span[1] << 16;
    std::vector<cd> t = {cd(Q.rounds[0], Q.rounds[1]), cd(Q.span[0], Q.span[1])};
    for (const std::vector<cd>* v : {&Q.m, &Q.g, &Q.scan[0], &Q.scan[1]}) t.insert(t.end(), v->begin(), v->end());
    return t;
}

// Strip tables of the fixed-point step (soft1d_fix.cuh, FxCn) from the LU of
// the block: thr threads of ch rows each.  gen: a multiplier above 1, a g
// above 1.9 (its halves still fit, and the rows it scales are below 2^59.5)
// or a growth of the sweeps above 2^10; the kernel then solves in FP64.
std::vector<int32_t> strip_tables_fx(const std::vector<cd>& mf, const std::vector<cd>& mb,
                                            const std::vector<cd>& g, int nb, int thr, bool* gen) {
    double grow = 1.0, gy = 0.0;
    std::vector<double> y(nb);
    *gen = false;
    for (int i = 0; i < nb; ++i) {
        gy = modulus(mf[i]) * gy + 1.0;
        y[i] = gy;
        grow = std::max(grow, gy);
        if (!(modulus(mf[i]) <= 1.0 + 1e-12 && modulus(g[i]) <= 1.9)) *gen = true;
    }
    double gx = 0.0;
    for (int i = nb - 1; i >= 0; --i) {
        gx = modulus(mb[i]) * gx + modulus(g[i]) * y[i];
        grow = std::max(grow, gx);
    }
    const int lg = (int)std::ceil(std::log2(grow));
    if (!(lg >= 0 && lg <= 10)) *gen = true;
    const StripScan Q = strip_scan(mf, g, nb, thr, 0x1p-70);
    const std::vector<cd> &m = Q.m, &gg = Q.g;
    const size_t nf = m.size() + gg.size() + Q.scan[0].size() + Q.scan[1].size();
    std::vector<int32_t> buf(4 + 4 * (nf + m.size() + gg.size()), 0);
    buf[0] = *gen ? 0 : lg;
    buf[1] = Q.rounds[0];
    buf[2] = Q.rounds[1];
    buf[3] = Q.span[0] | Q.span[1] << 16;
    if (!*gen) {
        int32_t* f = buf.data() + 4;
        for (const std::vector<cd>* v : {&m, &gg, &Q.scan[0], &Q.scan[1]}) {
            fx_fill(f, *v, 1.0);
            f += 4 * v->size();
        }
    }
    std::memcpy(buf.data() + 4 + 4 * nf, m.data(), 16 * m.size());
    std::memcpy(buf.data() + 4 + 4 * (nf + m.size()), gg.data(), 16 * gg.size());
    return buf;
}

int upload_i32(void** dst, const std::vector<int32_t>& v) { return upload(dst, v.data(), v.size() * 4); }

void host_parallel(int64_t n, const std::function<void(int64_t, int64_t)>& fn, int64_t grain) {
    if (n < 2 * grain) return fn(0, n);
    static const int64_t cores = std::thread::hardware_concurrency();      // (the query reads a file)
    const int64_t nt = std::max<int64_t>(1, std::min<int64_t>({cores, 32, n / grain}));
    std::vector<std::thread> pool;
    int64_t done = 0;              // handed to threads; the rest runs here
    try {
        for (int64_t t = 0; t + 1 < nt; ++t) {
            const int64_t b = n * t / nt, e = n * (t + 1) / nt;
            pool.emplace_back([&fn, b, e] { fn(b, e); });
            done = e;
        }
    } catch (...) {                // no thread could be started: no exception crosses the C ABI
    }
    if (done < n) fn(done, n);
    for (auto& th : pool) th.join();
}

// FxMeta of soft2d_fix.cuh
struct FxMetaHost { int p, gen; const void* d; };
static int fx_potential_fill(FxPotential& P, const std::vector<cd>& lv) {
    const int64_t n = (int64_t)lv.size();
    const LogRange r = log_range(lv);
    FxMetaHost h{0, P.cn_gen || fx_gen_factors(r), nullptr};
    h.p = !h.gen && std::exp(r.gain) > 1.01;
    const std::unique_ptr<int32_t[]> buf(new int32_t[4 * (size_t)n]);      // (pages first touched by the threads)
    host_parallel(n, [&](int64_t b, int64_t e) {
        for (int64_t i = b; i < e; ++i) {
            if (h.gen) {
                const cd v = std::exp(lv[i]);
                std::memcpy(&buf[4 * i], &v, 16);
                continue;
            }
            fx_put_factor(&buf[4 * i], lv[i], h.p, false);
        }
    });
    // gen plans read the same buffer as double2
    if (h.gen) h.d = P.tab;
    int rc = cuda_status(cudaMemcpy(P.tab, buf.get(), 16 * (size_t)n, cudaMemcpyHostToDevice));
    return rc ? rc : cuda_status(cudaMemcpy(P.meta, &h, sizeof(h), cudaMemcpyHostToDevice));
}
int FxPotential::build(const std::vector<cd>& lv) {
    int rc = cuda_status(cudaMalloc(&tab, 16 * lv.size()));
    if (rc) { tab = nullptr; return rc; }
    if ((rc = cuda_status(cudaMalloc(&meta, sizeof(FxMetaHost))))) { meta = nullptr; return rc; }
    return fx_potential_fill(*this, lv);
}
int FxPotential::refill(const std::vector<cd>& lv) { return fx_potential_fill(*this, lv); }
FxPotential::~FxPotential() { cudaFree(tab); cudaFree(meta); }

// the upload_* conversions into a temporary device buffer, then one copy
// into dst
static int refill_with(int (*up)(void**, const std::vector<cd>&, int), void* dst,
                       const std::vector<cd>& v, int prec) {
    if (v.empty()) return SOFT_OK;
    const size_t bytes = v.size() * (prec == SOFT_C128 ? 16 : 8);
    void* tmp = nullptr;
    int rc = up(&tmp, v, prec);
    if (rc == SOFT_OK) rc = cuda_status(cudaMemcpy(dst, tmp, bytes, cudaMemcpyDeviceToDevice));
    cudaFree(tmp);
    return rc;
}
int refill_c(void* dst, const std::vector<cd>& v, int prec) { return refill_with(upload_c, dst, v, prec); }
int refill_vtab(void* dst, const std::vector<cd>& v, int prec) { return refill_with(upload_vtab, dst, v, prec); }

// Logarithms of the potential factors of one step from U0 (Sec. II, the
// scheme after Eq. C_FD): e^{tv[j]} = e^{-iU0 tau} off the strip block (both
// half factors merged), e^{-iU0 tau/2} on it (the strip CN sits between the
// halves); tvs holds the block rows' in the chunk layout of the strip CN
// (thread t of the n >> loge threads owns rows t*ch .. t*ch + ch - 1, entry
// c*T + t).
static void potential_logs_1d(const Tables1D& T, int n, double tau, std::vector<cd>& tv, std::vector<cd>& tvs) {
    tv.resize(n);
    for (int j = 0; j < n; ++j) {
        const bool inblk = ((j - T.blk0 + n) % n) < T.nb;
        tv[j] = cd(0.0, -1.0) * T.U0[j] * tau * (inblk ? 0.5 : 1.0);
    }
    tvs.clear();
    if (T.nb > 0) {
        const int thr = n >> T.loge, nb = T.nb;
        const int ch = (nb + thr - 1) / thr;
        tvs.assign((size_t)ch * thr, 0.0);
        for (int t = 0; t < thr; ++t)
            for (int c = 0; c < ch; ++c) {
                const int i = t * ch + c;
                if (i < nb) tvs[(size_t)c * thr + t] = tv[(T.blk0 + i) % n];
            }
    }
}
static std::vector<cd> vexp(std::vector<cd> v) {
    for (cd& x : v) x = std::exp(x);
    return v;
}

static int ilog2(int64_t n) {
    int l = 0;
    while ((int64_t(1) << l) < n) ++l;
    return (int64_t(1) << l) == n ? l : -1;
}

static void free_tables(Tables1D* t) {
    cudaFree(t->TK); cudaFree(t->TKh); cudaFree(t->TV); cudaFree(t->W); cudaFree(t->cn);
    cudaFree(t->TVs);
}

// Build (host FP64) and upload the tables of one 1D problem.
int make_tables_1d(Tables1D* T, int n, double a, double b, double R0, double theta, double tau,
                   const soft_options& o, int loge, int logrm) {
    const int logn = ilog2(n);
    T->prec = o.prec; T->logn = logn; T->loge = loge; T->logrm = logrm;
    T->R0 = R0; T->theta = theta;
    ContourFn cf(o.contour, R0, b, theta, o.tfecs_alpha, o.cap_energy, o.tfap_kmin);
    build_axis(T->ax, n, a, b, cf, tau);
    const Axis1D& A = T->ax;
    int rc = find_block(A, &T->blk0, &T->nb);
    if (rc) return rc;
    T->iL = 0; T->iR = 0;
    for (int j = 0; j < n; ++j) {
        if (A.x[j] <= -R0) T->iL = j + 1;
        if (A.x[j] < R0) T->iR = j + 1;
    }
    T->U0.resize(n);
    T->Uabs.resize(n);
    for (int j = 0; j < n; ++j) {
        T->Uabs[j] = cf.absorber(A.x[j]);
        T->U0[j] = soft_coulomb(&A.z[j], 1, o.soft_a2, o.charge) + T->Uabs[j];
    }
    // kinetic tables in the forward FFT's output order, 1/N folded in
    // (complex128: the fixed-point passes carry the 1/N)
    const std::vector<int> perm = dif_output_order(logn, logrm);
    std::vector<cd> tv, tvs;
    std::vector<double> ph(n), phh(n);        // their phases
    const std::vector<cd> w = o.prec == SOFT_C64 ? pass_twiddles(logn, logrm) : std::vector<cd>();
    // The step kernel reads them in its last forward pass, whose butterflies
    // hold R consecutive positions b*R + m (R its radix): entry (b, m) is
    // stored at m*(n/R) + b, so that a warp's reads are contiguous.
    const int lrl = (logn % logrm) ? logn % logrm : logrm;
    const int Rl = 1 << lrl, nbf = n >> lrl;
    for (int p = 0; p < n; ++p) {
        const double k = A.k[perm[p]];
        const int q = (p % Rl) * nbf + p / Rl;
        ph[q] = -0.5 * k * k * tau;
        phh[q] = -0.25 * k * k * tau;
    }
    potential_logs_1d(*T, n, tau, tv, tvs);
    // Strip CN tables of the T = n >> loge threads; M is complex symmetric, so
    // mb_i = mf_{i+1} (tvs holds the rows' potential factors in chunk order)
    std::vector<cd> mf, mb, g, cnv;
    std::vector<int32_t> cnfx;
    if (T->nb > 0) {
        double err = 0;
        rc = strip_factor(A, T->blk0, T->nb, mf, mb, g, &err);
        if (rc) return rc;
        const int thr = n >> loge, nb = T->nb;
        for (int i = 0; i + 1 < nb; ++i)
            if (std::abs(mb[i] - mf[i + 1]) > 1e-12 * (std::abs(mb[i]) + 1e-300)) return SOFT_ERR_SETUP;
        if (o.prec == SOFT_C128) cnfx = strip_tables_fx(mf, mb, g, nb, thr, &T->cn_gen);
        else cnv = strip_tables_c(mf, g, nb, thr, &T->cnr);
    }
    if (o.prec == SOFT_C128) {
        const bool gen = T->cn_gen || fx_gen_factors(log_range(tv, T->blk0, T->nb));
        if ((rc = upload_i32(&T->cn, cnfx))) return rc;
        const bool s2 = fx_center(lrl, logrm).s2;
        if ((rc = upload_fx_phases(&T->TK, ph, s2))) return rc;
        if ((rc = upload_fx_phases(&T->TKh, phh, s2))) return rc;
        if ((rc = upload_i32(&T->W, pass_twiddles_fx(logn, logrm, FXFULL_MAXS)))) return rc;
        if ((rc = upload_i32(&T->TV, fxv_table(tv, gen, logrm & 1)))) return rc;
        return tvs.empty() ? SOFT_OK : upload_i32(&T->TVs, fxv_table(tvs, gen, false));
    }
    if ((rc = upload_c(&T->cn, cnv, o.prec))) return rc;
    std::vector<cd> tk(n), tkh(n);
    for (int q = 0; q < n; ++q) {
        tk[q] = std::polar(1.0 / n, ph[q]);
        tkh[q] = std::polar(1.0 / n, phh[q]);
    }
    if ((rc = upload_tab(&T->TK, tk, o.prec))) return rc;
    if ((rc = upload_tab(&T->TKh, tkh, o.prec))) return rc;
    if ((rc = upload_vtab(&T->TV, vexp(tv), o.prec))) return rc;
    if ((rc = upload_tw_comp(&T->W, w, o.prec))) return rc;
    if ((rc = upload_vtab(&T->TVs, vexp(tvs), o.prec))) return rc;
    return SOFT_OK;
}

}  // namespace soft

// ------------------------------------------------------------------------ ABI
extern "C" {

void soft_default_options(soft_options* opt) {
    if (!opt) return;
    opt->prec = SOFT_C128;
    opt->contour = SOFT_CONTOUR_SHARP;
    opt->tfecs_alpha = 0.5;
    opt->soft_a2 = 2.0;
    opt->charge = 1.0;
    opt->band_width = 10;
    opt->autotune = 0;
    opt->cap_energy = 2.0;
    opt->tfap_kmin = 0.25;
    opt->persistent = 1;
}

const char* soft_strerror(int s) {
    switch (s) {
    case SOFT_OK: return "ok";
    case SOFT_ERR_INVALID_ARG: return "invalid argument";
    case SOFT_ERR_NOT_POW2: return "grid size must be a power of two in the supported range";
    case SOFT_ERR_OOM: return "device memory allocation failed";
    case SOFT_ERR_CUDA: return "CUDA runtime error";
    case SOFT_ERR_NOT_CONVERGED: return "PCG did not reach the tolerance within maxit";
    case SOFT_ERR_BREAKDOWN: return "PCG breakdown (vanishing bilinear form)";
    case SOFT_ERR_TIMEOUT: return "device wait timed out";
    case SOFT_ERR_NONFINITE: return "non-finite value in input or result";
    case SOFT_ERR_UNSUPPORTED: return "size/precision combination not supported";
    case SOFT_ERR_SETUP: return "plan tables failed a self-check";
    case SOFT_ERR_TOO_LARGE: return "request exceeds the fixed scratch of the no-allocation entry point";
    }
    return "unknown status";
}

static int check_opts(const soft_options* opt, soft_options* o) {
    soft_default_options(o);
    if (opt) *o = *opt;
    if (o->prec != SOFT_C64 && o->prec != SOFT_C128) return SOFT_ERR_INVALID_ARG;
    if (o->contour < 0 || o->contour > SOFT_ABSORB_TFAP) return SOFT_ERR_INVALID_ARG;
    if (!(o->cap_energy >= 0) || !(o->tfap_kmin >= 0) || !std::isfinite(o->cap_energy) ||
        !std::isfinite(o->tfap_kmin))
        return SOFT_ERR_INVALID_ARG;
    if (!(o->soft_a2 > 0) && o->charge != 0) return SOFT_ERR_INVALID_ARG;
    if (o->band_width < 1) return SOFT_ERR_INVALID_ARG;
    if (o->persistent != 0 && o->persistent != 1) return SOFT_ERR_INVALID_ARG;
    return SOFT_OK;
}

static int check_axis(int64_t n, double a, double b, double R0) {
    const int l = ilog2(n);
    if (l < 6 || l > 14) return SOFT_ERR_NOT_POW2;
    if (!(b > 0) || std::fabs(a + b) > 1e-12 * b) return SOFT_ERR_INVALID_ARG;
    if (!(R0 > 0 && R0 < b)) return SOFT_ERR_INVALID_ARG;
    return SOFT_OK;
}

// Time every built kernel variant of one 1D size on a sample of instances
// (up to four waves of the device's SMs) and return the fastest configuration.
static int autotune_size(const soft_options& o, int n, double a, double b, double R0, double theta,
                         double dt, int count, int* best_e, int* best_r) {
    int le[16], lr[16];
    const int logn = ilog2(n);
    const int nv = soft1d_variants(o.prec, logn, le, lr, 16);
    if (nv <= 1) return SOFT_OK;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0)
        return SOFT_ERR_CUDA;
    const int ns = std::min(count, 4 * nsm);
    const size_t eb = o.prec == SOFT_C64 ? 8 : 16;
    void* psi = nullptr;
    int rc = cuda_status(cudaMalloc(&psi, eb * (size_t)ns * n));
    if (rc) return rc;
    cudaMemset(psi, 0x3c, eb * (size_t)ns * n);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    float best = 1e30f;
    for (int v = 0; v < nv && rc == SOFT_OK; ++v) {
        Tables1D T;
        if (make_tables_1d(&T, n, a, b, R0, theta, dt, o, le[v], lr[v]) == SOFT_OK) {
            const int thr = n >> le[v];
            if ((T.nb + thr - 1) / thr <= (1 << le[v]) / 4 + 2) {
                std::vector<Inst1D> d(ns);
                for (int i = 0; i < ns; ++i) {
                    std::memset(&d[i], 0, sizeof(Inst1D));
                    d[i].off = (int64_t)i * n;
                    d[i].TK = T.TK; d[i].TKh = T.TKh; d[i].TV = T.TV; d[i].W = T.W; d[i].cn = T.cn; d[i].cnr = T.cnr;
                    d[i].TVs = T.TVs;
                    d[i].nb = T.nb; d[i].blk0 = T.blk0; d[i].x0 = T.ax.x[0]; d[i].h = T.ax.h;
                    d[i].R0 = R0; d[i].tau = dt; d[i].iL = T.iL; d[i].iR = T.iR; d[i].n = n;
                }
                void* dd = nullptr;
                if (upload(&dd, d.data(), d.size() * sizeof(Inst1D)) == SOFT_OK) {
                    launch_soft1d(o.prec, logn, le[v], lr[v], (Inst1D*)dd, ns, psi, 2, nullptr, 0,
                                  nullptr, 0, nullptr);
                    cudaEventRecord(e0, 0);
                    launch_soft1d(o.prec, logn, le[v], lr[v], (Inst1D*)dd, ns, psi, 8, nullptr, 0,
                                  nullptr, 0, nullptr);
                    cudaEventRecord(e1, 0);
                    if (cudaEventSynchronize(e1) == cudaSuccess) {
                        float ms = 0;
                        cudaEventElapsedTime(&ms, e0, e1);
                        if (ms < best) { best = ms; *best_e = le[v]; *best_r = lr[v]; }
                    } else {
                        rc = SOFT_ERR_CUDA;
                    }
                }
                cudaFree(dd);
            }
        }
        free_tables(&T);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(psi);
    return rc;
}

// shared by soft_create (1D) and soft_create_batch
static int create_1d(int count, const soft_grid* grids, const double* boxes, const double* R0,
                     const double* theta, const soft_field* fields, double dt,
                     const soft_options& o, bool single, soft_plan** out) {
    std::unique_ptr<soft_plan> P(new soft_plan());
    P->kind = 1;
    P->single = single;
    P->prec = o.prec;
    P->opt = o;
    P->dt = dt;
    std::map<std::tuple<int64_t, double, double, double, double>, int> seen;
    std::map<std::pair<double, double>, int> cls;
    int64_t off = 0;
    for (int i = 0; i < count; ++i) {
        if (grids[i].ndim != 1) return SOFT_ERR_INVALID_ARG;
        const int64_t n = grids[i].n[0];
        const double a = boxes[2 * i], b = boxes[2 * i + 1];
        int rc = check_axis(n, a, b, R0[i]);
        if (rc) return rc;
        const int logn = ilog2(n);
        int loge, logrm, pgroups;
        if (single) soft1d_single_cfg(o.prec, logn, &loge, &logrm);
        else soft1d_default_cfg(o.prec, logn, &loge, &logrm);
        // sizes of the persistent kernel keep its (elements per thread, radix)
        const bool persist = !single && o.persistent &&
                             persist_config(o.prec, logn, &loge, &logrm, &pgroups) >= 0;
        if (!persist && !soft1d_supported(o.prec, logn, loge, logrm)) return SOFT_ERR_UNSUPPORTED;
        auto key = std::make_tuple(n, a, b, R0[i], theta[i]);
        int tab;
        auto it = seen.find(key);
        if (it == seen.end()) {
            if (o.autotune && !persist) {
                int cnt = 0;
                for (int j = i; j < count; ++j)
                    if (grids[j].n[0] == n) ++cnt;
                rc = autotune_size(o, (int)n, a, b, R0[i], theta[i], dt, cnt, &loge, &logrm);
                if (rc) return rc;
            }
            std::unique_ptr<Tables1D> T(new Tables1D());
            rc = make_tables_1d(T.get(), (int)n, a, b, R0[i], theta[i], dt, o, loge, logrm);
            if (rc) { free_tables(T.get()); return rc; }
            // strip rows per thread must fit the kernel's register budget
            const int thr = (int)(n >> loge);
            const int chunk = (T->nb + thr - 1) / thr;
            if (chunk > (1 << loge) / 4 + 2) { free_tables(T.get()); return SOFT_ERR_UNSUPPORTED; }
            tab = (int)P->tabs.size();
            P->tabs.push_back(std::move(T));
            seen[key] = tab;
        } else {
            tab = it->second;
        }
        soft_plan::InstHost ih;
        ih.tab = tab; ih.off = off; ih.n = (int)n;
        ih.has_field = 0; ih.fcls = 0; ih.E0 = 0;
        if (fields) {
            const soft_field& f = fields[i];
            if (f.E0 != 0.0) {
                if (!(f.omega > 0 && f.ncycles > 0)) return SOFT_ERR_INVALID_ARG;
                const double Tp = f.ncycles * 2 * 3.14159265358979323846 / f.omega;
                auto k = std::make_pair(f.omega, Tp);
                auto c = cls.find(k);
                if (c == cls.end()) {
                    const int id = (int)P->h_cls.size() / 2;
                    P->h_cls.push_back(f.omega);
                    P->h_cls.push_back(Tp);
                    cls[k] = id;
                    ih.fcls = id;
                } else {
                    ih.fcls = c->second;
                }
                if (o.contour >= SOFT_ABSORB_CAP) return SOFT_ERR_UNSUPPORTED;   // absorbers: no field
                ih.has_field = 1;
                ih.E0 = f.E0;
            }
        }
        P->inst.push_back(ih);
        off += n;
    }
    P->total = off;
    int rc = P->build_1d_device();
    if (rc) return rc;
    if (!single && o.persistent && o.autotune && P->npacks > 0 && (rc = P->time_schedules())) return rc;
    *out = P.release();
    return SOFT_OK;
}

static int soft_create_impl(const soft_grid* grid, const double* box, double R0, double theta, double dt,
                            const soft_options* opt, soft_plan** out) {
    if (!grid || !box || !out) return SOFT_ERR_INVALID_ARG;
    *out = nullptr;
    if (!std::isfinite(dt) || dt == 0.0 || !std::isfinite(theta)) return SOFT_ERR_INVALID_ARG;
    soft_options o;
    int rc = check_opts(opt, &o);
    if (rc) return rc;
    if (grid->ndim == 1) return create_1d(1, grid, box, &R0, &theta, nullptr, dt, o, true, out);
    if (grid->ndim == 2) return create_2d(grid, box, R0, theta, dt, o, out);
    if (grid->ndim == 3) return create_3d(grid, box, R0, theta, dt, o, out);
    return SOFT_ERR_INVALID_ARG;
}
int soft_create(const soft_grid* grid, const double* box, double R0, double theta, double dt,
                const soft_options* opt, soft_plan** out) {
    return abi_guard([&] { return soft_create_impl(grid, box, R0, theta, dt, opt, out); });
}

static int soft_create_batch_impl(int count, const soft_grid* grids, const double* boxes, const double* R0,
                                  const double* theta, const soft_field* fields, double dt,
                                  const soft_options* opt, soft_plan** out) {
    if (count <= 0 || !grids || !boxes || !R0 || !theta || !out) return SOFT_ERR_INVALID_ARG;
    *out = nullptr;
    if (!std::isfinite(dt) || dt == 0.0) return SOFT_ERR_INVALID_ARG;
    soft_options o;
    int rc = check_opts(opt, &o);
    if (rc) return rc;
    return create_1d(count, grids, boxes, R0, theta, fields, dt, o, false, out);
}
int soft_create_batch(int count, const soft_grid* grids, const double* boxes, const double* R0,
                      const double* theta, const soft_field* fields, double dt,
                      const soft_options* opt, soft_plan** out) {
    return abi_guard([&] { return soft_create_batch_impl(count, grids, boxes, R0, theta, fields, dt, opt, out); });
}

int soft_batch_layout(const soft_plan* P, int64_t* offsets, int64_t* total) {
    if (!P || P->kind != 1) return SOFT_ERR_INVALID_ARG;
    if (offsets)
        for (size_t i = 0; i < P->inst.size(); ++i) offsets[i] = P->inst[i].off;
    if (total) *total = P->total;
    return SOFT_OK;
}

// 1D steps are not recorded into a caller's stream capture: a replay would use
// the start time, and the host copies of a new field, of the call that
// recorded it (soft_step_noalloc takes both by value)
static int not_capturing(cudaStream_t st) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(st, &cs);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess && cs == cudaStreamCaptureStatusNone ? SOFT_OK : SOFT_ERR_CUDA;
}

static int soft_step_impl(soft_plan* P, void* psi, int64_t nsteps, const soft_field* field, double* t_inout,
                          void* stream) {
    if (!P || !psi || !t_inout || nsteps < 0) return SOFT_ERR_INVALID_ARG;
    if (P->kind == 2) return P->step_2d(psi, nsteps, t_inout, (cudaStream_t)stream);
    if (P->kind == 3) return P->step_3d(psi, nsteps, t_inout, (cudaStream_t)stream);
    if (P->kind != 1) return SOFT_ERR_INVALID_ARG;
    if (P->single) {
        int rc = nsteps > 0 ? not_capturing((cudaStream_t)stream) : SOFT_OK;
        if (rc == SOFT_OK) rc = P->set_single_field(field, (cudaStream_t)stream);
        if (rc) return rc;
    }
    return P->step_1d(psi, nsteps, t_inout, (cudaStream_t)stream);
}
int soft_step(soft_plan* P, void* psi, int64_t nsteps, const soft_field* field, double* t_inout,
              void* stream) {
    return abi_guard([&] { return soft_step_impl(P, psi, nsteps, field, t_inout, stream); });
}

static int soft_step_batch_impl(soft_plan* P, void* psi, int64_t nsteps, double* t_inout, void* stream) {
    if (!P || !psi || !t_inout || nsteps < 0 || P->kind != 1) return SOFT_ERR_INVALID_ARG;
    const int rc = P->single && nsteps > 0 ? not_capturing((cudaStream_t)stream) : SOFT_OK;
    if (rc) return rc;
    return P->step_1d(psi, nsteps, t_inout, (cudaStream_t)stream);
}
int soft_step_batch(soft_plan* P, void* psi, int64_t nsteps, double* t_inout, void* stream) {
    return abi_guard([&] { return soft_step_batch_impl(P, psi, nsteps, t_inout, stream); });
}

int soft_observe(const soft_plan* P, const void* psi, double* norm_in, double* flux, void* stream) {
    if (!P || !psi || !norm_in || !flux || P->kind != 1) return SOFT_ERR_INVALID_ARG;
    int rc = launch_observe1d(P->prec, P->d_inst_obs, (int)P->inst.size(), psi, norm_in, flux,
                              (cudaStream_t)stream);
    const_cast<soft_plan*>(P)->last_launches = 1;
    return rc;
}

int soft_step_status(soft_plan* P, void* stream) {
    if (!P || P->kind != 1) return P ? SOFT_ERR_UNSUPPORTED : SOFT_ERR_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int h = 0;
    int rc = cuda_status(cudaMemcpyAsync(&h, P->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
    if (rc == SOFT_OK) rc = cuda_status(cudaStreamSynchronize(st));
    if (rc) return rc;
    if (h == 0) return SOFT_OK;
    rc = cuda_status(cudaMemsetAsync(P->d_status, 0, sizeof(int), st));
    return rc ? rc : SOFT_ERR_NONFINITE;
}

static int soft_set_potential_impl(soft_plan* P, const double* U, int64_t n) {
    if (!P || !U || n <= 0) return SOFT_ERR_INVALID_ARG;
    for (int64_t i = 0; i < 2 * n; ++i)
        if (!std::isfinite(U[i])) return SOFT_ERR_NONFINITE;
    if (P->kind == 2) {
        if (n != (int64_t)P->p2->nx * P->p2->ny) return SOFT_ERR_INVALID_ARG;
        return P->p2->set_potential(U);
    }
    if (P->kind == 3) {
        if (n != P->points_3d()) return SOFT_ERR_INVALID_ARG;
        return P->p3->set_potential(U);
    }
    if (P->kind != 1 || !P->single || P->tabs.size() != 1) return SOFT_ERR_UNSUPPORTED;
    Tables1D* T = P->tabs[0].get();
    const int nn = 1 << T->logn;
    if (n != nn) return SOFT_ERR_INVALID_ARG;
    int rc = cuda_status(cudaDeviceSynchronize());      // no step may still read the tables
    if (rc) return rc;
    for (int j = 0; j < nn; ++j) T->U0[j] = cd(U[2 * j], U[2 * j + 1]) + T->Uabs[j];
    std::vector<cd> tv, tvs;
    potential_logs_1d(*T, nn, P->dt, tv, tvs);
    if (T->prec == SOFT_C128) {
        const bool gen = T->cn_gen || fx_gen_factors(log_range(tv, T->blk0, T->nb));
        for (int i = 0; i < 2; ++i) {
            const std::vector<cd>& v = i ? tvs : tv;
            if (v.empty()) continue;
            const std::vector<int32_t> b = fxv_table(v, gen, !i && (T->logrm & 1));
            rc = cuda_status(cudaMemcpy(i ? T->TVs : T->TV, b.data(), b.size() * 4, cudaMemcpyHostToDevice));
            if (rc) return rc;
        }
        return sse1d_refill_potential(P);
    }
    if ((rc = refill_vtab(T->TV, vexp(tv), T->prec))) return rc;
    if ((rc = refill_vtab(T->TVs, vexp(tvs), T->prec))) return rc;
    return sse1d_refill_potential(P);
}
int soft_set_potential(soft_plan* P, const double* U, int64_t n) {
    return abi_guard([&] { return soft_set_potential_impl(P, U, n); });
}

void soft_destroy(soft_plan* P) { delete P; }

int soft_plan_count(const soft_plan* P) {
    if (!P) return 0;
    return P->kind == 1 ? (int)P->inst.size() : 1;
}
int64_t soft_plan_points(const soft_plan* P, int i) {
    if (!P) return 0;
    if (P->kind == 1) return (i >= 0 && i < (int)P->inst.size()) ? P->inst[i].n : 0;
    return P->kind == 3 ? P->points_3d() : P->points_2d();
}
int soft_plan_prec(const soft_plan* P) { return P ? P->prec : 0; }
int64_t soft_last_launches(const soft_plan* P) { return P ? P->last_launches : 0; }

}  // extern "C"

// ---------------------------------------------------------------- soft_plan
soft_plan::~soft_plan() {
    for (auto& t : tabs) free_tables(t.get());
    for (auto& g : groups) cudaFree(g.d_inst);
    cudaFree(d_pinst);
    cudaFree(d_packs);
    cudaFree(d_pcount);
    cudaFree(d_inst_obs);
    cudaFree(d_cls);
    cudaFree(d_ftab);
    cudaFree(d_status);
    cudaFree(d_t0);
    delete nn;
    sse1d_free(s1);
    surf1d_free(sf);
    if (gexec) cudaGraphExecDestroy(gexec);
    if (side_ready) {
        for (size_t g = 0; g < groups.size() && g < MAX_SIDE; ++g) {
            cudaStreamDestroy(side[g]);
            cudaEventDestroy(ev_join[g]);
        }
        cudaEventDestroy(ev_fork);
    }
    free_2d();
    free_3d();
}

Inst1D soft_plan::descriptor(int i) const {
    const InstHost& ih = inst[i];
    const Tables1D& T = *tabs[ih.tab];
    Inst1D d;
    std::memset(&d, 0, sizeof(d));
    d.off = ih.off;
    d.TK = T.TK; d.TKh = T.TKh; d.TV = T.TV; d.W = T.W; d.cn = T.cn; d.cnr = T.cnr; d.TVs = T.TVs;
    d.nb = T.nb; d.blk0 = T.blk0;
    d.x0 = T.ax.x[0]; d.h = T.ax.h; d.R0 = T.R0; d.tau = dt;
    d.E0 = ih.E0; d.has_field = ih.has_field; d.fcls = ih.fcls;
    d.iL = T.iL; d.iR = T.iR; d.n = ih.n;
    return d;
}

// the instances of the persistent kernel's sizes as packs of same-size
// instances, largest N first
int soft_plan::build_packs(size_t cap) {
    std::vector<Pack1D> packs;
    std::vector<Inst1D> pd;
    for (auto& g : groups) {
        int le, lr, G;
        const int v = persist_config(prec, g.logn, &le, &lr, &G);
        if (v < 0 || le != g.loge || lr != g.logrm) continue;
        g.in_persist = true;
        G = (int)std::min<size_t>(G, cap);
        for (size_t k = 0; k < g.members.size(); k += G) {
            Pack1D pk;
            pk.var = v;
            pk.first = (int)pd.size();
            pk.count = (int)std::min<size_t>(G, g.members.size() - k);
            pk.pad_ = 0;
            for (int j = 0; j < pk.count; ++j) pd.push_back(descriptor(g.members[k + j]));
            packs.push_back(pk);
        }
    }
    std::stable_sort(packs.begin(), packs.end(), [](const Pack1D& a, const Pack1D& b) { return a.var < b.var; });
    cudaFree(d_pinst); cudaFree(d_packs); cudaFree(d_pcount);
    d_pinst = nullptr; d_packs = nullptr; d_pcount = nullptr;
    npacks = (int)packs.size();
    use_persist = npacks > 0;
    if (npacks == 0) return SOFT_OK;
    int rc;
    if ((rc = upload((void**)&d_pinst, pd.data(), pd.size() * sizeof(Inst1D)))) return rc;
    if ((rc = upload(&d_packs, packs.data(), packs.size() * sizeof(Pack1D)))) return rc;
    if ((rc = cuda_status(cudaMalloc((void**)&d_pcount, sizeof(int))))) return rc;
    // sets the kernel's shared-memory attribute outside any capture
    return launch_persist(prec, nullptr, 0, nullptr, nullptr, nullptr, 0, nullptr, 0, nullptr, 0, nullptr);
}

int soft_plan::build_1d_device() {
    // groups by kernel configuration, largest N first
    std::map<std::pair<int, int>, int> gid;
    for (size_t i = 0; i < inst.size(); ++i) {
        const Tables1D& T = *tabs[inst[i].tab];
        auto key = std::make_pair(-T.logn, T.loge * 8 + T.logrm);
        auto it = gid.find(key);
        if (it == gid.end()) {
            Group1D g;
            g.logn = T.logn; g.loge = T.loge; g.logrm = T.logrm;
            gid[key] = (int)groups.size();
            groups.push_back(g);
            it = gid.find(key);
        }
        groups[it->second].members.push_back((int)i);
    }
    std::sort(groups.begin(), groups.end(), [](const Group1D& a, const Group1D& b) { return a.logn > b.logn; });
    int rc;
    if (!single && opt.persistent) {
        int dev = 0, nsm = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return SOFT_ERR_CUDA;
        // the fewest instances per pack that still give at most one pack per SM:
        // SMs left idle cost more than part-filled CTAs (24 steps of 8 complex64
        // instances, full packs / one each: N = 2048 474 / 371 us, N = 8192 880 / 670)
        auto packs_for = [&](size_t cap) {
            size_t k = 0;
            int le, lr, G;
            for (const auto& g : groups)
                if (persist_config(prec, g.logn, &le, &lr, &G) >= 0 && le == g.loge && lr == g.logrm)
                    k += (g.members.size() + std::min<size_t>(G, cap) - 1) / std::min<size_t>(G, cap);
            return k;
        };
        size_t cap = 1;
        while (cap < 8 && packs_for(cap) > (size_t)nsm) cap *= 2;
        if ((rc = build_packs(cap))) return rc;
        // By default the queue runs batches of at most one instance per SM, in one
        // launch.  One kernel for four sizes spills registers and keeps one CTA of 512
        // threads per SM, so one launch per size takes less time at every batch
        // size (24 steps, persistent / per size, us, 8, 152 and 300 instances):
        //   complex64   N = 2048: 372/169, 402/191, 417/191    N = 4096: 404/248, 419/258, 503/327
        //               N = 8192: 671/509, 691/525, 899/717    N = 16384: 849/708, 867/719, 1713/1420
        //               2048 to 16384 mixed: 877/773, 890/773, 997/863
        //   complex128  N = 2048: 588/486, 594/494, 812/691    N = 4096: 1001/856, 1026/873, 1373/1204
        //               N = 8192: 1461/1365, 1474/1375, 2922/2734   N = 16384: 3679/3043, 3766/3083, 7508/6160
        //               mixed: 3640/3043, 3748/3058, 3776/3066
        // A caller who counts time and not launches sets persistent = 0, or autotune,
        // which times both, also the packs of several instances of larger batches.
        use_persist = npacks > 0 && npacks <= nsm && cap == 1;
    }
    for (auto& g : groups) {
        std::vector<Inst1D> d;
        for (int i : g.members) d.push_back(descriptor(i));
        if ((rc = upload((void**)&g.d_inst, d.data(), d.size() * sizeof(Inst1D)))) return rc;
    }
    h_obs.clear();
    for (size_t i = 0; i < inst.size(); ++i) h_obs.push_back(descriptor((int)i));
    if ((rc = upload((void**)&d_inst_obs, h_obs.data(), h_obs.size() * sizeof(Inst1D)))) return rc;
    ncls = (int)h_cls.size() / 2;
    // room for one extra class used by soft_step's per-call field
    std::vector<double> c = h_cls;
    c.push_back(1.0); c.push_back(1.0);
    if ((rc = upload((void**)&d_cls, c.data(), c.size() * sizeof(double)))) return rc;
    ftab_cap = 4096;
    if ((rc = cuda_status(cudaMalloc((void**)&d_ftab, sizeof(double) * ftab_cap * (ncls + 1))))) return rc;
    if ((rc = cuda_status(cudaMalloc((void**)&d_status, sizeof(int))))) return rc;
    if ((rc = cuda_status(cudaMemset(d_status, 0, sizeof(int))))) return rc;
    if ((rc = cuda_status(cudaMalloc((void**)&d_t0, sizeof(double))))) return rc;
    return SOFT_OK;
}

// soft_step on a single-instance plan: the call's field replaces the plan's.
// The descriptor and pulse-class copies are queued on the call's stream, so
// they take effect after every step already queued there (a step still
// waiting on a non-blocking stream keeps the field it was called with);
// pageable sources are staged before cudaMemcpyAsync returns.
int soft_plan::set_single_field(const soft_field* f, cudaStream_t st) {
    InstHost& ih = inst[0];
    int has = 0, fc = 0;
    double E0 = 0;
    if (f && f->E0 != 0.0) {
        if (!(f->omega > 0 && f->ncycles > 0)) return SOFT_ERR_INVALID_ARG;
        if (opt.contour >= SOFT_ABSORB_CAP) return SOFT_ERR_UNSUPPORTED;   // absorbers: no field
        const double Tp = f->ncycles * 2 * 3.14159265358979323846 / f->omega;
        if (call_cls[0] != f->omega || call_cls[1] != Tp) {
            call_cls[0] = f->omega;
            call_cls[1] = Tp;
            int rc = cuda_status(cudaMemcpyAsync(d_cls + 2 * ncls, call_cls, 2 * sizeof(double),
                                                 cudaMemcpyHostToDevice, st));
            if (rc) return rc;
        }
        has = 1; fc = ncls; E0 = f->E0;
    }
    if (has != ih.has_field || fc != ih.fcls || E0 != ih.E0) {
        ih.has_field = has; ih.fcls = fc; ih.E0 = E0;
        Inst1D d = descriptor(0);
        for (auto& g : groups) {
            int rc = cuda_status(cudaMemcpyAsync(g.d_inst, &d, sizeof(d), cudaMemcpyHostToDevice, st));
            if (rc) return rc;
        }
        h_obs[0] = d;
        int rc = cuda_status(cudaMemcpyAsync(d_inst_obs, &d, sizeof(d), cudaMemcpyHostToDevice, st));
        if (rc) return rc;
    }
    return SOFT_OK;
}

// one chunk of steps on the given stream: pulse table from the device start
// time, the persistent kernel (if used) and the size groups on parallel
// branches, then the start time advanced
int soft_plan::enqueue_chunk(void* psi, int64_t chunk, cudaStream_t st) {
    const int nc = ncls + (single ? 1 : 0);
    int rc;
    if (nc > 0) {
        if ((rc = launch_field_table_dev(d_cls, nc, d_t0, dt, chunk, d_ftab, ftab_cap, st))) return rc;
        ++last_launches;
    }
    const bool persist = use_persist && npacks > 0;
    int nlaunch = persist ? 1 : 0;
    for (const auto& G : groups)
        if (!(persist && G.in_persist)) ++nlaunch;
    const bool fork = nlaunch > 1;
    if (fork && (rc = cuda_status(cudaEventRecord(ev_fork, st)))) return rc;
    if (persist) {           // the persistent kernel on the call's stream, the groups beside it
        if ((rc = cuda_status(cudaMemsetAsync(d_pcount, 0, sizeof(int), st)))) return rc;
        if ((rc = launch_persist(prec, d_packs, npacks, d_pcount, d_pinst, psi, chunk, d_ftab, ftab_cap, d_status,
                                 st, nullptr)))
            return rc;
        last_launches += 1;
    }
    for (size_t g = 0; g < groups.size(); ++g) {
        if (persist && groups[g].in_persist) continue;
        cudaStream_t gs = fork ? side[g] : st;
        if (fork && (rc = cuda_status(cudaStreamWaitEvent(gs, ev_fork, 0)))) return rc;
        const Group1D& G = groups[g];
        rc = launch_soft1d(prec, G.logn, G.loge, G.logrm, G.d_inst, (int)G.members.size(), psi, chunk,
                           d_ftab, ftab_cap, d_status, gs, nullptr);
        if (rc) return rc;
        ++last_launches;
        if (fork) {
            if ((rc = cuda_status(cudaEventRecord(ev_join[g], gs)))) return rc;
            if ((rc = cuda_status(cudaStreamWaitEvent(st, ev_join[g], 0)))) return rc;
        }
    }
    if ((rc = launch_advance_time(d_t0, (double)chunk * dt, st))) return rc;
    ++last_launches;
    return SOFT_OK;
}

int soft_plan::ensure_side() {
    int rc;
    if (!side_ready) {
        for (size_t g = 0; g < groups.size() && g < MAX_SIDE; ++g) {
            if ((rc = cuda_status(cudaStreamCreateWithFlags(&side[g], cudaStreamNonBlocking)))) return rc;
            if ((rc = cuda_status(cudaEventCreateWithFlags(&ev_join[g], cudaEventDisableTiming)))) return rc;
        }
        if ((rc = cuda_status(cudaEventCreateWithFlags(&ev_fork, cudaEventDisableTiming)))) return rc;
        side_ready = true;
    }
    return groups.size() > MAX_SIDE ? SOFT_ERR_UNSUPPORTED : SOFT_OK;
}

// The schedule autotuner of a batch plan: one chunk of 16 steps on a constant,
// non-zero state (as autotune_size: a zero one is not a step's usual work) with
// the persistent kernel and with one kernel per size group (each timed after a
// warm-up run); the faster is kept.
int soft_plan::time_schedules() {
    int rc = ensure_side();
    if (rc) return rc;
    const size_t eb = prec == SOFT_C64 ? 8 : 16;
    void* tmp = nullptr;
    if ((rc = cuda_status(cudaMalloc(&tmp, eb * (size_t)total)))) return rc;
    cudaStream_t st = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    float ms[2] = {0, 0};
    rc = cuda_status(cudaMemset(tmp, 0x3c, eb * (size_t)total));
    if (!rc) rc = cuda_status(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    if (!rc) rc = cuda_status(cudaEventCreate(&e0));
    if (!rc) rc = cuda_status(cudaEventCreate(&e1));
    for (int mode = 0; mode < 2 && !rc; ++mode) {
        use_persist = mode == 0;
        const double zero = 0.0;
        rc = cuda_status(cudaMemcpyAsync(d_t0, &zero, sizeof(double), cudaMemcpyHostToDevice, st));
        for (int rep = 0; rep < 2 && !rc; ++rep) {
            if (rep == 1) rc = cuda_status(cudaEventRecord(e0, st));
            if (!rc) rc = enqueue_chunk(tmp, 16, st);
            if (!rc && rep == 1) rc = cuda_status(cudaEventRecord(e1, st));
        }
        if (!rc) rc = cuda_status(cudaEventSynchronize(e1));
        if (!rc) rc = cuda_status(cudaEventElapsedTime(&ms[mode], e0, e1));
    }
    use_persist = rc == SOFT_OK && ms[0] <= ms[1];
    last_launches = 0;
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (st) cudaStreamDestroy(st);
    cudaFree(tmp);
    return rc;
}

int soft_plan::step_1d(void* psi, int64_t nsteps, double* t_inout, cudaStream_t st) {
    last_launches = 0;
    if (nsteps == 0) return SOFT_OK;
    int rc;
    if (single) {
        // one instance: the pulse table (with a field) and the step kernel per
        // chunk, launched directly.  The graph of the batch path would add the
        // start time's copy, a table and a time kernel, and a new capture for
        // every new buffer: one step at N = 128 20.5 -> 16.0 us, on a new
        // buffer 88 -> 38.
        for (int64_t done = 0; done < nsteps;) {
            const int64_t chunk = std::min<int64_t>(ftab_cap, nsteps - done);
            if (inst[0].has_field) {
                rc = launch_field_table(d_cls, ncls + 1, *t_inout + (double)done * dt, dt, chunk, d_ftab, ftab_cap, st);
                if (rc) return rc;
                ++last_launches;
            }
            const Group1D& G = groups[0];
            rc = launch_soft1d(prec, G.logn, G.loge, G.logrm, G.d_inst, 1, psi, chunk, d_ftab, ftab_cap, d_status, st,
                               nullptr);
            if (rc) return rc;
            ++last_launches;
            done += chunk;
        }
        *t_inout += (double)nsteps * dt;
        return SOFT_OK;
    }
    if ((rc = ensure_side())) return rc;
    // start time: a pageable copy is consumed before the call returns
    const double t0 = *t_inout;
    if ((rc = cuda_status(cudaMemcpyAsync(d_t0, &t0, sizeof(double), cudaMemcpyHostToDevice, st)))) return rc;
    int64_t done = 0;
    while (done < nsteps) {
        const int64_t chunk = std::min<int64_t>(ftab_cap, nsteps - done);
        if (!gexec || gpsi != psi || gchunk != chunk || gstream != st) {
            if (gexec) { cudaGraphExecDestroy(gexec); gexec = nullptr; }
            cudaStream_t cap;
            if ((rc = cuda_status(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking)))) return rc;
            cudaGraph_t graph;
            const int64_t before = last_launches;
            rc = cuda_status(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal));
            if (rc == SOFT_OK) rc = enqueue_chunk(psi, chunk, cap);
            cudaError_t e = cudaStreamEndCapture(cap, &graph);
            if (rc == SOFT_OK) rc = cuda_status(e);
            if (rc == SOFT_OK) rc = cuda_status(cudaGraphInstantiate(&gexec, graph, 0));
            if (e == cudaSuccess) cudaGraphDestroy(graph);
            cudaStreamDestroy(cap);
            if (rc) { gexec = nullptr; return rc; }
            glaunches = last_launches - before;
            last_launches = before;
            gpsi = psi; gchunk = chunk; gstream = st;
        }
        if ((rc = cuda_status(cudaGraphLaunch(gexec, st)))) return rc;
        last_launches += glaunches;
        done += chunk;
    }
    *t_inout = t0 + (double)nsteps * dt;
    return SOFT_OK;
}
