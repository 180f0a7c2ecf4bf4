// The gate functions of the ionic models tabulated in V (host side).
//
// Each gate q has w_inf,q(V) and Lambda_q(V), smooth functions of the
// membrane potential alone:
//   SYN19 (12 gates): w_inf,q(V) = 1/(1 + e^{-(V - Vh_q)/k_q}),
//                     Lambda_q(V) = -r_q exp(ln rho_q / (1 + e^{-(V - Vr_q)/sr_q}));
//   HH1952 (3 gates): Lambda = -(alpha + beta), w_inf = alpha/(alpha + beta)
//                     with the 1952 rates at v = V - V_rest.
// Evaluated directly a SYN19 gate costs three exponentials and two
// reciprocals (about 35 FP64 operations), an HH gate about as much; on a GPU
// with two FP64 lane operations per SM and clock that is most of the node
// kernel.  Here each function is replaced, on each interval of width
// w = ESDC_VTAB_W (1/128 mV) centred at V_lo + i w, by its Chebyshev interpolant of
// degree 3 (4 Chebyshev points, values in long double), a cubic in t = V -
// centre that esdc_tabeval.h evaluates in FP32 pairs and integers.  The functions are
// analytic in a strip about the real axis of half-width about pi k (k, sr >= 4 mV
// on the models' parameter ranges), so the interpolation error falls like
// (w / (4 pi k))^4: narrow intervals allow a low degree and leave a small bracket
// for the FP32 pairs.  The evaluation against long double, 9 points per interval:
// at most 5.1e-16 for w_inf (b's error over |Lambda|) and 1.5e-16 relative for
// Lambda on SYN19, 1.5e-16 and 1.9e-16 on HH; FP64 Horner steps on the same cubics
// made 5.4e-16, 2.3e-16, 2.2e-16 and 2.5e-16.  The table is 24 MB, held in L2.
// A table whose evaluation misses by more than ESDC_VTAB_TOL is refused (the
// kernels then evaluate directly).  The oracle keeps the direct formulas; the
// table is a way of computing the same functions.
//
// Row i of the table (ESDC_VTAB_ROW doubles): for each gate q the cubics of b_q =
// -Lambda_q w_inf,q (for HH, alpha_q) and of Lambda_q.  The kernels need the
// gate's rate Lambda (u - w_inf) = Lambda u + b, one FMA from (Lambda, b);
// w_inf itself (diagnostics) is -b / Lambda.  The error check scales b's error
// by |Lambda|, which makes it the error in w_inf.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <thread>
#include <vector>

#include "esdc_internal.h"
#include "esdc_tabeval.h"

namespace {

using LD = long double;

LD logistic(LD x) { return 1.0L / (1.0L + expl(-x)); }

LD x_over_expm1(LD x) { return x == 0.0L ? 1.0L : x / expm1l(x); }

// alpha, beta of HH gate q (0 = m, 1 = h, 2 = n) at v = V - V_rest (mV, 1/ms).
void hh_rates(int q, LD v, LD& al, LD& be)
{
    if (q == 0) { al = x_over_expm1((25.0L - v) / 10.0L); be = 4.0L * expl(-v / 18.0L); }
    else if (q == 1) { al = 0.07L * expl(-v / 20.0L); be = 1.0L / (expl((30.0L - v) / 10.0L) + 1.0L); }
    else { al = 0.1L * x_over_expm1((10.0L - v) / 10.0L); be = 0.125L * expl(-v / 80.0L); }
}

// Chebyshev interpolant of f on [m - h, m + h] at d + 1 Chebyshev points,
// returned as monomial coefficients in t = V - m.
template <class F>
void cheb_monomial(F f, LD m, LD h, int d, LD* out)
{
    const int n = d + 1;
    std::vector<LD> fx(n), a(n, 0.0L);
    const LD pi = 3.14159265358979323846264338327950288L;
    for (int j = 0; j < n; ++j) fx[j] = f(m + h * cosl(pi * (j + 0.5L) / n));
    for (int k = 0; k < n; ++k) {
        LD s = 0.0L;
        for (int j = 0; j < n; ++j) s += fx[j] * cosl(pi * k * (j + 0.5L) / n);
        a[k] = (k == 0 ? 1.0L : 2.0L) * s / n;
    }
    // sum_k a_k T_k(tau) in powers of tau (T_{k+1} = 2 tau T_k - T_{k-1}), then tau = t/h
    std::vector<LD> tkm(n, 0.0L), tk(n, 0.0L), b(n, 0.0L);
    tkm[0] = 1.0L;                       // T_0 = 1
    tk[1] = 1.0L;                        // T_1 = tau (n >= 2)
    b[0] = a[0];
    b[1] = a[1];
    for (int k = 2; k < n; ++k) {
        std::vector<LD> tn(n, 0.0L);
        for (int p = 0; p < n; ++p) {
            if (p + 1 < n) tn[p + 1] += 2.0L * tk[p];
            tn[p] -= tkm[p];
        }
        for (int p = 0; p < n; ++p) b[p] += a[k] * tn[p];
        tkm = tk;
        tk = tn;
    }
    LD s = 1.0L;
    for (int p = 0; p < n; ++p) {
        out[p] = b[p] * s;
        s /= h;
    }
}

// Rows [i0, i1) of the table; returns the largest errors of their
// evaluation against the direct long-double values.
void build_rows(int model, const double* params, int i0, int i1, double* out, double& ew, double& el)
{
    const int d = 3, NG = model == ESDC_MODEL_SYN19 ? 12 : 3;
    ew = 0.0;
    el = 0.0;
    LD coef[4];
    for (int i = i0; i < i1; ++i) {
        const LD mid = (LD)ESDC_VTAB_VLO + (LD)i * ESDC_VTAB_W, h = 0.5L * ESDC_VTAB_W;
        auto* row = reinterpret_cast<esdc::TabPoly*>(out + (size_t)i * ESDC_VTAB_ROW);
        for (int q = 0; q < NG; ++q) {
            const bool syn = model == ESDC_MODEL_SYN19;
            const double* p = params + (syn ? 6 * q : 0);     // SYN19: Vh, k, r, ln rho, Vr, sr
            const LD Vrest = syn ? 0.0L : (LD)params[6];
            auto winf = [&](LD V) {
                if (syn) return logistic((V - (LD)p[0]) / (LD)p[1]);
                LD al, be;
                hh_rates(q, V - Vrest, al, be);
                return al / (al + be);
            };
            auto lam = [&](LD V) {
                if (syn) return -(LD)p[2] * expl((LD)p[3] * logistic((V - (LD)p[4]) / (LD)p[5]));
                LD al, be;
                hh_rates(q, V - Vrest, al, be);
                return -(al + be);
            };
            auto bfun = [&](LD V) { return -lam(V) * winf(V); };
            esdc::TabPoly &pb = row[2 * q], &pl = row[2 * q + 1];
            cheb_monomial(bfun, mid, h, d, coef);
            bool ok = esdc::tab_pack(coef, h, pb);
            cheb_monomial(lam, mid, h, d, coef);
            ok = esdc::tab_pack(coef, h, pl) && ok;
            if (!ok) ew = HUGE_VAL;
            for (int s = 0; s <= 8; ++s) {            // the evaluation against the direct values
                const double V = (double)(mid + h * (s - 4) / 4.0L);
                float th, tl;
                esdc::tab_split(V - (double)mid, th, tl);
                const LD l0 = lam((LD)V), b0 = -l0 * winf((LD)V);
                // b's error relative to |Lambda|: the error it makes in w_inf
                ew = std::fmax(ew, (double)(fabsl((LD)esdc::tab_eval(pb, th, tl) - b0) / fabsl(l0)));
                el = std::fmax(el, (double)(fabsl((LD)esdc::tab_eval(pl, th, tl) - l0) / fabsl(l0)));
            }
        }
    }
}

// Tables already built in this process, keyed by the model and the parameters
// the gate functions depend on (SYN19: the six of each gate; HH: V_rest), so
// that handles of the same model and a change of conductances reuse them.
struct Cached {
    int model;
    std::vector<double> key;
    TableRows rows;
    double ew, el;
};
std::mutex g_cache_mu;
std::vector<Cached> g_cache;            // most recent last, at most kCacheSize
constexpr size_t kCacheSize = 8;

}  // namespace

int esdc_vtab_build(int model, const double* params, TableRows& rows, double* err_winf, double* err_lam)
{
    rows.reset();
    if (model != ESDC_MODEL_SYN19 && model != ESDC_MODEL_HH1952) return -1;
    const std::vector<double> key = model == ESDC_MODEL_SYN19 ? std::vector<double>(params, params + 72)
                                                               : std::vector<double>{params[6]};
    double ew = 0.0, el = 0.0;
    bool hit = false;
    {
        std::lock_guard<std::mutex> lk(g_cache_mu);
        for (size_t k = 0; k < g_cache.size(); ++k)
            if (g_cache[k].model == model && g_cache[k].key == key) {
                Cached c = g_cache[k];
                g_cache.erase(g_cache.begin() + (long)k);
                g_cache.push_back(c);
                rows = c.rows;
                ew = c.ew;
                el = c.el;
                hit = true;
                break;
            }
    }
    if (!hit) {
        std::vector<double> v((size_t)ESDC_VTAB_N * ESDC_VTAB_ROW, 0.0);
        // rows are independent: split them over the host's cores; the maxima
        // do not depend on the split
        unsigned nt = std::thread::hardware_concurrency();
        nt = std::max(1u, std::min(nt, 16u));
        std::vector<double> tw(nt, 0.0), tl(nt, 0.0);
        std::vector<std::thread> th;
        const int per = (ESDC_VTAB_N + (int)nt - 1) / (int)nt;
        for (unsigned t = 0; t < nt; ++t) {
            const int i0 = (int)t * per, i1 = std::min(ESDC_VTAB_N, i0 + per);
            if (i0 >= i1) break;
            th.emplace_back(build_rows, model, params, i0, i1, v.data(), std::ref(tw[t]), std::ref(tl[t]));
        }
        for (auto& x : th) x.join();
        rows = std::make_shared<const std::vector<double>>(std::move(v));
        for (unsigned t = 0; t < nt; ++t) {
            ew = std::fmax(ew, tw[t]);
            el = std::fmax(el, tl[t]);
        }
        std::lock_guard<std::mutex> lk(g_cache_mu);
        if (g_cache.size() >= kCacheSize) g_cache.erase(g_cache.begin());
        g_cache.push_back(Cached{model, key, rows, ew, el});
    }
    if (err_winf) *err_winf = ew;
    if (err_lam) *err_lam = el;
    if (!(ew <= ESDC_VTAB_TOL) || !(el <= ESDC_VTAB_TOL)) {
        rows.reset();
        return -2;
    }
    return 0;
}
