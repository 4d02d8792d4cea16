// Test harness: the fixed-point hops of csrc/fixed.cuh, compiled for the host
// and driven with the eight hops of a site.  Not part of the
// library.
#include <algorithm>
#include <cmath>

#include "../paper_1204_1306_gb300/csrc/fixed.cuh"

using namespace psms;

namespace {

template <bool DAG>
bool hops(const double *u, const double *psi, FxAcc &acc) {
    bool ok = true;
    for (int d = 0; d < 8; ++d) {
        cpx<double> e[9];
        int4 v[9], w[9];
        for (int k = 0; k < 9; ++k) e[k] = {u[(d * 9 + k) * 2], u[(d * 9 + k) * 2 + 1]};
        const int ue = fx_link(e, w);
        for (int a = 0; a < 3; ++a)
            for (int c = 0; c < 3; ++c) v[3 * a + c] = (d & 1) ? w[3 * c + a] : w[3 * a + c];
        uint64_t p[12][2];
        for (int c = 0; c < 12; ++c)
            for (int k = 0; k < 2; ++k) p[c][k] = f64_bits(psi[(d * 12 + c) * 2 + k]);
        int64_t x[12][2];
        const int ep = fx_spinor(p, x);
        if (ep == FX_BAD || ue == FX_BAD) ok = false;
        else if (ep != 0 && ue != 0) {
            int2 hl[2][3][2];
            fx_half<DAG>(d, x, hl);
            fx_hop<DAG>(d, false, hl, ep, v, ue, acc);
        }
    }
    return ok;
}

}  // namespace

// the eight hops of n sites: links u[n][8][9] and spinors psi[n][8][12] complex
// (interleaved doubles); out[n][12]; returns the number of sites left to the
// FP64 form
extern "C" int fx_hops_host(const double *u, const double *psi, int dag, int n, double b, double *out) {
    int left = 0;
    for (int i = 0; i < n; ++i) {
        FxAcc acc;
        fx_zero(acc);
        const double *ui = u + (long long)i * 8 * 18, *pi = psi + (long long)i * 8 * 24;
        double f = 0;
        const bool ok = (dag ? hops<true>(ui, pi, acc) : hops<false>(ui, pi, acc)) && fx_factor(acc, b, f);
        left += !ok;
        for (int c = 0; c < 12; ++c)
            for (int k = 0; k < 2; ++k) {
                const int64_t s = c < 6 ? acc.up[c / 3][c % 3][k] : acc.dn[(c - 6) / 3][c % 3][k];
                out[(i * 12 + c) * 2 + k] = ok ? f * (double)s : 0.0;
            }
    }
    return left;
}

// out[i] = 1 where the hops take spinor i (psi[n][12] complex) in fixed point
extern "C" void fx_alike_host(const double *psi, int n, int *out) {
    for (int i = 0; i < n; ++i) {
        uint64_t p[12][2];
        for (int c = 0; c < 12; ++c)
            for (int k = 0; k < 2; ++k) p[c][k] = f64_bits(psi[(i * 12 + c) * 2 + k]);
        int64_t x[12][2];
        bool alike;
        const int e = fx_spinor(p, x, alike);
        out[i] = e != 0 && e != FX_BAD && alike;
    }
}

// a link through its fixed-point form and back
extern "C" int fx_link_host(const double *u, double *out) {
    cpx<double> e[9];
    int4 w[9];
    for (int k = 0; k < 9; ++k) e[k] = {u[2 * k], u[2 * k + 1]};
    const int ue = fx_link(e, w);
    for (int k = 0; k < 9; ++k) {
        out[2 * k] = fx_value(w[k].x, w[k].y, ue);
        out[2 * k + 1] = fx_value(w[k].z, w[k].w, ue);
    }
    return ue;
}

// one element of the LU's trailing update: w complex products of a row l (on
// its largest exponent) and a column u; out = the value subtracted
extern "C" void lu_sum_host(const double *l, const double *u, int w, double *out) {
    int el = 0, eu = 0;
    for (int q = 0; q < 2 * w; ++q) {
        el = std::max(el, (int)(f64_bits(l[q]) >> 52) & 0x7FF);
        eu = std::max(eu, (int)(f64_bits(u[q]) >> 52) & 0x7FF);
    }
    int64_t hr = 0, hi = 0, mr = 0, mi = 0;
    for (int q = 0; q < w; ++q) {
        const LuLimbs a = lu_limbs(l[2 * q], el), b = lu_limbs(l[2 * q + 1], el), c = lu_limbs(u[2 * q], eu),
                      d = lu_limbs(u[2 * q + 1], eu);
        fx_mad(hr, a.hi, c.hi), fx_mad(hr, -b.hi, d.hi);
        fx_mad(hi, a.hi, d.hi), fx_mad(hi, b.hi, c.hi);
        fx_mad(mr, a.hi, c.lo), fx_mad(mr, a.lo, c.hi), fx_mad(mr, -b.hi, d.lo), fx_mad(mr, -b.lo, d.hi);
        fx_mad(mi, a.hi, d.lo), fx_mad(mi, a.lo, d.hi), fx_mad(mi, b.hi, c.lo), fx_mad(mi, b.lo, c.hi);
    }
    out[0] = std::ldexp((double)lu_join(hr, mr), el + eu - 2100);
    out[1] = std::ldexp((double)lu_join(hi, mi), el + eu - 2100);
}
