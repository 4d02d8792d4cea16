// Wilson hops of one output site in fixed point (fixed.cuh) on the library's
// fields: FP64 spinors, fixed-point links.
#pragma once

#include "fixed.cuh"

namespace psms {

// what the hops of one system read
struct FxHop {
    const double2 *in;   // component c of site s at in[c cs + s - off]
    long long cs, off;
    const int4 *U;       // fixed-point links
    int mode, dag;       // (dag: of the FP64 form; the integer hops take it as DAG)
    // the same spinors in fixed point (null: converted as they are read):
    // component c of site s at x[c xcs + s - xoff], exponents behind
    const longlong2 *x = nullptr;
    long long xcs = 0, xoff = 0;
    const double2 *U64 = nullptr;  // the FP64 links, if there are any (for the FP64 form)
};

// a spinor in fixed point and its exponent word (FX_BAD: out of range or not
// alike, left to the FP64 form)
__device__ __forceinline__ int fx_load_spinor(const double2 *q, long long cs, int64_t v[12][2]) {
    uint64_t w[12][2];
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        const double2 z = q[c * cs];
        w[c][0] = f64_bits(z.x);
        w[c][1] = f64_bits(z.y);
    }
    bool alike;
    const int e = fx_spinor(w, v, alike);
    return alike ? e : FX_BAD;
}

// FP64 form of one output site (with the fixed-point links if there are no others), for spinors that
// fixed point does not cover (fx_load_spinor).
static __device__ __noinline__ void fx_site_f64(const FxHop &a, const Geom &g, const BlockInfo &bi, int r, int p, int j,
                                                double2 out[12]) {
    int y[4];
    const int ll = local_lex(g, p, j, y);
    const long long s = (long long)p * g.Vh + (long long)r * g.Vbh + j;
    const double sg = a.dag ? -1.0 : 1.0;
    Spinor<double> acc;
    zero(acc);
    for (int mu = 0; mu < 4; ++mu)
        for (int b = 0; b < 2; ++b) {
            long long sn;
            int bs;
            if (!neighbour(g, bi, r, p, y, ll, mu, b ? -1 : 1, a.mode, sn, bs)) continue;
            const long long sl = b ? sn : s;
            SU3<double> u;
            if (a.U64) {
                u = load_link<Store<double>>(a.U64, g.V, mu, sl);
            } else {
                const int ue = fx_exps(a.U, g.V)[(long long)mu * g.V + sl];
                for (int e = 0; e < 9; ++e) {
                    const int4 v = a.U[((long long)mu * 9 + e) * g.V + sl];
                    u.e[e / 3][e % 3] = {fx_value(v.x, v.y, ue), fx_value(v.z, v.w, ue)};
                }
            }
            const Spinor<double> v = load_spinor<Store<double>>(a.in, a.cs, sn - a.off);
            const double tt = b ? sg : -sg;
            Half<double> h = project(mu, tt, v);
            for (int q = 0; q < 2; ++q)
                for (int c = 0; c < 3; ++c) h.c[q][c] = (double)bs * h.c[q][c];
            reconstruct_add(mu, tt, b ? su3_dag_mul(u, h) : su3_mul(u, h), acc);
        }
    for (int c = 0; c < 12; ++c) out[c] = make_double2(acc.c[c / 3][c % 3].re, acc.c[c / 3][c % 3].im);
}

// Hop d (2 mu + backward) of the output site (r, p, local coordinates yp
// packed 16 bits each, lexicographic ll, internal index s) onto acc; false
// when its numbers are out of the fixed-point range.  CONV: the spinor is
// converted here; else it is read in fixed point.
template <bool CONV, bool DAG>
__device__ __forceinline__ bool fx_dir(const FxHop &a, const Geom &g, const BlockInfo &bi, int r, int p, uint64_t yp,
                                       int ll, long long s, int d, FxAcc &acc) {
    const int mu = d >> 1, step = (d & 1) ? -1 : 1;
    const int y = (int)(yp >> (16 * mu)) & 0xFFFF;
    const bool inside = (unsigned)(y + step) < (unsigned)g.l[mu];
    if (inside ? a.mode == HOP_INTER : a.mode == HOP_INTRA) return true;
    int rn = r, lln = ll + step * g.lstride[mu];
    bool neg = false;
    if (!inside) {
        rn = bi.nbr[d];
        lln = ll - step * (g.l[mu] - 1) * g.lstride[mu];
        neg = mu == 0 && bi.B[0] == ((d & 1) ? 0 : g.nb[0] - 1);
    }
    const long long sn = (long long)(1 - p) * g.Vh + (long long)rn * g.Vbh + (lln >> 1);
    const long long sl = (d & 1) ? sn : s;
    const int ue = __ldg(fx_exps(a.U, g.V) + (long long)mu * g.V + sl);
    int2 hl[2][3][2];
    int ep;
    {
        int64_t w[12][2];
        if constexpr (CONV) {
            ep = fx_load_spinor(a.in + sn - a.off, a.cs, w);
        } else {
            const longlong2 *q = a.x + sn - a.xoff;
#pragma unroll
            for (int c = 0; c < 12; ++c) {
                const longlong2 z = q[c * a.xcs];
                w[c][0] = z.x;
                w[c][1] = z.y;
            }
            ep = reinterpret_cast<const uint16_t *>(a.x + 12 * a.xcs)[sn - a.xoff];
        }
        fx_half<DAG>(d, w, hl);
    }
    if (ep == FX_BAD || ue == FX_BAD) return false;
    if (ep == 0 || ue == 0) return true;  // a zero spinor or link adds nothing
    const long long sa = (d & 1) ? g.V : 3 * g.V, sb = (d & 1) ? 3 * g.V : g.V;  // transposed for a backward hop
    const int4 *lk = a.U + (long long)mu * 9 * g.V + sl;
    int4 v[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) v[3 * i + j] = __ldg(lk + i * sa + j * sb);
    fx_hop<DAG>(d, neg, hl, ep, v, ue, acc);
    return true;
}

// all eight, as a rolled loop: unrolled, the code misses the instruction
// cache (D_w of 32^3 x 64 3147 us instead of 1332; rolled, 0.15 stalls for
// instructions per issue)
template <bool CONV, bool DAG>
__device__ __forceinline__ bool fx_dirs(const FxHop &a, const Geom &g, const BlockInfo &bi, int r, int p, const int y[4],
                                        int ll, long long s, FxAcc &acc) {
    const uint64_t yp = (uint64_t)y[0] | (uint64_t)y[1] << 16 | (uint64_t)y[2] << 32 | (uint64_t)y[3] << 48;
    bool ok = true;
#pragma unroll 1
    for (int d = 0; d < 8; ++d) ok = fx_dir<CONV, DAG>(a, g, bi, r, p, yp, ll, s, d, acc) && ok;
    return ok;
}

// out = b (sum of the hops of D) of one output site, as one out-of-line function
// for callers whose own code is large
template <bool CONV>
static __device__ __noinline__ void fx_site(const FxHop &h, const Geom &g, const BlockInfo &bi, int r, int p, int j,
                                            double b, double2 out[12]) {
    const long long s = (long long)p * g.Vh + (long long)r * g.Vbh + j;
    int y[4];
    const int ll = local_lex(g, p, j, y);
    FxAcc acc;
    fx_zero(acc);
    double f;
    if (fx_dirs<CONV, false>(h, g, bi, r, p, y, ll, s, acc) && fx_factor(acc, b, f)) {
#pragma unroll
        for (int c = 0; c < 12; ++c)
            out[c] = c < 6 ? make_double2(f * (double)acc.up[c / 3][c % 3][0], f * (double)acc.up[c / 3][c % 3][1])
                           : make_double2(f * (double)acc.dn[c / 3 - 2][c % 3][0], f * (double)acc.dn[c / 3 - 2][c % 3][1]);
        return;
    }
    fx_site_f64(h, g, bi, r, p, j, out);
    for (int c = 0; c < 12; ++c) out[c] = make_double2(b * out[c].x, b * out[c].y);
}

}  // namespace psms
