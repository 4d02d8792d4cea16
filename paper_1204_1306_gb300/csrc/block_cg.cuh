// Dirichlet block solver for blocks of 256 sites (4^4 and the other shapes of
// that volume) with FP32 inner iterations on the even-odd operator Dhat inside
// the FP64 defect correction of block_solve.cuh, the whole solve of a (block,
// system) by one CTA of 128 threads.  The inner method is BiCGStab unless the
// context asks for CGNR: a 1e-6 reduction takes 10 iterations of two Dhat
// against 24 of Dhat and Dhat^dag (4^4 blocks, beta 5.3, kappa 0.156).  An
// item whose BiCGStab breaks down, does not get there in CG_BICG_MAX
// iterations or fails to reduce the true residual starts over with CGNR, with
// all of its iterations and steps.
//
// What bounds it: the FP32 pipe and shared memory (a hop direction is 108 FP32
// instructions on 11 shared-memory loads; an iteration has four half hops).
// So what the hops touch lives on the SM: thread j owns odd site j and keeps
// its parts of three vectors in registers, the links inside the block (59 KB
// at 4^4) and the vector that neighbours read (12 KB) are in shared memory,
// and three CTAs share an SM.  Vectors used once an iteration, and the FP64
// right-hand side, solution and residual of the defect correction are in
// global memory (L2).
//
// Measured with CGNR against the general solver: the block level of 16^4 with
// twelve systems 18.7 -> 10.8 ms, 243 blocks of 12^4 1.10 -> 0.52 ms; with
// BiCGStab 7.0 and 0.41 ms (960 us for the 512 blocks of a 16^3 x 32 lattice).
//
// FP64 has two lanes per SM here, a warp's FP64 instruction costs 16 clocks
// of them, so the iterations have none: the norms are summed exactly in
// integers (redux on two 25-bit limbs), the scalars are pairs of FP32 numbers,
// and the true residual is taken in fixed point (fixed_hop.cuh), its spinors
// converted once into the links' shared memory.
#pragma once

#include "fixed_hop.cuh"
#include "kernels.hpp"
#include "solver.hpp"

namespace psms {

constexpr int CG_NT = 128;
constexpr int CG_XF = 12 * 128 + 16;  // 16-byte elements of a parity's fixed-point spinors (fixed.cuh)
constexpr int CG_XS = 132;  // sites of an exchange row: 128, one zero site for hops that leave the block, padding

// BiCGStab iterations of one inner solve.  Where it suits the operator it needs
// far fewer (10 at kappa 0.156 and beta 5.3; 20 on a random field at kappa
// 0.25, where CGNR takes 130), where it takes more CGNR is the better one: on a
// smooth field (eps 0.3) 50 against 26 at kappa 0.2, 700 against 35 at 0.25, and
// at 0.4 it does not converge.
constexpr int CG_BICG_MAX = 48;

// sum of a CTA's FP32 numbers as hi + lo
struct ff {
    float hi, lo;
};

__device__ __forceinline__ float pow2f(int k) {  // 2^k, 0 below the normal range, k <= 127
    return k < -126 ? 0.0f : __int_as_float((k + 127) << 23);
}

// a / b to FP32 precision of the pairs
__device__ __forceinline__ float ff_div(ff a, ff b) {
    const float q = a.hi / b.hi;
    const float r = fmaf(-q, b.hi, a.hi) + (a.lo - q * b.lo);
    return q + r / b.hi;
}

// Sums over the CTA of N FP32 numbers per thread, exact for numbers down to
// 2^-26 of a warp's largest (50 bits below it): signed mantissas on the warp's
// largest exponent, two 25-bit limbs summed by redux, the four warps' sums as
// 64-bit integers, value i by lane i.  slot: one of two, alternating (one
// barrier per call).
constexpr int CG_SUMS = 7;

struct CgSums {
    int4 v[2][CG_NT / 32][CG_SUMS];  // exponent, high, low limb sums
};

template <int N>
__device__ __forceinline__ void cg_sum(const float *t, ff *out, CgSums &sm, int &slot) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const unsigned b = __float_as_uint(t[i]);
        const int e = (int)(b >> 23) & 255;
        const int em = __reduce_max_sync(0xffffffffu, e);
        const int64_t m =
            e == 0 ? 0 : (int64_t)fx_shr((uint64_t)((b & 0x7FFFFFu) | 0x800000u) << 26, (uint32_t)(em - e));
        const int64_t q = (int)b < 0 ? -m : m;
        const int hi = __reduce_add_sync(0xffffffffu, (int)(q >> 25)),
                  lo = __reduce_add_sync(0xffffffffu, (int)(q & 0x1FFFFFF));
        if (l == i) sm.v[slot][w][i] = make_int4(em, hi, lo, 0);
    }
    __syncthreads();
    float rh = 0, rl = 0;
    if (l < N) {
        int E = 0;
        int4 q[CG_NT / 32];
#pragma unroll
        for (int i = 0; i < CG_NT / 32; ++i) {
            q[i] = sm.v[slot][i][l];
            E = max(E, q[i].x);
        }
        int64_t s = 0;
#pragma unroll
        for (int i = 0; i < CG_NT / 32; ++i) {
            const int sh = min(E - q[i].x, 63);
            s += (((int64_t)q[i].y << 25) + (int64_t)q[i].z) >> sh;
        }
        // value = s 2^(E - 176), |s| < 2^57, as the exact sum of three floats
        const uint64_t a = s < 0 ? (uint64_t)-s : (uint64_t)s;
        const float p2 = (float)(int)(a >> 48) * pow2f(E - 128), p1 = (float)(int)((a >> 24) & 0xFFFFFF) * pow2f(E - 152),
                    p0 = (float)(int)(a & 0xFFFFFF) * pow2f(E - 176);
        const float x = p2 + p1, c = (p1 - (x - p2)) + p0;
        rh = x + c;
        rl = c - (rh - x);
        if (s < 0) rh = -rh, rl = -rl;
        if (E == 255) rh = rl = __int_as_float(0x7FC00000);  // infinity or NaN among them
    }
    slot ^= 1;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        out[i].hi = __shfl_sync(0xffffffffu, rh, i);
        out[i].lo = __shfl_sync(0xffffffffu, rl, i);
    }
}

__device__ __forceinline__ ff cg_sum1(float t, CgSums &sm, int &slot) {
    ff r;
    cg_sum<1>(&t, &r, sm, slot);
    return r;
}

// complex quotient, scaled against overflow of the squares
__device__ __forceinline__ cpx<float> cg_div(cpx<float> a, cpx<float> b) {
    const float m = fmaxf(fabsf(b.re), fabsf(b.im)), i = 1.0f / m;
    const float x = b.re * i, y = b.im * i, d = 1.0f / (x * x + y * y);
    return {(a.re * x + a.im * y) * d * i, (a.im * x - a.re * y) * d * i};
}

// FP64 sum over the CTA in a fixed order
__device__ __forceinline__ double cg_sum64(double v, double *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = sh[0];
#pragma unroll
    for (int i = 1; i < CG_NT / 32; ++i) t += sh[i];
    return t;
}

// Links in shared memory: direction mu holds, per parity, the sites whose link
// stays in the block (mu = 3: all), row by row of the FP32 field layout; at
// most 864 links for the shapes of 256 sites.
constexpr int CG_LINKS = 864;

struct CgLinks {
    int off[4];  // first link of direction mu
    int n[4];    // links per parity
    int sh[4];   // half index j -> j - (j >> sh) hs (sh = 31: j)
    int hs[4];
};

__device__ __forceinline__ CgLinks cg_links(const Geom &g) {
    CgLinks c;
    int o = 0;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const int h = g.lstride[mu] >> 1;  // 0 for mu = 3
        c.hs[mu] = h;
        c.sh[mu] = h ? 31 - __clz(h) + g.lsh[mu] : 31;
        c.n[mu] = 128 - (h ? h << (7 - c.sh[mu]) : 0);
        c.off[mu] = o;
        o += 2 * c.n[mu];
    }
    return c;
}

// Neighbours of a thread's site of one parity inside the block: the eight
// half indices (bytes of nb; 128, the zero site, for a hop that leaves) and
// the positions of their links (16 bits each of lk[0], lk[1])
struct CgSite {
    uint64_t nb, lk[2];
};

__device__ __forceinline__ CgSite cg_site(const Geom &g, int p, int j) {
    CgSite c;
    c.nb = c.lk[0] = c.lk[1] = 0;
    const CgLinks L = cg_links(g);
    int y[4];
    const int ll = local_lex(g, p, j, y);
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const int mu = d >> 1, sg = (d & 1) ? -1 : 1;
        const bool in = (unsigned)(y[mu] + sg) < (unsigned)g.l[mu];
        const int n = in ? (ll + sg * g.lstride[mu]) >> 1 : 128;
        c.nb |= (uint64_t)n << (8 * d);
        // the link's site: this one forward, the neighbour backward (any
        // valid link for a hop that leaves: its spinor is zero)
        const int q = (d & 1) ? 1 - p : p, i = (d & 1) ? n : j;
        const int l = in ? L.off[mu] + q * L.n[mu] + i - (i >> L.sh[mu]) * L.hs[mu] : L.off[mu];
        c.lk[d >> 2] |= (uint64_t)l << (16 * (d & 3));
    }
    return c;
}

struct CgShared {
    float4 links[4 * CG_LINKS];  // units of element pairs, [unit][link]; then the ninth elements
    float2 links9[CG_LINKS];
    float4 x[6 * CG_XS];         // the vector that neighbours read
    CgSums sums;
    double sh[CG_NT / 32];
};

__device__ __forceinline__ void cg_put(float4 *x, int j, const Spinor<float> &v) {
#pragma unroll
    for (int u = 0; u < 6; ++u) {
        const cpx<float> a = v.c[(2 * u) / 3][(2 * u) % 3], b = v.c[(2 * u + 1) / 3][(2 * u + 1) % 3];
        x[u * CG_XS + j] = make_float4(a.re, a.im, b.re, b.im);
    }
}

// sum of the hops (s = sg: +1 D, -1 D^dagger) onto the thread's site
__device__ __forceinline__ Spinor<float> cg_hop(const CgShared &sm, uint64_t nb, uint64_t lk0, uint64_t lk1, float sg) {
    Spinor<float> acc;
    zero(acc);
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const int mu = d >> 1;
        const bool fwd = (d & 1) == 0;
        const int n = (int)(nb >> (8 * d)) & 255;
        const int l = (int)((d < 4 ? lk0 : lk1) >> (16 * (d & 3))) & 0xFFFF;
        Spinor<float> v;
#pragma unroll
        for (int u = 0; u < 6; ++u) {
            const float4 w = sm.x[u * CG_XS + n];
            v.c[(2 * u) / 3][(2 * u) % 3] = {w.x, w.y};
            v.c[(2 * u + 1) / 3][(2 * u + 1) % 3] = {w.z, w.w};
        }
        const float t = fwd ? -sg : sg;
        const Half<float> h = project(mu, t, v);
        SU3<float> u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 w = sm.links[k * CG_LINKS + l];
            u.e[(2 * k) / 3][(2 * k) % 3] = {w.x, w.y};
            u.e[(2 * k + 1) / 3][(2 * k + 1) % 3] = {w.z, w.w};
        }
        const float2 w = sm.links9[l];
        u.e[2][2] = {w.x, w.y};
        reconstruct_add(mu, t, fwd ? su3_mul(u, h) : su3_dag_mul(u, h), acc);
    }
    return acc;
}

// a x + b y
__device__ __forceinline__ Spinor<float> cg_axpby(float a, const Spinor<float> &x, float b, const Spinor<float> &y) {
    Spinor<float> r;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            r.c[q][c] = {fmaf(a, x.c[q][c].re, b * y.c[q][c].re), fmaf(a, x.c[q][c].im, b * y.c[q][c].im)};
    return r;
}

// x += a y
__device__ __forceinline__ void cg_add(float a, const Spinor<float> &y, Spinor<float> &x) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x.c[q][c].re = fmaf(a, y.c[q][c].re, x.c[q][c].re);
            x.c[q][c].im = fmaf(a, y.c[q][c].im, x.c[q][c].im);
        }
}

__device__ __forceinline__ float cg_norm(const Spinor<float> &x) {
    float t = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) t = fmaf(x.c[q][c].re, x.c[q][c].re, fmaf(x.c[q][c].im, x.c[q][c].im, t));
    return t;
}

// x += a y, complex a
__device__ __forceinline__ void cg_cadd(cpx<float> a, const Spinor<float> &y, Spinor<float> &x) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) x.c[q][c] = cfma(a, y.c[q][c], x.c[q][c]);
}

// sum of conj(x) y
__device__ __forceinline__ void cg_dot(const Spinor<float> &x, const Spinor<float> &y, float *t) {
    t[0] = t[1] = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const cpx<float> a = x.c[q][c], b = y.c[q][c];
            t[0] = fmaf(a.re, b.re, fmaf(a.im, b.im, t[0]));
            t[1] = fmaf(a.re, b.im, fmaf(-a.im, b.re, t[1]));
        }
}

// The whole solve of item (block rl of the launch, system k).  The hop is one
// copy of code, used by every step of a small state machine (several inlined
// copies overflow the instruction cache).
template <class Args>
__device__ void block_cg_item(const Args &a, int rl, int k, bool bicg, CgShared &sm) {
    const Geom &g = a.g;
    const int j = threadIdx.x, r = a.rank_lo + rl;
    const long long out_i = (long long)k * a.n_ranks + rl;
    const BlockInfo &bi = a.binfo[r];
    const long long V = g.V, Vh = g.Vh;
    const long long site[2] = {(long long)r * g.Vbh + j, Vh + (long long)r * g.Vbh + j};
    const double2 *b = a.b.p + k * a.b.bs - a.b.off;
    double2 *x = a.x.p + k * a.x.bs - a.x.off;
    double2 *r64 = a.r64.p + k * a.r64.bs - a.r64.off;
    // FP32 vectors of the system in global memory: the even half of the inner
    // right-hand side (full layout), then e (full layout) and rho or rh (odd half)
    float2 *rhs_e = (float2 *)a.vin + k * a.vin_bs;
    float2 *ev = rhs_e + 12 * V, *rhov = rhs_e + 24 * V - 2 * Vh;  // (rho: odd site s at unit u Vh + s - Vh)
    bool skip = (a.sys_active && !a.sys_active[k]) || (a.block_active && !a.block_active[bi.lex]);
    double bn = 0;
    if (!skip) {
        for (int p = 0; p < 2; ++p)
            for (int q = 0; q < 12; ++q) {
                const double2 v = b[q * a.b.cs + site[p]];
                x[q * a.x.cs + site[p]] = make_double2(0, 0);
                bn = fma(v.x, v.x, fma(v.y, v.y, bn));
            }
        bn = cg_sum64(bn, sm.sh);
        skip = bn == 0.0;
    }
    if (skip) {
        if (j == 0) {
            a.iters[out_i] = 0;
            a.resid[out_i] = 0;
            a.status[out_i] = 0;
            if (a.xnorm2) a.xnorm2[out_i] = 0;
        }
        return;
    }
    if (j < 6) sm.x[j * CG_XS + 128] = make_float4(0, 0, 0, 0);
    const CgSite st_e = cg_site(g, 0, j), st_o = cg_site(g, 1, j);
    const float A = (float)a.A, c4 = (float)(-1.0 / (4.0 * a.A)), h2A = (float)(0.5 / a.A), iA = (float)(1.0 / a.A);
    int total_it = 0, spent = 0, status = 0, slot = 0;  // (spent: by BiCGStab, before CGNR started over)
    double rel = 0, rn = bn, rn_old = 0;
    double reach = 1;   // of the steps so far, with CGNR
    bool met = false;   // the tolerance, in the step before
    bool quit = false;  // BiCGStab gave up
    for (int outer = 0;; ++outer) {
        // FP64 true residual r64 = b - D_b x (r64 = b on the first step)
        if (outer > 0 && !quit) {
            // x in fixed point takes the place of the links in shared memory
            longlong2 *xs = reinterpret_cast<longlong2 *>(sm.links);
            rn = 0;
            __syncthreads();
#pragma unroll 1
            for (int p = 0; p < 2; ++p) {
                int64_t v[12][2];
                const int e = fx_load_spinor(x + site[p], a.x.cs, v);
                longlong2 *o = xs + p * CG_XF;
#pragma unroll
                for (int c = 0; c < 12; ++c) o[c * 128 + j] = make_longlong2(v[c][0], v[c][1]);
                reinterpret_cast<uint16_t *>(o + 12 * 128)[j] = (uint16_t)e;
            }
            __syncthreads();
#pragma unroll 1
            for (int p = 0; p < 2; ++p) {
                const FxHop h{x, a.x.cs, 0, a.fx + k * a.fx_bs, HOP_INTRA, 0, xs + (1 - p) * CG_XF, 128,
                              site[1 - p] - j, a.U64 ? a.U64 + k * a.U64_bs : nullptr};
                double2 hx[12];
                fx_site<false>(h, g, bi, r, p, j, 0.5, hx);
                for (int q = 0; q < 12; ++q) {
                    const double2 bv = b[q * a.b.cs + site[p]], xv = x[q * a.x.cs + site[p]];
                    const double2 v = make_double2(fma(-a.A, xv.x, bv.x + hx[q].x), fma(-a.A, xv.y, bv.y + hx[q].y));
                    r64[q * a.r64.cs + site[p]] = v;
                    rn = fma(v.x, v.x, fma(v.y, v.y, rn));
                }
            }
            rn = cg_sum64(rn, sm.sh);
        }
        // BiCGStab ends an inner solve anywhere below its target, up to a
        // decade, so that two steps of 1e-6 may land just below a tolerance of
        // 1e-13, where CGNR, which ends within a factor three of the target,
        // takes a third: one more step when aim asks for it and the tolerance is
        // below what that many steps of CGNR reach
        rel = sqrt(rn / bn);
        const double aim = bicg ? a.aim : a.tol;
        const bool last = outer >= a.max_outer || total_it >= a.maxit;
        if (!quit && (rel <= aim || (rel <= a.tol && (met || last || a.tol >= reach)))) break;
        if (bicg && (quit || last || (outer > 0 && !(rn <= 0.25 * rn_old)))) {
            // BiCGStab does not get there: the item starts over with CGNR
            bicg = quit = false;
            spent = total_it;
            total_it = outer = 0;
            for (int p = 0; p < 2; ++p)
                for (int q = 0; q < 12; ++q) x[q * a.x.cs + site[p]] = make_double2(0, 0);
            rn = bn;
            rel = 1.0;
        } else if (last) {
            status = 1;
            break;
        }
        rn_old = rn;
        met = rel <= a.tol;
        reach *= a.delta * (1.0 / 3.0);
        // inner reduction, no further than the rounding of FP64
        const float delta = (float)(bicg ? fmax(a.delta, 0x1.0p-54 / rel) : a.delta), delta2 = delta * delta;
        const double2 *src = outer ? r64 : b;
        const long long scs = outer ? a.r64.cs : a.b.cs;
        const double scale = 1.0 / sqrt(rn);
        __syncthreads();
        // links of the block
        {
            const float2 *U = (const float2 *)a.Uin + k * a.Uin_bs;
            const CgLinks L = cg_links(g);
#pragma unroll 1
            for (int t = 0; t < 8; ++t) {
                const int mu = t >> 1, q = t & 1;
                int y[4];
                local_lex(g, q, j, y);
                if (mu < 3 && y[mu] == g.l[mu] - 1) continue;
                const int l = L.off[mu] + q * L.n[mu] + j - (j >> L.sh[mu]) * L.hs[mu];
                const float2 *gb = U + (long long)mu * 9 * V;
                const float4 *g4 = reinterpret_cast<const float4 *>(gb);
#pragma unroll
                for (int u = 0; u < 4; ++u) sm.links[u * CG_LINKS + l] = __ldg(g4 + u * V + site[q]);
                sm.links9[l] = __ldg(gb + 8 * V + site[q]);
            }
        }
        // inner rhs = r64 / |r64| in FP32: even half to the exchange buffer
        // (and kept in global memory for the end), odd half in q
        Spinor<float> res, pp, q;
        for (int c = 0; c < 12; ++c) {
            const double2 v = src[c * scs + site[0]];
            q.c[c / 3][c % 3] = {(float)(v.x * scale), (float)(v.y * scale)};
        }
        store_spinor<Store<float>>(rhs_e, V, site[0], q);
        cg_put(sm.x, j, q);
        for (int c = 0; c < 12; ++c) {
            const double2 w = src[c * scs + site[1]];
            q.c[c / 3][c % 3] = {(float)(w.x * scale), (float)(w.y * scale)};
        }
        zero(res);
        zero(pp);
        store_spinor<Store<float>>(ev, V, site[1], res);  // e = 0
        __syncthreads();
        ff rr = {0, 0};
        float target = 0, alpha = 0;
        cpx<float> rho = {0, 0}, al = {0, 0};
        int it = 0;
        // steps: 0 bhat = rhs_o + H_o(rhs_e)/(2A) (kept in q).
        // CGNR (rho = bhat): 1, 2 res = Dhat^dag rho; 3, 4 q = Dhat p and the
        // updates of e, rho; 5, 6 Dhat^dag q and the updates of res, p.
        // BiCGStab (rh = bhat, r = res, v = q): 8, 9 v = Dhat p, s = r - alpha v;
        // 10, 11 t = Dhat s and the updates of e, r, p.
        // 7 e_e = (rhs_e + H_e(e)/2)/A
#pragma unroll 1
        for (int step = 0;;) {
            const bool odd = step < 8 ? (step & 1) == 0 : (step & 1) == 1;  // output parity
            const Spinor<float> acc = cg_hop(sm, odd ? st_o.nb : st_e.nb, odd ? st_o.lk[0] : st_e.lk[0],
                                             odd ? st_o.lk[1] : st_e.lk[1],
                                             step == 1 || step == 2 || step == 5 || step == 6 ? -1.0f : 1.0f);
            if (step == 0) {
                cg_add(h2A, acc, q);
                store_spinor<Store<float>>(rhov, Vh, site[1], q);
                const ff bb = cg_sum1(cg_norm(q), sm.sums, slot);
                target = bb.hi * delta2;
                step = !(bb.hi > 0) || total_it >= a.maxit ? 7 : bicg ? 8 : 1;  // (a zero right-hand side: e = 0)
                if (step == 7) q = res;
                if (step == 8) {
                    res = q;
                    pp = q;
                    rho = {bb.hi, 0};
                }
                cg_put(sm.x, j, q);
            } else if (odd == false && step != 7) {  // 1, 3, 5, 8, 10: the vector on even sites
                __syncthreads();
                cg_put(sm.x, j, acc);
                ++step;
            } else if (step == 2) {
                res = cg_axpby(A, q, c4, acc);
                pp = res;
                rr = cg_sum1(cg_norm(res), sm.sums, slot);
                cg_put(sm.x, j, pp);
                step = 3;
            } else if (step == 4) {
                q = cg_axpby(A, pp, c4, acc);
                Spinor<float> rhoc = load_spinor<Store<float>>(rhov, Vh, site[1]);
                Spinor<float> e = load_spinor<Store<float>>(ev, V, site[1]);
                const ff qq = cg_sum1(cg_norm(q), sm.sums, slot);
                alpha = ff_div(rr, qq);
                cg_add(alpha, pp, e);
                cg_add(-alpha, q, rhoc);
                store_spinor<Store<float>>(ev, V, site[1], e);
                store_spinor<Store<float>>(rhov, Vh, site[1], rhoc);
                const ff rhorho = cg_sum1(cg_norm(rhoc), sm.sums, slot);
                ++it;
                // converged, broken down (NaN included)
                const bool stop = !(rhorho.hi > target) || !(qq.hi > 0);
                cg_put(sm.x, j, stop ? e : q);
                step = stop ? 7 : 5;
            } else if (step == 6) {
                cg_add(-alpha, cg_axpby(A, q, c4, acc), res);
                const ff rn2 = cg_sum1(cg_norm(res), sm.sums, slot);
                const float beta = ff_div(rn2, rr);
                rr = rn2;
                pp = cg_axpby(beta, pp, 1.0f, res);
                const bool stop = total_it + it >= a.maxit;
                if (stop) q = load_spinor<Store<float>>(ev, V, site[1]);
                cg_put(sm.x, j, stop ? q : pp);
                step = stop ? 7 : 3;
            } else if (step == 9) {
                q = cg_axpby(A, pp, c4, acc);
                float t[2];
                cg_dot(load_spinor<Store<float>>(rhov, Vh, site[1]), q, t);
                ff d[2];
                cg_sum<2>(t, d, sm.sums, slot);
                if (!(fabsf(d[0].hi) + fabsf(d[1].hi) > 0)) {  // breakdown (NaN included)
                    quit = true;
                    break;
                } else {
                    al = cg_div(rho, {d[0].hi, d[1].hi});
                    cg_cadd({-al.re, -al.im}, q, res);  // s
                    cg_put(sm.x, j, res);
                    step = 10;
                }
            } else if (step == 11) {
                const Spinor<float> t = cg_axpby(A, res, c4, acc);
                float u[7];
                cg_dot(t, res, u);
                u[2] = cg_norm(t);
                const Spinor<float> rh = load_spinor<Store<float>>(rhov, Vh, site[1]);
                cg_dot(rh, t, u + 3);
                cg_dot(rh, res, u + 5);
                Spinor<float> e = load_spinor<Store<float>>(ev, V, site[1]);
                ff d[7];
                cg_sum<7>(u, d, sm.sums, slot);
                const float itt = d[2].hi > 0 ? 1.0f / d[2].hi : 0.0f;
                const cpx<float> om = {d[0].hi * itt, d[1].hi * itt};
                const cpx<float> w = cmul(om, cpx<float>{d[3].hi, d[4].hi});
                const cpx<float> rho1 = {d[5].hi - w.re, d[6].hi - w.im};
                const bool stalled = !(fabsf(om.re) + fabsf(om.im) > 0) || !(fabsf(rho1.re) + fabsf(rho1.im) > 0);
                cg_cadd(al, pp, e);
                cg_cadd(om, res, e);
                store_spinor<Store<float>>(ev, V, site[1], e);
                cg_cadd({-om.re, -om.im}, q, pp);    // p - omega v
                cg_cadd({-om.re, -om.im}, t, res);   // r
                const ff r2 = cg_sum1(cg_norm(res), sm.sums, slot);
                ++it;
                if (r2.hi <= target) {
                    q = e;
                    cg_put(sm.x, j, q);
                    step = 7;
                } else if (stalled || !(r2.hi == r2.hi) || it >= CG_BICG_MAX || total_it + it >= a.maxit) {
                    quit = true;
                    break;
                } else {
                    const cpx<float> be = cmul(cg_div(rho1, rho), cg_div(al, om));
                    rho = rho1;
#pragma unroll
                    for (int b = 0; b < 4; ++b)
#pragma unroll
                        for (int c = 0; c < 3; ++c) pp.c[b][c] = cfma(be, pp.c[b][c], res.c[b][c]);
                    cg_put(sm.x, j, pp);
                    step = 8;
                }
            } else {
                // the solution of the inner system, added to x in FP64
                const Spinor<float> e = load_spinor<Store<float>>(ev, V, site[1]);
                Spinor<float> ee = load_spinor<Store<float>>(rhs_e, V, site[0]);
                ee = cg_axpby(iA, ee, h2A, acc);
                const double unscale = sqrt(rn);
                for (int c = 0; c < 12; ++c) {
                    double2 v = x[c * a.x.cs + site[0]];
                    v.x = fma(unscale, (double)ee.c[c / 3][c % 3].re, v.x);
                    v.y = fma(unscale, (double)ee.c[c / 3][c % 3].im, v.y);
                    x[c * a.x.cs + site[0]] = v;
                    double2 w = x[c * a.x.cs + site[1]];
                    w.x = fma(unscale, (double)e.c[c / 3][c % 3].re, w.x);
                    w.y = fma(unscale, (double)e.c[c / 3][c % 3].im, w.y);
                    x[c * a.x.cs + site[1]] = w;
                }
                break;
            }
            __syncthreads();
        }
        total_it += it;
    }
    double xn = 0;
    if (a.xnorm2) {
        for (int p = 0; p < 2; ++p)
            for (int q = 0; q < 12; ++q) {
                const double2 v = x[q * a.x.cs + site[p]];
                xn = fma(v.x, v.x, fma(v.y, v.y, xn));
            }
        xn = cg_sum64(xn, sm.sh);
    }
    if (j == 0) {
        a.iters[out_i] = spent + total_it;
        a.resid[out_i] = rel;
        a.status[out_i] = status;
        if (a.xnorm2) a.xnorm2[out_i] = xn;
    }
}

}  // namespace psms
