// Wilson-Dirac hopping kernel, Eq. (Dw):
//   H(psi)(x) = sum_mu { U(x,mu)(1 - s gamma_mu) psi(x+mu)
//                      + U(x-mu,mu)^dagger (1 + s gamma_mu) psi(x-mu) },
// s = +1 for D and -1 for D^dagger, antiperiodic in time.  D = A - H/2 with
// A = 4 + m0.  One thread per output site; spin projection to half spinors
// (rank-2 projectors), SU(3) x half-spinor, reconstruction.  Fields use the
// structure-of-arrays even-odd block-major layout, so a warp reads each
// component of 32 consecutive sites in one coalesced transaction.
#include "bicgstab.cuh"
#include "fixed_hop.cuh"
#include "kernels.hpp"

#include <type_traits>

namespace psms {

template <class E>
struct HopArgs {
    Geom g;
    const BlockInfo *binfo;
    View<E> in, out, y, y2;
    double a, a2, b;
    const void *U;
    long long U_bs;
    int p, rank_lo, n_ranks, mode, dag;
    const int *active;
    double *partial;
    unsigned long long *prof_sites;  // profiling: output sites of active systems
    const int *sys_map;              // systems launched (null: all, k = blockIdx.y)
    const int *rank_active;          // per rank: 0 skips its output sites (null: none skipped)
    const longlong2 *fxs;            // P64: the input spinors in fixed point (fixed.cuh)
    long long fxs_bs;
    const double2 *u64;              // P64: the FP64 links beside the fixed-point ones in U (nullable)
    long long u64_bs;
    LinkInterp li;                   // shared-endpoint FP32 links (li.U0 null: U, U_bs)
    int nsf;                         // > 0: nsf systems fastest in blockIdx.x (gridDim.y = 1)
    int nct;                         // CTAs per system
    // fused BiCGStab reduction (dot 0: none; see HopDot)
    int dot;
    View<E> dx;
    BCS *dst;
    double *dpart;
    long long dpart_n;
    unsigned int *dcnt;
    int dstage, dmaxit;
    int *dflags;
};

// (launched system, CTA of that system) of this CTA
__device__ __forceinline__ void hop_cta(int nsf, int &ks, int &bx) {
    if (nsf > 0) {
        ks = (int)(blockIdx.x % (unsigned)nsf);
        bx = (int)(blockIdx.x / (unsigned)nsf);
    } else {
        ks = (int)blockIdx.y;
        bx = (int)blockIdx.x;
    }
}

// link (mu, idx) of system k: from its own field (LI = 0), or a_k U0 + b_k U1
// of the shared endpoints (LI = 1: U0 alone where the endpoints agree; LI =
// 2: always both, no flag and no divergent branch)
template <class SL, int LI, class E>
__device__ __forceinline__ SU3<typename SL::R> hop_link(const HopArgs<E> &a, const typename SL::elem *U, int k, int mu,
                                                       long long idx) {
    if constexpr (LI == 2 && SL::VSH == 1) {
        SU3<float> u = load_link<SL>(a.li.U0, a.g.V, mu, idx);
        const SU3<float> u1 = load_link<SL>(a.li.U1, a.g.V, mu, idx);
        const float2 ab = __ldg(a.li.ab + k);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                u.e[i][j].re = fmaf(ab.y, u1.e[i][j].re, ab.x * u.e[i][j].re);
                u.e[i][j].im = fmaf(ab.y, u1.e[i][j].im, ab.x * u.e[i][j].im);
            }
        return u;
    } else if constexpr (LI == 1 && SL::VSH == 1) {
        {
            SU3<float> u = load_link<SL>(a.li.U0, a.g.V, mu, idx);
            if (__ldg(a.li.flag + (long long)mu * a.g.V + idx)) {
                const SU3<float> u1 = load_link<SL>(a.li.U1, a.g.V, mu, idx);
                const float2 ab = __ldg(a.li.ab + k);
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        u.e[i][j].re = fmaf(ab.y, u1.e[i][j].re, ab.x * u.e[i][j].re);
                        u.e[i][j].im = fmaf(ab.y, u1.e[i][j].im, ab.x * u.e[i][j].im);
                    }
            }
            return u;
        }
    }
    return load_link<SL>(U, a.g.V, mu, idx);
}

// Output site of thread t (parity, rank, index in the block's half); false
// when there is none or its rank is switched off.
template <class E>
__device__ __forceinline__ bool hop_site(const HopArgs<E> &a, const Geom &g, long long t, long long total, int &p,
                                         int &r, int &j) {
    bool work = t < total;
    p = r = j = 0;
    if (work) {
        // both parities: block-major order (block, parity, site) so that the
        // two endpoints of a block's links are processed close in time and
        // each link is fetched from HBM about once per launch
        if (a.p < 0) {
            r = a.rank_lo + (int)(t >> (g.vbh_sh + 1));
            p = (int)((t >> g.vbh_sh) & 1);
            j = (int)(t & (g.Vbh - 1));
            if (a.n_ranks == g.nblocks) {
                // whole lattice: walk the blocks in lexicographic order, so
                // that a block's neighbours (opposite colour) are processed
                // soon after it and face data is still in L2
                int B[4], rem = r;
                for (int m = 3; m >= 0; --m) {
                    B[m] = rem % g.nb[m];
                    rem /= g.nb[m];
                }
                r = rank_of_lex(g, r, B);
            }
        } else {
            p = a.p;
            r = a.rank_lo + (int)(t >> g.vbh_sh);
            j = (int)(t & (g.Vbh - 1));
            if (a.n_ranks == g.nblocks && g.coloured) {
                // whole lattice, one parity: walk the blocks in lexicographic
                // order (colours interleaved), so that the faces a block
                // reads from its neighbours were loaded by CTAs that ran
                // just before and are still in L2
                int B[4], rem = r;
                for (int m = 3; m >= 0; --m) {
                    B[m] = rem % g.nb[m];
                    rem /= g.nb[m];
                }
                r = rank_of_lex(g, r, B);
            }
        }
        work = !a.rank_active || a.rank_active[r];
    }
    return work;
}

template <int NT>
__device__ __forceinline__ double block_sum(double v, double *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    double t = 0;
    if (threadIdx.x == 0) {
        for (int i = 0; i < NT / 32; ++i) t += sh[i];
    }
    return t;  // valid in thread 0
}

// Directions [D0, D1) of the branch-free whole-lattice hop of one output
// site (d = 2 mu + (0 forward, 1 backward)), accumulated into acc.
template <int D0, int D1, class S, class SL, int LI, class E>
__device__ __forceinline__ void hop_dirs(const HopArgs<E> &a, const Geom &g, const BlockInfo &bi, int r, int p,
                                         const int y[4], int ll, long long s, int k, const E *in,
                                         const typename SL::elem *U, typename SL::R sg,
                                         Spinor<typename SL::R> &acc) {
    using R = typename SL::R;
    // (below 2^31 sites: 32-bit indices keep the eight neighbours in registers)
    const int off = (int)a.in.off;
    int snb[8], bsg[8];
#pragma unroll
    for (int d = D0; d < D1; ++d) {
        long long sn;
        neighbour(g, bi, r, p, y, ll, d >> 1, (d & 1) ? -1 : 1, HOP_ALL, sn, bsg[d]);
        snb[d] = (int)sn;
    }
#pragma unroll
    for (int d = D0; d < D1; ++d) {
        const int mu = d >> 1;
        const bool fwd = (d & 1) == 0;
        Spinor<R> v = load_spinor_ro<S>(in, a.in.cs, snb[d] - off);
        const R tt = fwd ? -sg : sg;
        Half<R> h = project(mu, tt, v);
        if (mu == 0) {
            // antiperiodic time boundary: sign on the hop
            const R bsr = R(bsg[d]);
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c) h.c[q][c] = bsr * h.c[q][c];
        }
        SU3<R> u = hop_link<SL, LI>(a, U, k, mu, fwd ? s : (long long)snb[d]);
        reconstruct_add(mu, tt, fwd ? su3_mul(u, h) : su3_dag_mul(u, h), acc);
    }
}

// The dot products of an output spinor o, its 12 components summed in the
// inner precision (threads and CTAs in FP64): dot 1: <x, o>; dot 2: <o, y>,
// |o|^2, <x, o>, <x, y>
template <class R>
__device__ __forceinline__ void hop_dots(int dot, const Spinor<R> &o, const Spinor<R> &x, const Spinor<R> &y,
                                         R sum[BCG_SUMS]) {
    R xr = 0, xi = 0, yr = 0, yi = 0, aa = 0, zr = 0, zi = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const cpx<R> ov = o.c[q][c], xv = x.c[q][c];
            xr += xv.re * ov.re + xv.im * ov.im;
            xi += xv.re * ov.im - xv.im * ov.re;
            if (dot == 2) {
                const cpx<R> yv = y.c[q][c];
                yr += ov.re * yv.re + ov.im * yv.im;
                yi += ov.re * yv.im - ov.im * yv.re;
                aa += ov.re * ov.re + ov.im * ov.im;
                zr += xv.re * yv.re + xv.im * yv.im;
                zi += xv.re * yv.im - xv.im * yv.re;
            }
        }
    if (dot == 1) {
        sum[0] = xr;
        sum[1] = xi;
    } else {
        sum[0] = yr;
        sum[1] = yi;
        sum[2] = aa;
        sum[3] = xr;
        sum[4] = xi;
        sum[5] = zr;
        sum[6] = zi;
    }
}

template <int NT, class R, class E>
__device__ __forceinline__ void hop_stage(const HopArgs<E> &a, const R sum[BCG_SUMS], double (*sh)[NT / 32], int k,
                                          int bx) {
    if (a.dot == 1)
        bcg_partials_and_stage<NT, 0, 2>(a.dst, sum, a.dpart, a.dpart_n, a.dcnt, a.dstage, a.dmaxit, a.dflags, sh, k,
                                         bx, a.nct);
    else
        bcg_partials_and_stage<NT, 0, BCG_SUMS>(a.dst, sum, a.dpart, a.dpart_n, a.dcnt, a.dstage, a.dmaxit, a.dflags,
                                                sh, k, bx, a.nct);
}

// ALL = 1: specialised for HOP_ALL (every neighbour exists): the eight
// neighbour indices are computed first and the eight hops run as one
// branch-free sequence, so the compiler can issue later directions' loads
// before earlier directions' arithmetic (more loads in flight per thread).
// LI = 1: links from the shared endpoints (FP32 links only).
// SPLIT = 1 (whole lattice, FP32 arithmetic): two threads per output site in
// a CTA of NT = 256 (128 sites), the first half of the CTA summing the
// directions mu = 0, 1 and the second mu = 2, 3 (halves of whole warps, so
// no divergence); the second half's partial spinors join the first's
// through shared memory and the first half finishes the site -- half the
// per-thread state, twice the threads in flight.
// DOT = 1: with the reduction of a BiCGStab half iteration (a form of its own:
// its seven sums would cost the plain operator registers).
template <class S, class SL, int NT, int MINB, int ALL, int LI = 0, int SPLIT = 0, int DOT = 0>
__global__ void __launch_bounds__(NT, MINB) hop_kernel(const HopArgs<typename S::elem> a) {
    using R = typename SL::R;
    using E = typename S::elem;
    using EL = typename SL::elem;
    static_assert(!SPLIT || (ALL && NT == 256 && sizeof(R) == 4), "split form: whole lattice, 256 threads, FP32");
    constexpr int SN = SPLIT ? NT / 2 : NT;  // output sites per CTA
    __shared__ double sh[NT / 32];
    int ks, bx;
    hop_cta(a.nsf, ks, bx);
    const int k = a.sys_map ? a.sys_map[ks] : ks;
    if (a.active && !a.active[k]) {
        if (a.partial && threadIdx.x == 0) a.partial[(long long)k * a.nct + bx] = 0.0;
        return;
    }
    const Geom &g = a.g;
    const long long per_p = (long long)a.n_ranks * g.Vbh;
    const long long total = (a.p < 0 ? 2 : 1) * per_p;
    const int half = SPLIT ? (int)(threadIdx.x >= SN) : 0;
    const long long t = (long long)bx * SN + (threadIdx.x - half * SN);
    double nrm = 0.0;
    R dsum[BCG_SUMS] = {};  // fused BiCGStab dot partials
    int p, r, j;
    bool work = hop_site(a, g, t, total, p, r, j);
    if (a.prof_sites) {
        // output sites this warp computes (algorithmic-byte accounting)
        const unsigned cnt = __popc(__ballot_sync(0xffffffffu, work && !half));
        if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(a.prof_sites, (unsigned long long)cnt);
    }
    const long long s = (long long)p * g.Vh + (long long)r * g.Vbh + j;
    Spinor<R> acc;
    zero(acc);
    if (work) {
        int y[4];
        const int ll = local_lex(g, p, j, y);
        const BlockInfo &bi = a.binfo[r];
        const E *in = a.in.p + k * a.in.bs;
        const EL *U = (const EL *)a.U + k * a.U_bs;
        const R sg = a.dag ? R(-1) : R(1);
        if constexpr (SPLIT) {
            // warp-uniform halves: mu = 0, 1 in the first, mu = 2, 3 in the second
            if (half)
                hop_dirs<4, 8, S, SL, LI>(a, g, bi, r, p, y, ll, s, k, in, U, sg, acc);
            else
                hop_dirs<0, 4, S, SL, LI>(a, g, bi, r, p, y, ll, s, k, in, U, sg, acc);
        } else if constexpr (ALL) {
            hop_dirs<0, 8, S, SL, LI>(a, g, bi, r, p, y, ll, s, k, in, U, sg, acc);
        } else {
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
            long long sn;
            int bs;
            if (neighbour(g, bi, r, p, y, ll, mu, +1, a.mode, sn, bs)) {
                Spinor<R> v = load_spinor_ro<S>(in, a.in.cs, sn - a.in.off);
                const R tf = -sg;
                Half<R> h = project(mu, tf, v);
                if (bs < 0) {
#pragma unroll
                    for (int q = 0; q < 2; ++q)
#pragma unroll
                        for (int c = 0; c < 3; ++c) h.c[q][c] = R(-1) * h.c[q][c];
                }
                SU3<R> u = hop_link<SL, LI>(a, U, k, mu, s);
                reconstruct_add(mu, tf, su3_mul(u, h), acc);
            }
            if (neighbour(g, bi, r, p, y, ll, mu, -1, a.mode, sn, bs)) {
                Spinor<R> v = load_spinor_ro<S>(in, a.in.cs, sn - a.in.off);
                const R tb = sg;
                Half<R> h = project(mu, tb, v);
                if (bs < 0) {
#pragma unroll
                    for (int q = 0; q < 2; ++q)
#pragma unroll
                        for (int c = 0; c < 3; ++c) h.c[q][c] = R(-1) * h.c[q][c];
                }
                SU3<R> u = hop_link<SL, LI>(a, U, k, mu, sn);
                reconstruct_add(mu, tb, su3_dag_mul(u, h), acc);
            }
        }
        }
    }
    if constexpr (SPLIT) {
        // join the halves: the second half's partial spinor goes through
        // shared memory to the first, which finishes the site
        __shared__ float red[24][SN];
        if (half && work) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    red[2 * (3 * q + c)][threadIdx.x - SN] = acc.c[q][c].re;
                    red[2 * (3 * q + c) + 1][threadIdx.x - SN] = acc.c[q][c].im;
                }
        }
        __syncthreads();
        if (!half && work) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    acc.c[q][c].re += red[2 * (3 * q + c)][threadIdx.x];
                    acc.c[q][c].im += red[2 * (3 * q + c) + 1][threadIdx.x];
                }
        }
        work = work && !half;
    }
    if (work) {
        const R cb = (R)a.b;
        Spinor<R> o;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < 3; ++c) o.c[q][c] = cb * acc.c[q][c];
        if (a.y.p) {
            const R ca = (R)a.a;
            Spinor<R> v = load_spinor<S>(a.y.p + k * a.y.bs, a.y.cs, s - a.y.off);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c) o.c[q][c] = o.c[q][c] + ca * v.c[q][c];
        }
        if (a.y2.p) {
            const R ca = (R)a.a2;
            Spinor<R> v = load_spinor<S>(a.y2.p + k * a.y2.bs, a.y2.cs, s - a.y2.off);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c) o.c[q][c] = o.c[q][c] + ca * v.c[q][c];
        }
        store_spinor<S>(a.out.p + k * a.out.bs, a.out.cs, s - a.out.off, o);
        if constexpr (DOT) {
            const Spinor<R> x = load_spinor<S>(a.dx.p + k * a.dx.bs, a.dx.cs, s - a.dx.off);
            Spinor<R> yv;
            if (a.dot == 2) yv = load_spinor<S>(a.y.p + k * a.y.bs, a.y.cs, s - a.y.off);
            hop_dots(a.dot, o, x, yv, dsum);
        }
        if (a.partial) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c) nrm += (double)norm2(o.c[q][c]);
        }
    }
    if (a.partial) {
        double tot = block_sum<NT>(nrm, sh);
        if (threadIdx.x == 0) a.partial[(long long)k * a.nct + bx] = tot;
    }
    if constexpr (DOT) {
        __shared__ double shd[BCG_SUMS][NT / 32];
        hop_stage<NT, R>(a, dsum, shd, k, bx);
    }
}

// ---------------------------------------------------------------------------
// FP64 hops in fixed point (fixed.cuh, fixed_hop.cuh)
// ---------------------------------------------------------------------------
// The spinors a hop reads, in fixed point: n sites from `in` (sites [0, cs) of
// a field) of the launched systems.  A pass of its own, so that a site is
// converted once and not by each of its eight neighbours (the conversion is
// two thirds of a hop's instructions).
__global__ void __launch_bounds__(256) spinor_fx_kernel(View<double2> in, longlong2 *out, long long out_bs,
                                                        const int *sys_map, const int *active) {
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    const int k = sys_map ? sys_map[blockIdx.y] : (int)blockIdx.y;
    if (i >= in.cs || (active && !active[k])) return;
    int64_t v[12][2];
    const int e = fx_load_spinor(in.p + k * in.bs + i, in.cs, v);
    longlong2 *o = out + k * out_bs;
#pragma unroll
    for (int c = 0; c < 12; ++c) o[c * in.cs + i] = make_longlong2(v[c][0], v[c][1]);
    reinterpret_cast<uint16_t *>(o + 12 * in.cs)[i] = (uint16_t)e;
}

// one output site in FP64 (numbers out of the fixed-point range); |out|^2
static __device__ __noinline__ double hop_f64_site(const HopArgs<double2> &a, const FxHop &h, const BlockInfo &bi, int k,
                                                   int r, int p, int j) {
    const long long s = (long long)p * a.g.Vh + (long long)r * a.g.Vbh + j;
    double2 o[12];
    fx_site_f64(h, a.g, bi, r, p, j, o);
    double nrm = 0.0;
    for (int c = 0; c < 12; ++c) {
        double re = a.b * o[c].x, im = a.b * o[c].y;
        if (a.y.p) {
            const double2 w = a.y.p[k * a.y.bs + c * a.y.cs + s - a.y.off];
            re = fma(a.a, w.x, re);
            im = fma(a.a, w.y, im);
        }
        if (a.y2.p) {
            const double2 w = a.y2.p[k * a.y2.bs + c * a.y2.cs + s - a.y2.off];
            re = fma(a.a2, w.x, re);
            im = fma(a.a2, w.y, im);
        }
        a.out.p[k * a.out.bs + c * a.out.cs + s - a.out.off] = make_double2(re, im);
        nrm = fma(re, re, fma(im, im, nrm));
    }
    return nrm;
}

// One thread per output site: b (sum of hops) in integers, a y + a2 y2 and
// the result in FP64.  Latency and issue bound it (8.8k instructions per site,
// 43 % of the issue slots, FP64 pipe 38 %; the loop over directions is kept
// rolled: unrolled, its code misses the instruction cache and it is 2.4 times
// slower).  D_w of 32^3 x 64: 3340 us with FP64 arithmetic, 1332 us at three
// CTAs per SM, 1166 us at four (1.7 TB/s).
// CONV: without room for the converted input, each site is converted by the
// threads that read it.
template <int NT, int MINB, bool DAG, bool CONV>
__global__ void __launch_bounds__(NT, MINB) hop_fx_kernel(const HopArgs<double2> a) {
    __shared__ double sh[NT / 32];
    const int ks = (int)blockIdx.y, bx = (int)blockIdx.x;
    const int k = a.sys_map ? a.sys_map[ks] : ks;
    if (a.active && !a.active[k]) {
        if (a.partial && threadIdx.x == 0) a.partial[(long long)k * a.nct + bx] = 0.0;
        return;
    }
    const Geom &g = a.g;
    const long long total = (a.p < 0 ? 2 : 1) * (long long)a.n_ranks * g.Vbh;
    int p, r, j;
    const bool work = hop_site(a, g, (long long)bx * NT + threadIdx.x, total, p, r, j);
    if (a.prof_sites) {
        const unsigned cnt = __popc(__ballot_sync(0xffffffffu, work));
        if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(a.prof_sites, (unsigned long long)cnt);
    }
    double nrm = 0.0;
    if (work) {
        const long long s = (long long)p * g.Vh + (long long)r * g.Vbh + j;
        int y[4];
        const int ll = local_lex(g, p, j, y);
        const BlockInfo &bi = a.binfo[r];
        const FxHop h{a.in.p + k * a.in.bs, a.in.cs, a.in.off, (const int4 *)a.U + k * a.U_bs, a.mode, a.dag,
                      CONV ? nullptr : a.fxs + k * a.fxs_bs, a.in.cs, a.in.off,
                      a.u64 ? a.u64 + k * a.u64_bs : nullptr};
        FxAcc acc;
        fx_zero(acc);
        double f;
        if (fx_dirs<CONV, DAG>(h, g, bi, r, p, y, ll, s, acc) && fx_factor(acc, a.b, f)) {
            const double2 *yv = a.y.p ? a.y.p + k * a.y.bs + s - a.y.off : nullptr;
            const double2 *y2v = a.y2.p ? a.y2.p + k * a.y2.bs + s - a.y2.off : nullptr;
            double2 *o = a.out.p + k * a.out.bs + s - a.out.off;
#pragma unroll
            for (int c = 0; c < 12; ++c) {
                const int64_t *v = c < 6 ? acc.up[c / 3][c % 3] : acc.dn[(c - 6) / 3][c % 3];
                double re = f * (double)v[0], im = f * (double)v[1];
                if (yv) {
                    const double2 w = yv[c * a.y.cs];
                    re = fma(a.a, w.x, re);
                    im = fma(a.a, w.y, im);
                }
                if (y2v) {
                    const double2 w = y2v[c * a.y2.cs];
                    re = fma(a.a2, w.x, re);
                    im = fma(a.a2, w.y, im);
                }
                o[c * a.out.cs] = make_double2(re, im);
                if (a.partial) nrm = fma(re, re, fma(im, im, nrm));
            }
        } else {
            nrm = hop_f64_site(a, h, bi, k, r, p, j);
        }
    }
    if (a.partial) {
        const double tot = block_sum<NT>(nrm, sh);
        if (threadIdx.x == 0) a.partial[(long long)k * a.nct + bx] = tot;
    }
}

// Small launches: one warp per direction, 32 sites per CTA.  The eight
// partial sums meet in shared memory on their largest exponent, and warp w
// finishes components 3 w .. 3 w + 2.  (No partial sums of the norm.)
struct FxSplitShared {
    int64_t v[24][8][32];
    int E[8][32], ok[8][32];
};

template <bool DAG>
__global__ void __launch_bounds__(256) hop_fx_split_kernel(const HopArgs<double2> a) {
    extern __shared__ __align__(16) unsigned char fx_smem[];
    FxSplitShared &sm = *reinterpret_cast<FxSplitShared *>(fx_smem);
    const int k = a.sys_map ? a.sys_map[blockIdx.y] : (int)blockIdx.y;
    if (a.active && !a.active[k]) return;
    const Geom &g = a.g;
    const int d = (int)(threadIdx.x >> 5), l = (int)(threadIdx.x & 31);
    const long long total = (a.p < 0 ? 2 : 1) * (long long)a.n_ranks * g.Vbh;
    int p, r, j;
    const bool work = hop_site(a, g, (long long)blockIdx.x * 32 + l, total, p, r, j);
    if (a.prof_sites && d == 0) {
        const unsigned cnt = __popc(__ballot_sync(0xffffffffu, work));
        if (l == 0 && cnt) atomicAdd(a.prof_sites, (unsigned long long)cnt);
    }
    const long long s = (long long)p * g.Vh + (long long)r * g.Vbh + j;
    const FxHop h{a.in.p + k * a.in.bs, a.in.cs, a.in.off, (const int4 *)a.U + k * a.U_bs, a.mode, a.dag,
                  nullptr, 0, 0, a.u64 ? a.u64 + k * a.u64_bs : nullptr};
    FxAcc acc;
    fx_zero(acc);
    bool ok = true;
    if (work) {
        int y[4];
        const int ll = local_lex(g, p, j, y);
        const uint64_t yp = (uint64_t)y[0] | (uint64_t)y[1] << 16 | (uint64_t)y[2] << 32 | (uint64_t)y[3] << 48;
        ok = fx_dir<true, DAG>(h, g, a.binfo[r], r, p, yp, ll, s, d, acc);
    }
    sm.E[d][l] = acc.E;
    sm.ok[d][l] = ok;
    __syncthreads();
    int E = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        E = max(E, sm.E[w][l]);
        ok = ok && sm.ok[w][l];
    }
    const int sft = min(E - acc.E, 63);
#pragma unroll
    for (int c = 0; c < 12; ++c)
#pragma unroll
        for (int i = 0; i < 2; ++i)
            sm.v[2 * c + i][d][l] = (c < 6 ? acc.up[c / 3][c % 3][i] : acc.dn[(c - 6) / 3][c % 3][i]) >> sft;
    __syncthreads();
    if (!work) return;
    acc.E = E;
    double f = a.b;
    ok = ok && fx_factor(acc, a.b, f);
    double2 slow[12];
    if (!ok) fx_site_f64(h, g, a.binfo[r], r, p, j, slow);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int n = 3 * d + i, c = n >> 1, im = n & 1;  // real number n of the site's 24
        int64_t t = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += sm.v[n][w][l];
        double o = f * (double)t;
        if (!ok) o = a.b * (im ? slow[c].y : slow[c].x);
        if (a.y.p) {
            const double2 v = a.y.p[k * a.y.bs + c * a.y.cs + s - a.y.off];
            o = fma(a.a, im ? v.y : v.x, o);
        }
        if (a.y2.p) {
            const double2 v = a.y2.p[k * a.y2.bs + c * a.y2.cs + s - a.y2.off];
            o = fma(a.a2, im ? v.y : v.x, o);
        }
        reinterpret_cast<double *>(a.out.p + k * a.out.bs + c * a.out.cs + s - a.out.off)[im] = o;
    }
}

// Staged variant for whole-lattice launches on blocks of 2 x 128 sites (4^4):
// one CTA per (block, output parity, system).  The block's own input sites
// of the other parity (the neighbours of 3/4 of the hops) are copied into
// shared memory with asynchronous 16-byte copies (cp.async, past the
// registers and L1), then every direction reads its neighbour through one
// generic load sequence from shared memory (inside the block) or global
// memory (across a face), so the two cases do not split the warp.  Blocks
// are walked in lexicographic order (colours interleaved) as in the
// unstaged kernel.  Links are read from global memory as there.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// TMA = 1: the block's input rows (one contiguous 16-byte unit row of NT
// sites per spinor unit) are moved by the bulk-copy engine
// (cp.async.bulk, completion counted in bytes on an mbarrier) instead of
// per-thread 16-byte copies.  The wait is bounded; if it ran out, the
// neighbours are read from global memory instead (same values), after a
// second bounded wait for the copies in flight.
__device__ __forceinline__ bool bulk_wait(uint32_t bar, uint32_t parity) {
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred q;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, q;\n\t}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

template <class S, class SL, int NT, int MINB, int TMA = 0>
__global__ void __launch_bounds__(NT, MINB) hop_staged_kernel(const HopArgs<typename S::elem> a) {
    using R = typename SL::R;
    using E = typename S::elem;
    using EL = typename SL::elem;
    constexpr int NU = 12 >> S::VSH;  // 16-byte units per site
    __shared__ int4 stage[NU * NT];
    __shared__ double sh[NT / 32];
    const Geom &g = a.g;
    const int k = a.sys_map ? a.sys_map[blockIdx.y] : (int)blockIdx.y;
    if (a.active && !a.active[k]) {
        if (a.partial && threadIdx.x == 0) a.partial[(long long)k * gridDim.x + blockIdx.x] = 0.0;
        return;
    }
    // CTA -> (block, parity): both parities in block-major order, or one
    int p, bl;
    if (a.p < 0) {
        bl = blockIdx.x >> 1;
        p = blockIdx.x & 1;
    } else {
        bl = blockIdx.x;
        p = a.p;
    }
    int B[4], rem = bl;
    for (int m = 3; m >= 0; --m) {
        B[m] = rem % g.nb[m];
        rem /= g.nb[m];
    }
    const int r = rank_of_lex(g, bl, B);
    if (a.rank_active && !a.rank_active[r]) {
        if (a.partial && threadIdx.x == 0) a.partial[(long long)k * gridDim.x + blockIdx.x] = 0.0;
        return;
    }
    if (a.prof_sites && threadIdx.x == 0) atomicAdd(a.prof_sites, (unsigned long long)NT);
    const E *in = a.in.p + k * a.in.bs;
    // stage the block's input sites of the other parity (unit u of site s at
    // 16-byte unit u * cs + s - off)
    bool staged_ok = true;
    {
        const long long s0 = (long long)(1 - p) * g.Vh + (long long)r * g.Vbh - a.in.off;
        const int4 *src = reinterpret_cast<const int4 *>(in);
        if constexpr (TMA) {
            __shared__ __align__(8) uint64_t bar;
            const uint32_t sbar = (uint32_t)__cvta_generic_to_shared(&bar);
            if (threadIdx.x == 0) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(sbar) : "memory");
                asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(sbar),
                             "r"((uint32_t)(NU * NT * 16))
                             : "memory");
#pragma unroll
                for (int u = 0; u < NU; ++u) {
                    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&stage[u * NT]);
                    asm volatile(
                        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                            dst),
                        "l"(src + u * a.in.cs + s0), "r"((uint32_t)(NT * 16)), "r"(sbar)
                        : "memory");
                }
            }
            staged_ok = bulk_wait(sbar, 0);
            if (!staged_ok) bulk_wait(sbar, 0);
            staged_ok = __syncthreads_and(staged_ok);
            if (threadIdx.x == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(sbar) : "memory");
        } else {
#pragma unroll
            for (int u = 0; u < NU; ++u)
                cp_async16(&stage[u * NT + threadIdx.x], src + u * a.in.cs + s0 + threadIdx.x);
            cp_async_wait_all();
            __syncthreads();
        }
    }
    const int j = threadIdx.x;
    int y[4];
    const int ll = local_lex(g, p, j, y);
    const BlockInfo &bi = a.binfo[r];
    const long long s = (long long)p * g.Vh + (long long)r * g.Vbh + j;
    const EL *U = (const EL *)a.U + k * a.U_bs;
    const R sg = a.dag ? R(-1) : R(1);
    const E *sm = reinterpret_cast<const E *>(stage);
    // lattice volumes stay below 2^31 sites: 32-bit indices keep the eight
    // neighbours in registers
    const int base_opp = (int)((long long)(1 - p) * g.Vh + (long long)r * g.Vbh);
    int snb[8], idx_[8];
    unsigned inside = 0, neg = 0;
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const int mu = d >> 1, sgn = (d & 1) ? -1 : 1;
        long long sn;
        int bs;
        neighbour(g, bi, r, p, y, ll, mu, sgn, HOP_ALL, sn, bs);
        snb[d] = (int)sn;
        if (bs < 0) neg |= 1u << d;
        const int yn = y[mu] + sgn;
        if (staged_ok && (unsigned)yn < (unsigned)g.l[mu]) {
            inside |= 1u << d;
            idx_[d] = snb[d] - base_opp;
        } else {
            idx_[d] = snb[d] - (int)a.in.off;
        }
    }
    Spinor<R> acc;
    zero(acc);
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const int mu = d >> 1;
        const bool fwd = (d & 1) == 0;
        const bool ins = (inside >> d) & 1;
        Spinor<R> v = load_spinor<S>(ins ? sm : in, ins ? (long long)NT : a.in.cs, idx_[d]);
        const R tt = fwd ? -sg : sg;
        Half<R> h = project(mu, tt, v);
        if (mu == 0 && ((neg >> d) & 1)) {
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int c = 0; c < 3; ++c) h.c[q][c] = R(-1) * h.c[q][c];
        }
        SU3<R> u = load_link<SL>(U, g.V, mu, fwd ? s : (long long)snb[d]);
        reconstruct_add(mu, tt, fwd ? su3_mul(u, h) : su3_dag_mul(u, h), acc);
    }
    const R cb = (R)a.b;
    Spinor<R> o;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) o.c[q][c] = cb * acc.c[q][c];
    if (a.y.p) {
        const R ca = (R)a.a;
        Spinor<R> v = load_spinor<S>(a.y.p + k * a.y.bs, a.y.cs, s - a.y.off);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < 3; ++c) o.c[q][c] = o.c[q][c] + ca * v.c[q][c];
    }
    if (a.y2.p) {
        const R ca = (R)a.a2;
        Spinor<R> v = load_spinor<S>(a.y2.p + k * a.y2.bs, a.y2.cs, s - a.y2.off);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < 3; ++c) o.c[q][c] = o.c[q][c] + ca * v.c[q][c];
    }
    store_spinor<S>(a.out.p + k * a.out.bs, a.out.cs, s - a.out.off, o);
    if (a.partial) {
        double nrm = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < 3; ++c) nrm += (double)norm2(o.c[q][c]);
        double tot = block_sum<NT>(nrm, sh);
        if (threadIdx.x == 0) a.partial[(long long)k * gridDim.x + blockIdx.x] = tot;
    }
}

static constexpr int HOP_NT = 128;
constexpr long long FX_SPLIT_SITES = 152 * 128;  // output sites of all systems (hop_launch_t gives both sides)

// The FP32 forms, by the number psms_hop_variant takes.  part: general form,
// register caps 2, 6, 7, 8 CTAs/SM.  whole (whole lattice): the same, the
// branch-free form with caps 4 to 7, two threads per site (8, 9), staged forms
// (10 to 13: blocks of 2 x 128 sites only).
// li (whole lattice, links shared by the endpoints): caps 2 to 8, general and
// branch-free forms, flagged or unconditional U1 reads, two threads per site
// (13, 14).
template <class S, class SL, int D>
struct HopVars {
    using KFn = void (*)(const HopArgs<typename S::elem>);
    static constexpr int N = HOP_NT, W = 2 * HOP_NT;
    static constexpr KFn part[] = {hop_kernel<S, SL, N, 2, 0, 0, 0, D>, hop_kernel<S, SL, N, 6, 0, 0, 0, D>,
                                   hop_kernel<S, SL, N, 7, 0, 0, 0, D>, hop_kernel<S, SL, N, 8, 0, 0, 0, D>};
    static constexpr KFn whole[] = {part[0], part[1], part[2], part[3],
                                    hop_kernel<S, SL, N, 4, 1, 0, 0, D>, hop_kernel<S, SL, N, 5, 1, 0, 0, D>,
                                    hop_kernel<S, SL, N, 6, 1, 0, 0, D>, hop_kernel<S, SL, N, 7, 1, 0, 0, D>,
                                    hop_kernel<S, SL, W, 3, 1, 0, 1, D>, hop_kernel<S, SL, W, 4, 1, 0, 1, D>,
                                    hop_staged_kernel<S, SL, N, 4>, hop_staged_kernel<S, SL, N, 6>,
                                    hop_staged_kernel<S, SL, N, 4, 1>, hop_staged_kernel<S, SL, N, 6, 1>};
    static constexpr int whole_nt[] = {N, N, N, N, N, N, N, N, W, W, N, N, N, N};
    static constexpr KFn li[] = {hop_kernel<S, SL, N, 2, 0, 1, 0, D>, hop_kernel<S, SL, N, 4, 0, 1, 0, D>,
                                 hop_kernel<S, SL, N, 2, 1, 1, 0, D>, hop_kernel<S, SL, N, 3, 1, 1, 0, D>,
                                 hop_kernel<S, SL, N, 4, 1, 1, 0, D>, hop_kernel<S, SL, N, 5, 1, 1, 0, D>,
                                 hop_kernel<S, SL, N, 6, 0, 1, 0, D>, hop_kernel<S, SL, N, 8, 0, 1, 0, D>,
                                 hop_kernel<S, SL, N, 6, 1, 1, 0, D>, hop_kernel<S, SL, N, 4, 0, 2, 0, D>,
                                 hop_kernel<S, SL, N, 6, 0, 2, 0, D>, hop_kernel<S, SL, N, 4, 1, 2, 0, D>,
                                 hop_kernel<S, SL, N, 6, 1, 2, 0, D>, hop_kernel<S, SL, W, 2, 1, 1, 1, D>,
                                 hop_kernel<S, SL, W, 3, 1, 1, 1, D>};
    static constexpr int li_nt[] = {N, N, N, N, N, N, N, N, N, N, N, N, N, W, W};
};

int hop_ctas(psms_ctx *c, const HopCall &h) {
    const int nr = h.n_ranks < 0 ? c->g.nblocks : h.n_ranks;
    const long long total = (h.p < 0 ? 2LL : 1LL) * nr * c->g.Vbh;
    return (int)((total + HOP_NT - 1) / HOP_NT);
}

template <class S, class SL>
static int hop_launch_t(psms_ctx *c, const HopCall &h) {
    using E = typename S::elem;
    HopArgs<E> a;
    a.g = c->g;
    a.binfo = c->d_binfo;
    auto cv = [](const View<void> &v) {
        View<E> w;
        w.p = (E *)v.p;
        w.cs = v.cs;
        w.off = v.off;
        w.bs = v.bs;
        return w;
    };
    a.in = cv(h.in);
    a.out = cv(h.out);
    a.y = cv(h.y);
    a.y2 = cv(h.y2);
    a.a = h.a;
    a.a2 = h.a2;
    a.b = h.b;
    a.U = h.U;
    a.U_bs = h.U_bs;
    a.p = h.p;
    a.rank_lo = h.rank_lo;
    a.n_ranks = h.n_ranks < 0 ? c->g.nblocks : h.n_ranks;
    a.mode = h.mode;
    a.dag = h.dag;
    a.active = h.active;
    a.partial = h.partial;
    a.prof_sites = nullptr;
    a.sys_map = h.sys_map;
    a.rank_active = h.rank_active;
    a.fxs = nullptr;
    a.fxs_bs = 0;
    a.u64 = h.prec == P64 ? (const double2 *)h.U : nullptr;
    a.u64_bs = h.U_bs;
    const bool shared_links = h.li.U0 != nullptr;
    a.li = h.li;
    a.dot = h.dot.dot;
    a.dx = cv(h.dot.x);
    a.dst = h.dot.st;
    a.dpart = h.dot.part;
    a.dpart_n = h.dot.part_n;
    a.dcnt = h.dot.cnt;
    a.dstage = h.dot.stage;
    a.dmaxit = h.dot.maxit;
    a.dflags = h.dot.flags;
    if (a.dot && (h.prec != P32 || h.p < 0 || !h.dot.st || !h.dot.cnt || (a.dot == 2 && !h.y.p) ||
                  !h.dot.x.p))
        fail(PSMS_EINVAL, "hop_launch: a fused reduction needs FP32 storage, one parity and its vectors");
    if (shared_links) {
        if (h.prec == P64 || !h.li.U1 || !h.li.ab || !h.li.flag)
            fail(PSMS_EINVAL, "hop_launch: shared-endpoint links need FP32 storage, U1, ab and flags");
        a.U = h.li.U0;
        a.U_bs = 0;
    }
    const int nct = hop_ctas(c, h);
    const int nsys = h.sys_map ? h.n_map : h.n_sys;
    if (nct == 0 || nsys == 0) return 0;
    // FP64 hops in fixed point (fixed.cuh).  Few output sites, or a few blocks
    // of a large lattice (whose other sites need no conversion): the
    // directions of a site go to eight warps, which convert what they read;
    // else a pass converts the input first (no room for its copy: converted as
    // it is read, which needs no memory).  Directions / pass, us per D_w: 4096
    // sites 8.4 / 28.9, 8192 14.5 / 29.0, 16384 23.7 / 28.9, 32768 39.1 / 36.4,
    // 65536 77 / 54.
    const bool fixed = std::is_same<S, Store<double>>::value && h.fx != nullptr;
    const long long per = (h.p < 0 ? 2LL : 1LL) * a.n_ranks * c->g.Vbh;
    const bool fx_split = !h.partial && (per * nsys <= FX_SPLIT_SITES || 8LL * a.n_ranks <= c->g.nblocks);
    if (fixed && !fx_split) {
        fx_wait(c);  // (first: a smaller copy in use on another stream may be given back here)
        a.fxs_bs = fx_spinors(a.in.cs);
        a.fxs = (longlong2 *)scratch_try(c, "hop_fx", sizeof(longlong2) * (size_t)a.fxs_bs * h.n_sys);
    }
    if (fixed) {
        a.U = h.fx;
        a.U_bs = h.fx_bs;
    }
    a.nct = nct;
    // shared-endpoint links: the systems of a launch run side by side (CTA
    // index = cta * nsys + system), so each endpoint link leaves HBM once
    a.nsf = shared_links ? nsys : 0;
    const dim3 grid = shared_links ? dim3((unsigned)((long long)nct * nsys), 1) : dim3(nct, nsys);
    double bytes = 0;
    int slot = -1;
    if (c->prof && h.mode == HOP_ALL && (c->prof_prec < 0 || c->prof_prec == h.prec)) {
        // algorithmic bytes per output site of an active system: in + out
        // (+ y, y2, + the fused reduction's vector) spinors and 4 links
        // (both parities) or 8 (one parity) of that system's field -- also
        // with shared-endpoint links, whose HBM traffic is lower (the
        // systems share the endpoint links through L2); the device counts
        // the output sites of the systems still active
        const double sp = 12.0 * sizeof(E), lk = 9.0 * sizeof(typename SL::elem);
        const double links = 4 * lk * (h.p < 0 ? 1 : 2);
        bytes = 2 * sp + (h.y.p ? sp : 0) + (h.y2.p ? sp : 0) + (a.dot ? sp : 0) + links;
        slot = prof_begin(c);
        a.prof_sites = prof_counter(c, slot);
    }
    if constexpr (std::is_same<S, Store<double>>::value) {
        if (fixed) {
            if (fx_split) {
                const auto fn = h.dag ? hop_fx_split_kernel<true> : hop_fx_split_kernel<false>;
                cuda_check(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                (int)sizeof(FxSplitShared)),
                           "hop shared memory");
                fn<<<dim3((unsigned)((per + 31) / 32), nsys), 256, sizeof(FxSplitShared), c->stream>>>(a);
            } else if (a.fxs) {
                spinor_fx_kernel<<<dim3((unsigned)((a.in.cs + 255) / 256), nsys), 256, 0, c->stream>>>(
                    a.in, const_cast<longlong2 *>(a.fxs), a.fxs_bs, h.sys_map, h.active);
                PSMS_LAUNCH_CHECK("spinor_fx_kernel");
                const auto fn = h.dag ? hop_fx_kernel<HOP_NT, 4, true, false> : hop_fx_kernel<HOP_NT, 4, false, false>;
                fn<<<grid, HOP_NT, 0, c->stream>>>(a);
                fx_mark(c);
            } else {
                const auto fn = h.dag ? hop_fx_kernel<HOP_NT, 4, true, true> : hop_fx_kernel<HOP_NT, 4, false, true>;
                fn<<<grid, HOP_NT, 0, c->stream>>>(a);
            }
            PSMS_LAUNCH_CHECK("hop_fx_kernel");
            if (slot >= 0) prof_end(c, slot, bytes);
            return nct;
        }
    }
    // Register cap (minimum resident CTAs per SM) chosen by the autotuner:
    // on the first launch of each (precision, parity shape) every variant is
    // timed twice with CUDA events and the fastest is kept, among those that do
    // identical arithmetic: the forms with two threads per site add the hops in
    // another order, and a choice by time must not change the bits (an
    // ill-conditioned solve takes another number of steps with them).  A launch
    // is idempotent (out is a function of in, y, y2, U only), so the extra tuning
    // launches leave the result unchanged.
    using KFn = void (*)(const HopArgs<E>);
    constexpr bool f32 = sizeof(typename SL::R) == 4;
    const bool all = h.mode == HOP_ALL;
    // the staged kernel: whole lattice, 128 sites of each parity per block
    const bool staged = all && a.n_ranks == c->g.nblocks && h.rank_lo == 0 && c->g.Vbh == HOP_NT;
    const KFn *vars;
    const int *thr = nullptr;  // threads per CTA of each variant (null: all HOP_NT)
    int nvar;
    if constexpr (f32) {
        using V = HopVars<S, SL, 0>;
        vars = shared_links ? V::li : (all ? V::whole : V::part);
        thr = shared_links ? V::li_nt : (all ? V::whole_nt : nullptr);
        if constexpr (std::is_same<S, Store<float>>::value) {
            using D = HopVars<S, SL, 1>;
            if (a.dot) vars = shared_links ? D::li : (all ? D::whole : D::part);
        }
        if (shared_links && !all) fail(PSMS_EINVAL, "hop_launch: shared-endpoint links on whole-lattice hops only");
        nvar = shared_links ? 15 : (all ? (staged ? 14 : 10) : 4);
    } else {
        // FP64 arithmetic (captured calls, no room for the links in fixed point):
        // bound by the FP64 pipe, every register cap and the branch-free form
        // within 0.6 % (D_w of 32^3 x 64 3339 to 3359 us)
        static const KFn v64[] = {hop_kernel<S, SL, HOP_NT, 2, 0>};
        vars = v64;
        nvar = 1;
    }
    int &choice = c->hop_variant[h.prec][h.p < 0 ? 1 : 0][all ? 1 : 0][shared_links ? 1 : 0];
    // (launches with a fused reduction are not used for tuning: they advance
    // the solver's scalars; nor are captured ones, which cannot be timed)
    if (choice < 0 && c->autotune && nvar > 1 && slot < 0 && c->forced_hop_variant < 0 && !a.dot && !capturing(c)) {
        cudaEvent_t e0, e1;
        cuda_check(cudaEventCreate(&e0), "tune event");
        cuda_check(cudaEventCreate(&e1), "tune event");
        float best = 1e30f;
        for (int v = 0; v < nvar; ++v) {
            if (thr && thr[v] != HOP_NT) continue;  // (two threads per site)
            vars[v]<<<grid, thr ? thr[v] : HOP_NT, 0, c->stream>>>(a);
            cuda_check(cudaEventRecord(e0, c->stream), "tune record");
            vars[v]<<<grid, thr ? thr[v] : HOP_NT, 0, c->stream>>>(a);
            vars[v]<<<grid, thr ? thr[v] : HOP_NT, 0, c->stream>>>(a);
            cuda_check(cudaEventRecord(e1, c->stream), "tune record");
            cuda_check(cudaEventSynchronize(e1), "tune sync");
            launch_counter() += 3;
            float ms = 0;
            cuda_check(cudaEventElapsedTime(&ms, e0, e1), "tune elapsed");
            if (ms < best) {
                best = ms;
                choice = v;
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        PSMS_LAUNCH_CHECK("hop_kernel (autotune)");
    }
    int v = (choice >= 0 && choice < nvar) ? choice : (f32 ? 1 : 0);
    if (c->forced_hop_variant >= 0) v = c->forced_hop_variant % nvar;
    // the staged kernels (10 to 13) carry no fused reduction
    if (a.dot && !shared_links && all && v >= 10) v = 6;
    vars[v]<<<grid, thr ? thr[v] : HOP_NT, 0, c->stream>>>(a);
    PSMS_LAUNCH_CHECK("hop_kernel");
    if (slot >= 0) prof_end(c, slot, bytes);
    return nct;
}

int hop_launch(psms_ctx *c, const HopCall &h) {
    switch (h.prec) {
        case P64: return hop_launch_t<Store<double>, Store<double>>(c, h);
        case P32: return hop_launch_t<Store<float>, Store<float>>(c, h);
        case PB16: return hop_launch_t<Store<__nv_bfloat16>, Store<float>>(c, h);
    }
    fail(PSMS_EINVAL, "hop_launch: bad precision");
}

// --- deterministic reductions ------------------------------------------------

template <int NT>
__global__ void __launch_bounds__(NT) reduce_partials_kernel(const double *partial, int n, double *out) {
    __shared__ double sh[NT / 32];
    const int k = blockIdx.x;
    double v = 0;
    for (int i = threadIdx.x; i < n; i += NT) v += partial[(long long)k * n + i];
    double t = block_sum<NT>(v, sh);
    if (threadIdx.x == 0) out[k] = t;
}

void reduce_partials(psms_ctx *c, const double *partial, int n, int n_sys, double *out) {
    reduce_partials_kernel<256><<<n_sys, 256, 0, c->stream>>>(partial, n, out);
    PSMS_LAUNCH_CHECK("reduce_partials");
}

template <class S, int NT>
__global__ void __launch_bounds__(NT) norm2_kernel(View<typename S::elem> v, long long s_lo, long long n,
                                                   double *partial) {
    __shared__ double sh[NT / 32];
    const int k = blockIdx.y;
    double acc = 0;
    for (long long i = (long long)blockIdx.x * NT + threadIdx.x; i < n; i += (long long)gridDim.x * NT) {
        const long long s = s_lo + i;
        for (int q = 0; q < 12; ++q) acc += (double)norm2(S::ld(v.p + k * v.bs, q, v.cs, s - v.off));
    }
    double t = block_sum<NT>(acc, sh);
    if (threadIdx.x == 0) partial[(long long)k * gridDim.x + blockIdx.x] = t;
}

void norm2_batch(psms_ctx *c, int prec, View<void> v, long long s_lo, long long n, int n_sys, double *out) {
    const int NT = 256;
    int nct = (int)std::min<long long>((n + NT - 1) / NT, 1024);
    if (nct < 1) nct = 1;
    double *partial = (double *)scratch(c, "norm2_partial", sizeof(double) * (size_t)nct * n_sys);
    dim3 grid(nct, n_sys);
    switch (prec) {
        case P64: {
            View<double2> w{(double2 *)v.p, v.cs, v.off, v.bs};
            norm2_kernel<Store<double>, NT><<<grid, NT, 0, c->stream>>>(w, s_lo, n, partial);
            break;
        }
        case P32: {
            View<float2> w{(float2 *)v.p, v.cs, v.off, v.bs};
            norm2_kernel<Store<float>, NT><<<grid, NT, 0, c->stream>>>(w, s_lo, n, partial);
            break;
        }
        default: {
            View<__nv_bfloat162> w{(__nv_bfloat162 *)v.p, v.cs, v.off, v.bs};
            norm2_kernel<Store<__nv_bfloat16>, NT><<<grid, NT, 0, c->stream>>>(w, s_lo, n, partial);
            break;
        }
    }
    PSMS_LAUNCH_CHECK("norm2_kernel");
    reduce_partials(c, partial, nct, n_sys, out);
}

}  // namespace psms
