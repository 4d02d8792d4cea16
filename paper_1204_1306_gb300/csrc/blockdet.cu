// Exact determinants of the Dirichlet block operators (Sec. 3: the paper
// computes small-block determinants exactly by LU; Tables 1 and 2 put
// coefficients on this exact action).
//
// For a block b, D_b = [[A, D_eo], [D_oe, A]] over its even and odd sites
// (A = 4 + m0, D_eo = -H_eo / 2 the hops of Eq. (Dw) that stay in the block),
// so det D_b = A^{n_e} det(A - D_oe D_eo / A): the even-odd reduced operator
// Dhat_b on the block's odd sites, an n x n complex matrix with
// n = 12 Vb / 2 (1536 for a 4^4 block).  For all blocks of a batch:
//   1. assemble Dhat_b column by column (a thread per column applies the two
//      hops to a unit vector and scatters the result; column-major storage);
//   2. LU with partial pivoting, right-looking (below);
//   3. ln|det D_b| = n_e ln A + sum_j ln|u_jj|, summed in a fixed order.
// FP64 accuracy throughout (the update in integers, errors no larger than those
// of FP64 chains on such factors): the level built on it is exact, and its Delta is
// compared across devices.
#include <cmath>
#include <string>
#include <vector>

#include "blockdet.hpp"
#include "fixed.cuh"

namespace psms {
namespace {

constexpr int kNb = 16;       // panel width
constexpr int kSub = 8;       // sub-panel width (two rows of it per thread stay in registers)
constexpr int kPanelNT = 768; // 1536 rows (a 4^4 block) in two
constexpr int kTileR = 64, kTileC = 32;  // trailing-update tile (rows, columns)
constexpr int kUpdNT = 256;   // 16 x 16 threads, 4 x 2 outputs each
constexpr int kMaxBlockSites = 1024;  // n <= 6144: at most 0.6 GB and 6e11 flop per block

__device__ __forceinline__ cpx<double> ld(const double2 *p) {
    const double2 v = *p;
    return {v.x, v.y};
}
__device__ __forceinline__ void st(double2 *p, cpx<double> v) { *p = make_double2(v.re, v.im); }

// Column col of Dhat_b for rank r = rank_lo + blockIdx-derived matrix index.
// Row / column index of (odd site with half-block index j, component c):
// 12 j + c.
__global__ void assemble_kernel(Geom g, const BlockInfo *binfo, const double2 *U, int rank_lo, int n_mat, double A,
                                double2 *M) {
    const int n = 12 * g.Vbh;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)n_mat * n) return;
    const int m = (int)(t / n), col = (int)(t - (long long)m * n);
    const int r = rank_lo + m;
    const BlockInfo &bi = binfo[r];
    double2 *out = M + (long long)m * n * n + (long long)col * n;  // zeroed by the caller
    const int jy = col / 12, cy = col % 12;
    int y[4];
    const int lly = local_lex(g, 1, jy, y);
    const long long sy = (long long)g.Vh + (long long)r * g.Vbh + jy;
    Spinor<double> e;
    zero(e);
    e.c[cy / 3][cy % 3] = mk<double>(1.0, 0.0);
    const double f = -0.25 / A;  // -(1/A) (1/2)(1/2): Dhat = A - (H_oe/2)(H_eo/2)/A
    for (int mu = 0; mu < 4; ++mu)
        for (int sg = -1; sg <= 1; sg += 2) {
            // w = (H e)(z) at the even neighbour z = y + sg mu inside the block
            long long sz;
            int bsg;
            if (!neighbour(g, bi, r, 1, y, lly, mu, sg, HOP_INTRA, sz, bsg)) continue;
            Spinor<double> w;
            zero(w);
            if (sg > 0) {  // z - mu = y: backward term U(y,mu)^dag (1 + gamma_mu) e
                const Half<double> h = su3_dag_mul(load_link<Store<double>>(U, g.V, mu, sy), project(mu, 1.0, e));
                reconstruct_add(mu, 1.0, h, w);
            } else {       // z + mu = y: forward term U(z,mu) (1 - gamma_mu) e
                const Half<double> h = su3_mul(load_link<Store<double>>(U, g.V, mu, sz), project(mu, -1.0, e));
                reconstruct_add(mu, -1.0, h, w);
            }
            int z[4] = {y[0], y[1], y[2], y[3]};
            z[mu] += sg;
            const int llz = lly + sg * g.lstride[mu];
            for (int nu = 0; nu < 4; ++nu)
                for (int sh = -1; sh <= 1; sh += 2) {
                    long long sx;
                    int bsx;
                    if (!neighbour(g, bi, r, 0, z, llz, nu, sh, HOP_INTRA, sx, bsx)) continue;
                    Spinor<double> v;
                    zero(v);
                    if (sh > 0) {  // x - nu = z: U(z,nu)^dag (1 + gamma_nu) w
                        const Half<double> h =
                            su3_dag_mul(load_link<Store<double>>(U, g.V, nu, sz), project(nu, 1.0, w));
                        reconstruct_add(nu, 1.0, h, v);
                    } else {       // x + nu = z: U(x,nu) (1 - gamma_nu) w
                        const Half<double> h = su3_mul(load_link<Store<double>>(U, g.V, nu, sx), project(nu, -1.0, w));
                        reconstruct_add(nu, -1.0, h, v);
                    }
                    const int jx = (int)(sx - (long long)g.Vh - (long long)r * g.Vbh);
                    double2 *o = out + 12 * jx;
#pragma unroll
                    for (int q = 0; q < 12; ++q) {
                        const cpx<double> a = ld(o + q);
                        st(o + q, a + f * v.c[q / 3][q % 3]);
                    }
                }
        }
    double2 *d = out + col;
    const cpx<double> a = ld(d);
    st(d, a + mk<double>(A, 0.0));
}

// deterministic argmax of |a|^2 over a CTA: larger value wins, the lower
// row index on ties
__device__ __forceinline__ void argmax_pair(double &v, int &i, double v2, int i2) {
    if (v2 > v || (v2 == v && i2 < i)) {
        v = v2;
        i = i2;
    }
}

// 2^k (zero or infinity beyond the range)
__device__ __forceinline__ double lu_scale(int k) {
    if (k < -1022 || k > 1023) return ldexp(1.0, k);
    return f64_from_bits((uint64_t)(k + 1023) << 52);
}

// The LU is right-looking in panels of kNb columns, each factored as two
// sub-panels of kSub:
//   lu_panel_kernel   columns [k, k + kSub), one CTA per matrix;
//   lu_solve_kernel   row swaps and U12 = L11^-1 A12 on the columns to the right;
//   lu_update_kernel  A22 -= L21 U12 on the trailing matrix.
// Pivots (kSub or kNb of them per step) go through piv[m n + j].

// Sub-panel [k, k + kSub) of matrix blockIdx.x by partial pivoting; row swaps
// also on the columns [swap_lo, k) of the same panel.  logu[m n + j] = ln|u_jj|.
//
// FP64 lanes bound it (160 instructions per row, two lanes on the one SM that
// a matrix occupies: 59 us for 1536 rows), so a thread keeps its RPT rows in
// registers, the pivot search compares |a|^2 as integers (redux), the inverse
// of the pivot is formed once, by the thread that owns the row, and no FP64
// instruction is spent on bookkeeping.
template <int RPT>
__global__ void __launch_bounds__(kPanelNT) lu_panel_kernel(double2 *Mall, int n, int k, int swap_lo, int *piv,
                                                            double *logu) {
    __shared__ uint32_t s_hi[kPanelNT / 32], s_lo[kPanelNT / 32];
    __shared__ int s_row[kPanelNT / 32];
    __shared__ cpx<double> prow[kSub + 1], jrow[kSub];  // pivot row (and its inverse pivot), row j
    const int m = blockIdx.x, tid = threadIdx.x;
    double2 *M = Mall + (long long)m * n * n;
    cpx<double> a[RPT][kSub];
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const int i = k + tid + r * kPanelNT;
#pragma unroll
        for (int c = 0; c < kSub; ++c) a[r][c] = i < n ? ld(M + (long long)(k + c) * n + i) : mk<double>(0.0, 0.0);
    }
#pragma unroll
    for (int jj = 0; jj < kSub; ++jj) {
        const int j = k + jj;
        // largest |a_ij|^2 over the rows i >= j, the lowest row on ties
        unsigned long long best = 0;
        int row = 0x7FFFFFFF;
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const int i = k + tid + r * kPanelNT;
            if (i >= j && i < n) {
                const unsigned long long v = (unsigned long long)__double_as_longlong(norm2(a[r][jj]));
                if (row == 0x7FFFFFFF || v > best) {
                    best = v;
                    row = i;
                }
            }
        }
        uint32_t hi = row == 0x7FFFFFFF ? 0u : (uint32_t)(best >> 32), lo = (uint32_t)best;
        uint32_t mh = __reduce_max_sync(0xffffffffu, hi);
        bool top = hi == mh && row != 0x7FFFFFFF;
        uint32_t ml = __reduce_max_sync(0xffffffffu, top ? lo : 0u);
        int mr = __reduce_min_sync(0xffffffffu, top && lo == ml ? row : 0x7FFFFFFF);
        if ((tid & 31) == 0) {
            s_hi[tid >> 5] = mh;
            s_lo[tid >> 5] = ml;
            s_row[tid >> 5] = mr;
        }
        __syncthreads();
        {
            const int l = tid & 31;
            const bool in = l < kPanelNT / 32;
            hi = in ? s_hi[l] : 0u;
            lo = in ? s_lo[l] : 0u;
            row = in ? s_row[l] : 0x7FFFFFFF;
            mh = __reduce_max_sync(0xffffffffu, row == 0x7FFFFFFF ? 0u : hi);
            top = hi == mh && row != 0x7FFFFFFF;
            ml = __reduce_max_sync(0xffffffffu, top ? lo : 0u);
            mr = __reduce_min_sync(0xffffffffu, top && lo == ml ? row : 0x7FFFFFFF);
        }
        const int p = mr;  // rows j .. n - 1 are never empty
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const int i = k + tid + r * kPanelNT;
            if (i == p) {
                const cpx<double> pv = a[r][jj];
                const double pn = norm2(pv);
#pragma unroll
                for (int c = 0; c < kSub; ++c) prow[c] = a[r][c];
                // a singular pivot gives non-finite values the host detects
                prow[kSub] = {pv.re / pn, -pv.im / pn};
                piv[(long long)m * n + j] = p;
                logu[(long long)m * n + j] = 0.5 * log(pn);
            }
            if (i == j) {
#pragma unroll
                for (int c = 0; c < kSub; ++c) jrow[c] = a[r][c];
            }
        }
        __syncthreads();
        const cpx<double> inv = prow[kSub];
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            const int i = k + tid + r * kPanelNT;
            if (i == p && p != j) {
#pragma unroll
                for (int c = 0; c < kSub; ++c) a[r][c] = jrow[c];
            }
            if (i == j) {
#pragma unroll
                for (int c = 0; c < kSub; ++c) a[r][c] = prow[c];
            } else if (i > j && i < n) {
                const cpx<double> l = cmul(a[r][jj], inv);
                a[r][jj] = l;
#pragma unroll
                for (int c = jj + 1; c < kSub; ++c) {
                    const cpx<double> u = prow[c];
                    a[r][c] = cfma(mk<double>(-l.re, -l.im), u, a[r][c]);
                }
            }
        }
        // the same rows in the panel's earlier columns
        if (p != j && tid < k - swap_lo) {
            double2 *cc = M + (long long)(swap_lo + tid) * n;
            const double2 t = cc[j];
            cc[j] = cc[p];
            cc[p] = t;
        }
    }
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const int i = k + tid + r * kPanelNT;
        if (i < n)
#pragma unroll
            for (int c = 0; c < kSub; ++c) st(M + (long long)(k + c) * n + i, a[r][c]);
    }
}

// Sub-panels with more rows than the registers of one CTA hold (blocks of
// more than 256 sites): the same steps on global memory.
__global__ void __launch_bounds__(kPanelNT) lu_panel_tall_kernel(double2 *Mall, int n, int k, int swap_lo, int *piv,
                                                                 double *logu) {
    __shared__ double sv[kPanelNT / 32];
    __shared__ int si[kPanelNT / 32];
    __shared__ int piv_s;
    const int m = blockIdx.x, tid = threadIdx.x;
    double2 *M = Mall + (long long)m * n * n;
    for (int jj = 0; jj < kSub; ++jj) {
        const int j = k + jj;
        double2 *cj = M + (long long)j * n;
        double bv = -1.0;
        int bi = n;
        for (int i = j + tid; i < n; i += kPanelNT) {
            const double2 a = cj[i];
            argmax_pair(bv, bi, a.x * a.x + a.y * a.y, i);
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double v2 = __shfl_xor_sync(0xffffffffu, bv, o);
            const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
            argmax_pair(bv, bi, v2, i2);
        }
        if ((tid & 31) == 0) {
            sv[tid >> 5] = bv;
            si[tid >> 5] = bi;
        }
        __syncthreads();
        if (tid == 0) {
            double v = sv[0];
            int i = si[0];
            for (int q = 1; q < kPanelNT / 32; ++q) argmax_pair(v, i, sv[q], si[q]);
            piv_s = i < n ? i : j;  // (nothing but NaN below: the result is NaN)
            piv[(long long)m * n + j] = piv_s;
        }
        __syncthreads();
        const int p = piv_s;
        if (p != j && tid < k + kSub - swap_lo) {
            double2 *cc = M + (long long)(swap_lo + tid) * n;
            const double2 t = cc[j];
            cc[j] = cc[p];
            cc[p] = t;
        }
        __syncthreads();
        const double2 pv = cj[j];
        const double pn = pv.x * pv.x + pv.y * pv.y;
        if (tid == 0) logu[(long long)m * n + j] = 0.5 * log(pn);
        const cpx<double> inv = {pv.x / pn, -pv.y / pn};
        for (int i = j + 1 + tid; i < n; i += kPanelNT) {
            const cpx<double> l = cmul(ld(cj + i), inv);
            st(cj + i, l);
            for (int c = j + 1; c < k + kSub; ++c) {
                double2 *cc = M + (long long)c * n;
                st(cc + i, cfma(mk<double>(-l.re, -l.im), ld(cc + j), ld(cc + i)));
            }
        }
        __syncthreads();
    }
}

// Columns [c0, c1) of matrix blockIdx.y, a thread per column: the row swaps
// piv[k .. k + w), then U12 = L11^-1 A12 by forward substitution with the unit
// lower L11 of the w columns from k (a kernel of its own: over all SMs the
// substitution's FP64 work is small, on the panel's SM it cost as much as the
// panel).
template <int W>
__global__ void __launch_bounds__(64) lu_solve_kernel(double2 *Mall, int n, int k, int c0, int c1, const int *piv) {
    __shared__ cpx<double> L11[W][W];
    __shared__ int ps[W];
    const int m = blockIdx.y;
    double2 *M = Mall + (long long)m * n * n;
    for (int q = threadIdx.x; q < W * W; q += 64) L11[q % W][q / W] = ld(M + (long long)(k + q / W) * n + k + q % W);
    if (threadIdx.x < W) ps[threadIdx.x] = piv[(long long)m * n + k + threadIdx.x];
    __syncthreads();
    const int c = c0 + blockIdx.x * 64 + threadIdx.x;
    if (c >= c1) return;
    double2 *col = M + (long long)c * n;
    for (int jj = 0; jj < W; ++jj) {
        const int j = k + jj, p = ps[jj];
        if (p != j) {
            const double2 t = col[j];
            col[j] = col[p];
            col[p] = t;
        }
    }
    cpx<double> x[W];
#pragma unroll
    for (int r = 0; r < W; ++r) x[r] = ld(col + k + r);
#pragma unroll
    for (int r = 1; r < W; ++r) {
#pragma unroll
        for (int q = 0; q < r; ++q) x[r] = cfma(mk<double>(-L11[r][q].re, -L11[r][q].im), x[q], x[r]);
        st(col + k + r, x[r]);
    }
}

// A22 -= L21 U12 for the rows [k + w, n) and columns [c0, c1), w <= kNb: tile
// (blockIdx.x: rows, blockIdx.y: columns) of matrix blockIdx.z.
//
// In FP64 this update ran at the rate of the two FP64 lanes per SM (1.1
// TFLOP/s, 75 % of the time of a determinant).  Here the products are
// integer multiply-adds (fixed.cuh gives the rates) of the two limbs that
// lu_limbs makes of the rows of L21 and the columns of U12, and one conversion
// and one FP64 multiply-add per real number remain.  12 integer instead of 4
// FP64 instructions per complex multiply-add, at 32 times the rate.  16 blocks
// of 4^4: 135 -> 42 ms of updates (the whole determinant 181 -> 58 ms) with
// 256 threads of 4 x 2 outputs; 128 threads of 4 x 4 take 82 ms in all, panels
// of 32 columns 73.
struct LuShared {
    int4 L[kNb][kTileR];  // limbs (re hi, re lo, im hi, im lo) of L21 rows
    int4 U[kNb][kTileC];
    int El[kTileR], Eu[kTileC];
};

__global__ void __launch_bounds__(kUpdNT) lu_update_kernel(double2 *Mall, int n, int k, int w, int c0, int c1) {
    extern __shared__ __align__(16) unsigned char lu_smem[];
    LuShared &sm = *reinterpret_cast<LuShared *>(lu_smem);
    auto &Ls = sm.L;
    auto &Us = sm.U;
    int *El = sm.El, *Eu = sm.Eu;
    const int m = blockIdx.z;
    double2 *M = Mall + (long long)m * n * n;
    const int i0 = k + w + blockIdx.x * kTileR, b0 = c0 + blockIdx.y * kTileC;
    const int tid = threadIdx.x;
    for (int q = tid; q < (kTileR + kTileC) * w; q += kUpdNT) {
        // consecutive threads read consecutive rows of L, and the kNb
        // consecutive entries of a column of U
        const bool isl = q < kTileR * w;
        const int t = isl ? q : q - kTileR * w;
        const int ii = isl ? t % kTileR : t / w, qq = isl ? t / kTileR : t % w;
        const int i = isl ? i0 + ii : b0 + ii;
        double2 v = make_double2(0.0, 0.0);
        if (i < (isl ? n : c1)) v = isl ? M[(long long)(k + qq) * n + i] : M[(long long)i * n + k + qq];
        int4 raw;
        raw.x = __double2hiint(v.x), raw.y = __double2loint(v.x), raw.z = __double2hiint(v.y), raw.w = __double2loint(v.y);
        (isl ? Ls[qq] : Us[qq])[ii] = raw;
    }
    __syncthreads();
    for (int t = tid; t < kTileR + kTileC; t += kUpdNT) {
        int e = 0;
        for (int q = 0; q < w; ++q) {
            const int4 v = t < kTileR ? Ls[q][t] : Us[q][t - kTileR];
            e = max(e, max((v.x >> 20) & 0x7FF, (v.z >> 20) & 0x7FF));
        }
        if (t < kTileR) El[t] = e;
        else Eu[t - kTileR] = e;
    }
    __syncthreads();
    for (int q = tid; q < (kTileR + kTileC) * w; q += kUpdNT) {
        const bool isl = q < kTileR * w;
        const int t = isl ? q : q - kTileR * w;
        const int ii = isl ? t % kTileR : t % kTileC, qq = isl ? t / kTileR : t / kTileC;
        int4 &v = (isl ? Ls[qq] : Us[qq])[ii];
        const int E = isl ? El[ii] : Eu[ii];
        const LuLimbs re = lu_limbs(__hiloint2double(v.x, v.y), E), im = lu_limbs(__hiloint2double(v.z, v.w), E);
        v = make_int4(re.hi, re.lo, im.hi, im.lo);
    }
    __syncthreads();
    const int tr = tid % 16, tc = tid / 16;  // rows tr + 16 a, columns tc + kUpdNT / 16 b
    constexpr int NA = kTileR / 16, NB = kTileC * 16 / kUpdNT, CB = kUpdNT / 16;
    int64_t hr[NA][NB], hi[NA][NB], mr[NA][NB], mi[NA][NB];
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int b = 0; b < NB; ++b) hr[a][b] = hi[a][b] = mr[a][b] = mi[a][b] = 0;
#pragma unroll 1
    for (int q = 0; q < w; ++q) {
        int4 l[NA], u[NB];
#pragma unroll
        for (int a = 0; a < NA; ++a) l[a] = Ls[q][tr + 16 * a];
#pragma unroll
        for (int b = 0; b < NB; ++b) u[b] = Us[q][tc + CB * b];
        // product by product over the thread's outputs, so that consecutive
        // multiply-adds do not wait for each other
#define LU_MADS(ACC, X, Y)                                    \
    _Pragma("unroll") for (int a = 0; a < NA; ++a)            \
        _Pragma("unroll") for (int b = 0; b < NB; ++b) fx_mad(ACC[a][b], l[a].X, u[b].Y);
        LU_MADS(hr, x, x)
        LU_MADS(hi, x, z)
        LU_MADS(mr, x, y)
        LU_MADS(mi, x, w)
        LU_MADS(mr, y, x)
        LU_MADS(mi, y, z)
        LU_MADS(hi, z, x)
        LU_MADS(mi, z, y)
        LU_MADS(mi, w, x)
#pragma unroll
        for (int a = 0; a < NA; ++a) l[a].z = -l[a].z, l[a].w = -l[a].w;
        LU_MADS(hr, z, z)
        LU_MADS(mr, z, w)
        LU_MADS(mr, w, z)
#undef LU_MADS
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const int c = b0 + tc + CB * b;
        if (c >= c1) continue;
        const int eu = Eu[tc + CB * b];
        double2 *col = M + (long long)c * n;
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            const int i = i0 + tr + 16 * a;
            if (i >= n) continue;
            const int el = El[tr + 16 * a];
            // sum = t 2^(el + eu - 2046 - 54); non-finite numbers poison it
            double f = (el == 0x7FF || eu == 0x7FF) ? nan("") : lu_scale(el + eu - 2100);
            double2 v = col[i];
            v.x = fma(-f, (double)lu_join(hr[a][b], mr[a][b]), v.x);
            v.y = fma(-f, (double)lu_join(hi[a][b], mi[a][b]), v.y);
            col[i] = v;
        }
    }
}

// out[lex(rank_lo + m)] = n_e ln A + sum_j logu[m n + j], a warp per matrix in
// a fixed order
__global__ void __launch_bounds__(32) logdet_sum_kernel(const BlockInfo *binfo, const double *logu, int n, int rank_lo,
                                                        double base, double *out) {
    const int m = blockIdx.x;
    double s = 0;
    for (int j = threadIdx.x; j < n; j += 32) s += logu[(long long)m * n + j];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) out[binfo[rank_lo + m].lex] = base + s;
}

}  // namespace

int block_logdet_batch(const psms_ctx *c) {
    const long long n = 12LL * c->g.Vbh;
    const double per = 16.0 * (double)n * (double)n;
    size_t fr = 0, tot = 0;
    cudaMemGetInfo(&fr, &tot);
    const double budget = std::min(8e9, 0.25 * (double)tot);
    int k = (int)(budget / per);
    if (c->max_chunk > 0) k = std::min(k, c->max_chunk);
    return std::max(1, std::min(k, c->g.nblocks));
}

void block_logdet(psms_ctx *c, const double2 *U, double *d_out) {
    const Geom &g = c->g;
    if (2 * g.Vbh > kMaxBlockSites)
        fail(PSMS_EINVAL, "exact block determinants are for blocks of at most " + std::to_string(kMaxBlockSites) +
                              " sites (Sec. 3: small blocks)");
    const int n = 12 * g.Vbh;
    const int batch = block_logdet_batch(c);
    double2 *M = (double2 *)scratch(c, "bd_mat", sizeof(double2) * (size_t)n * n * batch);
    double *logu = (double *)scratch(c, "bd_logu", sizeof(double) * (size_t)n * batch);
    int *piv = (int *)scratch(c, "bd_piv", sizeof(int) * (size_t)n * batch);
    cuda_check(cudaFuncSetAttribute(lu_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LuShared)),
               "blockdet shared memory");
    const double base = 12.0 * g.Vbh * std::log(c->A);
    for (int r0 = 0; r0 < g.nblocks; r0 += batch) {
        const int nm = std::min(batch, g.nblocks - r0);
        const long long nt = (long long)nm * n;
        cuda_check(cudaMemsetAsync(M, 0, sizeof(double2) * (size_t)n * n * nm, c->stream), "blockdet memset");
        assemble_kernel<<<(unsigned)((nt + 127) / 128), 128, 0, c->stream>>>(g, c->d_binfo, U, r0, nm, c->A, M);
        PSMS_LAUNCH_CHECK("blockdet assemble");
        auto panel = [&](int k, int swap_lo) {
            const int rows = n - k;
            if (rows <= kPanelNT)
                lu_panel_kernel<1><<<nm, kPanelNT, 0, c->stream>>>(M, n, k, swap_lo, piv, logu);
            else if (rows <= 2 * kPanelNT)
                lu_panel_kernel<2><<<nm, kPanelNT, 0, c->stream>>>(M, n, k, swap_lo, piv, logu);
            else
                lu_panel_tall_kernel<<<nm, kPanelNT, 0, c->stream>>>(M, n, k, swap_lo, piv, logu);
            PSMS_LAUNCH_CHECK("blockdet panel");
        };
        auto update = [&](int k, int w, int c0, int c1) {
            const dim3 grid((n - k - w + kTileR - 1) / kTileR, (c1 - c0 + kTileC - 1) / kTileC, nm);
            lu_update_kernel<<<grid, kUpdNT, sizeof(LuShared), c->stream>>>(M, n, k, w, c0, c1);
            PSMS_LAUNCH_CHECK("blockdet update");
        };
        // n = 12 Vbh is a multiple of kNb = 16 (blocks have at least 16 sites)
        for (int k = 0; k < n; k += kNb) {
            const int end = k + kNb;
            for (int j = k; j < end; j += kSub) {
                panel(j, k);
                if (j + kSub < end) {
                    lu_solve_kernel<kSub><<<dim3(1, nm), 64, 0, c->stream>>>(M, n, j, j + kSub, end, piv);
                    PSMS_LAUNCH_CHECK("blockdet solve");
                    update(j, kSub, j + kSub, end);
                }
            }
            if (end < n) {
                lu_solve_kernel<kNb><<<dim3((n - end + 63) / 64, nm), 64, 0, c->stream>>>(M, n, k, end, n, piv);
                PSMS_LAUNCH_CHECK("blockdet solve");
                update(k, kNb, end, n);
            }
        }
        logdet_sum_kernel<<<nm, 32, 0, c->stream>>>(c->d_binfo, logu, n, r0, base, d_out);
        PSMS_LAUNCH_CHECK("blockdet sum");
    }
}

}  // namespace psms
