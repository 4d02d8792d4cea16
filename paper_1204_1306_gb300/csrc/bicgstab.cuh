// Shared state and scalar steps of the batched BiCGStab on Dhat (one system
// per interpolation step): the per-system scalars, the stage that turns a
// finished reduction into alpha, omega or (rho, beta, convergence), and the
// deterministic "last CTA finishes the reduction" pattern used by the BLAS
// kernels of the solver and by Wilson hops that fuse their dot products.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace psms {

struct BCS {
    double2 rho, alpha, omega, beta;
    double rr, target;
    int active, iters, stalled;
};

constexpr int BCG_SUMS = 7;  // sums of one reduction (see bcg_stage)

__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    const double d = b.x * b.x + b.y * b.y;
    return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double2 cmul2(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// stage 0: sums 0, 1: <rh, v>; alpha = rho / <rh, v>
// stage 1: sums 0, 1: <t, s>; 2: |t|^2; 3, 4: <rh, t>; 5, 6: <rh, s>;
//          omega = <t, s> / |t|^2, rho' = <rh, s - omega t> and beta = (rho' /
//          rho)(alpha / omega), so that x, r and p are updated in one pass.
//          (<rh, s> = 0 but for rounding; dropping it stalls the solver at
//          16^4.)
// stage 2: sum 2: |r|^2 of the new residual, convergence
__device__ __forceinline__ void bcg_stage(BCS *st, int k, const double v[BCG_SUMS], int stage, int maxit, int *flags) {
    BCS s = st[k];
    if (stage == 0) {
        if (!(v[0] * v[0] + v[1] * v[1] > 0.0)) {
            s.active = 0;  // breakdown: <rh, v> = 0
        } else {
            s.alpha = cdiv(s.rho, make_double2(v[0], v[1]));
        }
    } else if (stage == 1) {
        s.omega = v[2] > 0.0 ? make_double2(v[0] / v[2], v[1] / v[2]) : make_double2(0.0, 0.0);
        const double2 w = cmul2(s.omega, make_double2(v[3], v[4]));
        const double2 rho = make_double2(v[5] - w.x, v[6] - w.y);
        s.stalled = !(s.omega.x * s.omega.x + s.omega.y * s.omega.y > 0.0) || !(rho.x * rho.x + rho.y * rho.y > 0.0);
        s.beta = s.stalled ? make_double2(0.0, 0.0) : cmul2(cdiv(rho, s.rho), cdiv(s.alpha, s.omega));
        s.rho = rho;
    } else {
        s.iters += 1;
        s.rr = v[2];
        if (v[2] <= s.target || s.iters >= maxit || s.stalled || !(v[2] == v[2])) s.active = 0;
    }
    st[k] = s;
    flags[k] = s.active;
}

// The same for iterations that take rho' from the new residual (solver.cu says
// which).  stage 0 as above; 1: omega alone; 2: sums 0, 1: <rh, r>; 2: |r|^2;
// rho', beta, convergence
__device__ __forceinline__ void bcg_stage_direct(BCS *st, int k, const double v[BCG_SUMS], int stage, int maxit,
                                                 int *flags) {
    if (stage == 0) {
        bcg_stage(st, k, v, 0, maxit, flags);
        return;
    }
    BCS s = st[k];
    if (stage == 1) {
        s.omega = v[2] > 0.0 ? make_double2(v[0] / v[2], v[1] / v[2]) : make_double2(0.0, 0.0);
        s.stalled = !(s.omega.x * s.omega.x + s.omega.y * s.omega.y > 0.0);
    } else {
        const double2 rho = make_double2(v[0], v[1]);
        s.stalled = s.stalled || !(rho.x * rho.x + rho.y * rho.y > 0.0);
        s.beta = s.stalled ? make_double2(0.0, 0.0) : cmul2(cdiv(rho, s.rho), cdiv(s.alpha, s.omega));
        s.rho = rho;
        s.iters += 1;
        s.rr = v[2];
        if (v[2] <= s.target || s.iters >= maxit || s.stalled || !(v[2] == v[2])) s.active = 0;
    }
    st[k] = s;
    flags[k] = s.active;
}

// Sums over a warp of P values per lane (P = 1, 2, 4, 8): while there are
// several, half of them go to the other half of the lanes, so that 8 sums
// take 9 FP64 additions and not 40 (a warp's FP64 addition occupies the two
// FP64 lanes of an SM for 16 clocks).  Lane l ends with value wsum_index<P>(l).
template <int P>
__device__ __forceinline__ double wsum(const double *v) {
    const int l = threadIdx.x & 31;
    double r[P];
#pragma unroll
    for (int i = 0; i < P; ++i) r[i] = v[i];
    int o = 16;
#pragma unroll
    for (int m = P; m > 1; m >>= 1, o >>= 1) {
        const bool up = l & o;
#pragma unroll
        for (int i = 0; i < m / 2; ++i) {
            const double keep = up ? r[i + m / 2] : r[i], give = up ? r[i] : r[i + m / 2];
            r[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) r[0] += __shfl_xor_sync(0xffffffffu, r[0], o);
    return r[0];
}
// The same of FP32 numbers, without the FP64 pipe: signed mantissas on the
// largest exponent of the warp's numbers (57 bits below it), summed as 64-bit
// integers, so the error is below that of FP64 sums.
template <int P>
__device__ __forceinline__ double wsum(const float *v) {
    const int l = threadIdx.x & 31;
    int64_t r[P];
    unsigned em[P], top = 0;
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const unsigned b = __float_as_uint(v[i]), e = (b >> 23) & 255u;
        em[i] = max(__reduce_max_sync(0xffffffffu, e), 1u);
        top = max(top, em[i]);
        const unsigned m = (b & 0x7FFFFFu) | (e ? 0x800000u : 0u), sh = em[i] - max(e, 1u);
        const int64_t x = (int64_t)(((uint64_t)m << 33) >> min(sh, 63u));
        r[i] = (int)b < 0 ? -x : x;
    }
    if (top == 255u) {  // infinity or NaN
        double d[P];
#pragma unroll
        for (int i = 0; i < P; ++i) d[i] = (double)v[i];
        return wsum<P>(d);
    }
    int o = 16;
#pragma unroll
    for (int m = P; m > 1; m >>= 1, o >>= 1) {
        const bool up = l & o;
#pragma unroll
        for (int i = 0; i < m / 2; ++i) {
            const int64_t keep = up ? r[i + m / 2] : r[i], give = up ? r[i] : r[i + m / 2];
            r[i] = keep + __shfl_xor_sync(0xffffffffu, (long long)give, o);
            em[i] = up ? em[i + m / 2] : em[i];
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) r[0] += __shfl_xor_sync(0xffffffffu, (long long)r[0], o);
    return (double)r[0] * __hiloint2double((int)(em[0] + 1023u - 183u) << 20, 0);  // 2^(em - 127 - 23 - 33)
}
template <int P>
__device__ __forceinline__ int wsum_index(int l) {  // the leading bits of the lane number
    return P == 1 ? 0 : P == 2 ? l >> 4 : P == 4 ? l >> 3 : l >> 2;
}

// Writes this CTA's partials of system k; the last CTA of the system to
// finish (a counter per system, no waiting) sums all partials in a fixed
// order and applies the scalar stage, so the result does not depend on
// which CTA finishes last.  part: BCG_SUMS arrays of part_n doubles; the sums
// [LO, HI) are taken.  DIRECT: bcg_stage_direct.  Ends at a barrier.
template <int NT, int LO, int HI, bool DIRECT = false, class T>
__device__ __forceinline__ void bcg_partials_and_stage(BCS *st, const T in[BCG_SUMS], double *part,
                                                       long long part_n, unsigned int *counters, int stage, int maxit,
                                                       int *flags, double (*sh)[NT / 32], int k, int cta, int nct) {
    const long long slot = (long long)k * nct + cta;
    __shared__ int last;
    constexpr int N = HI - LO, P = N > 4 ? 8 : N > 2 ? 4 : N;
    const int l = threadIdx.x & 31, wi = wsum_index<P>(l);
    const bool lead = l == wi * (32 / P) && wi < N;
    auto warp_sums = [&](const auto *v) {
        std::decay_t<decltype(*v)> x[P];
#pragma unroll
        for (int a = 0; a < P; ++a) x[a] = a < N ? v[LO + a] : 0;
        const double t = wsum<P>(x);
        if (lead) sh[LO + wi][threadIdx.x >> 5] = t;
    };
    warp_sums(in);
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int a = LO; a < HI; ++a) {
            double t = 0;
            for (int w = 0; w < NT / 32; ++w) t += sh[a][w];
            part[a * part_n + slot] = t;
        }
        __threadfence();
        last = atomicAdd(&counters[k], 1u) == (unsigned int)nct - 1u;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the other CTAs' partials, read past L1 (written by other SMs)
    double v[BCG_SUMS];
#pragma unroll
    for (int a = 0; a < BCG_SUMS; ++a) v[a] = 0;
    for (int i = threadIdx.x; i < nct; i += NT) {
        const long long q = (long long)k * nct + i;
#pragma unroll
        for (int a = LO; a < HI; ++a) v[a] += __ldcg(part + a * part_n + q);
    }
    warp_sums(v);
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int a = LO; a < HI; ++a) {
            double t = 0;
            for (int w = 0; w < NT / 32; ++w) t += sh[a][w];
            v[a] = t;
        }
        counters[k] = 0;
        if constexpr (DIRECT) bcg_stage_direct(st, k, v, stage, maxit, flags);
        else bcg_stage(st, k, v, stage, maxit, flags);
    }
    __syncthreads();
}

}  // namespace psms
