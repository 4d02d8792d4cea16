// FP64 Wilson hops in fixed point.
//
// GB300 has two FP64 lanes per SM against 64 lanes of 32 x 32 -> 64 bit
// integer multiply-add (measured: 2 DFMA, 64 IMAD.WIDE per clock and SM), so
// a product of two 53-bit numbers is cheaper as three integer multiply-adds
// than as one DFMA.  Here a link is held as two signed limbs per real number,
//     u = (hi 2^29 + lo) 2^(e - 58),   |hi| <= 2^30, 0 <= lo < 2^29,
// e the binary exponent of the largest of its 18 numbers (59 bits below
// 2^(e+1), so the 53-bit mantissas are exact down to 2^-6 of the largest and
// the absolute error of a smaller one is below 2^-58 of it).  The spinor a
// hop reads is converted in the kernel, all 24 numbers on the exponent of the
// largest (58 bits and a sign), projected with 64-bit adds and split alike.
// A row of U h is then
//     sum u h = (HI 2^29 + MID) 2^29 + sum lo lo,
// HI = sum hi hi and MID = sum (hi lo + lo hi) exact in 64 bits (6 x 2^60 and
// 12 x 2^59 at most); the last sum, six products below 2^58 where the largest
// product is 2^114 at least (below 2^-53 of it in the worst case, 2^-57 in the
// mean), is dropped.  The eight hops add up as 64-bit integers on one exponent (the
// largest so far, give or take one), rounded to 2^-54 of the largest product of a link entry
// and a spinor entry, and become FP64 again once per output.
//
// The error of H psi against exact arithmetic is below that of the FP64
// chain, whose 2^-53 is relative to every partial sum: it is measured in
// tests/test_fixed_point_host.py.  That holds for the norm of the error; for
// every single output it holds where no colour or chirality of a spinor is
// small against the others, and spinors for which it is not so (fx_spinor),
// numbers outside 2^-823 .. 2^877, NaN and infinity are left to the FP64 form.
#pragma once

#include "common.cuh"

namespace psms {

// A field of spinors in fixed point: longlong2 {re, im} in the FP64 layout
// [c][s] (fx_spinor), then one exponent per site, uint16; fx_spinors(cs)
// 16-byte elements for cs sites.
__host__ __device__ __forceinline__ long long fx_spinors(long long cs) { return 12 * cs + (cs + 7) / 8; }

// A field of links in fixed point: int4 {re hi, re lo, im hi, im lo} in the
// FP64 layout [mu][e][s], then one exponent per link [mu][s] (biased; 0 for
// a zero link; FX_BAD outside the range: the four words are then the FP64 bits),
// uint16.
constexpr int FX_BAD = 0xFFFF;

// keeps the cases of a direction apart: merged, every case is computed and
// one selected (the direction is uniform, so a branch costs next to nothing)
#ifdef __CUDA_ARCH__
#define FX_BRANCH asm volatile("")
#else
#define FX_BRANCH (void)0
#endif
constexpr int FX_EMIN = 200, FX_EMAX = 1900;  // biased exponents handled

// 16-byte elements of one field (links, then 4 V exponents)
__host__ __device__ __forceinline__ long long fx_field(long long V) { return 36 * V + V / 2; }
__host__ __device__ __forceinline__ const uint16_t *fx_exps(const int4 *U, long long V) {
    return reinterpret_cast<const uint16_t *>(U + 36 * V);
}
__host__ __device__ __forceinline__ uint16_t *fx_exps(int4 *U, long long V) {
    return reinterpret_cast<uint16_t *>(U + 36 * V);
}

__host__ __device__ __forceinline__ uint64_t f64_bits(double v) {
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(v);
#else
    union {
        double d;
        uint64_t u;
    } x;
    x.d = v;
    return x.u;
#endif
}

__host__ __device__ __forceinline__ double f64_from_bits(uint64_t v) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)v);
#else
    union {
        double d;
        uint64_t u;
    } x;
    x.u = v;
    return x.d;
#endif
}

// x >> s, zero (or the sign) for s beyond 63
__host__ __device__ __forceinline__ uint64_t fx_shr(uint64_t x, uint32_t s) {
#ifdef __CUDA_ARCH__
    asm("shr.u64 %0, %1, %2;" : "=l"(x) : "l"(x), "r"(s));  // clamps
    return x;
#else
    return s > 63 ? 0 : x >> s;
#endif
}

// the number with bit pattern b as a multiple of 2^(E - UP - 1), E >= its
// exponent (both biased): |result| < 2^(UP + 2); the low 52 - UP bits and
// those shifted out are cut off
template <int UP>
__host__ __device__ __forceinline__ int64_t fx_convert(uint64_t b, int E) {
    const uint32_t h = (uint32_t)(b >> 32);
    const int e = (int)((h >> 20) & 0x7FF);
    const uint64_t m = ((uint64_t)((h & 0xFFFFFu) | 0x100000u) << 32) | (uint32_t)b;
    const uint64_t x = fx_shr(m << (UP - 51), (uint32_t)(E - e));
    const int64_t sg = (int64_t)((int32_t)h >> 31);
    return ((int64_t)x ^ sg) - sg;
}
// links: 59 bits below 2^(E+1) (UP 57); spinors: 58 bits (UP 56)
constexpr int FX_UP_LINK = 57, FX_UP_SPINOR = 56;

__host__ __device__ __forceinline__ int2 fx_limbs(int64_t y) {
    int2 l;
    l.x = (int)(y >> 29);
    l.y = (int)((uint32_t)y & 0x1FFFFFFFu);
    return l;
}

// Fixed-point form of one link (18 numbers); returns its exponent word.
__host__ __device__ __forceinline__ int fx_link(const cpx<double> u[9], int4 out[9]) {
    int E = 0;
    bool zero = true;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const uint64_t a = f64_bits(u[i].re), b = f64_bits(u[i].im);
        const int ea = (int)(a >> 52) & 0x7FF, eb = (int)(b >> 52) & 0x7FF;
        E = ea > E ? ea : E;
        E = eb > E ? eb : E;
        zero = zero && ((a | b) << 1) == 0;
    }
    const bool bad = !zero && (E < FX_EMIN || E > FX_EMAX);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        int2 re = make_int2(0, 0), im = make_int2(0, 0);
        if (!zero && !bad) {
            re = fx_limbs(fx_convert<FX_UP_LINK>(f64_bits(u[i].re), E));
            im = fx_limbs(fx_convert<FX_UP_LINK>(f64_bits(u[i].im), E));
        } else if (bad) {
            re = make_int2((int)(f64_bits(u[i].re) >> 32), (int)f64_bits(u[i].re));
            im = make_int2((int)(f64_bits(u[i].im) >> 32), (int)f64_bits(u[i].im));
        }
        out[i] = make_int4(re.x, re.y, im.x, im.y);
    }
    return bad ? FX_BAD : (zero ? 0 : E);
}

// one number of a link with exponent word E back in FP64
__host__ __device__ __forceinline__ double fx_value(int hi, int lo, int E) {
    if (E == FX_BAD) return f64_from_bits(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo);
    if (E == 0) return 0.0;
    // (hi 2^29 + lo) 2^(E - 1023 - 58)
    const double v = (double)(((int64_t)hi << 29) + lo);
    return v * f64_from_bits((uint64_t)(E - 58) << 52);
}

// Sum of hops of one output site: up and down spin halves as integers,
// value = v 2^(E - 2099)
struct FxAcc {
    int64_t up[2][3][2], dn[2][3][2];  // [spin][colour][re, im]
    int E;
};

__host__ __device__ __forceinline__ void fx_zero(FxAcc &a) {
    a.E = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int k = 0; k < 2; ++k) a.up[q][c][k] = a.dn[q][c][k] = 0;
}

// Hops are numbered d = 2 mu + (0 forward, 1 backward); the sign of the
// projector 1 + t gamma_mu is t = -s forward, +s backward, s = +1 for D and -1
// for D^dagger (dag).  A backward hop multiplies by U^dagger, which is done as
// the complex conjugate of U^T times the conjugate of the projected spinor:
// the conjugations only change signs of the additions here.

// one case of fx_project: (re, im) of e_mu d for the two spin components given
// as signed references, h = u + t e d, conjugated for CONJ
#define FX_CASE_PROJECT(A0, B0, A1, B1)                                        \
    {                                                                          \
        for (int c = 0; c < 3; ++c) {                                          \
            const int64_t *u0 = p[c], *u1 = p[3 + c], *d0 = p[6 + c], *d1 = p[9 + c]; \
            (void)d0, (void)d1;                                                \
            const int64_t a0 = A0, b0 = B0, a1 = A1, b1 = B1;                  \
            h[0][c][0] = T ? u0[0] + a0 : u0[0] - a0;                          \
            h[1][c][0] = T ? u1[0] + a1 : u1[0] - a1;                          \
            h[0][c][1] = C ? (T ? -u0[1] - b0 : b0 - u0[1]) : (T ? u0[1] + b0 : u0[1] - b0); \
            h[1][c][1] = C ? (T ? -u1[1] - b1 : b1 - u1[1]) : (T ? u1[1] + b1 : u1[1] - b1); \
        }                                                                      \
    }

// projected spinor of direction mu; T: t = +1, C: conjugated
template <bool T, bool C>
__host__ __device__ __forceinline__ void fx_project(int mu, const int64_t p[12][2], int64_t h[2][3][2]) {
    if (mu == 0) {
        FX_BRANCH;
#pragma unroll
        FX_CASE_PROJECT(-d0[0], -d0[1], -d1[0], -d1[1])
    } else if (mu == 1) {
        FX_BRANCH;
#pragma unroll
        FX_CASE_PROJECT(d1[1], -d1[0], d0[1], -d0[0])
    } else if (mu == 2) {
        FX_BRANCH;
#pragma unroll
        FX_CASE_PROJECT(-d1[0], -d1[1], d0[0], d0[1])
    } else {
        FX_BRANCH;
#pragma unroll
        FX_CASE_PROJECT(d0[1], -d0[0], -d1[1], d1[0])
    }
}
#undef FX_CASE_PROJECT

// acc += (w, t e_mu^dagger w), w (conjugated for C) = w[spin][colour][re, im]
template <bool T, bool C>
__host__ __device__ __forceinline__ void fx_reconstruct(int mu, const int64_t w[2][3][2], FxAcc &a) {
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            a.up[q][c][0] += w[q][c][0];
            a.up[q][c][1] += C ? -w[q][c][1] : w[q][c][1];
        }
#define FX_ADD(X, NEG, Y) X += ((NEG) != !T) ? -(Y) : (Y)
    // e^dagger w; sign flips: of e^dagger, and of a conjugated imaginary part
    if (mu == 0) {
        FX_BRANCH;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            FX_ADD(a.dn[0][c][0], true, w[0][c][0]);
            FX_ADD(a.dn[0][c][1], !C, w[0][c][1]);
            FX_ADD(a.dn[1][c][0], true, w[1][c][0]);
            FX_ADD(a.dn[1][c][1], !C, w[1][c][1]);
        }
    } else if (mu == 1) {
        FX_BRANCH;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            FX_ADD(a.dn[0][c][0], !C, w[1][c][1]);
            FX_ADD(a.dn[0][c][1], false, w[1][c][0]);
            FX_ADD(a.dn[1][c][0], !C, w[0][c][1]);
            FX_ADD(a.dn[1][c][1], false, w[0][c][0]);
        }
    } else if (mu == 2) {
        FX_BRANCH;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            FX_ADD(a.dn[0][c][0], false, w[1][c][0]);
            FX_ADD(a.dn[0][c][1], C, w[1][c][1]);
            FX_ADD(a.dn[1][c][0], true, w[0][c][0]);
            FX_ADD(a.dn[1][c][1], !C, w[0][c][1]);
        }
    } else {
        FX_BRANCH;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            FX_ADD(a.dn[0][c][0], !C, w[0][c][1]);
            FX_ADD(a.dn[0][c][1], false, w[0][c][0]);
            FX_ADD(a.dn[1][c][0], C, w[1][c][1]);
            FX_ADD(a.dn[1][c][1], true, w[1][c][0]);
        }
    }
#undef FX_ADD
}

// A spinor (24 FP64 numbers, raw bits) as integers on the exponent of its
// largest number; returns that exponent, 0 for a zero spinor, FX_BAD out of
// range (v is then zero).
//
// alike: whether its numbers are so alike that a common exponent costs none of
// the hops' outputs its FP64 accuracy: every colour of every chirality (spins
// 0, 1 and spins 2, 3) has a number within 2^-6 of the largest.  Each output
// number draws on all four numbers of its colour and the other chirality,
// whatever the links, so that it is then not small against what it is rounded
// to.  Spinors with a colour or a chirality that is zero or small are left to
// the FP64 form: in a field whose links do not mix the colours (the unit field,
// abelian fields) or for a point source an output may hold nothing else.
// Gaussian spinors are alike but for one in 10^5 (FX_ALIKE = 5: 3 in 10^4).
constexpr int FX_ALIKE = 6;

__host__ __device__ __forceinline__ int fx_spinor(const uint64_t p[12][2], int64_t v[12][2], bool &alike) {
    uint32_t em = 0, low = 0xFFFFFFFFu;
    uint64_t any = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            uint32_t m = 0;
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const uint64_t b = p[6 * h + 3 * q + c][k];
                    const uint32_t e = (uint32_t)(b >> 32) & 0x7FF00000u;
                    m = e > m ? e : m;
                    any |= b;
                }
            em = m > em ? m : em;
            low = m < low ? m : low;
        }
    const int ep = (int)(em >> 20);
    alike = em - low <= (uint32_t)FX_ALIKE << 20;
    if (ep < FX_EMIN || ep > FX_EMAX) {
#pragma unroll
        for (int c = 0; c < 12; ++c) v[c][0] = v[c][1] = 0;
        return (any << 1) == 0 ? 0 : FX_BAD;
    }
#pragma unroll
    for (int c = 0; c < 12; ++c)
#pragma unroll
        for (int k = 0; k < 2; ++k) v[c][k] = fx_convert<FX_UP_SPINOR>(p[c][k], ep);
    return ep;
}

__host__ __device__ __forceinline__ int fx_spinor(const uint64_t p[12][2], int64_t v[12][2]) {
    bool alike;
    return fx_spinor(p, v, alike);
}

// projected spinor of hop d as limbs
template <bool DAG>
__host__ __device__ __forceinline__ void fx_half(int d, const int64_t p[12][2], int2 hl[2][3][2]) {
    int64_t h[2][3][2];
    if (d & 1) fx_project<!DAG, true>(d >> 1, p, h);
    else fx_project<DAG, false>(d >> 1, p, h);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int k = 0; k < 2; ++k) hl[q][c][k] = fx_limbs(h[q][c][k]);
}

// a += x y
__host__ __device__ __forceinline__ void fx_mad(int64_t &a, int x, int y) {
#ifdef __CUDA_ARCH__
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a) : "r"(x), "r"(y));
#else
    a += (int64_t)x * y;
#endif
}

// One hop: acc += bsign (1 + t gamma_mu) part of psi transported by the link
// (U, or U^dagger for backward; bsign = -1 when neg).  hl, ep: the projected
// spinor and its exponent (fx_half, fx_spinor); v: the link's elements
// (transposed for a backward hop); ue: its exponent word.  Neither exponent
// is 0 or FX_BAD.
template <bool DAG>
__host__ __device__ __forceinline__ void fx_hop(int d, bool neg, const int2 hl[2][3][2], int ep, const int4 v[9], int ue,
                                                FxAcc &acc) {
    const int e = ue + ep;
    if (acc.E == 0) acc.E = e;  // the first hop
    if (e > acc.E + 1) {
        // a larger hop (one bit more still fits): the sum moves to its exponent
        const int sh = e - acc.E > 63 ? 63 : e - acc.E;
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int c = 0; c < 3; ++c)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    acc.up[q][c][k] >>= sh;
                    acc.dn[q][c][k] >>= sh;
                }
        acc.E = e;
    }
    const int s = 4 + (acc.E - e);  // >= 3
    if (s > 61) return;             // below the resolution of the sum
    const int64_t rnd = (int64_t)1 << (s - 1);
    int2 ny[2][3];  // -Im h
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int b = 0; b < 3; ++b) ny[q][b] = make_int2(-hl[q][b][1].x, -hl[q][b][1].y);
    int64_t w[2][3][2];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // eight independent chains, one product of each in turn
        int64_t hr[2], hi[2], mr[2], mi[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) hr[q] = hi[q] = rnd, mr[q] = mi[q] = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 u = v[3 * a + b];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                fx_mad(hr[q], u.x, hl[q][b][0].x);
                fx_mad(hi[q], u.x, hl[q][b][1].x);
                fx_mad(mr[q], u.x, hl[q][b][0].y);
                fx_mad(mi[q], u.x, hl[q][b][1].y);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                fx_mad(hr[q], u.z, ny[q][b].x);
                fx_mad(hi[q], u.z, hl[q][b][0].x);
                fx_mad(mr[q], u.z, ny[q][b].y);
                fx_mad(mi[q], u.z, hl[q][b][0].y);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                fx_mad(mr[q], u.y, hl[q][b][0].x);
                fx_mad(mi[q], u.y, hl[q][b][1].x);
            }
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                fx_mad(mr[q], u.w, ny[q][b].x);
                fx_mad(mi[q], u.w, hl[q][b][0].x);
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            w[q][a][0] = (hr[q] + (mr[q] >> 29)) >> s;
            w[q][a][1] = (hi[q] + (mi[q] >> 29)) >> s;
        }
    }
    if (neg) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int k = 0; k < 2; ++k) w[q][a][k] = -w[q][a][k];
    }
    if (d & 1) fx_reconstruct<!DAG, true>(d >> 1, w, acc);
    else fx_reconstruct<DAG, false>(d >> 1, w, acc);
}

// Products of the blocked LU's trailing update (blockdet.cu): each row of L21
// and each column of U12 is held as x 2^(E - 1078), |x| < 2^56, on the exponent
// E (biased) of its largest real number (exact for the numbers down to 2^-3
// of it, smaller ones and denormals are cut off at 2^-55 of 2^(E - 1023)), in
// two limbs
//     x = hi 2^28 + lo,  |hi| <= 2^28, -2^27 <= lo < 2^27,
// so that, with w <= 16 complex products,
//     sum x y = HI 2^56 + MID 2^28 + sum lo lo,
// HI = sum hi hi <= 2^61 and MID = sum (hi lo + lo hi) <= 2^61 exact in 64
// bits.  The last sum is dropped: at most 8 units of HI, in the root mean
// square half a unit and of no sign (lo is rounded, not cut off: with lo in 0
// .. 2^28 the imaginary part, whose products all add, was short by 8 units in
// the mean).  The error of a sum is below that of the FP64 chain
// (tests/test_fixed_point_host.py).
struct LuLimbs {
    int hi, lo;
};

__host__ __device__ __forceinline__ LuLimbs lu_limbs(double v, int E) {
    LuLimbs l;
    const int64_t x = E == 0 ? 0 : fx_convert<54>(f64_bits(v), E);
    l.hi = (int)((x + (1 << 27)) >> 28);
    l.lo = (int)(x - ((int64_t)l.hi << 28));
    return l;
}

// HI + MID 2^-28, rounded: the sum in units of 2^56
__host__ __device__ __forceinline__ int64_t lu_join(int64_t hi, int64_t mid) { return hi + ((mid + (1 << 27)) >> 28); }

// Factor that turns the integers of a finished sum into b times its value;
// false when it is out of the normal range.
__host__ __device__ __forceinline__ bool fx_factor(const FxAcc &acc, double b, double &f) {
    const int k = acc.E - 2099;  // value = v 2^k
    f = 0.0;
    if (acc.E == 0) return true;  // no hop contributed
    if (k < -960 || k > 900) return false;
    f = b * f64_from_bits((uint64_t)(k + 1023) << 52);
    return true;
}

}  // namespace psms
