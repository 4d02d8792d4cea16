// Box-Muller pairs z = sqrt(-ln u_a) e^{2 pi i u_b} of two Philox words in
// integer arithmetic.
//
// In FP64 a pair costs 86 instructions (log, sqrt, sincospi), which the two
// FP64 lanes of an SM here execute at one warp instruction per 16 clocks: the
// noise of twelve systems at 16^4 took 1.36 ms, 1.1 of them that.  The
// uniforms u = (2 m + 1) 2^-53 are fixed-point numbers, so the logarithm and the
// angle functions are evaluated in 64-bit fixed point (tables and short Taylor
// series, products by 64 x 64 -> 128 bit multiplication); 13 FP64 instructions
// remain (two Heron steps for the root, the final products and conversions):
// 0.38 ms.
//
// Errors (tests/test_gauss_host.py, on the device tests/test_gpu_gauss.py):
// |z - exact| below 1.6 x 2^-52 of the radius sqrt(-ln u_a); over 8e6 pairs the
// largest 2.9 and the rms 0.51 units of 2^-53, both those of the FP64
// functions.  The angle functions are good to 2 units of 2^-62 of the radius,
// so that a component next to an axis has fewer digits of its own than FP64
// functions give it (2^-53 of itself).
#pragma once

#include <math.h>

#include "fixed.cuh"

namespace psms {

constexpr int GA_SIN = 256;  // table steps per quarter turn, used up to the eighth
constexpr int GA_LOG = 512;  // table steps per octave

struct GaussTables {
    // sin, cos (scale 2^62) of i / GA_SIN of a quarter turn
    int64_t sn[GA_SIN / 2 + 1], cs[GA_SIN / 2 + 1];
    // c = round(2^10 / f) at the middle f in [1, 2) of step i, and ln(c 2^-10) (scale 2^62)
    int64_t lnc[GA_LOG];
    uint16_t c[GA_LOG];
};

// filled by the host in extended precision (at least 64 bits of mantissa)
inline void gauss_tables(GaussTables &t) {
    const long double q = 1.5707963267948966192313216916397514421L;
    for (int i = 0; i <= GA_SIN / 2; ++i) {
        t.sn[i] = llroundl(ldexpl(sinl(q * i / GA_SIN), 62));
        t.cs[i] = llroundl(ldexpl(cosl(q * i / GA_SIN), 62));
    }
    for (int i = 0; i < GA_LOG; ++i) {
        const long double f = 1.0L + (i + 0.5L) / GA_LOG;
        t.c[i] = (uint16_t)lroundl(1024.0L / f);
        t.lnc[i] = llroundl(ldexpl(logl((long double)t.c[i] / 1024.0L), 62));
    }
}

__host__ __device__ __forceinline__ uint64_t mulhi_u(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ int64_t mulhi_s(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (int64_t)(((__int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ uint32_t mulhi_u32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
__host__ __device__ __forceinline__ int32_t mulhi_s32(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}
__host__ __device__ __forceinline__ int clz64(uint64_t x) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}

// sin and cos (scale 2^62) of the angle (2 m + 1) 2^-53 turns, m = w >> 12
__host__ __device__ __forceinline__ void gauss_angle(const GaussTables &T, uint64_t w, int64_t &sn, int64_t &cs) {
    const uint64_t t = ((w >> 12) << 12) | (1ull << 11);  // fraction of a turn, 2^64
    const int quad = (int)(t >> 62);
    uint64_t r = t << 2;  // fraction of the quarter
    const bool refl = (int64_t)r < 0;
    if (refl) r = 0 - r;  // the angle from the next axis
    // r in (0, 2^63]: step i and the rest, delta = rest pi/2 2^-64 < pi/2 2^-8
    const int i = (int)(r >> 56);
    const uint64_t d = mulhi_u((r & 0xFFFFFFFFFFFFFFull) << 7, 0xC90FDAA22168C235ull);  // delta 2^70 (pi/2 2^63 = 0xC90F..)
    const uint64_t z = mulhi_u(d, d);                                                  // delta^2 2^76
    const uint32_t z32 = (uint32_t)(z >> 32);                                          // delta^2 2^44
    // sin d = d - d z (1/6 - z/120): C = (1/6 - z/120) 2^64
    const uint64_t C = 0x2AAAAAAAAAAAAAABull - ((uint64_t)mulhi_u32(z32, 0x88888889u) << (32 - 12 - 6));
    const uint64_t sd = d - (mulhi_u(d, mulhi_u(z, C)) >> 12);                          // 2^70
    // 1 - cos d = z (1/2 - z (1/24 - z/720))
    const uint64_t D = 0x0AAAAAAAAAAAAAABull - ((uint64_t)mulhi_u32(z32, 0xB60B60B6u) << (32 - 12 - 9));  // (1/24 - z/720) 2^64
    const uint64_t H = 0x8000000000000000ull - (mulhi_u(z, D) >> 12);                   // 2^64
    const uint64_t vd = mulhi_u(z, H);                                                  // (1 - cos d) 2^76
    // rotate the table's angle by delta
    const int64_t s0 = T.sn[i], c0 = T.cs[i];
    const int64_t s1 = s0 + mulhi_s(c0, (int64_t)(sd >> 6)) - (mulhi_s(s0, (int64_t)(vd >> 1)) >> 11);
    const int64_t c1 = c0 - mulhi_s(s0, (int64_t)(sd >> 6)) - (mulhi_s(c0, (int64_t)(vd >> 1)) >> 11);
    int64_t a = refl ? c1 : s1, b = refl ? s1 : c1;  // sin, cos within the quarter
    // quarters: (s, c), (c, -s), (-s, -c), (-c, s)
    const int64_t a2 = (quad & 1) ? b : a, b2 = (quad & 1) ? a : b;
    sn = (quad & 2) ? -a2 : a2;
    cs = ((quad + 1) & 2) ? -b2 : b2;
}

// -ln u of u = (2 m + 1) 2^-53, m = w >> 12, on scale 2^56, or 2^62 (half) for
// u > 1/2; near reports u above 1 - 2^-10, where the result is small and its
// relative error not
__host__ __device__ __forceinline__ int64_t gauss_log(const GaussTables &T, uint64_t w, bool &half, bool &near) {
    const uint64_t M = ((w >> 12) << 1) | 1;  // u 2^53
    const int lz = clz64(M);                  // >= 11
    const uint64_t f = M << lz;               // f 2^-63 in [1, 2); u = f 2^-63 2^(10 - lz)
    near = lz == 11 && (f >> 54) == 0x3FF;
    const int i = (int)(f >> 54) & (GA_LOG - 1);
    // r = f c 2^-10 - 1, exact (53 bits by 11): f >> 11 is f 2^-11
    const int64_t r = (int64_t)((f >> 11) * (uint64_t)T.c[i] - (1ull << 62));  // r 2^62, |r| < 2^-8.9
    // ln(1 + r) = r (1 - r/2 + r^2/3 - r^3/4 + r^4/5 - r^5/6), the last three terms in 32 bits
    const int32_t q = (int32_t)(r >> 23);  // r 2^39
    int32_t p = 0x33333333 - (mulhi_s32(q, 0x2AAAAAAB) >> 7);  // (1/5 - r/6) 2^32
    p = 0x40000000 - (mulhi_s32(q, p) >> 7);                    // (1/4 - r (..)) 2^32
    const int64_t p3 = 0x1555555555555555ll - (mulhi_s(r, (int64_t)p << 32) >> 0);     // (1/3 - r (1/4 - ..)) 2^62
    const int64_t p2 = 0x2000000000000000ll - (mulhi_s(r, p3) << 2);                   // (1/2 - r (..)) 2^62
    const int64_t p1 = 0x4000000000000000ll - (mulhi_s(r, p2) << 2);                   // (1 - r (..)) 2^62
    const int64_t ln1 = mulhi_s(r << 2, p1);                                           // ln(1 + r) 2^62
    // -ln u = (lz - 10) ln 2 + ln c - ln(1 + r); ln 2 2^64 = B17217F7 D1CF79AC
    const int e = lz - 10;
    const int64_t b = T.lnc[i] - ln1;  // 2^62
    half = e == 1;
    return half ? 0x2C5C85FDF473DE6Bll + b : (int64_t)e * 0x00B17217F7D1CF79ll + ((e * 0xAC) >> 8) + (b >> 6);
}

// the pair of words (wa, wb)
__host__ __device__ __forceinline__ void gauss_pair(const GaussTables &T, uint64_t wa, uint64_t wb, double &re,
                                                    double &im) {
    bool near, half;
    const int64_t L = gauss_log(T, wa, half, near);
    int64_t sn, cs;
    gauss_angle(T, wb, sn, cs);
    double s;
    if (near) {
        s = sqrt(-log(((double)(wa >> 12) + 0.5) * 0x1.0p-52)) * 0x1.0p-62;
    } else {
        // sqrt(L 2^-56) 2^-62 = sqrt(L) 2^-90 (scale 2^62: 2^-93) by two Heron
        // steps from the FP32 root
        const float lf = (float)(int32_t)(L >> 32);  // L 2^-32, at least 2^14
#ifdef __CUDA_ARCH__
        const double y = (double)(rsqrtf(lf) * 0x1.0p-16f);
#else
        const double y = (double)(1.0f / sqrtf(lf) * 0x1.0p-16f);
#endif
        const double l = (double)L, hy = 0.5 * y;
        double x = l * y;
        x = fma(fma(-x, x, l), hy, x);
        x = fma(fma(-x, x, l), hy, x);
        s = x * (half ? 0x1.0p-93 : 0x1.0p-90);
    }
    re = s * (double)cs;
    im = s * (double)sn;
}

}  // namespace psms
