// Host-side planning of the estimators' batched interpolation steps, pure
// arithmetic (no CUDA calls) so that host tests can check it against the
// oracle: the per-system coefficients of the shared-endpoint links, the
// balanced chunk sizes and the memory of a level.
#pragma once

namespace psms {

// (a_k, b_k) of system k = 0..n-1 of a chunk starting at interpolation step
// i0: the links of field i = i0 + k + shift of Eq. (gfparam),
// U_i = ((N - i)/N) U + (i/N) U' (shift 0: the first operator of the pair,
// 1: the second); in the independent mode every system pairs U (shift 0)
// with U' (shift 1).  ab holds 2n floats.
inline void interp_coefs(int N, int i0, int n, int shift, bool independent, float *ab) {
    for (int k = 0; k < n; ++k) {
        if (independent) {
            ab[2 * k] = shift ? 0.f : 1.f;
            ab[2 * k + 1] = shift ? 1.f : 0.f;
        } else {
            const int i = i0 + k + shift;
            ab[2 * k] = (float)((double)(N - i) / N);
            ab[2 * k + 1] = (float)((double)i / N);
        }
    }
}

// Device memory of a level in bytes per site and system (the system's own
// link fields among them; fields of the whole chunk and reductions, below 1 %,
// left out).  full: the level has whole-lattice solves; shared: their FP32
// links are interpolated from shared endpoint fields.
enum LevelKind { LV_BLOCK, LV_GLOBAL, LV_SUB, LV_OUTER };

inline double level_bytes(LevelKind lv, bool fp64_inner, bool shared) {
    const double fx = 584, f64 = 576, f32 = 288;      // a link field: fixed point, FP64, FP32
    const double sp = 192;                             // an FP64 spinor field
    const double num = fp64_inner ? 16 : 8;            // a complex number of the inner iterations
    const double hop = 194;                            // the hops' input in fixed point
    const double block = sp + (24 + 42) * num;         // block solver: residual, inner vectors
    const double full = sp + (12 + 12 + 42) * num;     // whole-lattice solver: residual, inner rhs and solution, vectors
    const double links = fx + (fp64_inner ? f64 : f32);  // one link set
    switch (lv) {
        case LV_BLOCK: return links + 3 * sp + hop + block;
        case LV_GLOBAL: return links + 7 * sp + hop + block + full;
        case LV_SUB: return links + 5 * sp + hop + block + full;
        // three sets of links: all and masked, and the crossing ones (hops only)
        default: return 2 * (fp64_inner || !shared ? links : fx) + fx + 5 * sp + hop + full;
    }
}

// systems per chunk when at most k fit: as many chunks as needed, of equal
// size (the last at most one smaller)
inline int balanced_chunk(int N, int k) {
    if (k < 1) k = 1;
    if (k > N) k = N;
    const int n_chunks = (N + k - 1) / k;
    return (N + n_chunks - 1) / n_chunks;
}

}  // namespace psms
