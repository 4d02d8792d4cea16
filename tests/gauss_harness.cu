// Test harness: the fixed-point Box-Muller pairs of csrc/gauss.cuh, compiled
// for the host.  Not part of the library.
#include "../paper_1204_1306_gb300/csrc/gauss.cuh"

using namespace psms;

// z[2 i], z[2 i + 1] = the pair of the words w[2 i], w[2 i + 1]
extern "C" void gauss_pairs_host(const uint64_t *w, int n, double *z) {
    static GaussTables t;
    gauss_tables(t);
    for (int i = 0; i < n; ++i) gauss_pair(t, w[2 * i], w[2 * i + 1], z[2 * i], z[2 * i + 1]);
}
