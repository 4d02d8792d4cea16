// Test harness: the fixed-point Box-Muller pairs of csrc/gauss.cuh, compiled
// for the host and for the device.  Not part of the library.
#include "../paper_1204_1306_gb300/csrc/gauss.cuh"

using namespace psms;

// z[2 i], z[2 i + 1] = the pair of the words w[2 i], w[2 i + 1]
extern "C" void gauss_pairs_host(const uint64_t *w, int n, double *z) {
    static GaussTables t;
    gauss_tables(t);
    for (int i = 0; i < n; ++i) gauss_pair(t, w[2 * i], w[2 * i + 1], z[2 * i], z[2 * i + 1]);
}

namespace {
__global__ void pairs_kernel(const GaussTables *t, const uint64_t *w, int n, double *z) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) gauss_pair(*t, w[2 * i], w[2 * i + 1], z[2 * i], z[2 * i + 1]);
}
}  // namespace

// the same on the device (w, z: device pointers); a CUDA error code
extern "C" int gauss_pairs_device(const uint64_t *w, int n, double *z) {
    static GaussTables t;
    gauss_tables(t);
    GaussTables *d = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof(t));
    if (e == cudaSuccess) e = cudaMemcpy(d, &t, sizeof(t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        pairs_kernel<<<(n + 127) / 128, 128>>>(d, w, n, z);
        e = cudaDeviceSynchronize();
    }
    cudaFree(d);
    return (int)e;
}
