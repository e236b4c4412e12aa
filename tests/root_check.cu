// Test helper (not part of the library): evaluates the FP64 square root that
// the per-node arithmetic uses on the device (lbm::root) next to CUDA's
// correctly rounded one, for tests/test_gpu_root.py.
#include <cuda_runtime.h>

#include "../paper_1809_08683_gb300/csrc/lbm_node.cuh"

__global__ void k_root(const double* x, double* r_lbm, double* r_ieee, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r_lbm[i] = lbm::root(x[i]);
    r_ieee[i] = __dsqrt_rn(x[i]);
}

// Host arrays of n doubles; returns 0 on success, else the CUDA error code.
extern "C" int root_check(const double* x, double* r_lbm, double* r_ieee, int n) {
    double* d = nullptr;
    const size_t bytes = (size_t)n * sizeof(double);
    cudaError_t e = cudaMalloc(&d, 3 * bytes);
    if (e != cudaSuccess) return (int)e;
    cudaMemcpy(d, x, bytes, cudaMemcpyHostToDevice);
    k_root<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, n);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) {
        cudaMemcpy(r_lbm, d + n, bytes, cudaMemcpyDeviceToHost);
        cudaMemcpy(r_ieee, d + 2 * n, bytes, cudaMemcpyDeviceToHost);
    }
    cudaFree(d);
    return (int)e;
}
