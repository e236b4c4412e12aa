// Test helper (not part of the library): the FP64 population sums of FP32
// nodes, for tests/test_gpu_population_sums.py.
#include <cuda_runtime.h>

#include "../paper_1809_08683_gb300/csrc/lbm_sums.cuh"

// exact[i]: whether both halves of node i are summed in integers.
__global__ void k_sums(const float* v, double* out, int* exact, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float w[18];
    for (int q = 0; q < 18; ++q) w[q] = v[18 * i + q];
    lbm::node_sums_fp64(w, out[4 * i], out[4 * i + 1], out[4 * i + 2], out[4 * i + 3]);
    lbm::Fixed9 f, g;
    const bool okf = f.set(w), okg = g.set(w + 9);
    exact[i] = okf && okg;
}

// Host arrays: n x 18 floats, n x 4 doubles, n ints; returns the CUDA error code.
extern "C" int sums_check(const float* v, double* out, int* exact, int n) {
    char* d = nullptr;
    const size_t bo = (size_t)n * 4 * sizeof(double), bv = (size_t)n * 18 * sizeof(float), be = (size_t)n * sizeof(int);
    cudaError_t e = cudaMalloc(&d, bo + bv + be);
    if (e != cudaSuccess) return (int)e;
    float* dv = (float*)(d + bo);
    int* de = (int*)(d + bo + bv);
    cudaMemcpy(dv, v, bv, cudaMemcpyHostToDevice);
    k_sums<<<(n + 127) / 128, 128>>>(dv, (double*)d, de, n);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) {
        cudaMemcpy(out, d, bo, cudaMemcpyDeviceToHost);
        cudaMemcpy(exact, de, be, cudaMemcpyDeviceToHost);
    }
    cudaFree(d);
    return (int)e;
}
