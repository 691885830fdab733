// The FP64 functions of the right-hand side and the adjoint on arrays, for
// test_fp64_math_gpu.py.
#include "fire_device.cuh"

__global__ void k_probe(int op, int n, const double *a, const double *b, double *o) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double x = a[k], y = b[k];
    o[k] = op == 0   ? wf::rsqrt64(x)
           : op == 1 ? wf::sqrt64(x)
           : op == 2 ? wf::rcp64(x)
           : op == 3 ? wf::Mth<double>::dv(x, y)
                     : wf::wind_power64(x, y);
}

extern "C" int probe(int op, int n, const double *a, const double *b, double *o) {
    double *d = nullptr;
    const size_t s = sizeof(double) * (size_t)n;
    if (cudaMalloc(&d, 3 * s) != cudaSuccess) return 1;
    cudaMemcpy(d, a, s, cudaMemcpyHostToDevice);
    cudaMemcpy(d + n, b, s, cudaMemcpyHostToDevice);
    k_probe<<<(n + 255) / 256, 256>>>(op, n, d, d + n, d + 2 * (size_t)n);
    const cudaError_t e = cudaMemcpy(o, d + 2 * (size_t)n, s, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e != cudaSuccess;
}
