// The FP64 tanh and reciprocal square root of the evaluation kernels over an array, for
// tests/test_gpu_math64.py.
#include "../paper_2603_01234_gb300/csrc/evaluate_math.cuh"

__global__ void k_math64(int which, int n, const double* x, double* y)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = which == 0 ? nep::tanh_r(x[i]) : nep::rsqrt_r(x[i]);
}

extern "C" int math64(int which, int n, const double* x, double* y)  // device arrays
{
    k_math64<<<(n + 127) / 128, 128>>>(which, n, x, y);
    const cudaError_t e = cudaDeviceSynchronize();
    return e != cudaSuccess ? (int)e : (int)cudaGetLastError();
}
