// -ln u of the FP32 sampler beside the same by CUDA's logf (u < 1/2) and log1pf of the
// complement, for the words x of u = (x + 1/2) 2^-32.
#include "bz_kernels.cuh"

static __global__ void k_neglog(int n, const uint32_t *x, float *a, float *b)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    a[i] = bzk::neglog_u01f(x[i]);
    b[i] = x[i] < 0x80000000u ? -logf(bzk::u01f(x[i])) : -log1pf(-bzk::u01f(~x[i]));
}

extern "C" int neglog_ref(int n, const uint32_t *x, float *a, float *b)
{
    uint32_t *dx = nullptr;
    float *d = nullptr;
    const size_t m = (size_t)n;
    if (cudaMalloc(&dx, 4 * m) != cudaSuccess || cudaMalloc(&d, 8 * m) != cudaSuccess) return 1;
    int bad = cudaMemcpy(dx, x, 4 * m, cudaMemcpyHostToDevice) != cudaSuccess;
    k_neglog<<<(n + 255) / 256, 256>>>(n, dx, d, d + m);
    bad |= cudaMemcpy(a, d, 4 * m, cudaMemcpyDeviceToHost) != cudaSuccess;
    bad |= cudaMemcpy(b, d + m, 4 * m, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(dx);
    cudaFree(d);
    return bad;
}
