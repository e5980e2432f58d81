// Test harness: the FP32 network's SiLU (act_math.cuh) on host inputs z, for
// tests/test_gpu_mlp_fp32.py.
#include <cstdint>
#include <cuda_runtime.h>

#include "../paper_2206_02937_gb300/csrc/act_math.cuh"

namespace {
__global__ void k_eval(const float* z, int64_t n, float* out)
{
    const int64_t i = 2 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= n) return;
    float a, b;
    compton::act::upk2(compton::act::silu2_f32(compton::act::pk2(z[i], i + 1 < n ? z[i + 1] : 0.0f)), a, b);
    out[i] = a;
    if (i + 1 < n) out[i + 1] = b;
}
}  // namespace

extern "C" int silu_f32_eval(const float* z_host, int64_t n, float* out_host)
{
    float* d = nullptr;
    const size_t b = (size_t)n * sizeof(float);
    if (n <= 0 || cudaMalloc(&d, 2 * b) != cudaSuccess) return 1;
    int rc = cudaMemcpy(d, z_host, b, cudaMemcpyHostToDevice) != cudaSuccess ? 2 : 0;
    if (!rc) {
        k_eval<<<(unsigned)(((n + 1) / 2 + 255) / 256), 256>>>(d, n, d + n);
        if (cudaGetLastError() != cudaSuccess || cudaMemcpy(out_host, d + n, b, cudaMemcpyDeviceToHost) != cudaSuccess)
            rc = 3;
    }
    cudaFree(d);
    return rc;
}
