// Checks f2d and i2d (exact conversions to double with integer instructions) against the hardware's on every 32-bit
// pattern (NaN to NaN).  Built and run by tests/test_gpu_convert.py; prints the number of mismatches of each.
#include <cstdio>

#include "../../paper_2405_02508_gb300/csrc/mer_device.cuh"

__global__ void k_check(unsigned long long* out) {
    unsigned long long f = 0ull, n = 0ull;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long b = blockIdx.x * blockDim.x + threadIdx.x; b < (1ull << 32); b += stride) {
        const float x = __uint_as_float((unsigned)b);
        const double got = mer::f2d(x), want = (double)x;
        f += isnan(want) ? !isnan(got) : __double_as_longlong(got) != __double_as_longlong(want);
        const int v = (int)(unsigned)b;
        n += __double_as_longlong(mer::i2d(v)) != __double_as_longlong((double)v);
    }
    atomicAdd(&out[0], f);
    atomicAdd(&out[1], n);
}

int main() {
    unsigned long long* out = nullptr;
    if (cudaMalloc(&out, 2 * sizeof(unsigned long long)) != cudaSuccess) return 2;
    if (cudaMemset(out, 0, 2 * sizeof(unsigned long long)) != cudaSuccess) return 2;
    k_check<<<4096, 256>>>(out);
    unsigned long long h[2] = {1ull, 1ull};
    if (cudaMemcpy(h, out, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu %llu\n", h[0], h[1]);
    cudaFree(out);
    return 0;
}
