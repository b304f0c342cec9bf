// Checks rcp_nr on every denormal, zero, the infinities and NaN against the correctly rounded reciprocal: the number of
// inputs that differ, and the largest difference in units in the last place (infinity counts as the unit after the largest
// float).  Built and run by tests/test_gpu_rcp_small.py.
#include <cstdio>
#include <cstdlib>

#include "../../paper_2405_02508_gb300/csrc/mer_device.cuh"

__global__ void k_check(unsigned long long* out) {
    unsigned long long diff = 0ull, worst = 0ull;
    const unsigned n = 0x00800000u;  // the denormals and zero, then +infinity and a NaN; both signs
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < 2u * (n + 2u); i += gridDim.x * blockDim.x) {
        const unsigned k = i >> 1, bits = k < n ? k : (k == n ? 0x7f800000u : 0x7fc00000u);
        const float x = __uint_as_float(bits | (i << 31));
        const float a = mer::rcp_nr(x), c = __frcp_rn(x);
        if (a != a && c != c) continue;
        const unsigned ua = __float_as_uint(a), uc = __float_as_uint(c);
        if (ua != uc) {
            ++diff;
            const unsigned long long d = (ua ^ uc) >> 31 || a != a || c != c ? ~0ull >> 1 : (ua > uc ? ua - uc : uc - ua);
            if (d > worst) worst = d;
        }
    }
    atomicAdd(&out[0], diff);
    atomicMax(&out[1], worst);
}

int main() {
    unsigned long long* out = nullptr;
    if (cudaMalloc(&out, 2 * sizeof(unsigned long long)) != cudaSuccess) return 2;
    if (cudaMemset(out, 0, 2 * sizeof(unsigned long long)) != cudaSuccess) return 2;
    k_check<<<4096, 256>>>(out);
    unsigned long long h[2] = {0ull, 0ull};
    if (cudaMemcpy(h, out, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu %llu\n", h[0], h[1]);
    cudaFree(out);
    return 0;
}
