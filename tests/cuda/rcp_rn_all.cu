// Test-only: compares rcp_rn of the sweeps with CUDA's division 1.0f / g for every significand and sign
// at the exponents [e0, e1], and counts where they differ.
#include "sweep_group.cuh"

__global__ void compare_kernel(int e0, int e1, unsigned long long *wrong) {
    const uint32_t m = blockIdx.x * blockDim.x + threadIdx.x;          // 2^23 significands
    unsigned n = 0;
    for (int e = e0; e <= e1; ++e)
        for (uint32_t sign = 0; sign < 2; ++sign) {
            const float g = __uint_as_float((sign << 31) | ((uint32_t)(e + 127) << 23) | m);
            n += __float_as_uint(sail::rcp_rn(g)) != __float_as_uint(1.0f / g);
        }
    if (n) atomicAdd(wrong, (unsigned long long)n);
}

extern "C" int rcp_rn_all(int e0, int e1, unsigned long long *d_wrong) {
    if (e0 < -126 || e1 > 127) return -1;
    compare_kernel<<<(1 << 23) / 256, 256>>>(e0, e1, d_wrong);
    if (cudaGetLastError() != cudaSuccess) return -1;
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : -1;
}
