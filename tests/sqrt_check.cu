// Compares sqrt_fast with sqrtf bit for bit: every mantissa at an even and an odd exponent, and a
// spread of mantissas at every exponent of its range, and 0.  Prints the number of differences.
#include <cstdio>

#include "lfsgm_internal.cuh"

__global__ void check(unsigned *bad) {
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x, n = gridDim.x * blockDim.x;
    unsigned b = 0;
    for (unsigned v = i; v < 2u << 23; v += n) {
        const float x = __uint_as_float((126u + (v >> 23)) << 23 | (v & 0x7fffffu));
        b += __float_as_uint(lfsgm::sqrt_fast(x)) != __float_as_uint(sqrtf(x));
    }
    for (unsigned v = i; v < 227u << 12; v += n) {          // 2^-100 .. 2^126
        const float x = __uint_as_float((27u + (v >> 12)) << 23 | ((v & 0xfffu) * 2047u & 0x7fffffu));
        b += __float_as_uint(lfsgm::sqrt_fast(x)) != __float_as_uint(sqrtf(x));
    }
    if (i == 0) b += lfsgm::sqrt_fast(0.f) != 0.f;
    if (b) atomicAdd(bad, b);
}

int main() {
    unsigned *d = nullptr, h = 0;
    if (cudaMalloc(&d, 4) != cudaSuccess || cudaMemset(d, 0, 4) != cudaSuccess) return 2;
    check<<<1024, 256>>>(d);
    if (cudaMemcpy(&h, d, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%u\n", h);
    return h ? 1 : 0;
}
