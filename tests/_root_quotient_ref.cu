// Compares the library's sqrt1, sqrt2 and div2 with CUDA's correctly rounded operations:
// every mantissa at the exponents given on the command line, and eight quotients by each
// root.  Prints the numbers of differing roots and quotients.
#include <cstdio>
#include <cstdlib>

#include "../paper_1804_06304_gb300/csrc/ac_internal.cuh"

__global__ void compare(int e0, int e1, unsigned long long *bad)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;   // mantissa, 2^23 threads
    unsigned h = i * 2654435761u;
    unsigned long long roots = 0, quotients = 0;
    for (int e = e0; e <= e1; ++e) {
        const float x = __uint_as_float(((unsigned)(127 + e) << 23) | i);
        float2 rs;
        const float2 r = ac::sqrt2(make_float2(x, x), rs);
        roots += r.x != __fsqrt_rn(x) || r.y != r.x || ac::sqrt1(x) != r.x;
        for (int j = 0; j < 8; ++j) {
            h = h * 1664525u + 1013904223u;
            const float n = __uint_as_float(((unsigned)(113 + (int)(h >> 27)) << 23) | ((h >> 3) & 0x7fffffu));
            const float2 q = ac::div2(make_float2(n, -n), r, rs);
            quotients += q.x != __fdiv_rn(n, r.x) || q.y != -q.x;
        }
    }
    if (roots) atomicAdd(&bad[0], roots);
    if (quotients) atomicAdd(&bad[1], quotients);
}

int main(int argc, char **argv)
{
    if (argc < 3) return 2;
    unsigned long long *d, h[2];
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 3;
    compare<<<(1u << 23) / 256, 256>>>(atoi(argv[1]), atoi(argv[2]), d);
    if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 4;
    printf("%llu %llu\n", h[0], h[1]);
    return 0;
}
