// Compares the library's div2 with CUDA's division at the ends of its range: numerators of
// QUOTIENT_MIN to QUOTIENT_MAX and zero, by roots of radicands of ROOT_MIN to 2^50, and zero by
// the root of zero; numerators whose mantissas are all zeros, all ones, next to these, or the
// root's own by every root of two octaves; and max3_abs with the largest magnitude, NaN first.  Prints the numbers of
// differing quotients and maxima (zeros of either sign agree).
#include <cstdio>

#include "../paper_1804_06304_gb300/csrc/ac_internal.cuh"

__device__ bool same(float a, float b) { return a == b || (a != a && b != b); }

__global__ void compare(unsigned long long *bad)
{
    unsigned h = (blockIdx.x * blockDim.x + threadIdx.x) * 2654435761u;
    auto next = [&]() {
        h = h * 1664525u + 1013904223u;
        return (h >> 9) * 0x9E3779B1u ^ h;
    };
    unsigned long long quotients = 0, maxima = 0;
    for (int j = 0; j < 512; ++j) {
        float n[2], x[2];
        for (int i = 0; i < 2; ++i) {
            const unsigned kind = next() % 16;
            n[i] = __uint_as_float((next() & 0x80000000u) | (27 + next() % 176) << 23 | (next() & 0x7fffffu));
            x[i] = __uint_as_float((31 + next() % 146) << 23 | (next() & 0x7fffffu));
            if (kind <= 1) n[i] = 0.0f;
            if (kind == 1) x[i] = 0.0f;
            if (kind == 2) n[i] = ac::QUOTIENT_MIN;
            if (kind == 3) n[i] = -ac::QUOTIENT_MAX;
            if (kind == 4) x[i] = ac::ROOT_MIN;
        }
        float2 rs;
        const float2 r = ac::sqrt2(make_float2(x[0], x[1]), rs), q = ac::div2(make_float2(n[0], n[1]), r, rs);
        for (int i = 0; i < 2; ++i) {
            quotients += (i ? r.y : r.x) != __fsqrt_rn(x[i]) || ac::sqrt1(x[i]) != __fsqrt_rn(x[i]);
            quotients += !same(i ? q.y : q.x, x[i] > 0.0f ? __fdiv_rn(n[i], __fsqrt_rn(x[i])) : 0.0f);
        }
        float v[3], want = 0.0f;
        for (int i = 0; i < 3; ++i) {
            v[i] = __uint_as_float(next());
            want = v[i] != v[i] || want != want ? __uint_as_float(0x7fffffffu) : fmaxf(want, fabsf(v[i]));
        }
        const float got = ac::max3_abs(v[0], v[1], v[2]);
        maxima += !same(got, want) || (__float_as_uint(got) >> 31) != 0;
    }
    if (quotients) atomicAdd(&bad[0], quotients);
    if (maxima) atomicAdd(&bad[1], maxima);
}

__global__ void special(unsigned long long *bad)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;   // 2^24 threads
    const float x = __uint_as_float((127u << 23) + i);
    float2 rs;
    const float2 r = ac::sqrt2(make_float2(x, x), rs);
    const unsigned own = __float_as_uint(r.x) & 0x7fffffu;
    const unsigned mantissas[] = {0u, 1u, 2u, 0x7ffffdu, 0x7ffffeu, 0x7fffffu, own, own ^ 1u};
    unsigned long long quotients = 0;
    for (unsigned m : mantissas) {
        const float n = __uint_as_float(127u << 23 | m);
        const float2 q = ac::div2(make_float2(n, -n), r, rs);
        quotients += q.x != __fdiv_rn(n, r.x) || q.y != -q.x;
    }
    if (quotients) atomicAdd(&bad[0], quotients);
}

int main()
{
    unsigned long long *d, h[2];
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 3;
    compare<<<1024, 256>>>(d);
    special<<<(1u << 24) / 256, 256>>>(d);
    if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 4;
    printf("%llu %llu\n", h[0], h[1]);
    return 0;
}
