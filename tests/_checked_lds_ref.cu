// Addresses given to checked_lds (compiled with AC_CHECKED) around an array of N elements:
// prints how many come back changed or reported wrongly.  Nothing is read through them.
#include <cstdio>

#include "../paper_1804_06304_gb300/csrc/ac_internal.cuh"

constexpr int N = 24;

template <typename T> __device__ void probe(const T *array, int32_t *st, int *wrong)
{
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(array);
    for (int far = 0; far < 4; ++far)
        for (int byte = -40; byte < (N + 4) * (int)sizeof(T); ++byte) {
            *st = 0;
            const uint32_t at = base + byte, got = ac::checked_lds(at, far * (uint32_t)sizeof(T), array, N, st);
            const bool inside = byte >= 0 && byte % (int)sizeof(T) == 0 && byte / (int)sizeof(T) + far < N;
            if (got != (inside ? at : base) || (*st != 0) != !inside) ++*wrong;
        }
}

__global__ void probes(int32_t *st, int *wrong)
{
    __shared__ double room[3 * N];
    probe(reinterpret_cast<const uint8_t *>(room + N), st, wrong);
    probe(reinterpret_cast<const uint16_t *>(room + N), st, wrong);
    probe(reinterpret_cast<const float *>(room + N), st, wrong);
    probe(room + N, st, wrong);
}

int main()
{
    int *d, h[2] = {0, 0};
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 3;
    probes<<<1, 1>>>(d, d + 1);
    if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 4;
    printf("%d\n", h[1]);
    return 0;
}
