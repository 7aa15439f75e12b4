// ac_bin.cu -- contours grouped by the brick their centre lies in, ahead of the
// brick kernel (arXiv:1804.06304, "Parallel Contour Evaluation": contours of one
// image region share its voxels).
//
// The brick kernel needs, per brick, the list of its contours; the order of the bricks'
// lists does not matter, because contours evolve independently.  Within a list the order
// decides which contours share a warp, and a warp takes the slowest gather path that any
// of its contours needs: in index order neighbours meet, and the path counters are the
// same in every run.  So this is a counting sort without the ordering: count
// (each contour also learns its rank in its brick), give every brick a range of the
// list, scatter.  A brick then finds its contours with one 8-byte load, and puts a list
// of up to LIST_MAX in index order itself, while its voxels are on their way; longer ones
// (bricks of the caller's choice, crowded explicit seeds) are ordered here.  Bound by launch
// latency for small sets and by the chain of dependent loads at the head of every brick
// for large ones.  Against a radix sort by brick (five launches) and two binary searches
// per brick, passes of 10 iterations went from 111 to 99 us (64x64x32, 2,048 contours),
// 226 to 189 us (512^2), 547 to 504 us (128^3), 2.07 to 2.00 ms (4096^2) and 53.8 to
// 52.7 ms (1024x1024x256, where a CTA has its SM alone while it searches).  Where bricks
// far outnumber contours, or hold hundreds each (see bin_by_sort), the contours are still
// sorted by brick.
#include <cub/cub.cuh>

#include "ac_host.h"

namespace ac {
namespace {

constexpr int SMALL_THREADS = 1024;
constexpr int SMALL_ITEMS = 12;                              // contours per thread
constexpr int SMALL_CONTOURS = SMALL_THREADS * SMALL_ITEMS;
constexpr int SMALL_BRICKS = 8192;                           // 32 KB of counters

__device__ __forceinline__ uint32_t brick_of(const VolDesc &V, int64_t k, int3 B)
{
    const int Bd[3] = {B.x, B.y, B.z};
    int bi[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float c = V.state[d * V.C + k];
        int idx = (int)floorf(c * V.inv_sp[d]);
        idx = idx < 0 ? 0 : (idx >= V.n[d] ? V.n[d] - 1 : idx);
        const int b = idx / Bd[d];
        bi[d] = b >= V.nb[d] ? V.nb[d] - 1 : b;
    }
    return (uint32_t)(V.brick_base + bi[0] + (int64_t)V.nb[0] * (bi[1] + (int64_t)V.nb[1] * bi[2]));
}

// The launch's counters of contour-iterations per gather path start from zero.
__device__ __forceinline__ void clear_counts(unsigned long long *c)
{
    if (blockIdx.x == 0 && threadIdx.x < 3) c[threadIdx.x] = 0;
}

// One-CTA grouping: a list of n > LIST_MAX contours put in index order by a warp, through
// a bitmap of the indices (all below 32 WARP_WORDS) in its own `words`; nothing to wait
// for but the warp.  ORDER_WARPS bitmaps take the space of the counters, which have served.
// Launches of 12,000 contours with 64 lists of 188: 90 us, with the block at one list after
// the other 201 us, sorted 89 us; with 8 lists of 1,500: 282, 300 and 288 us.
constexpr int WARP_WORDS = SMALL_CONTOURS / 32;
constexpr int ORDER_WARPS = SMALL_BRICKS / WARP_WORDS;
static_assert(SMALL_CONTOURS % 1024 == 0, "the same number of bitmap words for every lane");

__device__ __forceinline__ void order_list_warp(uint32_t *list, uint32_t n, uint32_t *words)
{
    constexpr int PER = WARP_WORDS / 32;
    const uint32_t lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < PER; ++j) words[j * 32 + lane] = 0;
    __syncwarp();
    for (uint32_t i = lane; i < n; i += 32) atomicOr(&words[list[i] >> 5], 1u << (list[i] & 31));
    __syncwarp();
    uint32_t mine = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) mine += __popc(words[lane * PER + j]);
    uint32_t at = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += y;
    }
    at -= mine;
    for (int j = 0; j < PER; ++j)
        for (uint32_t w = words[lane * PER + j]; w; w &= w - 1) list[at++] = 32 * (lane * PER + j) + (__ffs(w) - 1);
    __syncwarp();   // `words` is free again
}

// Few contours and bricks: one CTA counts in shared memory, scans and scatters, each
// thread keeping its contours' (brick, rank) in registers: one launch instead of a clear
// and three.  12 contours a thread is what its 64 registers hold without spills to speak of.
__global__ void __launch_bounds__(SMALL_THREADS) bin_small_kernel(const VolDesc *vols, int n_vols, int total, int3 B,
                                                                  int nb, uint2 *ranges, uint32_t *order,
                                                                  unsigned long long *path_counts)
{
    clear_counts(path_counts);
    __shared__ uint32_t warp_sums[32], count[SMALL_BRICKS];
    for (int i = threadIdx.x; i < nb; i += SMALL_THREADS) count[i] = 0;
    __syncthreads();
    uint32_t at[SMALL_ITEMS];   // brick << 16 | rank (brick < 2^13, rank < 2^14)
#pragma unroll
    for (int j = 0; j < SMALL_ITEMS; ++j) {
        const int g = j * SMALL_THREADS + threadIdx.x;
        if (g < total) {
            const VolDesc &V = vols[find_set(vols, n_vols, g)];
            const uint32_t b = brick_of(V, g - V.contour_base, B);
            at[j] = b << 16 | atomicAdd(&count[b], 1u);
        }
    }
    __syncthreads();
    // thread t scans bricks [t per, (t + 1) per)
    const int per = (nb + SMALL_THREADS - 1) / SMALL_THREADS;
    const int b0 = threadIdx.x * per, b1 = min(b0 + per, nb);
    uint32_t mine = 0, sum;
    for (int b = b0; b < b1; ++b) mine += count[b];
    uint32_t start = block_exclusive(mine, warp_sums, &sum);
    bool any_long = false;
    for (int b = b0; b < b1; ++b) {
        const uint32_t n = count[b];
        ranges[b] = make_uint2(start, n);
        count[b] = start;
        start += n;
        any_long = any_long || n > LIST_MAX;
    }
    any_long = __syncthreads_or(any_long);
#pragma unroll
    for (int j = 0; j < SMALL_ITEMS; ++j) {
        const int g = j * SMALL_THREADS + threadIdx.x;
        if (g < total) order[count[at[j] >> 16] + (at[j] & 0xFFFFu)] = (uint32_t)g;
    }
    if (!any_long) return;
    __syncthreads();
    // warp w: the long ones among bricks w, w + ORDER_WARPS, ..., 32 of them looked at in one load
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w >= ORDER_WARPS) return;
    for (int b = w; b < nb; b += 32 * ORDER_WARPS) {
        const uint2 r = b + lane * ORDER_WARPS < nb ? ranges[b + lane * ORDER_WARPS] : make_uint2(0, 0);
        for (unsigned todo = __ballot_sync(0xffffffffu, r.y > LIST_MAX); todo; todo &= todo - 1) {
            const int l = __ffs(todo) - 1;
            const uint32_t first = __shfl_sync(0xffffffffu, r.x, l), n = __shfl_sync(0xffffffffu, r.y, l);
            order_list_warp(order + first, n, count + w * WARP_WORDS);
        }
    }
}

__global__ void bin_count_kernel(const VolDesc *vols, int n_vols, int64_t total, int3 B, uint2 *ranges,
                                 uint32_t *keys, uint32_t *ranks, unsigned long long *path_counts)
{
    clear_counts(path_counts);
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
        const VolDesc &V = vols[find_set(vols, n_vols, g)];
        const uint32_t b = brick_of(V, g - V.contour_base, B);
        keys[g] = b;
        ranks[g] = atomicAdd(&ranges[b].y, 1u);
    }
}

// A range of the list for every brick, in whatever order the blocks get to it.  head[0]:
// the list's length so far; head[1]: whether there are lists that bin_order_kernel orders.
__global__ void __launch_bounds__(256) bin_alloc_kernel(uint2 *ranges, int64_t nb, uint32_t *head)
{
    __shared__ uint32_t warp_sums[32], base;
    for (int64_t b0 = blockIdx.x * (int64_t)blockDim.x; b0 < nb; b0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = b0 + threadIdx.x;
        uint32_t sum;
        const uint32_t n = b < nb ? ranges[b].y : 0u;
        const uint32_t off = block_exclusive(n, warp_sums, &sum);
        if (n > LIST_MAX) head[1] = 1;
        if (threadIdx.x == 0) base = atomicAdd(&head[0], sum);
        __syncthreads();
        if (b < nb) ranges[b].x = base + off;
        __syncthreads();
    }
}

__global__ void bin_scatter_kernel(const uint2 *ranges, const uint32_t *keys, const uint32_t *ranks, int64_t total,
                                   uint32_t *order)
{
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x)
        order[ranges[keys[g]].x + ranks[g]] = (uint32_t)g;
}

// A list of n > LIST_MAX contours put in index order by its block: up to one contour a
// thread by counting the smaller ones, more through a bitmap of the indices, 32 WORDS of
// them at a time, with the list in order going to `tmp` first.  Latency of one block per
// list: 64 lists of 3,125 contours 8.4 us, 216 of 4,630 (four bitmaps) 31 us, in launches
// whose brick kernels take 490 and 1,410 us.
constexpr int ORDER_THREADS = 1024;
constexpr int WORDS = 8192;

__device__ __forceinline__ void order_list(uint32_t *list, uint32_t *tmp, uint32_t n, uint32_t *words,
                                           uint32_t *warp_sums)
{
    const uint32_t t = threadIdx.x;
    if (n <= ORDER_THREADS) {
        if (t < n) words[t] = list[t];
        __syncthreads();
        if (t < n) {
            const uint32_t g = words[t];
            uint32_t rank = 0;
            for (uint32_t j = 0; j < n; ++j) rank += words[j] < g ? 1 : 0;
            list[rank] = g;
        }
        __syncthreads();   // `words` is free again
        return;
    }
    uint32_t lo = 0xffffffffu, hi = 0;
    for (uint32_t i = t; i < n; i += ORDER_THREADS) {
        lo = min(lo, list[i]);
        hi = max(hi, list[i]);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((t & 31) == 0) {
        words[t >> 5] = lo;
        words[32 + (t >> 5)] = hi;
    }
    __syncthreads();
    for (int w = 0; w < ORDER_THREADS / 32; ++w) {
        lo = min(lo, words[w]);
        hi = max(hi, words[32 + w]);
    }
    __syncthreads();
    constexpr int PER = WORDS / ORDER_THREADS;
    uint32_t done = 0;
    for (uint64_t base = lo; base <= hi; base += 32 * WORDS) {
#pragma unroll
        for (int j = 0; j < PER; ++j) words[j * ORDER_THREADS + t] = 0;
        __syncthreads();
        for (uint32_t i = t; i < n; i += ORDER_THREADS) {
            const uint32_t g = list[i], bit = g - (uint32_t)base;
            if (g >= base && bit < 32 * WORDS) atomicOr(&words[bit >> 5], 1u << (bit & 31));
        }
        __syncthreads();
        uint32_t mine = 0, sum;
#pragma unroll
        for (int j = 0; j < PER; ++j) mine += __popc(words[t * PER + j]);
        uint32_t at = done + block_exclusive(mine, warp_sums, &sum);
        for (int j = 0; j < PER; ++j)
            for (uint32_t w = words[t * PER + j]; w; w &= w - 1)
                tmp[at++] = (uint32_t)base + 32 * (t * PER + j) + (__ffs(w) - 1);
        done += sum;
        __syncthreads();   // `words` and `warp_sums` are free again, `tmp` is written
    }
    for (uint32_t i = t; i < n; i += ORDER_THREADS) list[i] = tmp[i];
    __syncthreads();
}

// A block looks at 32 bricks, gridDim.x apart, in one load.  `tmp` holds a word per contour.
// Most launches have nothing to order: the kernel is launched while the scatter still runs
// (programmatic dependent launch) and waits for it here, so that it costs them nothing
// (after the scatter: 4 us, 145 -> 149 us for 900x800 u16).
__global__ void __launch_bounds__(ORDER_THREADS) bin_order_kernel(const uint2 *ranges, int64_t nb, const uint32_t *head,
                                                                  uint32_t *order, uint32_t *tmp)
{
    __shared__ uint32_t words[WORDS], warp_sums[32];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (head[1] == 0) return;
    for (int64_t b = blockIdx.x; b < nb; b += 32 * (int64_t)gridDim.x) {
        const int64_t mine = b + (int64_t)(threadIdx.x & 31) * gridDim.x;
        const uint2 r = mine < nb ? ranges[mine] : make_uint2(0, 0);
        for (unsigned todo = __ballot_sync(0xffffffffu, r.y > LIST_MAX); todo; todo &= todo - 1) {   // the same in every warp
            const int l = __ffs(todo) - 1;
            const uint32_t first = __shfl_sync(0xffffffffu, r.x, l), n = __shfl_sync(0xffffffffu, r.y, l);
            order_list(order + first, tmp + first, n, words, warp_sums);
        }
    }
}

__global__ void bin_keys_kernel(const VolDesc *vols, int n_vols, int64_t total, int3 B, uint32_t *keys,
                                uint32_t *vals, unsigned long long *path_counts)
{
    clear_counts(path_counts);
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total; g += (int64_t)gridDim.x * blockDim.x) {
        const VolDesc &V = vols[find_set(vols, n_vols, g)];
        keys[g] = brick_of(V, g - V.contour_base, B);
        vals[g] = (uint32_t)g;
    }
}

unsigned blocks_of(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 1 << 16); }

int key_bits(int64_t bricks)
{
    int b = 1;
    while (((int64_t)1 << b) < bricks + 1) ++b;
    return b;
}

constexpr int64_t CROWDED = 512;   // contours per brick, on average

bool bin_small(int64_t total, int64_t bricks) { return total <= SMALL_CONTOURS && bricks <= SMALL_BRICKS; }

size_t align16(size_t n) { return (n + 15) / 16 * 16; }

}  // namespace

// The table of ranges costs 8 bytes and a clear per brick: not worth it when bricks
// outnumber contours several times (a few explicit seeds in a large volume).  Where the
// mean list is long, counting serialises on the few bricks' counters and every list has to
// be ordered after it.  Launches counted / sorted, in us: mean list 313 104 / 116, 438 125 /
// 131, 602 249 / 223, 751 1083 / 1037, 1852 588 / 518, 4630 1320 / 1150.  The one-CTA form
// counts in shared memory.
bool bin_by_sort(int64_t total, int64_t bricks)
{
    const bool crowded = total > CROWDED * bricks && !bin_small(total, bricks);
    return crowded || bricks > 4 * total + 65536;
}

cudaError_t bin_table_bytes(int64_t total, int64_t bricks, bool sort, size_t *bytes)
{
    if (!sort) {
        *bytes = 16 + sizeof(uint2) * (size_t)bricks;
        return cudaSuccess;
    }
    size_t tmp = 0;
    uint32_t *n = nullptr;
    const cudaError_t e = cub::DeviceRadixSort::SortPairs(nullptr, tmp, n, n, n, n, (int)total, 0, key_bits(bricks));
    *bytes = align16(sizeof(uint32_t) * (size_t)total) + tmp;
    return e;
}

void bin_bind(EvolveArgs &a, const BinSpace &s)
{
    a.order = s.order;
    a.ranges = s.sort ? nullptr : reinterpret_cast<const uint2 *>(static_cast<unsigned char *>(s.table) + 16);
    a.sorted_brick = s.sort ? static_cast<const uint32_t *>(s.table) : nullptr;
}

cudaError_t launch_bin(const EvolveArgs &a, const BinSpace &s, cudaStream_t st, int64_t *launches)
{
    const int3 B = make_int3(a.B[0], a.B[1], a.B[2]);
    const int64_t total = a.total_contours, bricks = a.total_bricks;
    if (s.sort) {
        bin_keys_kernel<<<blocks_of(total), 256, 0, st>>>(a.vols, a.n_vols, total, B, s.keys, s.ranks,
                                                         a.path_counts);
        *launches += 1;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        const size_t sorted = align16(sizeof(uint32_t) * (size_t)total);
        size_t tmp = s.table_bytes - sorted;
        return cub::DeviceRadixSort::SortPairs(static_cast<unsigned char *>(s.table) + sorted, tmp, s.keys,
                                               static_cast<uint32_t *>(s.table), s.ranks, s.order, (int)total, 0,
                                               key_bits(bricks), st);
    }
    uint2 *ranges = const_cast<uint2 *>(a.ranges);
    if (bin_small(total, bricks)) {
        bin_small_kernel<<<1, SMALL_THREADS, 0, st>>>(a.vols, a.n_vols, (int)total, B,
                                                                              (int)bricks, ranges, s.order, a.path_counts);
        *launches += 1;
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(s.table, 0, 16 + sizeof(uint2) * (size_t)bricks, st);
    if (e != cudaSuccess) return e;
    bin_count_kernel<<<blocks_of(total), 256, 0, st>>>(a.vols, a.n_vols, total, B, ranges, s.keys, s.ranks,
                                                      a.path_counts);
    bin_alloc_kernel<<<blocks_of(bricks), 256, 0, st>>>(ranges, bricks, static_cast<uint32_t *>(s.table));
    bin_scatter_kernel<<<blocks_of(total), 256, 0, st>>>(ranges, s.keys, s.ranks, total, s.order);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the keys have been read when it starts to order: their space serves it
    cudaLaunchConfig_t order{};
    order.gridDim = dim3((unsigned)std::min<int64_t>(bricks, 152));
    order.blockDim = dim3(ORDER_THREADS);
    order.stream = st;
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    order.attrs = &early;
    order.numAttrs = 1;
    e = cudaLaunchKernelEx(&order, bin_order_kernel, (const uint2 *)ranges, bricks, static_cast<const uint32_t *>(s.table),
                           s.order, s.keys);
    if (e != cudaSuccess) return e;
    *launches += 4;
    return cudaGetLastError();
}

}  // namespace ac
