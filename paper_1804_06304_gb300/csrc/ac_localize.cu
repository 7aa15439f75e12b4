// ac_localize.cu -- energy cull and overlap competition (stage a9).
//
// Section "Results and Discussion" of arXiv:1804.06304: contours with energy above
// E0 are removed, and overlapping contours (|c' - c''| < max(R', R'') / 2^(1/3))
// compete, the lower energy surviving.  Visiting survivors by increasing (E, k)
// and keeping a contour unless a kept one overlaps it defines the result.  The
// GPU computes exactly that set in parallel rounds: a contour is accepted once
// every overlapping contour of higher priority is rejected, and rejected as soon
// as one of them is accepted (the lexicographically first maximal independent
// set).  Neighbours are found through a uniform grid of cell size
// rho max(R), built by counting.  Within a round a contour whose higher-priority
// neighbours are still open looks again a bounded number of times, so one round settles
// nearly everything.
//
// Any number of contour sets is localized in one pass: their contours are
// indexed one after another (set-major), the cull and the selection of survivors
// run once over all of them, one sort by (set, E, k) gives every set's priority
// order, every set has its own grid, placed one after another in one cell index
// space, and each round decides survivors of all sets at once.  A batch costs the same
// few launches and two stream synchronisations (three when many survive) whatever the
// number of sets.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <cub/cub.cuh>
#include <math_constants.h>
#include <string>
#include <thrust/iterator/counting_iterator.h>
#include <vector>

#include "ac_host.h"

#define LC_FAIL(code, msg)        \
    do {                          \
        ac::set_error(msg);       \
        return code;              \
    } while (0)

#define LC_CUDA(call)                                                                                   \
    do {                                                                                                \
        cudaError_t e_ = (call);                                                                        \
        if (e_ != cudaSuccess) {                                                                        \
            ac::set_error(std::string("ac_localize: ") + #call + ": " + cudaGetErrorString(e_));         \
            return e_ == cudaErrorMemoryAllocation ? AC_ERR_OOM : AC_ERR_CUDA;                          \
        }                                                                                               \
    } while (0)

namespace ac {
namespace {

enum : uint8_t { UNDECIDED = 0, ACCEPTED = 1, REJECTED = 2 };

struct Grid {
    float inv_h;
    int nc[3];
};

// One contour set of a batch, as the kernels see it.
struct LocSet {
    const float *state;       // 5 x C
    const int32_t *status;    // the set's status word
    int64_t C;
    int64_t cbase;            // index of the set's first contour in the batch
    int64_t sbase;            // index of its first survivor (survivors in priority order)
    int64_t n;                // its survivors
    int64_t cellbase;         // index of its first grid cell
    Grid g;
    float E0, rho;
};

// The same by a whole warp, 32 sets looked at in one load (among 1,000 sets two loads that
// wait for each other instead of ten).
template <int64_t LocSet::*base>
__device__ __forceinline__ int set_of_warp(const LocSet *sets, int nsets, int64_t i)
{
    int lo = 0, n = nsets;   // the set is among lo .. lo + n - 1
    while (n > 1) {
        const int step = (n + 31) >> 5, at = (threadIdx.x & 31) * step;
        const bool below = at < n && sets[lo + at].*base <= i;
        const int k = __popc(__ballot_sync(0xffffffffu, below)) - 1;   // offsets increase: the lanes below come first
        lo += k * step;
        n = min(step, n - k * step);
    }
    return lo;
}

// Per-set counters, CNT_N int32 per set in one device array (and its page-locked
// copy); two batch totals follow them.  CNT_OPEN: survivors a round left undecided.
enum { CNT_SURV, CNT_MAXR, CNT_STATUS, CNT_ABASE, CNT_ACC, CNT_OPEN, CNT_N };

// the set holding batch position `i` of the index whose set offsets are `base`
// (sets in increasing order of their offsets)
template <int64_t LocSet::*base>
__device__ __forceinline__ int set_of(const LocSet *sets, int nsets, int64_t i)
{
    int lo = 0, hi = nsets - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (sets[mid].*base <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Survivors of the energy cull (flags over the batch's contours), their count
// and largest radius per set (float bits of R > 0 order like ints), and the set's
// status word.  Block row blockIdx.y is set blockIdx.y.  Reads 8 bytes a contour; one
// pair of atomics per block, since one per warp serialised on the set's two counters
// (1.4 M contours: 46 us).
__global__ void __launch_bounds__(256) flag_kernel(const LocSet *sets, uint8_t *flags, int32_t *cnt)
{
    const LocSet &S = sets[blockIdx.y];
    const float *E = S.state + 4 * S.C, *R = S.state + 3 * S.C;
    int32_t *c = cnt + (int64_t)blockIdx.y * CNT_N;
    if (blockIdx.x == 0 && threadIdx.x == 0) c[CNT_STATUS] = *S.status;
    int32_t nk = 0, mx = 0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < S.C; k += (int64_t)gridDim.x * blockDim.x) {
        const float e = E[k];
        const bool keep = isfinite(e) && !(e > S.E0);
        flags[S.cbase + k] = keep ? 1 : 0;
        if (keep) {
            ++nk;
            mx = max(mx, __float_as_int(R[k]));
        }
    }
    __shared__ int32_t wn[8], wm[8];
    nk = __reduce_add_sync(0xffffffffu, nk);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) {
        wn[threadIdx.x >> 5] = nk;
        wm[threadIdx.x >> 5] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            nk += wn[w];
            mx = max(mx, wm[w]);
        }
        if (nk) atomicAdd(&c[CNT_SURV], nk);
        if (mx > 0) atomicMax(&c[CNT_MAXR], mx);
    }
}

// The energy's bits, mapped so that unsigned order is the order of the floats (-0 folded
// into +0).
__device__ __forceinline__ uint32_t energy_key(float e)
{
    const uint32_t b = __float_as_uint(e + 0.0f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// One small set: the cull, the list of survivors, their sort keys and the set's counters
// (all of them: nothing is cleared before) by one CTA, a tile of contours at a time.
// Launch latency is what a small set pays for: this and collect_small_kernel replace a
// clear and nine launches (2,048 contours: 135 -> 92 us a call).
constexpr int SMALL_THREADS = 1024;
constexpr int SMALL_TILES = 16;
constexpr int64_t SMALL_CONTOURS = (int64_t)SMALL_THREADS * SMALL_TILES;

__global__ void __launch_bounds__(SMALL_THREADS) cull_small_kernel(const LocSet *set, int32_t *cnt, int32_t *surv,
                                                                   uint64_t *keys)
{
    __shared__ uint32_t warp_sums[32];
    __shared__ int32_t max_r;
    const LocSet &S = *set;
    const float *E = S.state + 4 * S.C, *R = S.state + 3 * S.C;
    const int C = (int)S.C;
    if (threadIdx.x == 0) max_r = 0;
    __syncthreads();
    uint32_t n = 0;
    int32_t mx = 0;
    for (int k0 = 0; k0 < C; k0 += SMALL_THREADS) {
        const int k = k0 + threadIdx.x;
        const float e = k < C ? E[k] : CUDART_INF_F;
        const bool keep = isfinite(e) && !(e > S.E0);
        uint32_t tile;
        const uint32_t at = n + block_exclusive(keep ? 1u : 0u, warp_sums, &tile);
        if (keep) {
            surv[at] = k;
            keys[at] = energy_key(e);
            mx = max(mx, __float_as_int(R[k]));
        }
        n += tile;
        __syncthreads();
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((threadIdx.x & 31) == 0) atomicMax(&max_r, mx);
    __syncthreads();
    if (threadIdx.x == 0) {
        cnt[CNT_SURV] = (int32_t)n;
        cnt[CNT_MAXR] = max_r;
        cnt[CNT_STATUS] = *S.status;
        cnt[CNT_ABASE] = cnt[CNT_ACC] = cnt[CNT_OPEN] = 0;
        cnt[CNT_N] = (int32_t)n;       // the totals of a batch of one
        cnt[CNT_N + 1] = 0;
    }
}

// Sort keys of the survivors: set index above the energy's key.  The survivors arrive by
// batch index, so a stable sort leaves equal energies by k.
__global__ void key_kernel(const LocSet *sets, int nsets, const int32_t *surv, int64_t n, uint64_t *keys)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = surv[i];
        const int s = set_of<&LocSet::cbase>(sets, nsets, g);
        const LocSet &S = sets[s];
        keys[i] = ((uint64_t)s << 32) | energy_key(S.state[4 * S.C + (g - S.cbase)]);
    }
}

__device__ __forceinline__ int cell_axis(float x, float inv_h, int nc)
{
    int i = (int)floorf(x * inv_h);
    return i < 0 ? 0 : (i >= nc ? nc - 1 : i);
}

// Positions in priority order, each survivor's grid cell and its rank in the cell
// (`count` per cell, cleared before)
__global__ void cell_count_kernel(const LocSet *sets, int nsets, const int32_t *order, int64_t n, float4 *pos,
                                  uint32_t *cell, uint32_t *rank, int32_t *count, uint8_t *status)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const LocSet &S = sets[set_of<&LocSet::sbase>(sets, nsets, p)];
        const int64_t k = order[p] - S.cbase;
        const float4 q = make_float4(S.state[k], S.state[S.C + k], S.state[2 * S.C + k], S.state[3 * S.C + k]);
        pos[p] = q;
        const int cx = cell_axis(q.x, S.g.inv_h, S.g.nc[0]);
        const int cy = cell_axis(q.y, S.g.inv_h, S.g.nc[1]);
        const int cz = cell_axis(q.z, S.g.inv_h, S.g.nc[2]);
        const int64_t c = S.cellbase + cx + (int64_t)S.g.nc[0] * (cy + (int64_t)S.g.nc[1] * cz);
        cell[p] = (uint32_t)c;
        rank[p] = (uint32_t)atomicAdd(&count[c], 1);
        status[p] = UNDECIDED;
    }
}

// The survivors, their positions and their states by cell (in any order within a cell);
// `rank` becomes a survivor's place in the list
__global__ void cell_scatter_kernel(int64_t n, const uint32_t *cell, uint32_t *rank, const int32_t *start,
                                    const float4 *pos, uint32_t *list, float4 *list_pos, uint8_t *list_status)
{
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = (int64_t)start[cell[p]] + rank[p];
        list[j] = (uint32_t)p;
        list_pos[j] = pos[p];
        list_status[j] = UNDECIDED;
        rank[p] = (uint32_t)j;
    }
}

// One round of the parallel greedy competition over the survivors of every set.
// A set's cells hold only its own survivors, and within a set batch order is
// priority order.  CNT_OPEN counts per set what is still open.
//
// A warp per survivor.  The three cells of a row along x are neighbours in the list, so
// a survivor's 27 cells are 9 ranges: lanes 0-8 read their bounds, and the lanes then
// share the entries.  Bound by the latency of the chain position -> bounds -> entry (the
// states lie by list place too, so that they come with the entry and not after it): one
// thread per survivor walked 27 cells of it one after the other, and every link of a
// chain of competing contours cost a launch.  Here a warp that waits for a neighbour
// looks again up to LOOKS times, re-reading only the neighbours still open (two per
// lane are kept; with more it reads everything again); what is open after that is left
// to the next round, so nothing depends on which blocks run together.  2,048 contours
// (about 770 survivors): the rounds of a call 168 -> 11 us; 1.4 M (540 thousand
// survivors): 557 -> 165 us (240 us with the states by priority alone).
//
// Several sets are taken in turn: blocks are launched in about the order of their number,
// and neighbours in priority order of one small set would all wait for each other.  The
// first heads * ROUND_WARPS survivors of every set come first, a block of every set after
// the other, then what the larger sets have beyond that.  Rounds of 1,000 sets of 2,000
// contours: set after set 2,105 us, in turn 401 us; of 1,000 sets of 500 398 and 101 us.
constexpr int LOOKS = 64;
constexpr int ROUND_WARPS = 8;
constexpr int64_t RESIDENT_WARPS = 152 * 64;
constexpr uint32_t NONE = 0xffffffffu;

__global__ void __launch_bounds__(32 * ROUND_WARPS) round_kernel(const LocSet *sets, int nsets, const float4 *pos, int64_t n,
                                                    const int32_t *start, const uint32_t *list, const float4 *list_pos,
                                                    const uint32_t *place, uint8_t *list_status, uint8_t *status,
                                                    int32_t *cnt, unsigned heads)
{
    const unsigned in_heads = heads * (unsigned)nsets;   // blocks
    int64_t p;
    int s = 0;
    if (blockIdx.x < in_heads) {
        s = (int)(blockIdx.x % (unsigned)nsets);
        p = (int64_t)(blockIdx.x / (unsigned)nsets) * ROUND_WARPS + (threadIdx.x >> 5);
        if (p >= sets[s].n) return;
        p += sets[s].sbase;
    } else {
        p = (int64_t)(blockIdx.x - in_heads) * ROUND_WARPS + (threadIdx.x >> 5);
        if (p >= n) return;
        s = set_of_warp<&LocSet::sbase>(sets, nsets, p);
        if (p < sets[s].sbase + (int64_t)heads * ROUND_WARPS) return;   // among the heads
    }
    const float4 a = pos[p];
    const uint32_t mine = place[p];
    if (status[p] != UNDECIDED) return;   // the same for the whole warp
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const LocSet &S = sets[s];
    const Grid &g = S.g;
    const float rho = S.rho;
    int from = 0, len = 0;   // lanes 0-8: a row of up to three cells
    if (lane < 9) {
        const int x = cell_axis(a.x, g.inv_h, g.nc[0]);
        const int y = cell_axis(a.y, g.inv_h, g.nc[1]) + lane % 3 - 1;
        const int z = cell_axis(a.z, g.inv_h, g.nc[2]) + lane / 3 - 1;
        if (y >= 0 && y < g.nc[1] && z >= 0 && z < g.nc[2]) {
            const int64_t row = S.cellbase + (int64_t)g.nc[0] * (y + (int64_t)g.nc[1] * z);
            from = start[row + max(x - 1, 0)];
            len = start[row + min(x + 1, g.nc[0] - 1) + 1] - from;
        }
    }
    int upto = len;   // entries up to and including this lane's row
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
        const int v = __shfl_up_sync(all, upto, o);
        if (lane >= o) upto += v;
    }
    const int total = __shfl_sync(all, upto, 8);
    const int shift = from - (upto - len);   // entry number to list index
    volatile uint8_t *st = list_status;
    auto settle = [&](uint8_t state) {
        if (lane == 0) {
            st[mine] = state;
            status[p] = state;
        }
    };
    bool rejected = false, full = false;   // full: more open neighbours than the lane keeps
    uint32_t q0 = NONE, q1 = NONE;         // places of open neighbours
    auto scan = [&]() {
        q0 = q1 = NONE;
        full = false;
        for (int base = 0; base < total; base += 32) {
            const int e = base + lane;
            int row = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) row += e >= __shfl_sync(all, upto, i) ? 1 : 0;
            const int j = e + __shfl_sync(all, shift, row);
            if (e < total) {
                const uint32_t q = list[j];
                const float4 b = list_pos[j];
                const uint8_t sq = st[j];
                if ((int64_t)q < p) {           // only higher priority
                    const float ex = a.x - b.x, ey = a.y - b.y, ez = a.z - b.z;
                    const float dist = sqrtf(ex * ex + ey * ey + ez * ez);
                    if (dist < rho * fmaxf(a.w, b.w)) {
                        if (sq == ACCEPTED) rejected = true;
                        if (sq == UNDECIDED) {
                            if (q0 == NONE) q0 = (uint32_t)j;
                            else if (q1 == NONE) q1 = (uint32_t)j;
                            else full = true;
                        }
                    }
                }
            }
            if (__any_sync(all, rejected)) return;
        }
    };
    scan();
    for (int look = 0; look < LOOKS; ++look) {
        if (__any_sync(all, rejected)) {
            settle(REJECTED);
            return;
        }
        if (!__any_sync(all, q0 != NONE || q1 != NONE)) {
            settle(ACCEPTED);
            return;
        }
        __nanosleep(100);
        if (__any_sync(all, full)) {
            scan();
            continue;
        }
        if (q0 != NONE) {
            const uint8_t sq = st[q0];
            if (sq == ACCEPTED) rejected = true;
            if (sq != UNDECIDED) q0 = NONE;
        }
        if (q1 != NONE) {
            const uint8_t sq = st[q1];
            if (sq == ACCEPTED) rejected = true;
            if (sq != UNDECIDED) q1 = NONE;
        }
    }
    if (lane == 0) atomicAdd(&cnt[(int64_t)s * CNT_N + CNT_OPEN], 1);
}

struct IsAccepted {
    const uint8_t *status;
    __device__ __forceinline__ bool operator()(int32_t p) const { return status[p] == ACCEPTED; }
};

__device__ __forceinline__ int64_t lower_bound_i32(const int32_t *a, int64_t n, int64_t key)
{
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int64_t)a[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Where each set's accepted survivors start in the accepted list (which is in
// batch order) and how many there are; *m is the list's length.
__global__ void accepted_ranges_kernel(const LocSet *sets, int nsets, const int32_t *acc, const int32_t *m,
                                       int32_t *cnt)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < nsets; s += gridDim.x * blockDim.x) {
        const int64_t b = s == 0 ? 0 : lower_bound_i32(acc, *m, sets[s].sbase);
        const int64_t e = s == nsets - 1 ? *m : lower_bound_i32(acc, *m, sets[s].sbase + sets[s].n);
        cnt[s * CNT_N + CNT_ABASE] = (int32_t)b;
        cnt[s * CNT_N + CNT_ACC] = (int32_t)(e - b);
    }
}

__device__ __forceinline__ ac_cell make_cell(const LocSet &S, float4 q, int64_t k)
{
    ac_cell c;
    c.c[0] = q.x;
    c.c[1] = q.y;
    c.c[2] = q.z;
    c.r = S.rho * q.w;
    c.E = S.state[4 * S.C + k];
    c.id = (int32_t)k;
    return c;
}

// the accepted contours as cells, in the order of the accepted list
__global__ void cells_kernel(const LocSet *sets, int nsets, const float4 *pos, const int32_t *order,
                             const int32_t *acc, const int32_t *m, ac_cell *out)
{
    const int64_t lim = *m;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < lim; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = acc[i];
        const LocSet &S = sets[set_of<&LocSet::sbase>(sets, nsets, p)];
        out[i] = make_cell(S, pos[p], order[p] - S.cbase);
    }
}

// One small set: the cells in acceptance order and their count
__global__ void __launch_bounds__(SMALL_THREADS) collect_small_kernel(const LocSet *set, const float4 *pos,
                                                                      const int32_t *order, int n,
                                                                      const uint8_t *status, int32_t *cnt, ac_cell *out)
{
    __shared__ uint32_t warp_sums[32];
    uint32_t m = 0;
    for (int p0 = 0; p0 < n; p0 += SMALL_THREADS) {
        const int p = p0 + threadIdx.x;
        const bool keep = p < n && status[p] == ACCEPTED;
        uint32_t tile;
        const uint32_t at = m + block_exclusive(keep ? 1u : 0u, warp_sums, &tile);
        if (keep) out[at] = make_cell(*set, pos[p], order[p]);
        m += tile;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        cnt[CNT_ACC] = (int32_t)m;
        cnt[CNT_N + 1] = (int32_t)m;
    }
}

unsigned blocks_for(int64_t n)
{
    int64_t b = (n + 255) / 256;
    return (unsigned)(b < 1 ? 1 : (b > 65536 ? 65536 : b));
}

int bits_for(uint64_t v)   // smallest b >= 1 with v < 2^b
{
    int b = 1;
    while (b < 64 && (v >> b) != 0) ++b;
    return b;
}

}  // namespace

ac_status localize_many(ac_contours *const *sets, const float *E0, ac_cell *const *out_host, const int64_t *cap,
                        int64_t *n_out, int nsets, cudaStream_t st)
{
    if (nsets <= 0) return AC_OK;
    if (nsets > 65535) LC_FAIL(AC_ERR_ARG, "ac_localize: at most 65535 sets per call");
    Scratch &sc = sets[0]->scratch;   // holds the batch's buffers
    std::vector<LocSet> L((size_t)nsets);
    int64_t total = 0, maxC = 0;
    for (int s = 0; s < nsets; ++s) {
        n_out[s] = 0;
        LocSet &S = L[(size_t)s];
        S.state = sets[s]->state;
        S.status = sets[s]->status;
        S.C = sets[s]->C;
        S.cbase = total;
        S.E0 = E0[s];
        S.rho = sets[s]->vol->ndim == 3 ? 0.79370052598409973738f : 0.70710678118654752440f;
        total += S.C;
        maxC = std::max(maxC, S.C);
    }
    if (total >= ((int64_t)1 << 31)) LC_FAIL(AC_ERR_ARG, "ac_localize: more than 2^31 - 1 contours in one call");
    const size_t cnt_ints = (size_t)nsets * CNT_N + 2;
    LC_CUDA(sc.lsets.ensure(sizeof(LocSet) * nsets));
    LC_CUDA(sc.hsets.ensure(sizeof(LocSet) * nsets));
    LC_CUDA(sc.counters.ensure(sizeof(int32_t) * cnt_ints));
    LC_CUDA(sc.hcount.ensure(sizeof(int32_t) * cnt_ints));
    LocSet *dsets = sc.lsets.as<LocSet>();
    int32_t *cnt = sc.counters.as<int32_t>();
    int32_t *h = sc.hcount.as<int32_t>();
    int32_t *tot = cnt + (size_t)nsets * CNT_N;   // [0] survivors, [1] accepted

    // 1. the cull over every set's contours: flags, per-set counts and largest
    //    radius, the survivors by batch index, and the status words
    std::memcpy(sc.hsets.p, L.data(), sizeof(LocSet) * nsets);
    LC_CUDA(cudaMemcpyAsync(dsets, sc.hsets.p, sizeof(LocSet) * nsets, cudaMemcpyHostToDevice, st));
    const bool small = nsets == 1 && total <= SMALL_CONTOURS;
    if (small) {
        LC_CUDA(sc.surv.ensure(sizeof(int32_t) * total));
        LC_CUDA(sc.ekeys.ensure(sizeof(uint64_t) * 2 * total));
        cull_small_kernel<<<1, SMALL_THREADS, 0, st>>>(dsets, cnt, sc.surv.as<int32_t>(), sc.ekeys.as<uint64_t>());
        count_launch();
        LC_CUDA(cudaGetLastError());
    } else {
        LC_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * cnt_ints, st));
        LC_CUDA(sc.flags.ensure(total));
        const unsigned bx = (unsigned)std::max<int64_t>(1, std::min<int64_t>((maxC + 255) / 256, 1216));
        flag_kernel<<<dim3(bx, (unsigned)nsets), 256, 0, st>>>(dsets, sc.flags.as<uint8_t>(), cnt);
        count_launch();
        LC_CUDA(cudaGetLastError());
        if (total > 0) {
            LC_CUDA(sc.surv.ensure(sizeof(int32_t) * total));
            thrust::counting_iterator<int32_t> iota(0);
            size_t tmp = 0;
            LC_CUDA(cub::DeviceSelect::Flagged(nullptr, tmp, iota, sc.flags.as<uint8_t>(), sc.surv.as<int32_t>(), tot,
                                               (int)total, st));
            LC_CUDA(sc.cub.ensure(tmp));
            LC_CUDA(cub::DeviceSelect::Flagged(sc.cub.p, tmp, iota, sc.flags.as<uint8_t>(), sc.surv.as<int32_t>(), tot,
                                               (int)total, st));
        }
    }
    LC_CUDA(cudaMemcpyAsync(h, cnt, sizeof(int32_t) * cnt_ints, cudaMemcpyDeviceToHost, st));
    LC_CUDA(cudaStreamSynchronize(st));
    for (int s = 0; s < nsets; ++s) {
        const ac_status e = status_error(h[s * CNT_N + CNT_STATUS]);
        if (e != AC_OK) return e;
    }

    // 2. per set: survivors, the grid (cell size rho max R) and the offsets
    int64_t n = 0, ncells = 0, n_max = 0;
    for (int s = 0; s < nsets; ++s) {
        LocSet &S = L[(size_t)s];
        const ac_volume *v = sets[s]->vol;
        S.sbase = n;
        S.n = h[s * CNT_N + CNT_SURV];
        n += S.n;
        n_max = std::max(n_max, S.n);
        float maxR;
        std::memcpy(&maxR, &h[s * CNT_N + CNT_MAXR], sizeof(float));
        double hc = (double)S.rho * (double)maxR * 1.0001;
        if (!(hc > 0.0)) hc = 1.0;
        int64_t nc = 1;
        for (int pass = 0; pass < 64; ++pass) {
            nc = 1;
            for (int d = 0; d < 3; ++d) {
                const double top = d < v->ndim ? (double)(v->n[d] - 1) * v->sp[d] : 0.0;
                S.g.nc[d] = (int)std::floor(top / hc) + 1;
                nc *= S.g.nc[d];
            }
            if (nc <= ((int64_t)1 << 26)) break;
            hc *= 2.0;
        }
        S.g.inv_h = (float)(1.0 / hc);
        S.cellbase = ncells;
        ncells += S.n > 0 ? nc : 0;
    }
    if (total > 0 && n != h[(size_t)nsets * CNT_N]) LC_FAIL(AC_ERR_CUDA, "ac_localize: survivor counts disagree");
    if (n == 0) return AC_OK;
    if (ncells >= ((int64_t)1 << 31)) LC_FAIL(AC_ERR_OOM, "ac_localize: neighbour grids too large for one call");

    // 3. priority order by (set, E, k), positions, the grids' cells sorted
    std::memcpy(sc.hsets.p, L.data(), sizeof(LocSet) * nsets);
    LC_CUDA(cudaMemcpyAsync(dsets, sc.hsets.p, sizeof(LocSet) * nsets, cudaMemcpyHostToDevice, st));
    LC_CUDA(sc.ekeys.ensure(sizeof(uint64_t) * 2 * n));
    LC_CUDA(sc.surv_sorted.ensure(sizeof(int32_t) * n));
    uint64_t *ek = sc.ekeys.as<uint64_t>();
    int32_t *order = sc.surv_sorted.as<int32_t>();
    if (!small) {
        key_kernel<<<blocks_for(n), 256, 0, st>>>(dsets, nsets, sc.surv.as<int32_t>(), n, ek);
        count_launch();
        LC_CUDA(cudaGetLastError());
    }
    const int key_bits = nsets > 1 ? 32 + bits_for((uint64_t)(nsets - 1)) : 32;   // one set: the energy bits only
    size_t tmp = 0;
    LC_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, tmp, ek, ek + n, sc.surv.as<int32_t>(), order, (int)n, 0,
                                            key_bits, st));
    LC_CUDA(sc.cub.ensure(tmp));
    LC_CUDA(cub::DeviceRadixSort::SortPairs(sc.cub.p, tmp, ek, ek + n, sc.surv.as<int32_t>(), order, (int)n, 0,
                                            key_bits, st));
    LC_CUDA(sc.stat.ensure(2 * n));
    LC_CUDA(sc.pos.ensure(sizeof(float4) * n));
    LC_CUDA(sc.list_pos.ensure(sizeof(float4) * n));
    LC_CUDA(sc.cellk.ensure(sizeof(uint32_t) * n));
    LC_CUDA(sc.celli.ensure(sizeof(uint32_t) * n));
    LC_CUDA(sc.list.ensure(sizeof(uint32_t) * n));
    LC_CUDA(sc.cell_start.ensure(sizeof(int32_t) * (ncells + 1)));
    float4 *pos = sc.pos.as<float4>();
    int32_t *start = sc.cell_start.as<int32_t>();
    LC_CUDA(cudaMemsetAsync(start, 0, sizeof(int32_t) * (ncells + 1), st));
    cell_count_kernel<<<blocks_for(n), 256, 0, st>>>(dsets, nsets, order, n, pos, sc.cellk.as<uint32_t>(),
                                                     sc.celli.as<uint32_t>(), start, sc.stat.as<uint8_t>());
    count_launch();
    LC_CUDA(cudaGetLastError());
    const uint32_t n_starts = (uint32_t)(ncells + 1);   // up to 2^31: not an int
    tmp = 0;
    LC_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tmp, start, start, n_starts, st));
    LC_CUDA(sc.cub.ensure(tmp));
    LC_CUDA(cub::DeviceScan::ExclusiveSum(sc.cub.p, tmp, start, start, n_starts, st));
    cell_scatter_kernel<<<blocks_for(n), 256, 0, st>>>(n, sc.cellk.as<uint32_t>(), sc.celli.as<uint32_t>(), start, pos,
                                                       sc.list.as<uint32_t>(), sc.list_pos.as<float4>(),
                                                       sc.stat.as<uint8_t>() + n);
    count_launch();
    LC_CUDA(cudaGetLastError());

    // 4. rounds until every survivor is decided.  Each round decides at least the
    //    undecided survivor of highest priority of every set, so the largest set's
    //    n rounds settle all; the bound (that n + 8 unless a test lowers it) is
    //    checked between rounds.  After each round the kept survivors are collected in
    //    batch (= per set, acceptance) order, with each set's range of them, on the
    //    assumption that it was the last; few cells are copied back with the counts.
    LC_CUDA(sc.acc.ensure(sizeof(int32_t) * n));
    LC_CUDA(sc.cells.ensure(sizeof(ac_cell) * n));
    LC_CUDA(sc.hcells.ensure(sizeof(ac_cell) * n));
    uint8_t *status = sc.stat.as<uint8_t>();
    int32_t *acc = sc.acc.as<int32_t>();
    thrust::counting_iterator<int32_t> iota(0);
    const IsAccepted accepted{status};
    tmp = 0;
    LC_CUDA(cub::DeviceSelect::If(nullptr, tmp, iota, acc, tot + 1, (int)n, accepted, st));
    LC_CUDA(sc.cub.ensure(tmp));
    const int64_t max_rounds = localize_round_limit(n_max);
    // blocks of the sets' heads: the largest set whole if at most three in four blocks then
    // have nothing to do; none where the GPU holds nearly all survivors at once anyway (8 sets
    // of 2,000 among 40: 40 us set after set, 50 us in turn)
    const int64_t in_order = (n + ROUND_WARPS - 1) / ROUND_WARPS, largest = (n_max + ROUND_WARPS - 1) / ROUND_WARPS;
    const int64_t heads = nsets > 1 && n > 2 * RESIDENT_WARPS ? std::min(largest, 4 * in_order / nsets) : 0;
    const unsigned round_blocks = (unsigned)(heads * nsets + (heads < largest ? in_order : 0));
    const bool few = n <= 16384;   // 400 KB of cells: less than another synchronisation costs
    int64_t rounds = 0;
    for (bool open = true; open; ++rounds) {
        if (rounds >= max_rounds) {
            const int32_t bit = STATUS_LOCALIZE_LIMIT;
            for (int s = 0; s < nsets; ++s)
                if (L[(size_t)s].n > 0 && (rounds == 0 || h[s * CNT_N + CNT_OPEN] > 0))
                    LC_CUDA(cudaMemcpyAsync(sets[s]->status, &bit, sizeof(bit), cudaMemcpyHostToDevice, st));
            LC_CUDA(cudaStreamSynchronize(st));
            LC_FAIL(AC_ERR_TIMEOUT, "ac_localize: competition did not settle within its round bound");
        }
        if (rounds > 0)
            LC_CUDA(cudaMemset2DAsync(cnt + CNT_OPEN, sizeof(int32_t) * CNT_N, 0, sizeof(int32_t), nsets, st));
        round_kernel<<<round_blocks, 32 * ROUND_WARPS, 0, st>>>(dsets, nsets, pos, n, start, sc.list.as<uint32_t>(),
                                                                sc.list_pos.as<float4>(), sc.celli.as<uint32_t>(),
                                                                status + n, status, cnt, (unsigned)heads);
        count_launch();
        LC_CUDA(cudaGetLastError());
        if (small) {
            collect_small_kernel<<<1, SMALL_THREADS, 0, st>>>(dsets, pos, order, (int)n, status, cnt,
                                                              sc.cells.as<ac_cell>());
            count_launch();
            LC_CUDA(cudaGetLastError());
        } else {
            LC_CUDA(cub::DeviceSelect::If(sc.cub.p, tmp, iota, acc, tot + 1, (int)n, accepted, st));
            accepted_ranges_kernel<<<blocks_for(nsets), 256, 0, st>>>(dsets, nsets, acc, tot + 1, cnt);
            count_launch();
            LC_CUDA(cudaGetLastError());
            cells_kernel<<<blocks_for(n), 256, 0, st>>>(dsets, nsets, pos, order, acc, tot + 1, sc.cells.as<ac_cell>());
            count_launch();
            LC_CUDA(cudaGetLastError());
        }
        LC_CUDA(cudaMemcpyAsync(h, cnt, sizeof(int32_t) * cnt_ints, cudaMemcpyDeviceToHost, st));
        if (few)
            LC_CUDA(cudaMemcpyAsync(sc.hcells.p, sc.cells.p, sizeof(ac_cell) * n, cudaMemcpyDeviceToHost, st));
        LC_CUDA(cudaStreamSynchronize(st));
        open = false;
        for (int s = 0; s < nsets; ++s) open = open || h[s * CNT_N + CNT_OPEN] > 0;
    }

    // 5. the cells, contiguous, set by set
    const int64_t M = h[(size_t)nsets * CNT_N + 1];
    if (M > 0 && !few) {
        LC_CUDA(cudaMemcpyAsync(sc.hcells.p, sc.cells.p, sizeof(ac_cell) * M, cudaMemcpyDeviceToHost, st));
        LC_CUDA(cudaStreamSynchronize(st));
    }
    const ac_cell *cells = sc.hcells.as<ac_cell>();
    for (int s = 0; s < nsets; ++s) {
        const int64_t m = h[s * CNT_N + CNT_ACC];
        n_out[s] = m;
        const int64_t k = std::min(m, cap[s]);
        if (k > 0) std::memcpy(out_host[s], cells + h[s * CNT_N + CNT_ABASE], sizeof(ac_cell) * (size_t)k);
    }
    return AC_OK;
}

}  // namespace ac
