// ac_grid.cu -- the voxel-grid form of Eq. 5 (the paper's integration before it
// moved to Monte-Carlo sampling): the sums of Eqs. 5 and 7-10 run over every
// voxel centre inside the ball of radius R + dR/2, each weighted by one voxel
// volume, instead of over N random samples.  No interpolation and no random
// numbers; the image beyond the volume is clamp-to-edge, as for the samples.
//
// One group of G lanes per contour keeps the state in registers for every
// iteration of its window.  The group walks the rows of the ball's bounding box
// (y, z), skips rows that miss the ball, and its lanes take consecutive voxels of
// a row's chord, so a row is read with neighbouring addresses.  Gathers go
// through the read-only cache from global memory.
//
// Bound by instruction issue (1024^2 u8: 76 % of the slots; 256x250x64 u16: 80 %).  With a
// voxel after the other, sqrtf and the division (76 and 72 %), 10 iterations took 2.11e8
// and 1.31e9 warp instructions; in 3D a row whose chord ends between a lane's two voxels
// ran once for the lanes with both and once for the others.  Now the two voxels of a step
// share packed instructions, the reciprocal root serves both root and quotient, and a lane
// without a second voxel adds its first in the same instructions: 1.14e8 and 9.47e8, the
// kernel 263 -> 133 us and 1720 -> 1022 us.
#include "ac_evolve.cuh"
#include "ac_host.h"

namespace ac {
namespace {

// Whether the voxel nearest to c lies off it, but nearer than the root of ROOT_MIN (a little
// more, for rounding)
template <int DIM> __device__ __forceinline__ bool near_centre(const VolDesc &V, const float *c)
{
    float d2 = 0.0f, least = 0.0f;
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        const float off = fabsf(fmaf(rintf(c[d] * V.inv_sp[d]), V.sp[d], -c[d]));
        d2 = fmaf(off, off, d2);
        least = fmaxf(least, off);
    }
    return least > 0.0f && d2 < 4.0f * ROOT_MIN;
}

// Whether the roots and quotients of an evaluation with centre c and radius R are Newton
// steps.  Voxels nearer to the centre than the root of ROOT_MIN (but not on it) have a root that
// is only near enough: they must lie inside both bands, where the root plays no part, or not
// be there (none but the nearest can).  Squared distances, also of the
// voxel beside a chord's last, squared half chords (zero, or at least 2^-48 of the squared
// radius in 2D, where the difference is fused, 2^-25 in 3D) and (integer voxels) k I stay
// within the ranges of sqrt2 and div2.  What remains (radii below 1e-7 in 2D and 3e-11 in 3D,
// spacings above 3e7) takes the operations for any operand.
template <int DIM>
__device__ __forceinline__ bool newton_range(const EvolveArgs &a, const VolDesc &V, const float *c, float R)
{
    constexpr float NEAR = 7.105427357601002e-15f;   // 2^-47
    const float Ro = R + 0.5f * a.dR, Ro2 = __fmul_rn(Ro, Ro);
    const float kmin = fminf(fabsf(a.kr1), fabsf(a.kr2)), kmax = fmaxf(fabsf(a.kr1), fabsf(a.kr2));
    return Ro2 > (DIM == 2 ? 1.4210854715202004e-14f : 8.470329472543003e-22f) &&   // 2^-46, 2^-70
           Ro2 < 1.125899906842624e15f && V.sp[0] < 33554432.0f &&                  // 2^50, 2^25
           kmin > 9.094947017729282e-13f && kmax < 1.099511627776e12f &&            // 2^-40, 2^40
           ((fmaf(-a.rho * R + NEAR, a.inv_dr, 0.5f) < -0.001f && fmaf(NEAR - R, a.inv_dR, 0.5f) < -0.001f) ||
            !near_centre<DIM>(V, c));
}

// Whether div2 was right for all numerators of a ball, known after it (`s`: the evaluation).
// Integer voxels cannot leave its range.  binary16: none infinite or NaN, which leave no
// finite energy.  float: by the largest numerator.  (Numerators below QUOTIENT_MIN have an
// error in their last place: 2^-48 of the largest one is where the compensated sums end, so
// that one has to be 2^24 above.)
template <typename T> struct Numerators {
    __device__ __forceinline__ void add(float2) {}
    template <int G> __device__ __forceinline__ bool fine(const Step &, unsigned) const { return true; }
};
template <> struct Numerators<__half> {
    __device__ __forceinline__ void add(float2) {}
    template <int G> __device__ __forceinline__ bool fine(const Step &s, unsigned) const { return isfinite(s.E); }
};
template <> struct Numerators<float> {
    float top = 0.0f;
    __device__ __forceinline__ void add(float2 n) { top = max3_abs(top, n.x, n.y); }
    template <int G> __device__ __forceinline__ bool fine(const Step &, unsigned mask) const
    {
        uint32_t t = __float_as_uint(top);
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) t = max(t, __shfl_xor_sync(mask, t, o));
        return t == 0 || (t >= __float_as_uint(QUOTIENT_MIN * 16777216.0f) && t <= __float_as_uint(QUOTIENT_MAX));
    }
};

template <int DIM, typename T, int G, bool COMP, bool NEWTON>
__device__ __forceinline__ Step eval_grid(const VolDesc &V, const EvolveArgs &a, const float *c, float R, int lig,
                                          unsigned mask, Numerators<T> &numerators)
{
    const float Ro = R + 0.5f * a.dR;
    const float Ro2 = __fmul_rn(Ro, Ro);
    int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
        lo[d] = (int)ceilf((c[d] - Ro) * V.inv_sp[d]);
        hi[d] = (int)floorf((c[d] + Ro) * V.inv_sp[d]);
    }
    const float B1 = fmaf(-a.rho * R, a.inv_dr, 0.5f);   // inner band coordinate: r / dr + B1
    const float B2 = fmaf(-R, a.inv_dR, 0.5f);           // outer band coordinate: r / dR + B2
    const T *data = reinterpret_cast<const T *>(V.data);
    const int64_t nvox = V.pitch_z * V.n[2];   // extent for the checked build
    KSum acc[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
    for (int kz = lo[2]; kz <= hi[2]; ++kz) {
        const float dz = DIM == 3 ? fmaf((float)kz, V.sp[2], -c[2]) : 0.0f;
        const int zz = DIM == 3 ? min(max(kz, 0), V.n[2] - 1) : 0;
        for (int jy = lo[1]; jy <= hi[1]; ++jy) {
            const float dy = fmaf((float)jy, V.sp[1], -c[1]);
            const float q = __fmaf_rn(dy, dy, __fmul_rn(dz, dz));
            // fused in 2D, not in 3D: decides which voxels a chord ends on
            const float rem = DIM == 2 ? __fmaf_rn(Ro, Ro, -q) : __fsub_rn(Ro2, q);
            if (rem < 0.0f) continue;   // the row misses the ball (same for the whole group)
            const float chord = NEWTON ? sqrt1(rem) : sqrtf(rem);
            const int i0 = (int)ceilf((c[0] - chord) * V.inv_sp[0]);
            const int i1 = (int)floorf((c[0] + chord) * V.inv_sp[0]);
            const int yy = min(max(jy, 0), V.n[1] - 1);
            const int64_t row = (int64_t)zz * V.pitch_z + (int64_t)yy * V.pitch_y;
            // Two voxels of the row per step (ix and ix + G), side by side in packed
            // instructions: two independent chains of work per lane, and the products are
            // summed in one rounding before the compensated addition.  In 2D a second voxel
            // beyond the chord adds zero; in 3D, whose rows are shorter, the first is then
            // added alone, in the same instructions.
            for (int ix = i0 + lig; ix <= i1; ix += 2 * G) {
                const bool two = ix + G <= i1;
                const float fx = (float)ix;
                const float2 dx = fma2(make_float2(fx, fx + (float)G), dup2(V.sp[0]), dup2(-c[0]));
                const float Iv = ldg_f<T>(data + checked(row + min(max(ix, 0), V.n[0] - 1), nvox, V.status));
                const float Iw = two ? ldg_f<T>(data + checked(row + min(max(ix + G, 0), V.n[0] - 1), nvox, V.status))
                                     : 0.0f;
                const float2 d2 = fma2(dx, dx, dup2(q));
                float2 rs;
                const float2 r = NEWTON ? sqrt2(d2, rs) : make_float2(sqrtf(d2.x), sqrtf(d2.y));
                const float2 t1 = fma2(r, dup2(a.inv_dr), dup2(B1)), t2 = fma2(r, dup2(a.inv_dR), dup2(B2));
                const float2 s1 = make_float2(__saturatef(t1.x), __saturatef(t1.y));
                const float2 s2 = make_float2(__saturatef(t2.x), __saturatef(t2.y));
                const float2 S = sub2(fma2(dup2(2.0f), s1, dup2(-1.0f)), s2);
                // voxel inside the inner / outer band
                const bool v1 = s1.x == t1.x, v2 = s2.x == t2.x, w1 = s1.y == t1.y, w2 = s2.y == t2.y;
                const float2 dSdR = add2(make_float2(v1 ? a.kR1 : 0.0f, w1 ? a.kR1 : 0.0f),
                                         make_float2(v2 ? a.kR2 : 0.0f, w2 ? a.kR2 : 0.0f));
                // -S'(r) I / r, for the direction (x - c) / r (zero for a voxel on the centre)
                const float2 k = add2(make_float2(v1 ? a.kr1 : 0.0f, w1 ? a.kr1 : 0.0f),
                                      make_float2(v2 ? a.kr2 : 0.0f, w2 ? a.kr2 : 0.0f));
                const float2 kI = make_float2(__fmul_rn(k.x, Iv), __fmul_rn(k.y, Iw));
                float2 g;
                if constexpr (!NEWTON)
                    g = make_float2(d2.x > 0.0f ? kI.x / r.x : 0.0f, d2.y > 0.0f ? kI.y / r.y : 0.0f);
                else
                    g = div2(kI, r, rs);
                if (NEWTON) numerators.add(kI);
                const float gv = g.x, gw = g.y;
                const float fv[5] = {S.x, dSdR.x, gv, gv, gv}, xv[5] = {Iv, Iv, dx.x, dy, dz};
                const float fw[5] = {S.y, dSdR.y, gw, gw, gw}, xw[5] = {Iw, Iw, dx.y, dy, dz};
                // which voxel's product is fused with the sum of the two
                constexpr bool w_first[5] = {true, false, true, false, false};
#pragma unroll
                for (int m = 0; m < (DIM == 3 ? 5 : 4); ++m) {
                    const bool alone = DIM == 3 && !two;
                    const float w = w_first[m] ? __fmul_rn(fv[m], xv[m]) : __fmul_rn(fw[m], xw[m]);
                    const float ff = w_first[m] && !alone ? fw[m] : fv[m], fi = w_first[m] && !alone ? xw[m] : xv[m];
                    if (COMP) {
                        float y = __fmaf_rn(ff, fi, alone ? -acc[m].c : w);
                        if (!alone) y = y - acc[m].c;
                        const float t = acc[m].s + y;
                        acc[m].c = (t - acc[m].s) - y;
                        acc[m].s = t;
                    } else {
                        const float y = __fmaf_rn(ff, fi, alone ? acc[m].s : w);
                        acc[m].s = alone ? y : acc[m].s + y;
                    }
                }
            }
        }
    }
    float sums[5];
    sums[4] = 0.0f;
    group_reduce_all<G, COMP, DIM == 3 ? 5 : 4>(acc, sums, mask);
    // Eqs. 5-11 in centre/radius form with the voxel volume as the measure
    float vox = V.sp[0] * V.sp[1];
    if (DIM == 3) vox *= V.sp[2];
    const float w = vox * V.scale;
    const float inv2R = __frcp_rn(2.0f * R);
    const float inv = DIM == 3 ? inv2R * inv2R * inv2R : inv2R * inv2R;   // (2R)^-d
    Step s;
    const float J = sums[0] * w;
    s.E = J * inv;
    s.dEdR = (sums[1] * w - (float)DIM * 2.0f * J * inv2R) * inv;
    s.g[0] = sums[2] * w * inv;
    s.g[1] = sums[3] * w * inv;
    s.g[2] = DIM == 3 ? sums[4] * w * inv : 0.0f;
    return s;
}

// Iterations n, n + 1, ... of a contour in registers, to the last of its window or until it
// stops (returns last_iter + 1), or (NEWTON) until one that is beyond the Newton steps
// (returns its number, nothing done).
template <int DIM, typename T, int G, bool COMP, bool NEWTON>
__device__ __forceinline__ int run_grid(const VolDesc &V, const EvolveArgs &a, int v, int64_t k, int n, int lig, unsigned mask,
                                        float *c, float &R, int32_t &h, Step &s, unsigned int &evals)
{
    for (; n <= V.last_iter; ++n) {
        // bounded work per evaluation: a radius beyond the grid bound (possible
        // only through an explicitly set state) stops the contour with a status
        const float Ro = R + 0.5f * a.dR;
        bool wide = false;
#pragma unroll
        for (int d = 0; d < DIM; ++d) wide = wide || !(Ro * V.inv_sp[d] <= GRID_MAX_RADIUS_VOXELS);
        if (wide) {
            if (lig == 0) atomicOr(V.status, STATUS_GRID_RANGE);
            s.E = V.state[4 * V.C + k];
            break;
        }
        if (NEWTON && !newton_range<DIM>(a, V, c, R)) return n;
        Numerators<T> numerators;
        const Step t = eval_grid<DIM, T, G, COMP, NEWTON>(V, a, c, R, lig, mask, numerators);
        if (NEWTON && !numerators.template fine<G>(t, mask)) return n;
        s = t;
        ++evals;
        if (lig == 0) write_trace(a, v, k, n, c, R, s);
        if (!finite_step(s)) {
            if (lig == 0) atomicOr(V.status, STATUS_NONFINITE);
            break;
        }
        if (step_or_stop<DIM>(s, n, a, V, c, R, h)) break;
    }
    return V.last_iter + 1;
}

template <int DIM, typename T, int G, bool COMP>
__global__ void __maxnreg__(80) evolve_grid_kernel(const __grid_constant__ EvolveArgs a)
{
    unsigned int evals = 0;
    const int lig = threadIdx.x % G;
    const unsigned mask = group_mask<G>();
    const int64_t groups = (int64_t)gridDim.x * (blockDim.x / G);
    for (int64_t gi = (int64_t)blockIdx.x * (blockDim.x / G) + threadIdx.x / G; gi < a.total_contours; gi += groups) {
        const int v = find_set(a.vols, a.n_vols, gi);
        const VolDesc &V = a.vols[v];
        if (V.first_iter > V.last_iter) continue;   // no iterations for this set in this launch
        const int64_t k = gi - V.contour_base;
        const int64_t C = V.C;
        int32_t h = V.hold ? V.hold[k] : 0;
        if (h & HOLD_STOPPED) continue;
        float c[3] = {V.state[k], V.state[C + k], DIM == 3 ? V.state[2 * C + k] : 0.0f};
        float R = V.state[3 * C + k];
        Step s{0.0f, 0.0f, {0.0f, 0.0f, 0.0f}};
        const int n = run_grid<DIM, T, G, COMP, true>(V, a, v, k, V.first_iter, lig, mask, c, R, h, s, evals);
        if (n <= V.last_iter)   // the rest of its window in the general form
            run_grid<DIM, T, G, COMP, false>(V, a, v, k, n, lig, mask, c, R, h, s, evals);
        if (lig == 0) {
            V.state[k] = c[0];
            V.state[C + k] = c[1];
            if (DIM == 3) V.state[2 * C + k] = c[2];
            V.state[3 * C + k] = R;
            V.state[4 * C + k] = s.E;
            if (!(isfinite(s.E) && isfinite(R) && isfinite(c[0]) && isfinite(c[1]) && isfinite(c[2])))
                atomicOr(V.status, STATUS_NONFINITE);
            if (V.hold && rules_on(a)) V.hold[k] = h;
        }
    }
    // contour-iterations, counted once per group, one atomic per warp
    const unsigned int tot = __reduce_add_sync(0xffffffffu, lig == 0 ? evals : 0u);
    if ((threadIdx.x & 31) == 0 && tot) atomicAdd(&a.path_counts[2], (unsigned long long)tot);
}

template <int DIM, typename T, int G, bool COMP>
cudaError_t launch_grid_t(const EvolveArgs &a, int warps, int64_t grid, cudaStream_t st)
{
    evolve_grid_kernel<DIM, T, G, COMP><<<(unsigned)grid, warps * 32, 0, st>>>(a);
    return cudaGetLastError();
}

// 8 and 16 lanes, compensated and plain sums, 2D and 3D; 4 lanes in 2D (compensated).
template <typename T>
cudaError_t launch_grid_dtype(const EvolveArgs &a, int G, bool comp, int warps, int64_t grid, cudaStream_t st)
{
#define AC_GRID(DIM, GG, CC) \
    if (a.ndim == DIM && G == GG && comp == CC) return launch_grid_t<DIM, T, GG, CC>(a, warps, grid, st);
    AC_GRID(3, 8, true) AC_GRID(3, 16, true) AC_GRID(3, 8, false) AC_GRID(3, 16, false)
    AC_GRID(2, 8, true) AC_GRID(2, 16, true) AC_GRID(2, 8, false) AC_GRID(2, 16, false) AC_GRID(2, 4, true)
#undef AC_GRID
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_grid(ac_dtype t, const EvolveArgs &a, int G, bool comp, int warps, int64_t grid, cudaStream_t st)
{
    switch (t) {
    case AC_U8: return launch_grid_dtype<uint8_t>(a, G, comp, warps, grid, st);
    case AC_U16: return launch_grid_dtype<uint16_t>(a, G, comp, warps, grid, st);
    case AC_F16: return launch_grid_dtype<__half>(a, G, comp, warps, grid, st);
    default: return launch_grid_dtype<float>(a, G, comp, warps, grid, st);
    }
}

}  // namespace ac
