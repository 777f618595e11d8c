// tti_stencil.cuh -- first-derivative building blocks shared by the TTI
// kernels (two-pass, fused and recompute schemes): tap tables t[d + R] for
// offsets d = -R..R (centred, forward- or backward-staggered), float4 cells
// of four consecutive x points, and the z accumulator pipeline.
#pragma once

#include "common.cuh"
#include "f32x2.cuh"

namespace fdsweep {
namespace tti {

__device__ __forceinline__ float4 lds4(const float *p) {
    return *reinterpret_cast<const float4 *>(p);
}

// Stencil kinds: 0 centred (taps -R..R without the centre), +1 forward-
// staggered D+ (taps -R+1..R), -1 backward-staggered D- (taps -R..R-1).
template <int KIND>
__host__ __device__ constexpr bool tap_used(int d, int R) {
    return KIND == 0 ? d != 0 : (KIND > 0 ? d > -R : d < R);
}

// First derivative along x of 4 consecutive points from a row that starts RA
// points left of them: sum_d t[d + R] q[d].
template <int R, int RA, int KIND>
__device__ __forceinline__ float4 dx4(const float *row, const float *t) {
    float xs[2 * RA + 4];
#pragma unroll
    for (int i = 0; i < (2 * RA + 4) / 4; ++i) {
        const float4 f = lds4(row + 4 * i);
        xs[4 * i] = f.x;
        xs[4 * i + 1] = f.y;
        xs[4 * i + 2] = f.z;
        xs[4 * i + 3] = f.w;
    }
    float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = -R; k <= R; ++k) {
        if (!tap_used<KIND>(k, R)) continue;
        const float w = t[k + R];
        d.x = fmaf(w, xs[RA + 0 + k], d.x);
        d.y = fmaf(w, xs[RA + 1 + k], d.y);
        d.z = fmaf(w, xs[RA + 2 + k], d.z);
        d.w = fmaf(w, xs[RA + 3 + k], d.w);
    }
    return d;
}

// ---- cells of four points as two packed pairs
using f32x2::f2;
using f32x2::f2_add;
using f32x2::f2_fma;
using f32x2::f2_mul;
using f32x2::f2_pack;
using f32x2::f2_splat;
using f32x2::f2_sub;
using f32x2::lds_q4;
using f32x2::Q4;

__device__ __forceinline__ Q4 q4_fma(Q4 a, Q4 b, Q4 c) {
    return Q4{f2_fma(a.lo, b.lo, c.lo), f2_fma(a.hi, b.hi, c.hi)};
}
__device__ __forceinline__ Q4 q4_fma(f2 w, Q4 b, Q4 c) {
    return Q4{f2_fma(w, b.lo, c.lo), f2_fma(w, b.hi, c.hi)};
}
__device__ __forceinline__ Q4 q4_mul(Q4 a, Q4 b) {
    return Q4{f2_mul(a.lo, b.lo), f2_mul(a.hi, b.hi)};
}
__device__ __forceinline__ Q4 q4_add(Q4 a, Q4 b) {
    return Q4{f2_add(a.lo, b.lo), f2_add(a.hi, b.hi)};
}
__device__ __forceinline__ Q4 q4_sub(Q4 a, Q4 b) {
    return Q4{f2_sub(a.lo, b.lo), f2_sub(a.hi, b.hi)};
}
__device__ __forceinline__ Q4 q4_neg(Q4 a) {
    const f2 m1 = f2_splat(-1.f);
    return Q4{f2_mul(a.lo, m1), f2_mul(a.hi, m1)};
}
__device__ __forceinline__ Q4 q4_from(float4 v) { return Q4{f2_pack(v.x, v.y), f2_pack(v.z, v.w)}; }

// First derivative along y: `centre` points at the thread's four points in the
// centre row, rows `pitch` floats apart.
template <int R, int KIND>
__device__ __forceinline__ Q4 dy_q4(const float *centre, int pitch, const float *t) {
    Q4 d = Q4{0ull, 0ull};
#pragma unroll
    for (int k = -R; k <= R; ++k) {
        if (!tap_used<KIND>(k, R)) continue;
        d = q4_fma(f2_splat(t[k + R]), lds_q4(centre + k * pitch), d);
    }
    return d;
}
// z accumulator pipeline: acc[i] is output plane p-R+i when plane p arrives
// with values c (plane p is at offset R - i from it); acc[0] is then complete.
template <int R, int KIND>
__device__ __forceinline__ void dz_feed_q4(Q4 (&acc)[2 * R], Q4 c, const float *t) {
#pragma unroll
    for (int i = 0; i < 2 * R; ++i) {
        if (!tap_used<KIND>(R - i, R)) continue;
        acc[i] = q4_fma(f2_splat(t[2 * R - i]), c, acc[i]);
    }
}
// rotate: the new last entry is output p+R, for which plane p is offset -R
template <int R, int KIND>
__device__ __forceinline__ void dz_shift_q4(Q4 (&acc)[2 * R], Q4 c, const float *t) {
#pragma unroll
    for (int i = 0; i < 2 * R - 1; ++i) acc[i] = acc[i + 1];
    const f2 w = f2_splat(tap_used<KIND>(-R, R) ? t[0] : 0.f);
    acc[2 * R - 1] = Q4{f2_mul(w, c.lo), f2_mul(w, c.hi)};
}

// TMA tiled load of a 5-D box (several fields at once) into shared memory.
__device__ __forceinline__ void tma_load_5d(void *dst, const CUtensorMap *map, uint64_t *bar,
                                            int x, int y, int z, int v, int w) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(v), "r"(w),
        "r"(smem_u32(bar))
        : "memory");
}

}  // namespace tti
}  // namespace fdsweep
