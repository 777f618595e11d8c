// tti.cu -- K2a/K2b: one leapfrog step of the pseudo-acoustic TTI system.
//
// The rotated operators are built from central first derivatives D_i of
// radius R (section "Test case setup": two coupled acoustic equations whose
// Laplacians come from spatially rotated first-derivative operators):
//   Hz q = sum_i D_i(n_i (n . grad q)),   Hxy q = sum_i D_i D_i q - Hz q.
// Since D is linear, Hxy p = sum_i D_i f_i with f_i = D_i p - n_i (n . grad p)
// and Hz r = sum_i D_i e_i with e_i = n_i (n . grad r).  Only Hxy p and Hz r
// enter the update
//   m p_tt + damp p_t = a Hxy p + s Hz r,   m r_tt + damp r_t = s Hxy p + Hz r,
// (a = 1 + 2 eps, s = sqrt(1 + 2 delta)), so pass 1 (K2a) writes the six
// first-derivative temporaries f (of p) and e (of r), computed once per point
// and reused by every stencil point of pass 2 -- the shift-invariant reuse the
// paper's SIE pass performs -- and pass 2 (K2b) applies the second
// first-derivative and the centred damped leapfrog
//   q+ = q + (1 - zeta)(q - q-) + b * rhs_q,  b = dt^2/(m + damp dt/2),
//   zeta = damp * b / dt.
// Temporaries outside the grid are zero ghosts, like the fields.
//
// GB300 design (both passes, like the acoustic step): one CTA owns a BX x BY
// column and marches it through z.  The z-derivatives use an accumulator
// pipeline (2R pending outputs per point and field in registers, fed by the
// interior tile of each arriving plane); the x/y derivatives of the output
// plane s = p - R come from tiles staged with their halo.  Every operand
// arrives by cp.async.bulk.tensor, several fields per copy (three copies per
// plane in K2a, five in K2b), issued by a producer warp into a ring of stages
// with full/empty mbarriers.  A thread owns four x points of BOTH fields: it
// reads n (K2a) and b, a, s (K2b) once for the two, and K2b needs no exchange
// of Hxy p and Hz r between threads, so warps never meet at a barrier.  (With
// one thread group per field, one copy per field and tile and a consumer
// thread as the producer, a plane of both passes took 1.4 us for a lone CTA;
// see the launch tables for what this layout measures.)
//
// A time step is two launches, chained to each other: K2a's extra blocks
// record the receivers of p^n (or (p + r)/2), K2b's CTAs inject the sources
// into the nodes they own.
#include <string.h>

#include "kernels.cuh"
#include "receive.cuh"
#include "ring.cuh"
#include "runtime.cuh"
#include "tti_inject.cuh"
#include "tti_stencil.cuh"

namespace fdsweep {
namespace {
using namespace tti;

constexpr int round32(int n) { return (n + 31) / 32 * 32; }

template <int R, int TX, int TY, int D>
struct TtiCfg {
    static constexpr int BX = 4 * TX;
    static constexpr int BY = TY;
    static constexpr int RA = (R + 3) / 4 * 4;
    static constexpr int PW = BX + 2 * RA;       // x-halo width
    static constexpr int PH = BY + 2 * R;        // y-halo height
    static constexpr int NSL = D + 1;
    static constexpr int CONSUMERS = TX * TY;
    static constexpr int WARPS = CONSUMERS / 32;
    static constexpr int THREADS = CONSUMERS + 32;
    static constexpr int INT = BX * BY;
    static constexpr int HXY = PW * PH;  // x+y halo tile
    static constexpr int HX = PW * BY;   // x-halo tile
    static constexpr int HY = BX * PH;   // y-halo tile
    // pass 1 stage: [p | r](j) interiors, [p | r](s) xy-halo, [nx | ny | nz](s)
    static constexpr int OFF1_H = round32(2 * INT);
    static constexpr int OFF1_N = OFF1_H + round32(2 * HXY);
    static constexpr int STAGE1 = OFF1_N + round32(3 * INT);
    // pass 2 stage: [fz | ez](j), [fx | ex](s) x-halo, [fy | ey](s) y-halo,
    //               [p0 | p1 | r0 | r1](s) both levels, [b | a | s](s)
    static constexpr int OFF2_X = round32(2 * INT);
    static constexpr int OFF2_Y = OFF2_X + round32(2 * HX);
    static constexpr int OFF2_W = OFF2_Y + round32(2 * HY);
    static constexpr int OFF2_C = OFF2_W + round32(4 * INT);
    static constexpr int STAGE2 = OFF2_C + round32(3 * INT);
    static constexpr size_t SMEM1 = (size_t)NSL * STAGE1 * 4 + NSL * 16 + 16 + 128;
    static constexpr size_t SMEM2 = (size_t)NSL * STAGE2 * 4 + NSL * 16 + 16 + 128;
    static_assert(PW <= 256 && PH <= 256, "TMA box dimension limit");
    static_assert(CONSUMERS % 32 == 0, "whole consumer warps");
    static_assert(WARPS <= kMaxRingWarps, "room behind the abort flag");
};

struct Ring {
    float *smem;
    uint64_t *full, *empty;
    volatile int *abort_flag;
};

template <int NSL, int WARPS>
__device__ __forceinline__ Ring ring_init(unsigned char *raw, size_t stage_floats) {
    Ring r;
    r.smem = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(raw) + 127) &
                                       ~static_cast<uintptr_t>(127));
    r.full = reinterpret_cast<uint64_t *>(r.smem + NSL * stage_floats);
    r.empty = r.full + NSL;
    r.abort_flag = reinterpret_cast<volatile int *>(r.empty + NSL);
    if (threadIdx.x == 0) {
        for (int s = 0; s < NSL; ++s) {
            mbar_init(&r.full[s], 1);
            mbar_init(&r.empty[s], WARPS);
        }
        fence_mbar_init();
        init_ring_abort(r.abort_flag);
    }
    return r;
}

// The producer lane's loop: waits for each stage to be released by every
// consumer warp and fills it with fill(jj, stage, barrier) (which announces
// its bytes first).  Returns the number of stages issued.
template <int NSL, class Fill>
__device__ __forceinline__ int produce(const Ring &ring, size_t stage_floats, int nplanes,
                                       unsigned int *err, Fill fill) {
    int issued = 0;
    RingPos<NSL> pos;
    for (int jj = 0; jj < nplanes && !*ring.abort_flag; ++jj, pos.next()) {
        const int slot = pos.slot(jj);
        if (jj >= NSL && !mbar_wait_bounded(&ring.empty[slot], pos.phase(jj) ^ 1u)) {
            if (!*ring.abort_flag) atomicOr(err, DEV_ERR_TIMEOUT);
            *ring.abort_flag = 1;
            break;
        }
        fill(jj, ring.smem + slot * stage_floats, &ring.full[slot]);
        issued = jj + 1;
    }
    chain_trigger();  // the next launch may move in (see acoustic.cu)
    return issued;
}

// After an aborted column: the copies in flight get a bounded chance to land
// before the CTA's shared memory is released.
template <int NSL>
__device__ __forceinline__ void drain(const Ring &ring, int issued) {
    for (int jj = issued - NSL; jj < issued; ++jj)
        if (jj >= 0)
            mbar_wait_bounded(&ring.full[jj % NSL], (uint32_t)((jj / NSL) & 1), 200000000ull);
}

// ---------------------------------------------------------------- pass 1

template <int R, int TX, int TY, int D, int KIND, int U, int MINB>
__global__ void __launch_bounds__(TX *TY + 32, MINB)
    tti_pass1_kernel(const __grid_constant__ CUtensorMap map_wint,
                     const __grid_constant__ CUtensorMap map_whalo,
                     const __grid_constant__ CUtensorMap map_cint,
                     const __grid_constant__ TtiArgs a, const __grid_constant__ ReceiveArgs rec,
                     int zchunk, int nzc) {
    using C = TtiCfg<R, TX, TY, D>;
    if (blockIdx.z >= gridDim.z - rec.slices) {
        chain_trigger();
        chain_wait();
        if (!(__ldcg(a.err) & DEV_ERR_NONFINITE))
            record_receivers(&rec, a.wave, 4, a.cur, 2 + a.cur, &a.L);
        return;
    }
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Ring ring = ring_init<C::NSL, C::WARPS>(smem_raw, C::STAGE1);
    const int tid = threadIdx.x, lane = tid & 31;
    const int tx = tid % TX, ty = tid / TX;
    const int shot = blockIdx.z / nzc, chunk = blockIdx.z - shot * nzc;
    const int x0 = blockIdx.x * C::BX, y0 = blockIdx.y * C::BY;
    const int za = chunk * zchunk, zb = min(a.L.nz, za + zchunk);
    const int nplanes = zb - za + 2 * R;
    __syncthreads();
    chain_wait();
    if (__ldcg(a.err) & DEV_ERR_NONFINITE) return;  // stopped by the divergence watchdog

    int issued = 0;
    if (tid >= C::CONSUMERS) {
        if (lane == 0) {
            prefetch_tensormap(&map_wint);
            prefetch_tensormap(&map_whalo);
            prefetch_tensormap(&map_cint);
            issued = produce<C::NSL>(
                ring, C::STAGE1, nplanes, a.err, [&](int jj, float *st, uint64_t *full) {
                    const bool out = jj >= 2 * R;
                    mbar_arrive_expect_tx(
                        full, (2 * C::INT + (out ? 2 * C::HXY + 3 * C::INT : 0)) * 4);
                    const int zj = za - R + jj;
                    tma_load_5d(st, &map_wint, full, x0, y0, zj, a.cur, 2 * shot);
                    if (out) {
                        tma_load_5d(st + C::OFF1_H, &map_whalo, full, x0 - C::RA, y0 - R, zj - R,
                                    a.cur, 2 * shot);
                        tma_load_4d(st + C::OFF1_N, &map_cint, full, x0, y0, zj - R, 3);
                    }
                });
        }
    } else {
        const int gx = x0 + 4 * tx, gy = y0 + ty;
        const bool ok = gx < a.L.nxp && gy < a.L.ny;
        const int q = ty * C::BX + 4 * tx;
        float *out = a.tmp + (int64_t)6 * shot * a.L.vol + (int64_t)gy * a.L.nxp + gx;
        Q4 acc[2][2 * R];
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int i = 0; i < 2 * R; ++i) acc[f][i] = Q4{0ull, 0ull};
        RingPos<C::NSL> pos;
#pragma unroll U
        for (int j = 0; j < nplanes; ++j, pos.next()) {
            const int slot = pos.slot(j);
            if (*ring.abort_flag || !mbar_wait_bounded(&ring.full[slot], pos.phase(j))) {
                leave_ring(ring.abort_flag, j, a.err);
                break;
            }
            const float *st = ring.smem + slot * C::STAGE1;
            const Q4 cp = lds_q4(st + q), cr = lds_q4(st + C::INT + q);
            dz_feed_q4<R, KIND>(acc[0], cp, a.t1[2]);
            dz_feed_q4<R, KIND>(acc[1], cr, a.t1[2]);
            if (j >= 2 * R) {
                const float *N = st + C::OFF1_N + q;
                const Q4 nx = lds_q4(N), ny = lds_q4(N + C::INT), nz = lds_q4(N + 2 * C::INT);
                const int64_t off = (int64_t)(za - 2 * R + j) * a.L.plane;
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const float *H = st + C::OFF1_H + f * C::HXY + (R + ty) * C::PW + 4 * tx;
                    const Q4 gxv = q4_from(dx4<R, C::RA, KIND>(H, a.t1[0]));
                    const Q4 gyv = dy_q4<R, KIND>(H + C::RA, C::PW, a.t1[1]);
                    const Q4 gzv = acc[f][0];
                    const Q4 h = q4_fma(nz, gzv, q4_fma(nx, gxv, q4_mul(ny, gyv)));
                    Q4 o[3];
                    if (f == 0) {  // f_i = D_i p - n_i h
                        const Q4 mh = q4_neg(h);
                        o[0] = q4_fma(nx, mh, gxv);
                        o[1] = q4_fma(ny, mh, gyv);
                        o[2] = q4_fma(nz, mh, gzv);
                    } else {  // e_i = n_i h
                        o[0] = q4_mul(nx, h);
                        o[1] = q4_mul(ny, h);
                        o[2] = q4_mul(nz, h);
                    }
                    // streaming stores: the temporaries are read once, by
                    // pass 2, and must not push the p/r halo planes out of L2
                    if (ok)
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const float4 v =
                                make_float4(f32x2::f2_lo(o[c].lo), f32x2::f2_hi(o[c].lo),
                                            f32x2::f2_lo(o[c].hi), f32x2::f2_hi(o[c].hi));
                            __stcs(reinterpret_cast<float4 *>(out + (3 * f + c) * a.L.vol + off),
                                   v);
                        }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&ring.empty[slot]);
            dz_shift_q4<R, KIND>(acc[0], cp, a.t1[2]);
            dz_shift_q4<R, KIND>(acc[1], cr, a.t1[2]);
        }
    }
    __syncthreads();
    if (*ring.abort_flag && tid == C::CONSUMERS) drain<C::NSL>(ring, issued);
}

// ---------------------------------------------------------------- pass 2

template <int R, int TX, int TY, int D, int KIND, int U, int MINB>
__global__ void __launch_bounds__(TX *TY + 32, MINB)
    tti_pass2_kernel(const __grid_constant__ CUtensorMap map_tint,
                     const __grid_constant__ CUtensorMap map_tx,
                     const __grid_constant__ CUtensorMap map_ty,
                     const __grid_constant__ CUtensorMap map_wlev,
                     const __grid_constant__ CUtensorMap map_cint,
                     const __grid_constant__ TtiArgs a, const __grid_constant__ AcousticInject inj,
                     int zchunk, int nzc) {
    using C = TtiCfg<R, TX, TY, D>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Ring ring = ring_init<C::NSL, C::WARPS>(smem_raw, C::STAGE2);
    const int tid = threadIdx.x, lane = tid & 31;
    const int tx = tid % TX, ty = tid / TX;
    const int shot = blockIdx.z / nzc, chunk = blockIdx.z - shot * nzc;
    const int x0 = blockIdx.x * C::BX, y0 = blockIdx.y * C::BY;
    const int za = chunk * zchunk, zb = min(a.L.nz, za + zchunk);
    const int nplanes = zb - za + 2 * R;
    // For R <= 2 the x/y derivatives of a plane enter the z pipeline when the
    // plane arrives, between the contributions of the planes below and above
    // it, as in the fused scheme: the automatic scheme then gives the same
    // bits on either side of its size limit.  Wider stencils take them with
    // the output plane.
    constexpr bool EARLY = R <= 2;
    __syncthreads();
    chain_wait();
    if (__ldcg(a.err) & DEV_ERR_NONFINITE) return;  // stopped by the divergence watchdog

    int issued = 0;
    if (tid >= C::CONSUMERS) {
        if (lane == 0) {
            issued = produce<C::NSL>(
                ring, C::STAGE2, nplanes, a.err, [&](int jj, float *st, uint64_t *full) {
                    const bool out = jj >= 2 * R;
                    const bool xy = EARLY ? jj >= R && jj < nplanes - R : out;
                    mbar_arrive_expect_tx(full, (2 * C::INT + (xy ? 2 * C::HX + 2 * C::HY : 0) +
                                                 (out ? 7 * C::INT : 0)) *
                                                    4);
                    const int zj = za - R + jj, zs = zj - R, zxy = EARLY ? zj : zs;
                    tma_load_5d(st, &map_tint, full, x0, y0, zj, 2, 2 * shot);  // f_z, e_z
                    if (xy) {
                        tma_load_5d(st + C::OFF2_X, &map_tx, full, x0 - C::RA, y0, zxy, 0,
                                    2 * shot);  // f_x, e_x
                        tma_load_5d(st + C::OFF2_Y, &map_ty, full, x0, y0 - R, zxy, 1,
                                    2 * shot);  // f_y, e_y
                    }
                    if (out) {
                        tma_load_5d(st + C::OFF2_W, &map_wlev, full, x0, y0, zs, 0, 2 * shot);
                        tma_load_4d(st + C::OFF2_C, &map_cint, full, x0, y0, zs, 0);  // b, a, s
                    }
                });
        }
    } else {
        const int gx = x0 + 4 * tx, gy = y0 + ty;
        const bool ok = gx < a.L.nxp && gy < a.L.ny;
        const int q = ty * C::BX + 4 * tx;
        float dpx4[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) dpx4[i] = (gx + i < a.L.nx) ? a.dpx[gx + i] : 0.f;
        const f2 dpx_lo = f2_pack(dpx4[0], dpx4[1]), dpx_hi = f2_pack(dpx4[2], dpx4[3]);
        const float dpy = gy < a.L.ny ? a.dpy[gy] : 0.f;
        const f2 one2 = f2_splat(1.f);
        // q^{n+1} overwrites q^{n-1}
        float *qn = a.wave + (int64_t)(4 * shot + 1 - a.cur) * a.L.vol +
                    (int64_t)gy * a.L.nxp + gx;
        Q4 acc[2][2 * R];
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int i = 0; i < 2 * R; ++i) acc[f][i] = Q4{0ull, 0ull};
        RingPos<C::NSL> pos;
#pragma unroll U
        for (int j = 0; j < nplanes; ++j, pos.next()) {
            const int slot = pos.slot(j);
            const int zs = za - 2 * R + j;
            const float dz = j >= 2 * R ? __ldg(a.dpz + zs) : 0.f;
            if (*ring.abort_flag || !mbar_wait_bounded(&ring.full[slot], pos.phase(j))) {
                leave_ring(ring.abort_flag, j, a.err);
                break;
            }
            const float *st = ring.smem + slot * C::STAGE2;
            const Q4 cf = lds_q4(st + q), ce = lds_q4(st + C::INT + q);
            dz_feed_q4<R, KIND>(acc[0], cf, a.t2[2]);
            dz_feed_q4<R, KIND>(acc[1], ce, a.t2[2]);
            Q4 dxy[2];
            if (EARLY ? j >= R && j < nplanes - R : j >= 2 * R) {
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const float *hx = st + C::OFF2_X + f * C::HX + ty * C::PW + 4 * tx;
                    const float *hy = st + C::OFF2_Y + f * C::HY + (R + ty) * C::BX + 4 * tx;
                    const Q4 dxv = q4_from(dx4<R, C::RA, KIND>(hx, a.t2[0]));
                    const Q4 dyv = dy_q4<R, KIND>(hy, C::BX, a.t2[1]);
                    dxy[f] = q4_add(dxv, dyv);
                    if (EARLY) acc[f][R] = q4_add(acc[f][R], dxy[f]);
                }
            }
            if (j >= 2 * R) {
                Q4 H[2];  // Hxy p, Hz r
#pragma unroll
                for (int f = 0; f < 2; ++f)
                    H[f] = EARLY ? acc[f][0] : q4_add(dxy[f], acc[f][0]);
                const float *w = st + C::OFF2_W + q, *cc = st + C::OFF2_C + q;
                const Q4 b = lds_q4(cc), av = lds_q4(cc + C::INT), sv = lds_q4(cc + 2 * C::INT);
                const f2 dyz = f2_splat(-(dpy + dz));
                // 1 - zeta, zeta = (dx + dy + dz) b
                const Q4 keep = Q4{f2_fma(f2_sub(dyz, dpx_lo), b.lo, one2),
                                   f2_fma(f2_sub(dyz, dpx_hi), b.hi, one2)};
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const Q4 rhs = f == 0 ? q4_fma(av, H[0], q4_mul(sv, H[1]))  // a Hxy p + s Hz r
                                          : q4_fma(sv, H[0], H[1]);             // s Hxy p + Hz r
                    const Q4 qc = lds_q4(w + (2 * f + a.cur) * C::INT);
                    const Q4 qm = lds_q4(w + (2 * f + 1 - a.cur) * C::INT);
                    const Q4 o = q4_fma(b, rhs, q4_fma(keep, q4_sub(qc, qm), qc));
                    if (ok)
                        *reinterpret_cast<ulonglong2 *>(qn + 2 * f * a.L.vol +
                                                        (int64_t)zs * a.L.plane) =
                            make_ulonglong2(o.lo, o.hi);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&ring.empty[slot]);
            dz_shift_q4<R, KIND>(acc[0], cf, a.t2[2]);
            dz_shift_q4<R, KIND>(acc[1], ce, a.t2[2]);
        }
    }
    __syncthreads();
    if (*ring.abort_flag && tid == C::CONSUMERS) drain<C::NSL>(ring, issued);
    if (inj.nsrc > 0 && tid == 0 && !*ring.abort_flag)
        tti_inject_column<C::BX, C::BY>(&a, &inj, zchunk, nzc);
}

// ---------------------------------------------------------------- small grids

// Both passes with one block of 32 x 8 x 8 points per CTA instead of a march
// (see acoustic_direct_kernel): a pass of a small grid is latency, and here it
// is one set of copies and one pass of arithmetic.  The block's operands with
// halos come in one copy (p and r) or three (the x, y and z temporaries of
// both fields), the rest are plain loads under them; the launch lets the next
// one set itself up at once.  Same operations in the same order per point as
// the marching passes.
// us per step, best march and this: so 4 48^3 10.1 and 9.6, 80^3 18.8 and 12.9,
// 96^3 22.0 and 17.2; so 8 80^3 22.6 and 16.3; so 16 64^3 21.9 and 14.9; past
// about 100^3 the halos of the blocks lose (so 8 128^3 37.9 and 51.5).  The
// cost model takes either kernel for each pass by itself.
template <int R>
struct TtiDirect {
    static constexpr int BX = 32, BY = 8, BZ = 8;
    static constexpr int RA = (R + 3) / 4 * 4;
    static constexpr int PW = BX + 2 * RA, PH = BY + 2 * R, PD = BZ + 2 * R;
    static constexpr int THREADS = BX / 4 * BY * BZ;
    static constexpr int F1 = PW * PH * PD;                       // a field of pass 1
    static constexpr int FX = PW * BY * BZ, FY = BX * PH * BZ, FZ = BX * BY * PD;  // of pass 2
    static constexpr size_t SMEM1 = (size_t)2 * F1 * 4 + 16 + 128;
    static constexpr size_t SMEM2 = (size_t)2 * (FX + FY + FZ) * 4 + 16 + 128;
    static_assert(FX % 16 == 0 && FY % 16 == 0, "128-byte aligned copies");
};

// First derivative along z of the float4 at `centre`, planes `pitch` floats
// apart, summed as the z pipeline does (`mid` is added when the centre plane
// arrives).
template <int R, int KIND, bool MID>
__device__ __forceinline__ Q4 dz_direct(const float *centre, int pitch, const float *t, Q4 mid) {
    const f2 w0 = f2_splat(tap_used<KIND>(-R, R) ? t[0] : 0.f);
    const Q4 c0 = lds_q4(centre - R * pitch);
    Q4 s = Q4{f2_mul(w0, c0.lo), f2_mul(w0, c0.hi)};
#pragma unroll
    for (int d = -R + 1; d <= R; ++d) {
        if (tap_used<KIND>(d, R)) s = q4_fma(f2_splat(t[d + R]), lds_q4(centre + d * pitch), s);
        if (MID && d == 0) s = q4_add(s, mid);
    }
    return s;
}

__device__ __forceinline__ Q4 ldg_q4(const float *p) {
    return q4_from(__ldg(reinterpret_cast<const float4 *>(p)));
}

template <int R, int KIND>
__global__ void __launch_bounds__(TtiDirect<R>::THREADS)
    tti_direct1_kernel(const __grid_constant__ CUtensorMap map_wint,
                       const __grid_constant__ CUtensorMap map_whalo,
                       const __grid_constant__ CUtensorMap map_cint,
                       const __grid_constant__ TtiArgs a, const __grid_constant__ ReceiveArgs rec,
                       int zchunk, int nzc) {
    using C = TtiDirect<R>;
    if (blockIdx.z >= gridDim.z - rec.slices) {
        chain_trigger();
        chain_wait();
        if (!(__ldcg(a.err) & DEV_ERR_NONFINITE))
            record_receivers(&rec, a.wave, 4, a.cur, 2 + a.cur, &a.L);
        return;
    }
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *tile = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) &
                                            ~static_cast<uintptr_t>(127));
    uint64_t *full = reinterpret_cast<uint64_t *>(tile + 2 * C::F1);
    const int tid = threadIdx.x;
    const int tx = tid % 8, ty = tid / 8 % C::BY, tz = tid / (8 * C::BY);
    const int shot = blockIdx.z / nzc, chunk = blockIdx.z - shot * nzc;
    const int x0 = blockIdx.x * C::BX, y0 = blockIdx.y * C::BY, z0 = chunk * C::BZ;
    const int gx = x0 + 4 * tx, gy = y0 + ty, gz = z0 + tz;
    if (tid == 0) {
        prefetch_tensormap(&map_whalo);
        mbar_init(full, 1);
        fence_mbar_init();
    }
    __syncthreads();
    chain_trigger();
    chain_wait();
    if (tid == 0) {
        mbar_arrive_expect_tx(full, 2 * C::F1 * 4);
        tma_load_5d(tile, &map_whalo, full, x0 - C::RA, y0 - R, z0 - R, a.cur, 2 * shot);
    }
    const bool ok = gx < a.L.nxp && gy < a.L.ny && gz < a.L.nz;
    const int64_t off = (int64_t)gz * a.L.plane + (int64_t)gy * a.L.nxp + gx;
    Q4 nx = Q4{0ull, 0ull}, ny = nx, nz = nx;
    if (ok) {
        nx = ldg_q4(a.nvec + off);
        ny = ldg_q4(a.nvec + a.L.vol + off);
        nz = ldg_q4(a.nvec + 2 * a.L.vol + off);
    }
    // set by the divergence watchdog to stop the run: nothing is stored then
    const bool stopped = __ldcg(a.err) & DEV_ERR_NONFINITE;
    if (!mbar_wait_bounded(full, 0)) {
        atomicOr(a.err, DEV_ERR_TIMEOUT);
        // the copy gets a bounded chance to land
        if (tid == 0) mbar_wait_bounded(full, 0, 200000000ull);
        return;
    }
    if (!ok || stopped) return;
    constexpr int SY = C::PW, SZ = C::PW * C::PH;
    float *out = a.tmp + (int64_t)6 * shot * a.L.vol + off;
#pragma unroll
    for (int f = 0; f < 2; ++f) {
        const float *H = tile + f * C::F1 + (R + tz) * SZ + (R + ty) * SY + 4 * tx;
        const Q4 gxv = q4_from(dx4<R, C::RA, KIND>(H, a.t1[0]));
        const Q4 gyv = dy_q4<R, KIND>(H + C::RA, SY, a.t1[1]);
        const Q4 gzv = dz_direct<R, KIND, false>(H + C::RA, SZ, a.t1[2], gxv);
        const Q4 h = q4_fma(nz, gzv, q4_fma(nx, gxv, q4_mul(ny, gyv)));
        Q4 o[3];
        if (f == 0) {  // f_i = D_i p - n_i h
            const Q4 mh = q4_neg(h);
            o[0] = q4_fma(nx, mh, gxv);
            o[1] = q4_fma(ny, mh, gyv);
            o[2] = q4_fma(nz, mh, gzv);
        } else {  // e_i = n_i h
            o[0] = q4_mul(nx, h);
            o[1] = q4_mul(ny, h);
            o[2] = q4_mul(nz, h);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
            *reinterpret_cast<ulonglong2 *>(out + (3 * f + c) * a.L.vol) =
                make_ulonglong2(o[c].lo, o[c].hi);
    }
}

template <int R, int KIND>
__global__ void __launch_bounds__(TtiDirect<R>::THREADS)
    tti_direct2_kernel(const __grid_constant__ CUtensorMap map_tint,
                       const __grid_constant__ CUtensorMap map_tx,
                       const __grid_constant__ CUtensorMap map_ty,
                       const __grid_constant__ CUtensorMap map_wlev,
                       const __grid_constant__ CUtensorMap map_cint,
                       const __grid_constant__ TtiArgs a,
                       const __grid_constant__ AcousticInject inj, int zchunk, int nzc) {
    using C = TtiDirect<R>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *tile = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) &
                                            ~static_cast<uintptr_t>(127));
    float *tile_y = tile + 2 * C::FX, *tile_z = tile_y + 2 * C::FY;
    uint64_t *full = reinterpret_cast<uint64_t *>(tile_z + 2 * C::FZ);
    const int tid = threadIdx.x;
    const int tx = tid % 8, ty = tid / 8 % C::BY, tz = tid / (8 * C::BY);
    const int shot = blockIdx.z / nzc, chunk = blockIdx.z - shot * nzc;
    const int x0 = blockIdx.x * C::BX, y0 = blockIdx.y * C::BY, z0 = chunk * C::BZ;
    const int gx = x0 + 4 * tx, gy = y0 + ty, gz = z0 + tz;
    if (tid == 0) {
        prefetch_tensormap(&map_tint);
        prefetch_tensormap(&map_tx);
        prefetch_tensormap(&map_ty);
        mbar_init(full, 1);
        fence_mbar_init();
    }
    __syncthreads();
    chain_trigger();
    chain_wait();
    if (tid == 0) {
        mbar_arrive_expect_tx(full, 2 * (C::FX + C::FY + C::FZ) * 4);
        tma_load_5d(tile, &map_tx, full, x0 - C::RA, y0, z0, 0, 2 * shot);      // f_x, e_x
        tma_load_5d(tile_y, &map_ty, full, x0, y0 - R, z0, 1, 2 * shot);        // f_y, e_y
        tma_load_5d(tile_z, &map_tint, full, x0, y0, z0 - R, 2, 2 * shot);      // f_z, e_z
    }
    const bool ok = gx < a.L.nxp && gy < a.L.ny && gz < a.L.nz;
    const int64_t off = (int64_t)gz * a.L.plane + (int64_t)gy * a.L.nxp + gx;
    float *wave = a.wave + (int64_t)4 * shot * a.L.vol + off;
    Q4 b = Q4{0ull, 0ull}, av = b, sv = b, keep = b, qc[2] = {b, b}, qm[2] = {b, b};
    if (ok) {
        b = ldg_q4(a.bcoef + off);
        av = ldg_q4(a.acoef + off);
        sv = ldg_q4(a.scoef + off);
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            qc[f] = lds_q4(wave + (2 * f + a.cur) * a.L.vol);
            qm[f] = lds_q4(wave + (2 * f + 1 - a.cur) * a.L.vol);
        }
        float dpx4[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) dpx4[i] = (gx + i < a.L.nx) ? a.dpx[gx + i] : 0.f;
        const f2 dyz = f2_splat(-(a.dpy[gy] + a.dpz[gz]));
        const f2 one2 = f2_splat(1.f);
        // 1 - zeta, zeta = (dx + dy + dz) b
        keep = Q4{f2_fma(f2_sub(dyz, f2_pack(dpx4[0], dpx4[1])), b.lo, one2),
                  f2_fma(f2_sub(dyz, f2_pack(dpx4[2], dpx4[3])), b.hi, one2)};
    }
    const bool stopped = __ldcg(a.err) & DEV_ERR_NONFINITE;
    bool landed = mbar_wait_bounded(full, 0);
    if (!landed) {
        atomicOr(a.err, DEV_ERR_TIMEOUT);
        // the copies get a bounded chance to land
        if (tid == 0) mbar_wait_bounded(full, 0, 200000000ull);
    } else if (ok && !stopped) {
        constexpr bool EARLY = R <= 2;  // see the marching pass
        Q4 H[2];                        // Hxy p, Hz r
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const float *hx = tile + f * C::FX + (tz * C::BY + ty) * C::PW + 4 * tx;
            const float *hy = tile_y + f * C::FY + (tz * C::PH + R + ty) * C::BX + 4 * tx;
            const float *hz = tile_z + f * C::FZ + ((R + tz) * C::BY + ty) * C::BX + 4 * tx;
            const Q4 dxy = q4_add(q4_from(dx4<R, C::RA, KIND>(hx, a.t2[0])),
                                  dy_q4<R, KIND>(hy, C::BX, a.t2[1]));
            H[f] = dz_direct<R, KIND, EARLY>(hz, C::BX * C::BY, a.t2[2], dxy);
            if (!EARLY) H[f] = q4_add(dxy, H[f]);
        }
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            const Q4 rhs = f == 0 ? q4_fma(av, H[0], q4_mul(sv, H[1]))  // a Hxy p + s Hz r
                                  : q4_fma(sv, H[0], H[1]);             // s Hxy p + Hz r
            const Q4 o = q4_fma(b, rhs, q4_fma(keep, q4_sub(qc[f], qm[f]), qc[f]));
            float4 v = make_float4(f32x2::f2_lo(o.lo), f32x2::f2_hi(o.lo), f32x2::f2_lo(o.hi),
                                   f32x2::f2_hi(o.hi));
            // the row's padding stays zero
            if (gx >= a.L.nx) v.x = 0.f;
            if (gx + 1 >= a.L.nx) v.y = 0.f;
            if (gx + 2 >= a.L.nx) v.z = 0.f;
            if (gx + 3 >= a.L.nx) v.w = 0.f;
            *reinterpret_cast<float4 *>(wave + (2 * f + 1 - a.cur) * a.L.vol) = v;
        }
    }
    if (inj.nsrc > 0) {
        __syncthreads();
        if (tid == 0 && landed && !stopped)
            tti_inject_column<C::BX, C::BY>(&a, &inj, zchunk, nzc);
    }
}

// ---------------------------------------------------------------- recompute

// The "no temporaries" scheme of the ablation (the paper's `advanced` level:
// common sub-expressions eliminated, but no shift-invariant temporaries): for
// every outer stencil point of Hxy p = sum_i D_i f_i and Hz r = sum_i D_i e_i
// the inner gradients of p and r, and from them f_i and e_i, are recomputed
// from scratch.  Work per point grows as (stencil points)^2 instead of
// linearly; the loads are served by L1/L2.  One thread per grid point; CHECK
// adds the zero-ghost tests near the boundary (block-uniform choice).
template <int R, int K1, int K2, bool CHECK>
__device__ __forceinline__ void recompute_ops(const TtiArgs &a, const float *__restrict__ p,
                                              const float *__restrict__ r, int i, int j, int k,
                                              float &A, float &B) {
    const WaveLayout &L = a.L;
    const int64_t o0 = (int64_t)k * L.plane + (int64_t)j * L.nxp + i;
    const int64_t stride[3] = {1, L.nxp, L.plane};
    const int n3[3] = {L.nx, L.ny, L.nz};
    const int c0[3] = {i, j, k};
    A = 0.f;
    B = 0.f;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
#pragma unroll 1
        for (int d = -R; d <= R; ++d) {
            if (!tap_used<K2>(d, R)) continue;
            if (CHECK && (c0[ax] + d < 0 || c0[ax] + d >= n3[ax])) continue;  // zero ghost
            const int64_t o2 = o0 + d * stride[ax];
            float gp[3] = {0.f, 0.f, 0.f}, gr[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const int cb = c0[b] + (b == ax ? d : 0);
#pragma unroll
                for (int e = -R; e <= R; ++e) {
                    if (!tap_used<K1>(e, R)) continue;
                    if (CHECK && (cb + e < 0 || cb + e >= n3[b])) continue;
                    const int64_t o3 = o2 + e * stride[b];
                    const float w = a.t1[b][e + R];
                    gp[b] = fmaf(w, __ldg(p + o3), gp[b]);
                    gr[b] = fmaf(w, __ldg(r + o3), gr[b]);
                }
            }
            const float nx = __ldg(a.nvec + o2), ny = __ldg(a.nvec + L.vol + o2),
                        nz = __ldg(a.nvec + 2 * L.vol + o2);
            const float hp = nx * gp[0] + ny * gp[1] + nz * gp[2];
            const float hr = nx * gr[0] + ny * gr[1] + nz * gr[2];
            const float na = ax == 0 ? nx : (ax == 1 ? ny : nz);
            const float w2 = a.t2[ax][d + R];
            A = fmaf(w2, gp[ax] - na * hp, A);  // f_ax = D_ax p - n_ax (n . grad p)
            B = fmaf(w2, na * hr, B);           // e_ax = n_ax (n . grad r)
        }
    }
}

constexpr int kRecBX = 32, kRecBY = 8;

template <int R, int K1, int K2>
__global__ void __launch_bounds__(kRecBX *kRecBY) tti_recompute_kernel(const TtiArgs a) {
    if (__ldcg(a.err) & DEV_ERR_NONFINITE) return;  // stopped by the divergence watchdog
    const WaveLayout &L = a.L;
    const int i = blockIdx.x * kRecBX + threadIdx.x;
    const int j = blockIdx.y * kRecBY + threadIdx.y;
    const int shot = blockIdx.z / L.nz;
    const int k = blockIdx.z - shot * L.nz;
    // every tap of the block (outer + inner: 2R) inside the grid?
    const int bx0 = blockIdx.x * kRecBX, by0 = blockIdx.y * kRecBY;
    const bool interior = bx0 >= 2 * R && bx0 + kRecBX + 2 * R <= L.nx && by0 >= 2 * R &&
                          by0 + kRecBY + 2 * R <= L.ny && k >= 2 * R && k + 2 * R < L.nz;
    if (i >= L.nx || j >= L.ny) return;
    const float *p = a.wave + (int64_t)(4 * shot + a.cur) * L.vol;
    const float *r = a.wave + (int64_t)(4 * shot + 2 + a.cur) * L.vol;
    float A, B;
    if (interior)
        recompute_ops<R, K1, K2, false>(a, p, r, i, j, k, A, B);
    else
        recompute_ops<R, K1, K2, true>(a, p, r, i, j, k, A, B);
    const int64_t o = (int64_t)k * L.plane + (int64_t)j * L.nxp + i;
    const float b = __ldg(a.bcoef + o), av = __ldg(a.acoef + o), sv = __ldg(a.scoef + o);
    const float zeta = (a.dpx[i] + (a.dpy[j] + a.dpz[k])) * b;
    const float *pm = a.wave + (int64_t)(4 * shot + 1 - a.cur) * L.vol;
    const float *rm = a.wave + (int64_t)(4 * shot + 3 - a.cur) * L.vol;
    const float pc = __ldg(p + o), pp = pm[o], rc = __ldg(r + o), rp = rm[o];
    const float rhs_p = av * A + sv * B, rhs_r = sv * A + B;
    // q+ overwrites q- (each point reads q- only at itself)
    a.wave[(int64_t)(4 * shot + 1 - a.cur) * L.vol + o] = pc + (1.f - zeta) * (pc - pp) + b * rhs_p;
    a.wave[(int64_t)(4 * shot + 3 - a.cur) * L.vol + o] = rc + (1.f - zeta) * (rc - rp) + b * rhs_r;
}

// ---------------------------------------------------------------- host side

// A launch configuration of one pass with its cost constants (microseconds),
// as in acoustic.cu.
struct PassEntry {
    const void *fn;
    size_t smem;
    int bx, by, pw, ph, threads;
    float launch, lat, thr, warm;
    int bz, pd;  // z extent of a block and of its copy (marching passes: 0 and 1)
};

template <int PASS, int R, int STAG>
PassEntry direct_entry(float launch, float lat, float thr) {
    using C = TtiDirect<R>;
    constexpr int KIND = STAG ? (PASS == 1 ? 1 : -1) : 0;
    const void *fn;
    if constexpr (PASS == 1)
        fn = (const void *)&tti_direct1_kernel<R, KIND>;
    else
        fn = (const void *)&tti_direct2_kernel<R, KIND>;
    return PassEntry{fn,    PASS == 1 ? C::SMEM1 : C::SMEM2,
                     C::BX, C::BY, C::PW, C::PH, C::THREADS, launch, lat, thr, 0.f, C::BZ, C::PD};
}

template <int PASS, int R, int TX, int TY, int D, int U, int MINB, int STAG>
PassEntry pass_entry(float launch, float lat, float thr, float warm) {
    using C = TtiCfg<R, TX, TY, D>;
    constexpr int KIND = STAG ? (PASS == 1 ? 1 : -1) : 0;  // D+ inner, D- outer, or centred
    const void *fn;
    if constexpr (PASS == 1)
        fn = (const void *)&tti_pass1_kernel<R, TX, TY, D, KIND, U, MINB>;
    else
        fn = (const void *)&tti_pass2_kernel<R, TX, TY, D, KIND, U, MINB>;
    return PassEntry{fn,    PASS == 1 ? C::SMEM1 : C::SMEM2,
                     C::BX, C::BY, C::PW, C::PH, C::THREADS, launch, lat, thr, warm, 0, 1};
}

struct PassTable {
    const PassEntry *e;
    int n;
};
constexpr int kMaxPassEntries = 4;  // of a table

#define FD_TTI_ENTRY(PASS, R, TX, TY, D, U, MB, ...) \
    pass_entry<PASS, R, TX, TY, D, U, MB, STAG>(__VA_ARGS__)

// Per radius (template arguments TX, TY, D, U, minimum CTAs per SM), fitted
// and chosen on 13 problems from 48^3 to 512^3 with centred derivatives (the
// staggered ones have as many taps but one; so 2 takes so 4's costs).  Both fields' pending z
// outputs take 16R registers of a thread, which decides the tile: 64 x 8 with
// two or three CTAs per SM up to so 12, one CTA of 64 x 14 (224 + 32 threads
// with 255 registers) at so 16, a smaller one beside it for small grids.
// 512^3, pass 1 + pass 2, so 4 / 8 / 12 / 16: 880 + 1153, 892 + 1169, 927 +
// 1171 and 1039 + 1188 us, within 8 % of 104 bytes per point at the copy
// bandwidth (2065 us); before (one thread group per field): 2112 / 2110 /
// 2264 / 2570 us in all.
template <int STAG>
PassTable pass1_table(int radius) {
    static const PassEntry r1[] = {
        FD_TTI_ENTRY(1, 1, 16, 8, 3, 4, 0, 5.74f, 0.050f, 0.467f, 0.10f)};
    static const PassEntry r2[] = {
        FD_TTI_ENTRY(1, 2, 16, 8, 3, 4, 0, 5.74f, 0.050f, 0.467f, 0.10f),
        FD_TTI_ENTRY(1, 2, 16, 16, 3, 4, 0, 2.59f, 0.771f, 0.249f, 0.66f),
        direct_entry<1, 2, STAG>(5.96f, 0.62f, 2.09f)};
    static const PassEntry r4[] = {
        FD_TTI_ENTRY(1, 4, 16, 8, 3, 4, 0, 6.43f, 0.275f, 0.453f, 0.21f),
        direct_entry<1, 4, STAG>(5.67f, 0.05f, 3.05f)};
    static const PassEntry r6[] = {
        FD_TTI_ENTRY(1, 6, 16, 8, 3, 4, 2, 6.84f, 0.449f, 0.465f, 0.25f),
        FD_TTI_ENTRY(1, 6, 16, 14, 3, 4, 1, 4.65f, 0.828f, 0.145f, 0.41f),
        direct_entry<1, 6, STAG>(5.04f, 3.26f, 3.50f)};
    static const PassEntry r8[] = {
        FD_TTI_ENTRY(1, 8, 16, 14, 3, 2, 1, 5.46f, 0.529f, 0.851f, 0.39f),
        FD_TTI_ENTRY(1, 8, 16, 6, 3, 2, 2, 7.26f, 0.548f, 0.423f, 0.30f),
        direct_entry<1, 8, STAG>(4.89f, 4.79f, 3.82f)};
    switch (radius) {
        case 1: return {r1, 1};
        case 2: return {r2, 3};
        case 4: return {r4, 2};
        case 6: return {r6, 3};
        case 8: return {r8, 3};
        default: return {nullptr, 0};
    }
}

template <int STAG>
PassTable pass2_table(int radius) {
    static const PassEntry r1[] = {
        FD_TTI_ENTRY(2, 1, 16, 8, 2, 4, 0, 5.87f, 0.050f, 0.632f, 0.27f)};
    static const PassEntry r2[] = {
        FD_TTI_ENTRY(2, 2, 16, 8, 2, 4, 0, 5.87f, 0.050f, 0.632f, 0.27f),
        direct_entry<2, 2, STAG>(5.03f, 3.28f, 1.99f)};
    static const PassEntry r4[] = {
        FD_TTI_ENTRY(2, 4, 16, 8, 2, 4, 0, 7.16f, 0.199f, 0.631f, 0.20f),
        direct_entry<2, 4, STAG>(4.95f, 4.53f, 2.84f)};
    static const PassEntry r6[] = {
        FD_TTI_ENTRY(2, 6, 16, 8, 2, 4, 2, 7.92f, 0.408f, 0.622f, 0.25f),
        direct_entry<2, 6, STAG>(4.11f, 5.05f, 4.27f)};
    static const PassEntry r8[] = {
        FD_TTI_ENTRY(2, 8, 16, 14, 2, 4, 1, 4.78f, 0.652f, 0.881f, 0.40f),
        FD_TTI_ENTRY(2, 8, 16, 6, 1, 1, 2, 7.03f, 0.648f, 0.499f, 0.32f),
        direct_entry<2, 8, STAG>(5.21f, 3.93f, 4.39f)};
    switch (radius) {
        case 1: return {r1, 1};
        case 2: return {r2, 2};
        case 4: return {r4, 2};
        case 6: return {r6, 2};
        case 8: return {r8, 3};
        default: return {nullptr, 0};
    }
}

PassTable pass_table(int pass, int radius, int stag) {
    return pass == 1 ? (stag ? pass1_table<1>(radius) : pass1_table<0>(radius))
                     : (stag ? pass2_table<1>(radius) : pass2_table<0>(radius));
}

const void *recompute_fn(int radius, int stag) {
    switch (radius) {
        case 1: return stag ? (const void *)&tti_recompute_kernel<1, 1, -1>
                            : (const void *)&tti_recompute_kernel<1, 0, 0>;
        case 2: return stag ? (const void *)&tti_recompute_kernel<2, 1, -1>
                            : (const void *)&tti_recompute_kernel<2, 0, 0>;
        case 4: return stag ? (const void *)&tti_recompute_kernel<4, 1, -1>
                            : (const void *)&tti_recompute_kernel<4, 0, 0>;
        case 6: return stag ? (const void *)&tti_recompute_kernel<6, 1, -1>
                            : (const void *)&tti_recompute_kernel<6, 0, 0>;
        case 8: return stag ? (const void *)&tti_recompute_kernel<8, 1, -1>
                            : (const void *)&tti_recompute_kernel<8, 0, 0>;
        default: return nullptr;
    }
}

// The entry and chunk count with the smallest estimated time for one pass.
fd_status plan_pass(int pass, int radius, int stag, int config, const WaveLayout &L, int nshots,
                    TtiPassPlan *p) {
    const PassTable t = pass_table(pass, radius, stag);
    if (!t.e) return set_error(FD_ERR_SO, "no TTI kernel for radius %d", radius);
    int dev = 0, nsm = 0;
    FD_CUDA_TRY(cudaGetDevice(&dev));
    FD_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    PlanEntry cand[kMaxPassEntries];
    for (int i = 0; i < t.n; ++i) {
        const PassEntry &e = t.e[i];
        int per_sm = 0;
        FD_TRY(raise_smem_limit(e.fn, e.smem));
        FD_CUDA_TRY(
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, e.fn, e.threads, e.smem));
        if (per_sm < 1) return set_error(FD_ERR_CUDA, "TTI pass-%d kernel does not fit", pass);
        cand[i] = PlanEntry{e.bx,  e.by, e.bz, per_sm, e.launch, e.lat, e.thr,
                            e.warm * 2.0 * radius, INT_MAX, 0, false};
    }
    const int forced = config < 0 ? -1 : (config < t.n ? config : t.n - 1);
    const PlanChoice best = choose_plan(cand, t.n, forced, L.nx, L.ny, L.nz, nshots, nsm);
    if (best.entry < 0)
        return set_error(FD_ERR_ARG, "grid too large for the TTI launch configuration");
    const PassEntry &e = t.e[best.entry];
    const int ntx = (L.nx + e.bx - 1) / e.bx, nty = (L.ny + e.by - 1) / e.by;
    p->fn = e.fn;
    p->grid = dim3(ntx, nty, nshots * best.nzc);
    p->block = dim3(e.threads, 1, 1);
    p->smem = e.smem;
    p->zchunk = best.zchunk;
    p->nzc = best.nzc;
    p->bx = e.bx;
    p->by = e.by;
    p->pw = e.pw;
    p->ph = e.ph;
    p->bz = e.bz ? e.bz : 1;
    p->pd = e.pd;
    p->est_us = best.us;
    return FD_OK;
}

}  // namespace

int tti_num_configs(int radius) {
    const PassTable a = pass_table(1, radius, 0), b = pass_table(2, radius, 0);
    const int n = a.n > b.n ? a.n : b.n;
    return a.e && radius <= 2 && n < 2 ? 2 : n;  // the fused scheme has two tiles
}

fd_status tti_plan(int radius, const WaveLayout &L, int nshots, float *wave, float *tmp,
                   const float *coef, TtiPlan *plan, int stag, int scheme, int config) {
    plan->radius = radius;
    plan->stag = stag ? 1 : 0;
    plan->scheme = scheme;
    if (scheme == kTtiRecompute) {
        if (!recompute_fn(radius, stag))
            return set_error(FD_ERR_SO, "no TTI kernel for radius %d", radius);
        if ((int64_t)nshots * L.nz > 65535)
            return set_error(FD_ERR_ARG, "grid too large for the TTI recompute launch");
        plan->p1.grid = dim3((L.nx + kRecBX - 1) / kRecBX, (L.ny + kRecBY - 1) / kRecBY,
                             nshots * L.nz);
        plan->p1.block = dim3(kRecBX, kRecBY, 1);
        return FD_OK;
    }
    if (scheme != kTtiTwoPass) return set_error(FD_ERR_ARG, "unknown TTI scheme %d", scheme);
    FD_TRY(plan_pass(1, radius, stag, config, L, nshots, &plan->p1));
    FD_TRY(plan_pass(2, radius, stag, config, L, nshots, &plan->p2));
    const uint64_t sy = (uint64_t)L.nxp * 4, sz = (uint64_t)L.plane * 4, sv = (uint64_t)L.vol * 4;
    const uint64_t nx = L.nx, ny = L.ny, nz = L.nz, nf = 2ull * nshots;
    // p/r buffers [shot][field][level], temporaries [shot][field][component]
    const uint64_t wdim[5] = {nx, ny, nz, 2, nf}, wstr[4] = {sy, sz, sv, 2 * sv};
    const uint64_t tdim[5] = {nx, ny, nz, 3, nf}, tstr[4] = {sy, sz, sv, 3 * sv};
    const uint32_t bx1 = plan->p1.bx, by1 = plan->p1.by, bx2 = plan->p2.bx, by2 = plan->p2.by;
    const uint32_t wint[5] = {bx1, by1, 1, 1, 2};
    const uint32_t bz2 = plan->p2.bz;
    const uint32_t whalo[5] = {(uint32_t)plan->p1.pw, (uint32_t)plan->p1.ph,
                               (uint32_t)plan->p1.pd, 1, 2};
    const uint32_t wlev[5] = {bx2, by2, 1, 2, 2};
    const uint32_t tint[5] = {bx2, by2, (uint32_t)plan->p2.pd, 1, 2};
    const uint32_t txb[5] = {(uint32_t)plan->p2.pw, by2, bz2, 1, 2};
    const uint32_t tyb[5] = {bx2, (uint32_t)plan->p2.ph, bz2, 1, 2};
    FD_TRY(make_tensor_map_5d(&plan->map_wint, wave, wdim, wstr, wint));
    FD_TRY(make_tensor_map_5d(&plan->map_whalo, wave, wdim, wstr, whalo));
    FD_TRY(make_tensor_map_5d(&plan->map_wlev, wave, wdim, wstr, wlev));
    FD_TRY(make_tensor_map_5d(&plan->map_tint, tmp, tdim, tstr, tint));
    FD_TRY(make_tensor_map_5d(&plan->map_tx, tmp, tdim, tstr, txb));
    FD_TRY(make_tensor_map_5d(&plan->map_ty, tmp, tdim, tstr, tyb));
    FD_TRY(make_tensor_map_4d(&plan->map_c1, coef, L.nx, L.ny, L.nz, 6, sy, sz, sv, bx1, by1, 1,
                              3));
    return make_tensor_map_4d(&plan->map_c2, coef, L.nx, L.ny, L.nz, 6, sy, sz, sv, bx2, by2, 1,
                              3);
}

fd_status tti_choose_scheme(int radius, int stag, const WaveLayout &L, int nshots, int *scheme) {
    *scheme = kTtiTwoPass;
    // from so 8 on the cross cells of the fused scheme cost more than the
    // temporaries' 56 bytes per point
    if (radius > 2 || !tti_fused_supported(radius)) return FD_OK;
    double fused_us = 0.0;
    FD_TRY(tti_fused_time(radius, stag, L, nshots, &fused_us));
    TtiPassPlan p1, p2;
    FD_TRY(plan_pass(1, radius, stag, -1, L, nshots, &p1));
    FD_TRY(plan_pass(2, radius, stag, -1, L, nshots, &p2));
    // so 4: two passes up to about 128^3 (48^3 10.0 against 15.5 us per step,
    // 96^3 17.4 and 22.9, 128^3 35.9 and 32.5), fused above (256^3 204 against
    // 268, 512^3 1430 against 2025).  The pass tables were fitted to launches
    // between events, 3.7 us each longer than chained ones.  The six
    // temporaries are not spent on many small shots at once.
    const bool cheap = (int64_t)6 * nshots * L.vol * 4 <= (int64_t)1 << 30;
    if (!cheap || fused_us <= p1.est_us + p2.est_us - 7.5) *scheme = kTtiFused;
    return FD_OK;
}

bool tti_records_receivers(const TtiPlan &plan) {
    return plan.scheme != kTtiRecompute && plan.p1.grid.z < 65535;
}

fd_status tti_launch(const TtiPlan &plan, const TtiArgs &a, cudaStream_t stream,
                     cudaEvent_t *ev, const AcousticInject *inject, const ReceiveArgs *receive) {
    if (ev) FD_CUDA_TRY(cudaEventRecord(ev[0], stream));
    if (plan.scheme == kTtiRecompute) {
        void *pr[] = {(void *)&a};
        FD_CUDA_TRY(cudaLaunchKernel(recompute_fn(plan.radius, plan.stag), plan.p1.grid,
                                     plan.p1.block, pr, 0, stream));
        note_launch(stream);
        if (ev) {
            FD_CUDA_TRY(cudaEventRecord(ev[1], stream));
            FD_CUDA_TRY(cudaEventRecord(ev[2], stream));
        }
        return FD_OK;
    }
    AcousticInject inj;
    memset(&inj, 0, sizeof(inj));
    if (inject) inj = *inject;
    ReceiveArgs rec;
    memset(&rec, 0, sizeof(rec));
    dim3 grid1 = plan.p1.grid;
    if (receive) rec = *receive;
    if (plan.scheme == kTtiFused) {
        FD_TRY(tti_fused_launch(plan, a, stream, inj, rec));
        if (ev) {
            FD_CUDA_TRY(cudaEventRecord(ev[1], stream));
            FD_CUDA_TRY(cudaEventRecord(ev[2], stream));
        }
        return FD_OK;
    }
    if (rec.nrec > 0) {
        rec.slices = receive_slices(rec, grid1.x, grid1.y, plan.p1.block.x);
        if (grid1.z >= 65535) return set_error(FD_ERR_ARG, "no grid slice left for receivers");
        if ((int64_t)grid1.z + rec.slices > 65535) rec.slices = 65535 - grid1.z;
        grid1.z += rec.slices;
    }
    int zc1 = plan.p1.zchunk, nzc1 = plan.p1.nzc, zc2 = plan.p2.zchunk, nzc2 = plan.p2.nzc;
    void *p1[] = {(void *)&plan.map_wint, (void *)&plan.map_whalo, (void *)&plan.map_c1,
                  (void *)&a, (void *)&rec, (void *)&zc1, (void *)&nzc1};
    FD_CUDA_TRY(launch_chained(plan.p1.fn, grid1, plan.p1.block, p1, plan.p1.smem, stream));
    note_launch(stream);
    if (ev) FD_CUDA_TRY(cudaEventRecord(ev[1], stream));
    void *p2[] = {(void *)&plan.map_tint, (void *)&plan.map_tx, (void *)&plan.map_ty,
                  (void *)&plan.map_wlev, (void *)&plan.map_c2, (void *)&a, (void *)&inj,
                  (void *)&zc2, (void *)&nzc2};
    FD_CUDA_TRY(launch_chained(plan.p2.fn, plan.p2.grid, plan.p2.block, p2, plan.p2.smem, stream));
    note_launch(stream);
    if (ev) FD_CUDA_TRY(cudaEventRecord(ev[2], stream));
    return FD_OK;
}

}  // namespace fdsweep
