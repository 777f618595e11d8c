// acoustic.cu -- K1: one leapfrog step of the damped isotropic acoustic wave
// equation (Eq. WE; Listing fd-3) with the compact central Laplacian of
// radius R = so/2 (Listing fd-1/fd-2), over every grid point (Dirichlet: zero
// ghosts outside the grid).
//
//   u+ = u + (1 - zeta)(u - u-) + b * lap(u),   b = dt^2 / (m + damp dt/2),
//   zeta = damp * b / dt,
// which is the centred discretisation m (u+ - 2u + u-)/dt^2 +
// damp (u+ - u-)/(2 dt) = lap(u) rearranged for u+; with damp = 0 it is
// u+ = 2u - u- + dt^2 lap(u) / m.
//
// GB300 design.  One CTA owns a BX x BY column of the grid and marches it
// through z.  Every plane p of u^n (tile plus an R-wide halo, zero-filled
// outside the grid by the TMA unit) is brought into a small ring of shared-
// memory stages by cp.async.bulk.tensor, D planes ahead of use; the same stage
// also receives the interior tiles of u^n, u^{n-1} and b for the output plane
// p - R.  Each stage has a "full" mbarrier (TMA transaction count) and an
// "empty" mbarrier (one arrival per warp), so warps run decoupled; a producer
// warp refills a stage as soon as every consumer warp has released it.  (With
// a consumer thread as the producer, the wait for the stage and the four copy
// issues, about 460 cycles, preceded that warp's share of every plane and set
// the pace of all: 1024 cycles (0.5 us) per plane for a lone CTA of any
// radius. With its own warp a plane takes 0.28 - 0.39 us.)
//
// One launch is one time step: extra blocks record the receivers of u^n, the
// sources are injected by the CTAs that own their nodes, and the launch is
// chained to the previous one (its prologue overlaps the other's last planes).
//
// The z-direction uses an accumulator pipeline: when plane p arrives, each
// thread adds w_|p-z| u(p) to the 2R pending outputs z in [p-R, p+R) it holds
// in registers, adds the x/y part of the Laplacian of plane p (read from the
// staged plane) to output p, and completes output p-R.  Per point this keeps
// 2R floats of state (instead of a 2R+1-plane queue plus R staged planes), so
// the shared-memory ring is only D+1 planes deep.  Every thread owns a 4 (x,
// one float4) by VY (y) micro-tile.  Algorithmic HBM traffic: 16 bytes per
// point (read u^n, u^{n-1}, b; write u^{n+1}); halo and centre re-reads are
// served by L2.
#include <stdio.h>
#include <string.h>

#include "f32x2.cuh"
#include "kernels.cuh"
#include "receive.cuh"
#include "ring.cuh"
#include "runtime.cuh"

namespace fdsweep {
namespace {
using namespace f32x2;

// DF: the damping is a 3-D field; the stage then also carries the interior
// tile of the per-point coefficient zeta = damp b / dt (stored after b as a
// second field of the coefficient tensor) instead of forming zeta from the
// per-axis profiles: 20 instead of 16 bytes per point.
template <int R, int TX, int TY, int VY, int D, bool DF = false>
struct AcCfg {
    static constexpr int BX = 4 * TX;
    static constexpr int BY = VY * TY;
    static constexpr int RA = (R + 3) / 4 * 4;  // x halo rounded to 16 bytes (TMA rule)
    static constexpr int PW = BX + 2 * RA;
    static constexpr int PH = BY + 2 * R;
    static constexpr int NSL = D + 1;           // ring slots
    static constexpr int HALO = (PW * PH + 31) / 32 * 32;
    static constexpr int INT = BX * BY;         // interior tile (multiple of 32)
    static constexpr int NINT = DF ? 4 : 3;     // interior tiles per stage
    static constexpr int STAGE = HALO + NINT * INT;  // [halo u^n][u^n][u^{n-1}][b][zeta]
    static constexpr uint32_t HALO_BYTES = PW * PH * 4;
    static constexpr uint32_t INT_BYTES = INT * 4;
    static constexpr int CONSUMERS = TX * TY;        // threads that own points
    static constexpr int WARPS = CONSUMERS / 32;
    static constexpr int THREADS = CONSUMERS + 32;   // + the producer warp
    // stages, full/empty mbarriers, abort flag; + damp_z of the z chunk
    // (added at launch) and 128 bytes to align the base
    static constexpr size_t SMEM = (size_t)NSL * STAGE * 4 + NSL * 16 + 16 + 128;
    static_assert(PW <= 256 && PH <= 256 && BX <= 256 && BY <= 256, "TMA box dimension limit");
    static_assert(INT % 32 == 0 && CONSUMERS % 32 == 0, "tile shape");
    static_assert(WARPS <= kMaxRingWarps, "room behind the abort flag");
};

// Source injection by the CTA that wrote a source's corners, after its
// column is complete: thread 0 adds w_c b q to each corner node inside the
// column and z chunk, sources in order, with the sparse kernel's operations
// (w_c = wx wy wz, times b, times q, added to the stored value).  The block
// barrier before it makes the column's stores visible to thread 0; no other
// CTA touches these nodes in this launch.  Out of line, with the column
// recomputed from the block index, so that nothing stays live across the
// plane loop for it.
template <int BX, int BY>
__device__ __noinline__ void inject_column(const AcousticStepArgs *a, const AcousticInject *inj,
                                           int zchunk, int nzc) {
    const int n = inj->step + (inj->step_base ? *inj->step_base : 0);
    if (n < 0 || n >= inj->nt) return;
    const int shot = blockIdx.z / nzc;
    const int za = (blockIdx.z - shot * nzc) * zchunk;
    const int zb = min(a->L.nz, za + zchunk);
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    const int x1 = min(x0 + BX, a->L.nx), y1 = min(y0 + BY, a->L.ny);
    float *u = a->wave + (int64_t)(shot * a->lps + a->lev_out) * a->L.vol;
    for (int s = 0; s < inj->nsrc; ++s) {
        const SparsePoint p = inj->src_tab[shot * inj->nsrc + s];
        const int i = (int)(p.base % (uint32_t)a->L.nxp);
        const int j = (int)((p.base / (uint32_t)a->L.nxp) % (uint32_t)a->L.ny);
        const int k = (int)(p.base / (uint32_t)a->L.plane);
        if (i + 1 < x0 || i >= x1 || j + 1 < y0 || j >= y1 || k + 1 < za || k >= zb) continue;
        const float q = inj->src_wav[((int64_t)shot * inj->nt + n) * inj->nsrc + s];
        for (int c = 0; c < 8; ++c) {
            const int ci = i + (c & 1), cj = j + ((c >> 1) & 1), ck = k + ((c >> 2) & 1);
            if (ci < x0 || ci >= x1 || cj < y0 || cj >= y1 || ck < za || ck >= zb) continue;
            const float wx = (c & 1) ? p.fx : __fsub_rn(1.f, p.fx);
            const float wy = (c & 2) ? p.fy : __fsub_rn(1.f, p.fy);
            const float wz = (c & 4) ? p.fz : __fsub_rn(1.f, p.fz);
            const int64_t off = (int64_t)ck * a->L.plane + (int64_t)cj * a->L.nxp + ci;
            const float val =
                __fmul_rn(__fmul_rn(__fmul_rn(__fmul_rn(wx, wy), wz), a->bcoef[off]), q);
            u[off] = __fadd_rn(u[off], val);
        }
    }
}

// x part of the Laplacian of 4 consecutive points (centre weight of all axes
// included) from a row that starts RA points left of them; *cen: the points.
template <int R, int RA>
__device__ __forceinline__ Q4 laplace_x(const float *row, const AcousticStepArgs &a, Q4 *cen) {
    constexpr int NP = (2 * RA + 4) / 2;  // packed pairs in the x span
    f2 xp[NP];
#pragma unroll
    for (int t = 0; t < NP / 2; ++t) {
        const Q4 q = lds_q4(row + 4 * t);
        xp[2 * t] = q.lo;
        xp[2 * t + 1] = q.hi;
    }
    constexpr int c0 = RA / 2;  // pair index of points 0,1
    const Q4 c = Q4{xp[c0], xp[c0 + 1]};
    const f2 wc2 = f2_splat(a.wc);
    Q4 s = Q4{f2_mul(wc2, c.lo), f2_mul(wc2, c.hi)};
    // even shifts keep the pair alignment: packed arithmetic
#pragma unroll
    for (int k = 2; k <= R; k += 2) {
        const f2 w2 = f2_splat(a.wx[k]);
        s.lo = f2_fma(w2, f2_add(xp[c0 + k / 2], xp[c0 - k / 2]), s.lo);
        s.hi = f2_fma(w2, f2_add(xp[c0 + 1 + k / 2], xp[c0 + 1 - k / 2]), s.hi);
    }
    // odd shifts straddle the pairs: scalar arithmetic
    float o0 = 0.f, o1 = 0.f, o2 = 0.f, o3 = 0.f;
#pragma unroll
    for (int k = 1; k <= R; k += 2) {
        auto el = [&](int idx) -> float {
            return (idx & 1) ? f2_hi(xp[idx >> 1]) : f2_lo(xp[idx >> 1]);
        };
        const float w = a.wx[k];
        o0 = fmaf(w, el(RA + 0 + k) + el(RA + 0 - k), o0);
        o1 = fmaf(w, el(RA + 1 + k) + el(RA + 1 - k), o1);
        o2 = fmaf(w, el(RA + 2 + k) + el(RA + 2 - k), o2);
        o3 = fmaf(w, el(RA + 3 + k) + el(RA + 3 - k), o3);
    }
    s.lo = f2_add(s.lo, f2_pack(o0, o1));
    s.hi = f2_add(s.hi, f2_pack(o2, o3));
    *cen = c;
    return s;
}

// U: unroll factor of the plane loop.  The pending-output registers shift by
// one plane per iteration; unrolling by U turns U - 1 of every U shifts into
// register renaming instead of moves (U = 2R removes them all).
// WL: the pipeline waits take their limit from the arguments (the
// failure-injection setting of fd_set_wait_limit_ns); otherwise it is the
// constant 2 s, which keeps the limit out of the plane loop's registers (a
// limit read at run time cost 13 % at so 8).
// EDGE: the R planes before and behind a chunk, which only feed its outputs
// along z, are loaded as interior tiles without a halo and skip the x/y part.
template <int R, int TX, int TY, int VY, int D, int U, bool DF, int MINB = 0, bool EDGE = false,
          bool WL = false>
__global__ void __launch_bounds__(TX *TY + 32, MINB)
    acoustic_step_kernel(const __grid_constant__ CUtensorMap map_halo,
                         const __grid_constant__ CUtensorMap map_int,
                         const __grid_constant__ CUtensorMap map_b,
                         const __grid_constant__ AcousticStepArgs a,
                         const __grid_constant__ AcousticInject inj,
                         const __grid_constant__ ReceiveArgs rec, int zchunk, int nzc) {
    using C = AcCfg<R, TX, TY, VY, D, DF>;
    if (blockIdx.z >= gridDim.z - rec.slices) {
        chain_trigger();
        chain_wait();
        if (!(__ldcg(a.err) & DEV_ERR_NONFINITE))
            record_receivers(&rec, a.wave, a.lps, a.lev_cur, a.lev_cur, &a.L);
        return;
    }
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *smem = reinterpret_cast<float *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~static_cast<uintptr_t>(127));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + C::NSL * C::STAGE);
    uint64_t *empty = full + C::NSL;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(empty + C::NSL);
    float *sdz = reinterpret_cast<float *>(empty + C::NSL + 2);  // damp_z / dt of this chunk

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int tx = tid % TX, ty = tid / TX;
    const int shot_i = blockIdx.z / nzc;
    const int chunk = blockIdx.z - shot_i * nzc;
    const int shot = a.slot_map ? a.slot_map[shot_i] : shot_i;
    const int x0 = blockIdx.x * C::BX, y0 = blockIdx.y * C::BY;
    const int za = chunk * zchunk;
    const int zb = min(a.L.nz, za + zchunk);
    const int nplanes = zb - za + 2 * R;  // arriving planes za-R .. zb+R-1
    const int wcur = shot * a.lps + a.lev_cur, wprev = shot * a.lps + a.lev_prev;
    const int wout = shot * a.lps + a.lev_out;
    const int gx = x0 + 4 * tx;
    const uint64_t wait_ns = WL ? (a.wait_ns ? a.wait_ns : 2000000000ull) : 2000000000ull;

    if (tid == 0) {
        prefetch_tensormap(&map_halo);
        prefetch_tensormap(&map_int);
        prefetch_tensormap(&map_b);
        for (int s = 0; s < C::NSL; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], C::WARPS);
        }
        fence_mbar_init();
        init_ring_abort(abort_flag);
    }
    for (int z = za + tid; z < zb; z += C::THREADS) sdz[z - za] = a.dpz[z];
    __syncthreads();
    chain_wait();
    // the divergence watchdog stopped the run: nothing more to compute
    if (__ldcg(a.err) & DEV_ERR_NONFINITE) return;

    int issued = 0;
    if (tid >= C::CONSUMERS) {
        // Producer warp (one lane): stage jj = halo plane za-R+jj, plus the
        // interior tiles of output plane za-2R+jj once jj >= 2R.
        if (lane == 0) {
            RingPos<C::NSL> pos;
            for (int jj = 0; jj < nplanes && !*abort_flag; ++jj, pos.next()) {
                const int slot = pos.slot(jj);
                if (jj >= C::NSL &&
                    !mbar_wait_bounded(&empty[slot], pos.phase(jj) ^ 1u, wait_ns)) {
                    if (!*abort_flag) atomicOr(a.err, DEV_ERR_TIMEOUT);
                    *abort_flag = 1;
                    break;
                }
                const bool with_out = jj >= 2 * R;
                const bool edge = EDGE && (jj < R || jj >= nplanes - R);
                mbar_arrive_expect_tx(&full[slot], (edge ? C::INT_BYTES : C::HALO_BYTES) +
                                                       (with_out ? C::NINT * C::INT_BYTES : 0));
                float *st = smem + slot * C::STAGE;
                if (edge)
                    tma_load_4d(st, &map_int, &full[slot], x0, y0, za - R + jj, wcur);
                else
                    tma_load_4d(st, &map_halo, &full[slot], x0 - C::RA, y0 - R, za - R + jj, wcur);
                if (with_out) {
                    const int zo = za - 2 * R + jj;
                    tma_load_4d(st + C::HALO, &map_int, &full[slot], x0, y0, zo, wcur);
                    tma_load_4d(st + C::HALO + C::INT, &map_int, &full[slot], x0, y0, zo, wprev);
                    tma_load_4d(st + C::HALO + 2 * C::INT, &map_b, &full[slot], x0, y0, zo, 0);
                    if (DF)
                        tma_load_4d(st + C::HALO + 3 * C::INT, &map_b, &full[slot], x0, y0, zo, 1);
                }
                issued = jj + 1;
            }
            // the next launch may move in while the last planes are computed;
            // earlier, its waiting blocks would take the place of this one's
            chain_trigger();
        }
    } else {
    const bool xok = gx < a.L.nxp;
    float dpx4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) dpx4[i] = (gx + i < a.L.nx) ? a.dpx[gx + i] : 0.f;
    const f2 dpx_lo = f2_pack(dpx4[0], dpx4[1]), dpx_hi = f2_pack(dpx4[2], dpx4[3]);
    int gy[VY];
    bool yok[VY];
    float dpyv[VY];
#pragma unroll
    for (int v = 0; v < VY; ++v) {
        gy[v] = y0 + ty * VY + v;
        yok[v] = gy[v] < a.L.ny;
        dpyv[v] = yok[v] ? a.dpy[gy[v]] : 0.f;
    }
    float *__restrict__ unew = a.wave + (int64_t)wout * a.L.vol;
    const f2 one2 = f2_splat(1.f);

    // acc[i][v]: pending output plane p - R + i (p = arriving plane)
    Q4 acc[2 * R][VY];
#pragma unroll
    for (int i = 0; i < 2 * R; ++i)
#pragma unroll
        for (int v = 0; v < VY; ++v) acc[i][v] = Q4{0ull, 0ull};

    RingPos<C::NSL> pos;
#pragma unroll U
    for (int j = 0; j < nplanes; ++j, pos.next()) {
        const int slot = pos.slot(j);
        if (*abort_flag || !mbar_wait_bounded(&full[slot], pos.phase(j), wait_ns)) {
            leave_ring(abort_flag, j, a.err);
            break;
        }
        const float *H = smem + slot * C::STAGE;
        const int rbase = R + ty * VY;

        // x/y part of the Laplacian of plane p (centre weight of all axes
        // included) and the centre values
        Q4 cen[VY], lxy[VY];
        if (EDGE && (j < R || j >= nplanes - R)) {
#pragma unroll
            for (int v = 0; v < VY; ++v) {
                cen[v] = lds_q4(H + (ty * VY + v) * C::BX + 4 * tx);
                lxy[v] = Q4{0ull, 0ull};
            }
        } else {
#pragma unroll
        for (int v = 0; v < VY; ++v) {
            lxy[v] = laplace_x<R, C::RA>(H + (rbase + v) * C::PW + 4 * tx, a, &cen[v]);
        }
#pragma unroll
        for (int dy = -R; dy < VY + R; ++dy) {
            bool needed = false;
#pragma unroll
            for (int v = 0; v < VY; ++v) {
                const int k = dy > v ? dy - v : v - dy;
                if (k >= 1 && k <= R) needed = true;
            }
            if (!needed) continue;
            const Q4 f = lds_q4(H + (rbase + dy) * C::PW + C::RA + 4 * tx);
#pragma unroll
            for (int v = 0; v < VY; ++v) {
                const int k = dy > v ? dy - v : v - dy;
                if (k >= 1 && k <= R) {
                    const f2 w2 = f2_splat(a.wy[k]);
                    lxy[v].lo = f2_fma(w2, f.lo, lxy[v].lo);
                    lxy[v].hi = f2_fma(w2, f.hi, lxy[v].hi);
                }
            }
        }

        }

        // z part: plane p feeds the pending outputs p-R .. p+R-1 and starts p+R
#pragma unroll
        for (int v = 0; v < VY; ++v) {
            const Q4 c = cen[v];
#pragma unroll
            for (int i = 0; i < 2 * R; ++i) {
                if (i == R) {
                    acc[i][v].lo = f2_add(acc[i][v].lo, lxy[v].lo);
                    acc[i][v].hi = f2_add(acc[i][v].hi, lxy[v].hi);
                } else {
                    const f2 w2 = f2_splat(a.wz[i < R ? R - i : i - R]);
                    acc[i][v].lo = f2_fma(w2, c.lo, acc[i][v].lo);
                    acc[i][v].hi = f2_fma(w2, c.hi, acc[i][v].hi);
                }
            }
        }

        // output plane zo = p - R is complete:
        //   u+ = u + (1 - zeta)(u - u-) + b * acc,  zeta = (dx + dy + dz) b
        if (j >= 2 * R) {
            const int zo = za - 2 * R + j;
            const float dz = sdz[zo - za];
            const float *Ui = H + C::HALO;
            const float *Pi = Ui + C::INT;
            const float *Bi = Pi + C::INT;
#pragma unroll
            for (int v = 0; v < VY; ++v) {
                if (!(xok && yok[v])) continue;
                const int q = (ty * VY + v) * C::BX + 4 * tx;
                const Q4 c = lds_q4(Ui + q);
                const Q4 p = lds_q4(Pi + q);
                const Q4 b = lds_q4(Bi + q);
                const Q4 s = acc[0][v];
                f2 zl, zh;
                if constexpr (DF) {
                    const Q4 zt = lds_q4(Bi + C::INT + q);
                    zl = zt.lo;
                    zh = zt.hi;
                } else {
                    const f2 dyz = f2_splat(dpyv[v] + dz);
                    zl = f2_mul(f2_add(dpx_lo, dyz), b.lo);
                    zh = f2_mul(f2_add(dpx_hi, dyz), b.hi);
                }
                f2 ol = f2_fma(f2_sub(one2, zl), f2_sub(c.lo, p.lo), c.lo);
                f2 oh = f2_fma(f2_sub(one2, zh), f2_sub(c.hi, p.hi), c.hi);
                ol = f2_fma(b.lo, s.lo, ol);
                oh = f2_fma(b.hi, s.hi, oh);
                const int64_t off = (int64_t)zo * a.L.plane + (int64_t)gy[v] * a.L.nxp + gx;
                *reinterpret_cast<ulonglong2 *>(unew + off) = make_ulonglong2(ol, oh);
            }
        }
        // every thread is done with the stage: release it
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[slot]);

        // rotate the pending outputs; plane p + R starts with w_R u(p)
        const f2 wR2 = f2_splat(a.wz[R]);
#pragma unroll
        for (int v = 0; v < VY; ++v) {
#pragma unroll
            for (int i = 0; i < 2 * R - 1; ++i) acc[i][v] = acc[i + 1][v];
            acc[2 * R - 1][v] = Q4{f2_mul(wR2, cen[v].lo), f2_mul(wR2, cen[v].hi)};
        }
    }
    }
    __syncthreads();
    if (*abort_flag && tid == C::CONSUMERS) {
        // The last NSL issued stages may still be in flight: give them a
        // bounded chance to land before the CTA's shared memory is released.
        for (int jj = issued - C::NSL; jj < issued; ++jj)
            if (jj >= 0)
                mbar_wait_bounded(&full[jj % C::NSL], (uint32_t)((jj / C::NSL) & 1), 200000000ull);
    }
    if (inj.nsrc > 0 && tid == 0 && !*abort_flag)
        inject_column<C::BX, C::BY>(&a, &inj, zchunk, nzc);
}

// Small grids: one block of 32 x 8 x 8 points per CTA instead of a march, so
// that a launch is one copy and one pass of arithmetic long.  The block comes
// with its halo on all sides (one cp.async.bulk.tensor), a thread owns four x
// points of one plane, and u^{n-1} and b are plain loads under the copy.  Every
// point sums its neighbours in the order of the marching kernel: same bits.
// A step of a small grid is latency: launch, copy, arithmetic and store behind
// one another.  So the launch lets the next one set itself up at once (the
// grid is one or two waves, no block waits for a place) and the stop flag is
// read under the copy.  us per step, direct against the best march: 64^3 so 4
// 4.5 and 5.6, so 8 4.8 and 6.8, so 16 6.4 and 9.0; 80^3 so 8 6.0 and 8.1; two
// waves of it lose (128^3 so 8 14.9 and 9.8), and the halo of a block (13
// times its points at so 16) costs more than the march's above 96^3.
template <int R>
struct AcDirect {
    static constexpr int BX = 32, BY = 8, BZ = 8;
    static constexpr int RA = (R + 3) / 4 * 4;
    static constexpr int PW = BX + 2 * RA, PH = BY + 2 * R, PD = BZ + 2 * R;
    static constexpr int THREADS = BX / 4 * BY * BZ;
    static constexpr int TILE = (PW * PH * PD + 31) / 32 * 32;
    static constexpr size_t SMEM = (size_t)TILE * 4 + 16 + 128;
};

template <int R, bool DF, bool WL = false>
__global__ void __launch_bounds__(AcDirect<R>::THREADS)
    acoustic_direct_kernel(const __grid_constant__ CUtensorMap map_halo,
                           const __grid_constant__ CUtensorMap map_int,
                           const __grid_constant__ CUtensorMap map_b,
                           const __grid_constant__ AcousticStepArgs a,
                           const __grid_constant__ AcousticInject inj,
                           const __grid_constant__ ReceiveArgs rec, int zchunk, int nzc) {
    using C = AcDirect<R>;
    if (blockIdx.z >= gridDim.z - rec.slices) {
        chain_trigger();
        chain_wait();
        if (!(__ldcg(a.err) & DEV_ERR_NONFINITE))
            record_receivers(&rec, a.wave, a.lps, a.lev_cur, a.lev_cur, &a.L);
        return;
    }
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *tile = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) &
                                            ~static_cast<uintptr_t>(127));
    uint64_t *full = reinterpret_cast<uint64_t *>(tile + C::TILE);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(full + 1);
    const int tid = threadIdx.x;
    const int tx = tid % 8, ty = tid / 8 % C::BY, tz = tid / (8 * C::BY);
    const int shot_i = blockIdx.z / nzc;
    const int chunk = blockIdx.z - shot_i * nzc;
    const int shot = a.slot_map ? a.slot_map[shot_i] : shot_i;
    const int x0 = blockIdx.x * C::BX, y0 = blockIdx.y * C::BY, z0 = chunk * C::BZ;
    const int gx = x0 + 4 * tx, gy = y0 + ty, gz = z0 + tz;
    const uint64_t wait_ns = WL ? (a.wait_ns ? a.wait_ns : 2000000000ull) : 2000000000ull;
    if (tid == 0) {
        prefetch_tensormap(&map_halo);
        mbar_init(full, 1);
        fence_mbar_init();
        *abort_flag = 0;
    }
    __syncthreads();
    chain_trigger();
    chain_wait();
    if (tid == 0) {
        mbar_arrive_expect_tx(full, C::PW * C::PH * C::PD * 4);
        tma_load_4d(tile, &map_halo, full, x0 - C::RA, y0 - R, z0 - R,
                    shot * a.lps + a.lev_cur);
    }
    // set by the divergence watchdog to stop the run: nothing is stored then
    const bool stopped = __ldcg(a.err) & DEV_ERR_NONFINITE;
    const bool ok = gx < a.L.nxp && gy < a.L.ny && gz < a.L.nz;
    const int64_t off = (int64_t)gz * a.L.plane + (int64_t)gy * a.L.nxp + gx;
    float4 p4 = make_float4(0.f, 0.f, 0.f, 0.f), b4 = p4, z4 = p4;
    if (ok) {
        p4 = *reinterpret_cast<const float4 *>(
            a.wave + (int64_t)(shot * a.lps + a.lev_prev) * a.L.vol + off);
        b4 = __ldg(reinterpret_cast<const float4 *>(a.bcoef + off));
        if (DF) {
            z4 = __ldg(reinterpret_cast<const float4 *>(a.bcoef + a.L.vol + off));
        } else {
            const float dyz = a.dpy[gy] + a.dpz[gz];
            z4.x = (gx < a.L.nx ? a.dpx[gx] : 0.f) + dyz;
            z4.y = (gx + 1 < a.L.nx ? a.dpx[gx + 1] : 0.f) + dyz;
            z4.z = (gx + 2 < a.L.nx ? a.dpx[gx + 2] : 0.f) + dyz;
            z4.w = (gx + 3 < a.L.nx ? a.dpx[gx + 3] : 0.f) + dyz;
        }
        // the row's padding stays zero, as the copies of the march read it
        if (gx + 1 >= a.L.nx) p4.y = b4.y = 0.f;
        if (gx + 2 >= a.L.nx) p4.z = b4.z = 0.f;
        if (gx + 3 >= a.L.nx) p4.w = b4.w = 0.f;
        if (gx >= a.L.nx) p4.x = b4.x = 0.f;
    }
    if (!mbar_wait_bounded(full, 0, wait_ns)) {
        *abort_flag = 1;
        atomicOr(a.err, DEV_ERR_TIMEOUT);
    } else {
        constexpr int SY = C::PW, SZ = C::PW * C::PH;
        const float *c = tile + (R + tz) * SZ + (R + ty) * SY + C::RA + 4 * tx;
        Q4 u;
        Q4 lxy = laplace_x<R, C::RA>(c - C::RA, a, &u);
#pragma unroll
        for (int d = -R; d <= R; ++d) {
            if (d == 0) continue;
            const f2 w2 = f2_splat(a.wy[d < 0 ? -d : d]);
            const Q4 f = lds_q4(c + d * SY);
            lxy.lo = f2_fma(w2, f.lo, lxy.lo);
            lxy.hi = f2_fma(w2, f.hi, lxy.hi);
        }
        Q4 s;
#pragma unroll
        for (int d = -R; d <= R; ++d) {
            if (d == 0) {
                s.lo = f2_add(s.lo, lxy.lo);
                s.hi = f2_add(s.hi, lxy.hi);
                continue;
            }
            const f2 w2 = f2_splat(a.wz[d < 0 ? -d : d]);
            const Q4 f = lds_q4(c + d * SZ);
            if (d == -R) {
                s.lo = f2_mul(w2, f.lo);
                s.hi = f2_mul(w2, f.hi);
            } else {
                s.lo = f2_fma(w2, f.lo, s.lo);
                s.hi = f2_fma(w2, f.hi, s.hi);
            }
        }
        if (ok && !stopped) {
            const f2 one2 = f2_splat(1.f);
            const f2 blo = f2_pack(b4.x, b4.y), bhi = f2_pack(b4.z, b4.w);
            f2 zl = f2_pack(z4.x, z4.y), zh = f2_pack(z4.z, z4.w);
            if (!DF) {
                zl = f2_mul(zl, blo);
                zh = f2_mul(zh, bhi);
            }
            f2 ol = f2_fma(f2_sub(one2, zl), f2_sub(u.lo, f2_pack(p4.x, p4.y)), u.lo);
            f2 oh = f2_fma(f2_sub(one2, zh), f2_sub(u.hi, f2_pack(p4.z, p4.w)), u.hi);
            ol = f2_fma(blo, s.lo, ol);
            oh = f2_fma(bhi, s.hi, oh);
            *reinterpret_cast<ulonglong2 *>(
                a.wave + (int64_t)(shot * a.lps + a.lev_out) * a.L.vol + off) =
                make_ulonglong2(ol, oh);
        }
    }
    if (inj.nsrc > 0) __syncthreads();
    // a copy that was given up gets a bounded chance to land
    if (*abort_flag && tid == 0) mbar_wait_bounded(full, 0, 200000000ull);
    if (inj.nsrc > 0 && tid == 0 && !*abort_flag && !stopped)
        inject_column<C::BX, C::BY>(&a, &inj, zchunk, nzc);
}

// A launch configuration and what a launch of it costs (microseconds, fitted
// to measured steps of 21 problems from 48^3 to 512^3, ragged and with up to
// 8 shots, over all chunk counts): `launch` + (planes + warm 2R) x waves, a
// plane costing sqrt(lat^2 + (k thr)^2) with k CTAs on the SM; a block of the
// direct kernel counts as one plane.
struct ConfigEntry {
    int radius;
    const void *fn, *fn_wl;  // fn_wl: the variant with the wait limit from the arguments
    size_t smem;
    int bx, by, pw, ph, threads;
    float launch, lat, thr, warm;
    const char *name;
    int bz, pd;  // z extent of a block and of its copy (marching kernel: 0 and 1)
    bool spare = false;  // only for grids that no other entry can launch
};
constexpr int kMaxEntries = 8;  // of a configuration table

template <int R, int TX, int TY, int VY, int D, int U, bool DF, int MINB, bool EDGE>
ConfigEntry make_entry(const char *name, float launch, float lat, float thr, float warm) {
    using C = AcCfg<R, TX, TY, VY, D, DF>;
    const void *wl = nullptr;
    if constexpr (!DF)
        wl = (const void *)&acoustic_step_kernel<R, TX, TY, VY, D, U, DF, MINB, EDGE, true>;
    return ConfigEntry{R,      (const void *)&acoustic_step_kernel<R, TX, TY, VY, D, U, DF, MINB, EDGE>,
                       wl,     C::SMEM, C::BX, C::BY, C::PW, C::PH, C::THREADS,
                       launch, lat, thr, warm, name, 0, 1};
}

template <int R, bool DF>
ConfigEntry make_direct(const char *name, float launch, float lat, float thr) {
    using C = AcDirect<R>;
    const void *wl = nullptr;
    if constexpr (!DF) wl = (const void *)&acoustic_direct_kernel<R, DF, true>;
    return ConfigEntry{R,     (const void *)&acoustic_direct_kernel<R, DF>,
                       wl,    C::SMEM, C::BX, C::BY, C::PW, C::PH, C::THREADS,
                       launch, lat, thr, 0.f, name, C::BZ, C::PD};
}

ConfigEntry spare(ConfigEntry e) {
    e.spare = true;
    return e;
}

#define FD_AC_ENTRY(R, TX, TY, VY, D, U, MB, ED, ...)                                           \
    make_entry<R, TX, TY, VY, D, U, false, MB, ED>("acoustic_step<" #R "," #TX "," #TY "," #VY "," \
                                               #D "," #U ">",                                  \
                                               __VA_ARGS__)
#define FD_AC_ENTRY_DF(R, TX, TY, VY, D, U, MB, ED, ...)                                       \
    make_entry<R, TX, TY, VY, D, U, true, MB, ED>("acoustic_step<" #R "," #TX "," #TY "," #VY "," \
                                              #D "," #U ",damp field>",                       \
                                              __VA_ARGS__)

// The configurations of each radius (template arguments R, TX, TY, VY, D, U,
// minimum CTAs per SM, EDGE); acoustic_plan takes the one with the smallest
// estimated time for the grid (plan.h).  Ring sizes are powers of two (D = 3), so that
// the unrolled plane loop has constant stage addresses.
//  * Small tiles fill the machine on small grids (64 x 4 at so 16: 128^3 17.8
//    us per step, 64 x 8 19.4).
//  * Two rows per thread (VY = 2) halve the shared-memory reads of the y
//    neighbours, which bound the wide stencils: R y-rows above and below cost
//    R + 1 reads per point instead of 2R.  At so 12 and 16 a few large CTAs
//    pay best at large sizes: 64 x 28 tiles, one CTA of 224 + 32 threads with
//    255 registers per SM, run 512^3 so 16 in 378 us (442 with 64 x 8, 472
//    before the producer warp); 64 x 44 at so 12 in 331 us (387 and 402).
//  * so 4 and 8 are at the HBM limit at 512^3 (310 and 329 us for 2.15 GB).
//  * EDGE (see the kernel) halves what the 2R extra planes of a chunk cost, so
//    that wide stencils can be cut into more chunks: so 16 4 x 128^3 41.4 ->
//    37.5 us per step, 160^3 25.9 -> 22.4, 64^3 11.4 -> 9.4; so 12 4 x 128^3
//    31.0 -> 26.9, 160^3 21.3 -> 18.6; so 8 96^3 8.8 -> 8.1.  Without gain at
//    so 4; a 64 x 28 tile that marches the whole axis in one chunk (512^3 so
//    16) is 1 % faster without it.
const ConfigEntry *config_table(int radius, int *count) {
    static const ConfigEntry r1[] = {
        FD_AC_ENTRY(1, 16, 16, 1, 3, 4, 0, 0, 2.4f, 0.30f, 0.27f, 0.9f)};
    static const ConfigEntry r2[] = {
        FD_AC_ENTRY(2, 16, 8, 1, 3, 4, 0, 0, 3.57f, 0.278f, 0.162f, 0.40f),
        FD_AC_ENTRY(2, 16, 16, 1, 4, 2, 0, 0, 2.44f, 0.299f, 0.269f, 0.91f),
        make_direct<2, false>("acoustic_direct<2>", 2.50f, 1.41f, 1.20f)};
    static const ConfigEntry r4[] = {
        FD_AC_ENTRY(4, 16, 8, 1, 3, 8, 0, 0, 3.70f, 0.269f, 0.157f, 0.73f),
        FD_AC_ENTRY(4, 16, 4, 2, 3, 8, 0, 1, 3.02f, 0.455f, 0.124f, 0.57f),
        make_direct<4, false>("acoustic_direct<4>", 2.56f, 2.02f, 1.48f)};
    static const ConfigEntry r6[] = {
        FD_AC_ENTRY(6, 16, 8, 1, 3, 4, 0, 1, 3.71f, 0.356f, 0.161f, 0.59f),
        FD_AC_ENTRY(6, 16, 8, 2, 3, 4, 2, 1, 2.80f, 0.488f, 0.279f, 0.54f),
        FD_AC_ENTRY(6, 16, 22, 2, 3, 4, 1, 1, 1.29f, 0.785f, 0.436f, 0.59f),
        make_direct<6, false>("acoustic_direct<6>", 2.60f, 2.58f, 1.73f)};
    static const ConfigEntry r8[] = {
        FD_AC_ENTRY(8, 16, 8, 1, 3, 8, 3, 1, 4.20f, 0.351f, 0.182f, 0.55f),
        FD_AC_ENTRY(8, 16, 4, 1, 3, 4, 0, 1, 3.25f, 0.412f, 0.093f, 0.48f),
        FD_AC_ENTRY(8, 16, 14, 2, 3, 8, 1, 1, 1.76f, 0.609f, 0.325f, 0.59f),
        FD_AC_ENTRY(8, 16, 14, 2, 3, 8, 1, 0, 1.89f, 0.619f, 0.241f, 0.99f),
        make_direct<8, false>("acoustic_direct<8>", 2.80f, 2.68f, 2.20f)};
    switch (radius) {
        case 1: *count = 1; return r1;
        case 2: *count = 3; return r2;
        case 4: *count = 3; return r4;
        case 6: *count = 4; return r6;
        case 8: *count = 5; return r8;
        default: *count = 0; return nullptr;
    }
}

// 3-D damping field: a fourth interior tile per stage (64 x 44 tiles at so 12
// would need a shorter ring and measured slower than 64 x 16 up to 384^3); the
// costs of the marching entries fitted to 10 problems, the one-block entries
// with the per-axis kernels' costs.
const ConfigEntry *config_table_df(int radius, int *count) {
    static const ConfigEntry r1[] = {
        FD_AC_ENTRY_DF(1, 16, 16, 1, 3, 4, 0, 0, 2.7f, 0.28f, 0.38f, 0.5f)};
    static const ConfigEntry r2[] = {
        FD_AC_ENTRY_DF(2, 16, 8, 1, 3, 4, 0, 0, 3.17f, 0.286f, 0.185f, 0.42f),
        make_direct<2, true>("acoustic_direct<2,damp field>", 2.50f, 1.41f, 1.20f),
        // 16 rows: the only one beyond 524280 of them (65535 blocks of 8)
        spare(FD_AC_ENTRY_DF(2, 16, 16, 1, 3, 4, 0, 0, 2.44f, 0.30f, 0.31f, 0.9f))};
    static const ConfigEntry r4[] = {
        FD_AC_ENTRY_DF(4, 16, 8, 1, 3, 8, 0, 0, 3.33f, 0.291f, 0.193f, 0.57f),
        FD_AC_ENTRY_DF(4, 16, 4, 2, 3, 8, 0, 0, 3.91f, 0.342f, 0.181f, 0.42f),
        make_direct<4, true>("acoustic_direct<4,damp field>", 2.56f, 2.02f, 1.48f)};
    static const ConfigEntry r6[] = {
        FD_AC_ENTRY_DF(6, 16, 8, 1, 3, 4, 0, 1, 3.48f, 0.384f, 0.179f, 0.59f),
        FD_AC_ENTRY_DF(6, 16, 8, 2, 3, 4, 2, 1, 3.01f, 0.460f, 0.360f, 0.44f),
        make_direct<6, true>("acoustic_direct<6,damp field>", 2.60f, 2.58f, 1.73f)};
    static const ConfigEntry r8[] = {
        FD_AC_ENTRY_DF(8, 16, 8, 1, 3, 8, 3, 1, 3.83f, 0.387f, 0.196f, 0.54f),
        FD_AC_ENTRY_DF(8, 16, 4, 1, 3, 4, 0, 1, 2.87f, 0.402f, 0.088f, 0.66f),
        FD_AC_ENTRY_DF(8, 16, 14, 2, 3, 8, 1, 1, 1.12f, 0.536f, 0.509f, 0.56f),
        make_direct<8, true>("acoustic_direct<8,damp field>", 2.80f, 2.68f, 2.20f)};
    switch (radius) {
        case 1: *count = 1; return r1;
        case 2: *count = 3; return r2;
        case 4: *count = 3; return r4;
        case 6: *count = 3; return r6;
        case 8: *count = 4; return r8;
        default: *count = 0; return nullptr;
    }
}

}  // namespace

int acoustic_num_configs(int radius) {
    int n = 0;
    config_table(radius, &n);
    return n;
}

fd_status acoustic_plan(int radius, int config, const WaveLayout &L, int nshots, int lps,
                        float *wave, const float *bcoef, AcousticPlan *plan, int map_shots,
                        bool damp_field) {
    if (map_shots < nshots) map_shots = nshots;
    int n = 0;
    const ConfigEntry *tab =
        damp_field ? config_table_df(radius, &n) : config_table(radius, &n);
    if (!tab) return set_error(FD_ERR_SO, "no acoustic kernel for radius %d", radius);
    if (config >= n) config = -1;
    int dev = 0, nsm = 0, max_smem = 0;
    FD_CUDA_TRY(cudaGetDevice(&dev));
    FD_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    FD_CUDA_TRY(
        cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    PlanEntry cand[kMaxEntries];
    for (int i = 0; i < n; ++i) {
        const ConfigEntry &e = tab[i];
        int per_sm = 0;
        FD_TRY(raise_smem_limit(e.fn, e.smem));
        FD_CUDA_TRY(
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, e.fn, e.threads, e.smem));
        if (per_sm < 1) return set_error(FD_ERR_CUDA, "kernel %s does not fit on an SM", e.name);
        // damp_z of a chunk follows the stages in shared memory
        cand[i] = PlanEntry{e.bx, e.by, e.bz, per_sm, e.launch, e.lat, e.thr,
                            e.warm * 2.0 * radius, (max_smem - (int)e.smem) / 4, 0, e.spare};
    }
    const PlanChoice best = choose_plan(cand, n, config, L.nx, L.ny, L.nz, nshots, nsm);
    if (best.entry < 0)
        return set_error(FD_ERR_ARG, "grid too large for the launch configuration");
    const ConfigEntry &e = tab[best.entry];
    plan->radius = radius;
    plan->config = best.entry;
    plan->damp_field = damp_field;
    plan->name = e.name;
    plan->block = dim3(e.threads, 1, 1);
    const int ntx = (L.nx + e.bx - 1) / e.bx;
    const int nty = (L.ny + e.by - 1) / e.by;
    int nzc = 1;
    if (best.zchunk < L.nz) nzc = best.nzc;
    plan->grid = dim3(ntx, nty, nshots * nzc);
    plan->zchunk = best.zchunk;
    plan->nzc = nzc;
    plan->smem = e.smem + (size_t)best.zchunk * 4;
    FD_TRY(raise_smem_limit(e.fn, plan->smem));
    if (e.fn_wl) FD_TRY(raise_smem_limit(e.fn_wl, plan->smem));
    FD_TRY(make_tensor_map_4d(&plan->map_halo, wave, L.nx, L.ny, L.nz, (uint64_t)map_shots * lps,
                              (uint64_t)L.nxp * 4, (uint64_t)L.plane * 4, (uint64_t)L.vol * 4,
                              e.pw, e.ph, e.pd, 1));
    FD_TRY(make_tensor_map_4d(&plan->map_int, wave, L.nx, L.ny, L.nz, (uint64_t)map_shots * lps,
                              (uint64_t)L.nxp * 4, (uint64_t)L.plane * 4, (uint64_t)L.vol * 4,
                              e.bx, e.by, 1, 1));
    return make_tensor_map_4d(&plan->map_b, bcoef, L.nx, L.ny, L.nz, damp_field ? 2 : 1,
                              (uint64_t)L.nxp * 4, (uint64_t)L.plane * 4, (uint64_t)L.vol * 4,
                              e.bx, e.by, 1, 1);
}

fd_status acoustic_launch(const AcousticPlan &plan, const AcousticStepArgs &args,
                          cudaStream_t stream, const AcousticInject *inject,
                          const ReceiveArgs *receive) {
    int n = 0;
    const ConfigEntry *tab =
        plan.damp_field ? config_table_df(plan.radius, &n) : config_table(plan.radius, &n);
    if (!tab || plan.config >= n) return set_error(FD_ERR_SO, "bad acoustic plan");
    AcousticInject inj;
    memset(&inj, 0, sizeof(inj));
    if (inject && inject->nsrc > 0) {
        if (inject->nsrc > kInjectMaxSources || args.slot_map)
            return set_error(FD_ERR_ARG, "in-kernel injection: at most %d sources, no slot map",
                             kInjectMaxSources);
        inj = *inject;
    }
    ReceiveArgs rec;
    memset(&rec, 0, sizeof(rec));
    dim3 grid = plan.grid;
    if (receive && receive->nrec > 0) {
        rec = *receive;
        rec.slices = receive_slices(rec, grid.x, grid.y, plan.block.x);
        if (grid.z >= 65535) return set_error(FD_ERR_ARG, "no grid slice left for receivers");
        if ((int64_t)grid.z + rec.slices > 65535) rec.slices = 65535 - grid.z;
        grid.z += rec.slices;
    }
    int zchunk = plan.zchunk, nzc = plan.nzc;
    AcousticStepArgs a = args;
    if (!a.wait_ns) a.wait_ns = wait_limit_ns();
    void *params[] = {(void *)&plan.map_halo, (void *)&plan.map_int, (void *)&plan.map_b,
                      (void *)&a, (void *)&inj, (void *)&rec, (void *)&zchunk, (void *)&nzc};
    const void *fn = tab[plan.config].fn;
    if (a.wait_ns != 0 && tab[plan.config].fn_wl)
        fn = tab[plan.config].fn_wl;  // same tiles, ring and shared memory
    FD_CUDA_TRY(launch_chained(fn, grid, plan.block, params, plan.smem, stream));
    note_launch(stream);
    return FD_OK;
}

}  // namespace fdsweep
