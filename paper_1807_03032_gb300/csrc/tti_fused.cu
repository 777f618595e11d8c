// tti_fused.cu -- the TTI step in one kernel with the first-derivative
// temporaries kept on chip (the paper's shift-invariant temporaries, here in
// shared memory instead of HBM), for stencil radii R <= 4.
//
// Same operators as the two passes of tti.cu (Hxy p = sum_i D_i f_i,
// Hz r = sum_i D_i e_i, f_i = D_i p - n_i (n . grad p), e_i = n_i (n . grad r)).
// One CTA owns a 64 x 16 column and marches it through z; a thread owns one
// "cross" cell -- four x points of the tile, of the R rows above and below it
// or of the float4 column left and right of it, the points whose temporaries
// the tile's outer stencil reads -- for BOTH fields:
//   * every arriving plane of p and r comes with a halo of 2R rows and 2RA
//     columns (TMA, zero fill outside the grid) into a ring of R + 1 + D
//     planes and feeds the cell's z-derivative accumulators;
//   * R planes behind, the gradient of the cells is complete: f_x, e_x on the
//     x-extended tile and f_y, e_y on the y-extended tile go to shared memory
//     (zero outside the grid, as the ghosts of the two-pass scheme), f_z, e_z
//     stay with the tile cell's thread;
//   * after one barrier, the tile warps feed the outer derivatives to a second
//     accumulator pipeline, whose output R planes further behind is complete:
//     p and r are updated by the thread that holds Hxy p and Hz r.  The strip
//     warps meanwhile start the next plane (the temporaries have two buffers).
// A producer warp issues the four copies of a plane (both fields, n, both
// levels, coefficients).  HBM traffic per point: p, r and n_x, n_y, n_z once
// with halos, p, p-, r, r-, b, a, s for the update, p+, r+ out: 48 bytes
// against 104 for the two passes; the price is the gradient of the cross
// cells (1.38x the tile's at R = 2).  Bound by shared memory (about 85 floats
// per point, 87 % of its bandwidth at 512^3) and by the latency of a plane's
// chain (wait, gradient, barrier, outer derivative).
// 512^3 so 4: 1430 us per step; with one thread group per field
// exchanging Hxy p and Hz r at a second barrier, two cells for some threads
// and a consumer thread issuing twelve copies per plane, 1763 us.
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

template <int R, int TY_, int D>
struct TfCfg {
    static constexpr int TX = 16, TY = TY_;
    static constexpr int BX = 4 * TX, BY = TY;
    static constexpr int RA = 4;  // x halo in whole float4 cells (R <= 4)
    static_assert(R >= 1 && R <= 4, "the fused TTI kernel covers radii 1..4");
    // p/r plane box (its rows carry 4 extra columns so that the x-strip
    // cells, one per row and 8 rows per phase of a 128-bit shared access,
    // fall on distinct banks) and the cross bounding box
    static constexpr int PX = BX + 4 * RA + 4, PY = BY + 4 * R;
    static constexpr int NXW = BX + 2 * RA, NYH = BY + 2 * R;
    static constexpr int INT = BX * BY, TILE = TX * TY;
    static constexpr int NCELL = TILE + 2 * BY + 2 * R * TX;
    static constexpr int WARPS = (NCELL + 31) / 32;
    static constexpr int CONSUMERS = 32 * WARPS;
    static constexpr int THREADS = CONSUMERS + 32;  // + the producer warp
    static constexpr int BOX = PX * PY, NBOX = NXW * NYH;
    static constexpr int NP = R + 1 + D;  // plane ring: plane s .. arriving plane, + prefetch
    static constexpr int NQ = D + 1;      // per-iteration ring: n at s, update tiles at o
    static constexpr int PSLOT = round32(2 * BOX);
    static constexpr int OFF_W = round32(3 * NBOX);            // p0, p1, r0, r1
    static constexpr int OFF_C = OFF_W + round32(4 * INT);     // b, a, s
    static constexpr int QSLOT = OFF_C + round32(3 * INT);
    static constexpr int FX = round32(NXW * BY);  // f_x / e_x, x-extended
    static constexpr int FY = round32(BX * NYH);  // f_y / e_y, y-extended
    static constexpr int TMP = FX + FY;
    static constexpr uint32_t PBYTES = 2 * BOX * 4;
    static constexpr uint32_t NBYTES = 3 * NBOX * 4, UBYTES = 7 * INT * 4;
    static constexpr size_t SMEM = ((size_t)NP * PSLOT + (size_t)NQ * QSLOT + 4 * TMP) * 4 +
                                   (size_t)(2 * NP + NQ) * 8 + 16 + 128;
    static_assert(PX <= 256 && PY <= 256, "TMA box dimension limit");
    static_assert(TILE % 32 == 0, "whole tile warps");
};

// Barrier of the first `n` threads with the OR of a flag over them, so that
// all of them leave together after a failed wait.
__device__ __forceinline__ bool consumers_or(int n, bool flag) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(flag ? 1u : 0u), "r"(n)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ float4 masked(Q4 v, unsigned m) {
    return make_float4((m & 1u) ? f32x2::f2_lo(v.lo) : 0.f, (m & 2u) ? f32x2::f2_hi(v.lo) : 0.f,
                       (m & 4u) ? f32x2::f2_lo(v.hi) : 0.f, (m & 8u) ? f32x2::f2_hi(v.hi) : 0.f);
}

template <int R, int TY, int D, int K1, int K2, int U, int MINB>
__global__ void __launch_bounds__(TfCfg<R, TY, D>::THREADS, MINB)
    tti_fused_kernel(const __grid_constant__ CUtensorMap map_box,
                     const __grid_constant__ CUtensorMap map_nbox,
                     const __grid_constant__ CUtensorMap map_wlev,
                     const __grid_constant__ CUtensorMap map_cint,
                     const __grid_constant__ TtiArgs a, const __grid_constant__ AcousticInject inj,
                     const __grid_constant__ ReceiveArgs rec, int zchunk, int nzc) {
    using C = TfCfg<R, TY, D>;
    if (blockIdx.z >= gridDim.z - rec.slices) {
        chain_trigger();
        chain_wait();
        if (!(__ldcg(a.err) & DEV_ERR_NONFINITE))
            record_receivers(&rec, a.wave, 4, a.cur, 2 + a.cur, &a.L);
        return;
    }
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float *smem = reinterpret_cast<float *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~static_cast<uintptr_t>(127));
    float *ringP = smem;
    float *ringQ = ringP + C::NP * C::PSLOT;
    float *tmp = ringQ + C::NQ * C::QSLOT;  // [2 buffers][field][fx | fy]
    uint64_t *full = reinterpret_cast<uint64_t *>(tmp + 4 * C::TMP);  // one per P slot
    uint64_t *emptyP = full + C::NP;
    uint64_t *emptyQ = emptyP + C::NP;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(emptyQ + C::NQ);

    const int tid = threadIdx.x, lane = tid & 31;
    const int shot = blockIdx.z / nzc, chunk = blockIdx.z - shot * nzc;
    const int x0 = blockIdx.x * C::BX, y0 = blockIdx.y * C::BY;
    const int za = chunk * zchunk, zb = min(a.L.nz, za + zchunk);
    const int nplanes = zb - za + 4 * R;
    const int P0 = za - 2 * R;  // first arriving plane

    if (tid == 0) {
        for (int i = 0; i < C::NP; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&emptyP[i], C::WARPS);
        }
        for (int i = 0; i < C::NQ; ++i) mbar_init(&emptyQ[i], C::WARPS);
        fence_mbar_init();
        *abort_flag = 0;
    }
    __syncthreads();
    chain_wait();
    if (__ldcg(a.err) & DEV_ERR_NONFINITE) return;  // stopped by the divergence watchdog

    int issued = 0;
    if (tid >= C::CONSUMERS) {
        // Producer lane.  Ring P slot jj % NP: the plane's box of p and r;
        // ring Q slot jj % NQ: the n box at s = P0 + jj - R (from jj >= 2R)
        // and the update tiles at o = P0 + jj - 2R (from jj >= 4R).  One full
        // barrier covers both.
        if (lane == 0) {
            RingPos<C::NP> pp;
            RingPos<C::NQ> pq;
            for (int jj = 0; jj < nplanes && !*abort_flag; ++jj, pp.next(), pq.next()) {
                const int sp = pp.slot(jj), sq = pq.slot(jj);
                if ((jj >= C::NP && !mbar_wait_bounded(&emptyP[sp], pp.phase(jj) ^ 1u)) ||
                    (jj >= C::NQ && !mbar_wait_bounded(&emptyQ[sq], pq.phase(jj) ^ 1u))) {
                    if (!*abort_flag) atomicOr(a.err, DEV_ERR_TIMEOUT);
                    *abort_flag = 1;
                    break;
                }
                const bool qs = jj >= 2 * R, qo = jj >= 4 * R;
                mbar_arrive_expect_tx(&full[sp], C::PBYTES + (qs ? C::NBYTES : 0) +
                                                     (qo ? C::UBYTES : 0));
                tma_load_5d(ringP + sp * C::PSLOT, &map_box, &full[sp], x0 - 2 * C::RA,
                            y0 - 2 * R, P0 + jj, a.cur, 2 * shot);
                float *Q = ringQ + sq * C::QSLOT;
                if (qs)
                    tma_load_4d(Q, &map_nbox, &full[sp], x0 - C::RA, y0 - R, P0 + jj - R, 3);
                if (qo) {
                    const int o = P0 + jj - 2 * R;
                    tma_load_5d(Q + C::OFF_W, &map_wlev, &full[sp], x0, y0, o, 0, 2 * shot);
                    tma_load_4d(Q + C::OFF_C, &map_cint, &full[sp], x0, y0, o, 0);
                }
                issued = jj + 1;
            }
            chain_trigger();  // the next launch may move in (see acoustic.cu)
        }
    } else {
        // the thread's cross cell: float4 column qx in [-1, 16], row y in
        // [-R, BY + R); tile cells first, then the x strips, then the y strips
        const bool valid = tid < C::NCELL, tile = tid < C::TILE;
        int qx = tid % C::TX, y = tid / C::TX;
        bool to_x = tile, to_y = tile;  // whether f_x / f_y of the cell is needed
        if (!tile && tid < C::TILE + 2 * C::BY) {
            const int e = tid - C::TILE;
            qx = e < C::BY ? -1 : C::TX;
            y = e % C::BY;
            to_x = true;
        } else if (!tile && valid) {
            const int e = tid - C::TILE - 2 * C::BY;
            const int rr = e / C::TX;
            qx = e % C::TX;
            y = rr < R ? rr - R : C::BY + (rr - R);
            to_y = true;
        }
        const int cbox = (y + 2 * R) * C::PX + 4 * qx + 2 * C::RA;  // the cell in the p/r box
        const int cnb = (y + R) * C::NXW + 4 * qx + C::RA;          // the cell in the n box
        unsigned mask = 0u;  // elements inside the grid
        if (y0 + y >= 0 && y0 + y < a.L.ny)
            for (int e = 0; e < 4; ++e) {
                const int xe = x0 + 4 * qx + e;
                if (xe >= 0 && xe < a.L.nx) mask |= 1u << e;
            }
        const int gx = x0 + 4 * qx, gy = y0 + y;
        const bool ok = tile && gx < a.L.nxp && gy < a.L.ny;
        float dpx4[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            dpx4[i] = (tile && gx + i < a.L.nx) ? a.dpx[gx + i] : 0.f;
        const f2 dpx_lo = f2_pack(dpx4[0], dpx4[1]), dpx_hi = f2_pack(dpx4[2], dpx4[3]);
        const float dpy = ok ? a.dpy[gy] : 0.f;
        const f2 one2 = f2_splat(1.f);
        float *qn = a.wave + (int64_t)(4 * shot + 1 - a.cur) * a.L.vol +
                    (ok ? (int64_t)gy * a.L.nxp + gx : 0);
        const int q = y * C::BX + 4 * qx;

        Q4 acc1[2][2 * R], acc2[2][2 * R];
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int i = 0; i < 2 * R; ++i) acc1[f][i] = acc2[f][i] = Q4{0ull, 0ull};
        RingPos<C::NP> pp, ps;  // slots of the arriving plane and of plane s
        RingPos<C::NQ> pq;
#pragma unroll U
        for (int j = 0; j < nplanes; ++j) {
            const int sp = pp.slot(j), sq = pq.slot(j);
            const bool has_s = j >= 2 * R, has_o = j >= 4 * R;
            const int s = P0 + j - R, o = P0 + j - 2 * R;
            const float dz = has_o ? __ldg(a.dpz + o) : 0.f;
            const bool good = !*abort_flag && mbar_wait_bounded(&full[sp], pp.phase(j));
            const int ss = j >= R ? ps.slot(j - R) : 0;  // slot of plane s
            const float *Q = ringQ + sq * C::QSLOT;
            float *T = tmp + (j & 1) * 2 * C::TMP;

            // ---- stage 1: z-derivative feed; gradient and temporaries of plane s
            Q4 fz[2];
            if (good && valid) {
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const Q4 cv = lds_q4(ringP + sp * C::PSLOT + f * C::BOX + cbox);
                    dz_feed_q4<R, K1>(acc1[f], cv, a.t1[2]);
                    if (has_s) {
                        const float *B = ringP + ss * C::PSLOT + f * C::BOX + cbox;
                        const Q4 gxv = q4_from(dx4<R, C::RA, K1>(B - C::RA, a.t1[0]));
                        const Q4 gyv = dy_q4<R, K1>(B, C::PX, a.t1[1]);
                        const Q4 gzv = acc1[f][0];
                        const Q4 nx = lds_q4(Q + cnb), ny = lds_q4(Q + C::NBOX + cnb),
                                 nz = lds_q4(Q + 2 * C::NBOX + cnb);
                        const Q4 h = q4_fma(nz, gzv, q4_fma(nx, gxv, q4_mul(ny, gyv)));
                        Q4 o0, o1, o2;
                        if (f == 0) {  // f_i = D_i p - n_i h
                            const Q4 mh = q4_neg(h);
                            o0 = q4_fma(nx, mh, gxv);
                            o1 = q4_fma(ny, mh, gyv);
                            o2 = q4_fma(nz, mh, gzv);
                        } else {  // e_i = n_i h
                            o0 = q4_mul(nx, h);
                            o1 = q4_mul(ny, h);
                            o2 = q4_mul(nz, h);
                        }
                        // zero ghosts: temporaries outside the grid vanish
                        const unsigned m = s >= 0 && s < a.L.nz ? mask : 0u;
                        float *Tf = T + f * C::TMP;
                        if (to_x)
                            *reinterpret_cast<float4 *>(Tf + y * C::NXW + 4 * qx + C::RA) =
                                masked(o0, m);
                        if (to_y)
                            *reinterpret_cast<float4 *>(Tf + C::FX + (y + R) * C::BX + 4 * qx) =
                                masked(o1, m);
                        fz[f] = q4_from(masked(o2, m));
                    }
                    dz_shift_q4<R, K1>(acc1[f], cv, a.t1[2]);
                }
            }
            __syncwarp();
            // the temporaries of plane s are written (and those of two planes
            // before consumed); leave together after a failed wait
            if (consumers_or(C::CONSUMERS, !good)) {
                if (tid == 0) {
                    *abort_flag = 1;
                    atomicOr(a.err, DEV_ERR_TIMEOUT);
                }
                break;
            }
            // the box of plane s has been read by this warp (stage 2 reads
            // only temporaries and the Q slot)
            if (lane == 0 && j >= R) mbar_arrive(&emptyP[ss]);

            // ---- stage 2 (tile warps): outer derivatives of the temporaries
            //      of plane s feed the pending outputs; output o is complete
            if (tile && has_s) {
                Q4 H[2];
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    const float *Tf = T + f * C::TMP;
                    dz_feed_q4<R, K2>(acc2[f], fz[f], a.t2[2]);
                    const Q4 dxv =
                        q4_from(dx4<R, C::RA, K2>(Tf + y * C::NXW + 4 * qx, a.t2[0]));
                    const Q4 dyv =
                        dy_q4<R, K2>(Tf + C::FX + (y + R) * C::BX + 4 * qx, C::BX, a.t2[1]);
                    acc2[f][R] = q4_add(acc2[f][R], q4_add(dxv, dyv));
                    H[f] = acc2[f][0];
                    dz_shift_q4<R, K2>(acc2[f], fz[f], a.t2[2]);
                }
                if (has_o) {
                    const float *w = Q + C::OFF_W + q, *cc = Q + C::OFF_C + q;
                    const Q4 b = lds_q4(cc), av = lds_q4(cc + C::INT),
                             sv = lds_q4(cc + 2 * C::INT);
                    const f2 dyz = f2_splat(-(dpy + dz));
                    const Q4 keep = Q4{f2_fma(f2_sub(dyz, dpx_lo), b.lo, one2),
                                       f2_fma(f2_sub(dyz, dpx_hi), b.hi, one2)};
#pragma unroll
                    for (int f = 0; f < 2; ++f) {
                        const Q4 rhs = f == 0 ? q4_fma(av, H[0], q4_mul(sv, H[1]))
                                              : q4_fma(sv, H[0], H[1]);
                        const Q4 qc = lds_q4(w + (2 * f + a.cur) * C::INT);
                        const Q4 qm = lds_q4(w + (2 * f + 1 - a.cur) * C::INT);
                        const Q4 v = q4_fma(b, rhs, q4_fma(keep, q4_sub(qc, qm), qc));
                        if (ok)
                            *reinterpret_cast<ulonglong2 *>(qn + 2 * f * a.L.vol +
                                                            (int64_t)o * a.L.plane) =
                                make_ulonglong2(v.lo, v.hi);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&emptyQ[sq]);
            pp.next();
            pq.next();
            if (j >= R) ps.next();
        }
    }
    __syncthreads();
    if (*abort_flag && tid == C::CONSUMERS) {
        for (int jj = issued - C::NP; jj < issued; ++jj)
            if (jj >= 0)
                mbar_wait_bounded(&full[jj % C::NP], (uint32_t)((jj / C::NP) & 1), 200000000ull);
    }
    if (inj.nsrc > 0 && tid == 0 && !*abort_flag)
        tti_inject_column<C::BX, C::BY>(&a, &inj, zchunk, nzc);
}

struct FusedInfo {
    const void *fn;
    size_t smem;
    int px, py, nxw, nyh, by, threads;
    float launch, lat, thr, warm;  // cost constants (see acoustic.cu)
};

template <int R, int TY, int D, int U, int MINB>
FusedInfo fused_info_t(int stag, float launch, float lat, float thr, float warm) {
    using C = TfCfg<R, TY, D>;
    return FusedInfo{stag ? (const void *)&tti_fused_kernel<R, TY, D, 1, -1, U, MINB>
                          : (const void *)&tti_fused_kernel<R, TY, D, 0, 0, U, MINB>,
                     C::SMEM, C::PX,  C::PY, C::NXW, C::NYH, C::BY, C::THREADS,
                     launch,  lat,    thr,   warm};
}

// Built-in and configuration 1: 64 x 16 tiles, one CTA per SM (R <= 2; 1.38x the
// tile's gradients); configuration 0: 64 x 8 tiles, two CTAs (1.63x).  so 4, us per
// step: 96^3 23.0 and 26.7, 256^3 204 and 248, 384^3 598 and 711, 512^3 1430
// and 1664.  The costs are fitted to 13 problems.
bool fused_info(int radius, int stag, int config, FusedInfo *out) {
    const bool small = config == 0;
    switch (radius) {
        case 1:
            *out = small ? fused_info_t<1, 8, 1, 2, 2>(stag, 4.1f, 1.05f, 0.60f, 0.59f)
                         : fused_info_t<1, 16, 1, 2, 1>(stag, 2.2f, 1.30f, 0.05f, 0.72f);
            return true;
        case 2:
            *out = small ? fused_info_t<2, 8, 1, 2, 2>(stag, 4.1f, 1.18f, 0.715f, 0.59f)
                         : fused_info_t<2, 16, 1, 2, 1>(stag, 2.2f, 1.46f, 0.05f, 0.72f);
            return true;
        case 4:
            *out = fused_info_t<4, 8, 1, 1, 1>(stag, 3.f, 2.5f, 1.0f, 0.55f);
            return true;
        default: return false;
    }
}

}  // namespace

bool tti_fused_supported(int radius) {
    FusedInfo in;
    return fused_info(radius, 0, -1, &in);
}

// Chunk count of a fused step and its estimated time.
static fd_status fused_choice(const FusedInfo &in, int radius, const WaveLayout &L, int nshots,
                              PlanChoice *c) {
    FD_TRY(raise_smem_limit(in.fn, in.smem));
    int dev = 0, nsm = 0, per_sm = 0;
    FD_CUDA_TRY(cudaGetDevice(&dev));
    FD_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    FD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, in.fn, in.threads, in.smem));
    if (per_sm < 1) return set_error(FD_ERR_CUDA, "fused TTI kernel does not fit on an SM");
    // 4R warm-up planes, the first half of which only feed the z pipeline
    const PlanEntry e{64, in.by, 0, per_sm, in.launch, in.lat, in.thr,
                      in.warm * 4.0 * radius, INT_MAX, 0, false};
    *c = choose_plan(&e, 1, -1, L.nx, L.ny, L.nz, nshots, nsm);
    if (c->entry < 0) return set_error(FD_ERR_ARG, "grid too large for the fused TTI launch");
    return FD_OK;
}

fd_status tti_fused_time(int radius, int stag, const WaveLayout &L, int nshots, double *us) {
    FusedInfo in;
    if (!fused_info(radius, stag, -1, &in))
        return set_error(FD_ERR_ARG, "the fused TTI scheme covers space orders up to 8");
    PlanChoice c;
    FD_TRY(fused_choice(in, radius, L, nshots, &c));
    *us = c.us;
    return FD_OK;
}

fd_status tti_fused_plan(int radius, int stag, const WaveLayout &L, int nshots, float *wave,
                         const float *coef, TtiPlan *plan, int config) {
    FusedInfo in;
    if (!fused_info(radius, stag, config, &in))
        return set_error(FD_ERR_ARG, "the fused TTI scheme covers space orders up to 8");
    const uint32_t bx = 64, by = in.by;
    const int ntx = (L.nx + bx - 1) / bx, nty = (L.ny + by - 1) / by;
    PlanChoice c;
    FD_TRY(fused_choice(in, radius, L, nshots, &c));
    plan->radius = radius;
    plan->stag = stag ? 1 : 0;
    plan->scheme = kTtiFused;
    plan->p1.fn = in.fn;
    plan->p1.grid = dim3(ntx, nty, nshots * c.nzc);
    plan->p1.block = dim3(in.threads, 1, 1);
    plan->p1.smem = in.smem;
    plan->p1.zchunk = c.zchunk;
    plan->p1.nzc = c.nzc;
    plan->p1.est_us = c.us;
    const uint64_t sy = (uint64_t)L.nxp * 4, sz = (uint64_t)L.plane * 4, sv = (uint64_t)L.vol * 4;
    const uint64_t wdim[5] = {(uint64_t)L.nx, (uint64_t)L.ny, (uint64_t)L.nz, 2, 2ull * nshots};
    const uint64_t wstr[4] = {sy, sz, sv, 2 * sv};
    const uint32_t box[5] = {(uint32_t)in.px, (uint32_t)in.py, 1, 1, 2};
    const uint32_t lev[5] = {bx, by, 1, 2, 2};
    FD_TRY(make_tensor_map_5d(&plan->map_fbox, wave, wdim, wstr, box));
    FD_TRY(make_tensor_map_5d(&plan->map_wlev, wave, wdim, wstr, lev));
    FD_TRY(make_tensor_map_4d(&plan->map_fnbox, coef, L.nx, L.ny, L.nz, 6, sy, sz, sv, in.nxw,
                              in.nyh, 1, 3));
    return make_tensor_map_4d(&plan->map_c2, coef, L.nx, L.ny, L.nz, 6, sy, sz, sv, bx, by, 1, 3);
}

fd_status tti_fused_launch(const TtiPlan &plan, const TtiArgs &a, cudaStream_t stream,
                           const AcousticInject &inj, const ReceiveArgs &receive) {
    ReceiveArgs rec = receive;
    dim3 grid = plan.p1.grid;
    rec.slices = 0;
    if (rec.nrec > 0) {
        if (grid.z >= 65535) return set_error(FD_ERR_ARG, "no grid slice left for receivers");
        rec.slices = receive_slices(rec, grid.x, grid.y, plan.p1.block.x);
        if ((int64_t)grid.z + rec.slices > 65535) rec.slices = 65535 - grid.z;
        grid.z += rec.slices;
    }
    int zchunk = plan.p1.zchunk, nzc = plan.p1.nzc;
    void *params[] = {(void *)&plan.map_fbox, (void *)&plan.map_fnbox, (void *)&plan.map_wlev,
                      (void *)&plan.map_c2,   (void *)&a,              (void *)&inj,
                      (void *)&rec,           (void *)&zchunk,         (void *)&nzc};
    FD_CUDA_TRY(launch_chained(plan.p1.fn, grid, plan.p1.block, params, plan.p1.smem, stream));
    note_launch(stream);
    return FD_OK;
}

}  // namespace fdsweep
