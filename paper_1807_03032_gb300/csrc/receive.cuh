// receive.cuh -- receiver interpolation by the extra blocks of a stencil
// launch (Eq. interp), with the operations of the sparse kernel.
#pragma once

#include "kernels.cuh"

namespace fdsweep {

// z slices of receiver blocks behind a grid of ntx x nty columns: one
// receiver per thread.
inline int receive_slices(const ReceiveArgs &r, int ntx, int nty, int threads) {
    const int64_t blocks = ((int64_t)r.nshots * r.nrec + threads - 1) / threads;
    const int64_t per = (int64_t)ntx * nty;
    return (int)((blocks + per - 1) / per);
}

// rec[n][i] = sum_c w_c u^n(node_c), or of (u + u2) / 2.  Reads through L2:
// the launch may overlap the one that wrote u^n.
static __device__ __noinline__ void record_receivers(const ReceiveArgs *r, const float *wave, int lps,
                                              int lev, int lev2, const WaveLayout *L) {
    const int n = r->step + (r->step_base ? *r->step_base : 0);
    if (n < 0 || n >= r->nt) return;
    const int64_t total = (int64_t)r->nshots * r->nrec;
    const int64_t per = (int64_t)gridDim.x * gridDim.y;
    const int64_t block = (blockIdx.z - (gridDim.z - r->slices)) * per +
                          (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
    for (int64_t g = block * blockDim.x + threadIdx.x; g < total;
         g += r->slices * per * blockDim.x) {
        const int s = (int)(g / r->nrec);
        const int i = (int)(g - (int64_t)s * r->nrec);
        const SparsePoint p = r->tab[g];
        const float *u = wave + (int64_t)(s * lps + lev) * L->vol + p.base;
        const float *u2 = wave + (int64_t)(s * lps + lev2) * L->vol + p.base;
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int64_t o = ((c & 1) ? 1 : 0) + ((c & 2) ? L->nxp : 0) + ((c & 4) ? L->plane : 0);
            v[c] = r->mean ? 0.5f * (__ldcg(u + o) + __ldcg(u2 + o)) : __ldcg(u + o);
        }
        float acc = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float wx = (c & 1) ? p.fx : 1.f - p.fx;
            const float wy = (c & 2) ? p.fy : 1.f - p.fy;
            const float wz = (c & 4) ? p.fz : 1.f - p.fz;
            acc = fmaf(wx * wy * wz, v[c], acc);
        }
        r->out[((int64_t)s * r->nt + n) * r->nrec + i] = acc;
    }
}

}  // namespace fdsweep
