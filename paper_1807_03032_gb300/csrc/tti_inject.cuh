// tti_inject.cuh -- source injection by the TTI kernels that write p^{n+1}
// and r^{n+1}.
#pragma once

#include "kernels.cuh"

namespace fdsweep {
namespace tti {

// Source injection into p^{n+1} and r^{n+1} by the CTA that wrote a source's
// corners, after its column is complete (see inject_column in acoustic.cu):
// thread 0, sources in order, with the sparse kernel's operations.
template <int BX, int BY>
static __device__ __noinline__ void tti_inject_column(const TtiArgs *a, const AcousticInject *inj,
                                               int zchunk, int nzc) {
    const int n = inj->step + (inj->step_base ? *inj->step_base : 0);
    if (n < 0 || n >= inj->nt) return;
    const int shot = blockIdx.z / nzc;
    const int za = (blockIdx.z - shot * nzc) * zchunk;
    const int zb = min(a->L.nz, za + zchunk);
    const int x0 = blockIdx.x * BX, y0 = blockIdx.y * BY;
    const int x1 = min(x0 + BX, a->L.nx), y1 = min(y0 + BY, a->L.ny);
    float *p = a->wave + (int64_t)(4 * shot + 1 - a->cur) * a->L.vol;
    float *r = p + 2 * a->L.vol;
    for (int s = 0; s < inj->nsrc; ++s) {
        const SparsePoint t = inj->src_tab[shot * inj->nsrc + s];
        const int i = (int)(t.base % (uint32_t)a->L.nxp);
        const int j = (int)((t.base / (uint32_t)a->L.nxp) % (uint32_t)a->L.ny);
        const int k = (int)(t.base / (uint32_t)a->L.plane);
        if (i + 1 < x0 || i >= x1 || j + 1 < y0 || j >= y1 || k + 1 < za || k >= zb) continue;
        const float q = inj->src_wav[((int64_t)shot * inj->nt + n) * inj->nsrc + s];
        for (int c = 0; c < 8; ++c) {
            const int ci = i + (c & 1), cj = j + ((c >> 1) & 1), ck = k + ((c >> 2) & 1);
            if (ci < x0 || ci >= x1 || cj < y0 || cj >= y1 || ck < za || ck >= zb) continue;
            const float wx = (c & 1) ? t.fx : __fsub_rn(1.f, t.fx);
            const float wy = (c & 2) ? t.fy : __fsub_rn(1.f, t.fy);
            const float wz = (c & 4) ? t.fz : __fsub_rn(1.f, t.fz);
            const int64_t off = (int64_t)ck * a->L.plane + (int64_t)cj * a->L.nxp + ci;
            const float val =
                __fmul_rn(__fmul_rn(__fmul_rn(__fmul_rn(wx, wy), wz), a->bcoef[off]), q);
            p[off] = __fadd_rn(p[off], val);
            r[off] = __fadd_rn(r[off], val);
        }
    }
}

}  // namespace tti
}  // namespace fdsweep
