// sparse.cu -- K3/K4: sparse source injection and receiver interpolation.
//
// Trilinear interpolation (Eq. interp, the tensor product of the 1-D linear
// weights 1 - frac and frac along x, y and z) gathers
//   rec[n][i] = sum_c w_c u^n(node_c),
// and injection, its adjoint (Listing finject), scatters
//   u^{n+1}(node_c) += w_c * b(node_c) * q[n],  b = dt^2 / (m + damp dt/2),
// with atomicAdd so that sources sharing a node accumulate (injection is a
// reduction).  One launch does both: receiver threads first, then one thread
// per (source, corner).
#include "kernels.cuh"

namespace fdsweep {
namespace {

__device__ __forceinline__ float corner_weight(const SparsePoint &p, int c) {
    const float wx = (c & 1) ? p.fx : 1.f - p.fx;
    const float wy = (c & 2) ? p.fy : 1.f - p.fy;
    const float wz = (c & 4) ? p.fz : 1.f - p.fz;
    return wx * wy * wz;
}

__device__ __forceinline__ int64_t corner_offset(const SparsePoint &p, int c, const WaveLayout &L) {
    return (int64_t)p.base + ((c & 1) ? 1 : 0) + ((c & 2) ? L.nxp : 0) + ((c & 4) ? L.plane : 0);
}

// Threads [0, nrec_total) interpolate receivers (nrec_total = 0 when only
// injecting); the following nshots*nsrc*8 threads inject.
__global__ void sparse_kernel(const SparseArgs a, int step, int do_inject, int64_t nrec_total) {
    chain_wait();
    chain_trigger();
    const int n = step + (a.step_base ? *a.step_base : 0);
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid < nrec_total) {
        const int ro = a.rec_t0 + a.rec_dt * n;
        if (ro < 0 || ro >= a.nt) return;
        const int s = (int)(gid / a.nrec);
        const int i = (int)(gid - (int64_t)s * a.nrec);
        const SparsePoint p = a.rec_tab[gid];
        const float *u = a.wave + (int64_t)(s * a.fields_per_shot + a.rec_level) * a.L.vol;
        float acc = 0.f;
        if (a.rec_mean) {  // interpolate (u + u2) / 2
            const float *u2 = a.wave + (int64_t)(s * a.fields_per_shot + a.rec_level2) * a.L.vol;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int64_t o = corner_offset(p, c, a.L);
                acc = fmaf(corner_weight(p, c), 0.5f * (__ldcg(u + o) + __ldcg(u2 + o)), acc);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c)
                acc = fmaf(corner_weight(p, c), __ldcg(u + corner_offset(p, c, a.L)), acc);
        }
        a.rec_out[((int64_t)s * a.nt + ro) * a.nrec + i] = acc;
        return;
    }
    if (!do_inject) return;
    const int64_t k = gid - nrec_total;
    if (k >= (int64_t)a.nshots * a.nsrc * 8) return;
    const int c = (int)(k & 7);
    const int64_t ps = k >> 3;  // (shot, source)
    const int s = (int)(ps / a.nsrc);
    const int isrc = (int)(ps - (int64_t)s * a.nsrc);
    const int qi = a.inj_t0 + a.inj_dt * n;
    if (qi < 0 || qi >= a.nt) return;
    const SparsePoint p = a.src_tab[ps];
    const int64_t off = corner_offset(p, c, a.L);
    const float q = a.src_wav[((int64_t)s * a.nt + qi) * a.nsrc + isrc];
    const float val = corner_weight(p, c) * __ldg(a.bcoef + off) * q;
    atomicAdd(a.wave + (int64_t)(s * a.fields_per_shot + a.inj_level0) * a.L.vol + off, val);
    if (a.inj_level1 >= 0)
        atomicAdd(a.wave + (int64_t)(s * a.fields_per_shot + a.inj_level1) * a.L.vol + off, val);
}

__global__ void bump_kernel(int *counter, int by) { *counter += by; }

template <int V>
__device__ __forceinline__ void vec_load(float (&d)[V], const float *s) {
    static_assert(V == 4 || V == 2, "vectors of 2 or 4 floats");
    if (V == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(s);
        d[0] = t.x, d[1] = t.y, d[2 % V] = t.z, d[3 % V] = t.w;
    } else {
        const float2 t = *reinterpret_cast<const float2 *>(s);
        d[0] = t.x, d[1] = t.y;
    }
}

template <int V>
__device__ __forceinline__ void vec_store(float *d, const float (&s)[V]) {
    if (V == 4)
        *reinterpret_cast<float4 *>(d) = make_float4(s[0], s[1], s[2 % V], s[3 % V]);
    else
        *reinterpret_cast<float2 *>(d) = make_float2(s[0], s[1]);
}

// g += sum over steps j and shots b of w_jb (u_jb - 2 u_jb' + u_jb''), step j
// outside and shot b inside (the order of one launch per step), see
// grad_accumulate.  A stream kernel: the window u', u of every shot stays in
// registers, so a step reads one level of u and of w and g is read and
// written once in `steps` steps: 8 + 8/steps + 8/(nb steps) bytes per
// shot-point instead of 16 + 8/nb.  V floats per thread and NB >= nb shots
// trade the width of the loads against the registers of the window (2 NB V).
// 128^3, 239 steps, whole gradient: 4 shots 19.7 ms with one launch per step
// and 15.4 in eights, 8 shots 34.1 and 26.7.  Two blocks of 128 registers per
// SM and no unrolling: with unroll 2 (255 registers) 16.1 and 27.1 ms, and a
// 16-shot kernel of single floats was slower than two batches of 8 (29.4 ms
// against 27.1 for 119 steps).
template <int V, int NB>
__global__ void __launch_bounds__(256, 2) grad_steps_kernel(const GradArgs a) {
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V; i < a.vol;
         i += (int64_t)gridDim.x * blockDim.x * V) {
        float o[V], p[NB][V], q[NB][V];
        vec_load<V>(o, a.grad + i);
        const float *u = a.u + i;
#pragma unroll
        for (int b = 0; b < NB; ++b)
            if (b < a.nb) {
                vec_load<V>(p[b], u + b * a.u_stride);
                vec_load<V>(q[b], u + b * a.u_stride - a.vol);
            }
        u -= 2 * a.vol;
        int lev = a.w_level;
#pragma unroll 1
        for (int j = 0; j < a.steps; ++j) {
            const float *w = a.w + lev * a.vol + i;
            float x[NB][V], r[NB][V];
#pragma unroll
            for (int b = 0; b < NB; ++b)
                if (b < a.nb) {
                    vec_load<V>(x[b], w + b * a.w_stride);
                    vec_load<V>(r[b], u + b * a.u_stride);
                }
#pragma unroll
            for (int b = 0; b < NB; ++b)
                if (b < a.nb)
#pragma unroll
                    for (int e = 0; e < V; ++e) {
                        o[e] = fmaf(x[b][e], p[b][e] - 2.f * q[b][e] + r[b][e], o[e]);
                        p[b][e] = q[b][e];
                        q[b][e] = r[b][e];
                    }
            u -= a.vol;
            if (++lev == a.w_levels) lev = 0;
        }
        vec_store<V>(a.grad + i, o);
    }
}

__global__ void scale_kernel(float *__restrict__ f, float s, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        f[i] *= s;
}

int stream_grid(int64_t n, int threads) {
    int dev = 0, nsm = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int64_t b = (n + threads - 1) / threads;
    if (b > (int64_t)nsm * 16) b = (int64_t)nsm * 16;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

fd_status sparse_launch(const SparseArgs &a, int step, bool do_inject, bool do_interp,
                        cudaStream_t stream) {
    const int64_t nrec_total = do_interp ? (int64_t)a.nshots * a.nrec : 0;
    const int64_t ninj = do_inject ? (int64_t)a.nshots * a.nsrc * 8 : 0;
    const int64_t total = nrec_total + ninj;
    if (total == 0) return FD_OK;
    const int threads = 256;
    const int64_t blocks = (total + threads - 1) / threads;
    int inject = do_inject ? 1 : 0;
    int64_t nrec = nrec_total;
    void *params[] = {(void *)&a, (void *)&step, (void *)&inject, (void *)&nrec};
    FD_CUDA_TRY(launch_chained((const void *)&sparse_kernel, dim3((unsigned)blocks), dim3(threads),
                               params, 0, stream));
    note_launch(stream);
    return FD_OK;
}

fd_status bump_counter(int *counter, int by, cudaStream_t stream) {
    bump_kernel<<<1, 1, 0, stream>>>(counter, by);
    FD_CUDA_TRY(cudaGetLastError());
    note_launch(stream);
    return FD_OK;
}

fd_status grad_accumulate(const GradArgs &a, cudaStream_t stream) {
    if (a.vol % 4 || a.w_stride % 4 || a.u_stride % 4)
        return set_error(FD_ERR_ARG, "grad_accumulate: sizes not multiples of 4");
    if (a.nb > kGradShots)
        return set_error(FD_ERR_ARG, "grad_accumulate: %d shots in a batch", a.nb);
    if (a.nb <= 4)
        grad_steps_kernel<4, 4><<<stream_grid(a.vol / 4, 256), 256, 0, stream>>>(a);
    else
        grad_steps_kernel<2, kGradShots><<<stream_grid(a.vol / 2, 256), 256, 0, stream>>>(a);
    FD_CUDA_TRY(cudaGetLastError());
    note_launch(stream);
    return FD_OK;
}

fd_status scale_field(float *f, float s, int64_t n, cudaStream_t stream) {
    scale_kernel<<<stream_grid(n, 256), 256, 0, stream>>>(f, s, n);
    FD_CUDA_TRY(cudaGetLastError());
    note_launch(stream);
    return FD_OK;
}

}  // namespace fdsweep
