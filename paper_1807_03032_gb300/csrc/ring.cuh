// ring.cuh -- position in the shared-memory rings of the z-marching kernels, and
// how their consumer threads leave the plane loop when a wait ran out.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#include "common.cuh"
#define FD_RING __device__ __forceinline__
#else  // host build, for tests
#define FD_RING inline
#endif

namespace fdsweep {

// Position in a ring of N stages: from the plane index where N is a power of
// two (constant stage addresses in an unrolled loop), counted otherwise.
template <int N>
struct RingPos {
    int s = 0;
    uint32_t ph = 0;
    static constexpr bool POW2 = (N & (N - 1)) == 0;
    FD_RING int slot(int j) const { return POW2 ? j % N : s; }
    FD_RING uint32_t phase(int j) const { return POW2 ? (uint32_t)(j / N) & 1u : ph; }
    FD_RING void next() {
        if (POW2) return;
        if (++s == N) {
            s = 0;
            ph ^= 1u;
        }
    }
};

// The lanes of a warp need not give up a wait in the same iteration of the
// plane loop: each looks at the clock and at the block's abort mark for itself.
// A lane that is past its wait in iteration j still gets to the __syncwarp at
// the end of j, so the lanes that leave in j meet it there (it would wait for
// ever otherwise); it then sees the mark and leaves in j + 1, meeting nobody.
// *left: 1 + the parity of the iteration in which the first lanes of the warp
// left, 0 before.
template <class Sync>
FD_RING void meet_remaining_lanes(volatile unsigned char *left, int j, Sync sync) {
    if (*left == 1 + ((j + 1) & 1)) return;  // the others left in j - 1
    *left = (unsigned char)(1 + (j & 1));
    sync();
}

// The words behind a block's abort flag: one byte per consumer warp.
constexpr int kMaxRingWarps = 12;

#ifdef __CUDACC__
__device__ __forceinline__ void init_ring_abort(volatile int *abort_flag) {
    for (int i = 0; i < 1 + kMaxRingWarps / 4; ++i) abort_flag[i] = 0;
}

// A consumer thread leaves the plane loop in iteration j: the block is marked
// as aborted and the error reported.
__device__ __forceinline__ void leave_ring(volatile int *abort_flag, int j, unsigned int *err) {
    *abort_flag = 1;
    atomicOr(err, DEV_ERR_TIMEOUT);
    meet_remaining_lanes(
        reinterpret_cast<volatile unsigned char *>(abort_flag + 1) + (threadIdx.x >> 5), j,
        [] { __syncwarp(); });
}
#endif

}  // namespace fdsweep
