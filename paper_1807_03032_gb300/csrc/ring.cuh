// ring.cuh -- position in the shared-memory rings of the z-marching kernels.
#pragma once

#include <stdint.h>

namespace fdsweep {

// Position in a ring of N stages: from the plane index where N is a power of
// two (constant stage addresses in an unrolled loop), counted otherwise.
template <int N>
struct RingPos {
    int s = 0;
    uint32_t ph = 0;
    static constexpr bool POW2 = (N & (N - 1)) == 0;
    __device__ __forceinline__ int slot(int j) const { return POW2 ? j % N : s; }
    __device__ __forceinline__ uint32_t phase(int j) const {
        return POW2 ? (uint32_t)(j / N) & 1u : ph;
    }
    __device__ __forceinline__ void next() {
        if (POW2) return;
        if (++s == N) {
            s = 0;
            ph ^= 1u;
        }
    }
};

}  // namespace fdsweep
