// Order of a path's share of the receiver / sender state along the contraction axis.
#pragma once
#include <stdint.h>

namespace sobek {

// Position of (radial index q, multiplicity u) in the K * c values of a path.  zq = 1: q-major, q * c + u (what every producer but the
// moment stream writes, and the channelwise kernels read).  zq = 2, 4, 8: runs of 2 zq radial indices, in a run its even ones, then
// its odd ones, multiplicity by multiplicity with the zq radial indices of one multiplicity side by side: what one lane of the moment
// stream's read-out holds is one store.  A last run of fewer than 2 zq radial indices stays q-major.
__host__ __device__ inline int32_t state_pos(int zq, int K, int c, int q, int u) {
    const int q0 = q / (2 * zq) * (2 * zq), j = q - q0;
    return q0 * c + (q0 + 2 * zq <= K ? ((j & 1) * c + u) * zq + (j >> 1) : j * c + u);
}

}  // namespace sobek
