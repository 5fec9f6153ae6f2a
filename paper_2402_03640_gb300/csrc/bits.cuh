// Bit-matrix helper shared by the evaluation kernels (k_eval.cu, k_dense.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace msat {

// Transpose of a 32 x 32 bit matrix held one row per lane (bit c of lane
// r's word is entry (r, c)): five butterfly rounds, each exchanging with
// lane ^ j the half of the bits whose position has bit j set; afterwards
// bit r of lane l's word is entry (r, l).
__device__ __forceinline__ uint32_t transpose_bits32(uint32_t x, int lane) {
    uint32_t m = 0x0000FFFFu;
#pragma unroll
    for (int j = 16; j >= 1; j >>= 1, m ^= m << j) {
        const uint32_t t = __shfl_xor_sync(0xffffffffu, x, j);
        x = (lane & j) ? (((t >> j) & m) | (x & ~m)) : ((x & m) | ((t & m) << j));
    }
    return x;
}

}  // namespace msat
