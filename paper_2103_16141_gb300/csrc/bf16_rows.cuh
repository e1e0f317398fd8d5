// The 32-bit words of the BF16 dense rows: the even entry's BF16 bits in the
// lower half, the odd entry's upper half chosen such that the whole word, read
// as FP32, is the odd entry's stored value. Host code can include this file.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define SIVF_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define SIVF_HOST_DEVICE inline
#endif

namespace sivf {

// Upper half of the word with lower half `low` that is nearest, in the order of
// FP32 bits, to the value with bits u_bits (positive; taken as at least the
// smallest normal): within half of the upper half's step, as rounding to BF16 is
// (2^-8 relative).
SIVF_HOST_DEVICE uint16_t odd_upper_half(uint32_t u_bits, uint16_t low) {
    const uint32_t u = u_bits > 0x00800000u ? u_bits : 0x00800000u;
    return (uint16_t)((u - low + 0x8000u) >> 16);
}

}  // namespace sivf
