// lbp_codes.cuh -- A3 arithmetic shared by the feature kernels (Section 2.4, Eq. 2).
#pragma once

#include <stdint.h>

namespace rgbd {

// ---------------------------------------------------------------------------------------
// A3 helper: byte-SIMD "a > b" (or >=) on four packed pixels.  cb = (b & 0x7f7f7f7f) + 1 per
// byte for the strict test, without the +1 for >=.  Result: 0x80 in each byte where it holds.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cmp_msb(uint32_t a, uint32_t b, uint32_t cb) {
    const uint32_t d = (a | 0x80808080u) - cb;  // per byte: low 7 bits of a vs b, no borrows
    return ((a & ~b) | (~(a ^ b) & d)) & 0x80808080u;
}

}  // namespace rgbd
