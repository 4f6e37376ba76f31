// resample.cuh -- A1 arithmetic shared by the kernels that resample face rects (Section 2.1, Eq. 1):
// Q16.16 source coordinates, their clamped taps, and the bilinear grey sample.
#pragma once

#include <stdint.h>

namespace rgbd {

// ---------------------------------------------------------------------------------------
// A1 helpers: Q16.16 source coordinates, pixel centre to pixel centre.
// ---------------------------------------------------------------------------------------

// origin + (i + 1/2) * len / out_len - 1/2 in Q16.16 (len > 0, so the quotient is >= 0).
__device__ __forceinline__ int64_t rect_coord_q16(int origin, int len, int out_len, int i) {
    uint64_t num = (uint64_t)(2 * i + 1) * (uint64_t)len * 65536ull;
    return (int64_t)origin * 65536 + (int64_t)(num / (2ull * (uint64_t)out_len)) - 32768;
}

// Packs the taps of one coordinate: .x = a | (b - a) << 16 | frac << 24 (bilinear: clamped
// taps a = floor, b = floor + 1, Q8 fraction), .y = the clamped nearest index.
__device__ __forceinline__ uint2 make_tap(int64_t q, int lim) {
    const int64_t f0 = q >> 16;  // floor (arithmetic shift)
    const int frac = (int)((q >> 8) & 255);
    const int64_t nn = (q + 32768) >> 16;
    const int64_t hi = (int64_t)lim - 1;
    const int a = (int)(f0 < 0 ? 0 : (f0 > hi ? hi : f0));
    const int b = (int)(f0 + 1 < 0 ? 0 : (f0 + 1 > hi ? hi : f0 + 1));
    const int n = (int)(nn < 0 ? 0 : (nn > hi ? hi : nn));
    return make_uint2((uint32_t)a | ((uint32_t)(b - a) << 16) | ((uint32_t)frac << 24), (uint32_t)n);
}

// Bilinear grey sample with Q8 weights (they sum to 2^16), rounded half up.
__device__ __forceinline__ uint32_t bilerp(const uint8_t* img, int W, uint32_t cx, uint32_t ry) {
    const uint32_t xa = cx & 0xFFFFu, dx = (cx >> 16) & 1u, fx = cx >> 24;
    const uint32_t ya = ry & 0xFFFFu, dy = (ry >> 16) & 1u, fy = ry >> 24;
    const uint8_t* r0 = img + (size_t)ya * W + xa;
    const uint8_t* r1 = r0 + (size_t)dy * W;
    const uint32_t p00 = __ldg(r0), p01 = __ldg(r0 + dx);
    const uint32_t p10 = __ldg(r1), p11 = __ldg(r1 + dx);
    const uint32_t acc = (256u - fy) * ((256u - fx) * p00 + fx * p01) + fy * ((256u - fx) * p10 + fx * p11);
    return (acc + 32768u) >> 16;
}

}  // namespace rgbd
