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

// Taps of the column pair (2 i, 2 i + 1) of a crop `out` columns wide (past its edge: the last
// column again).  .c in general: {tap, 0, tap, 0}; with windows (rects at most twice as wide as the
// crop, frame rows word-aligned and at least 8 bytes: `windows` below): .x / .z = byte selector (o, o + dx, o) of each
// column in the aligned 8-byte window that starts at byte wb (kept above .x's selector), .y / .w =
// byte weights (255 - fx, fx, 1, 0), so that a permute and a 4-way dot product give
// 256 p(o) + fx (p(o + dx) - p(o)).  Neighbouring taps are at most 2 apart, so every offset is at
// most 7.  Rects no wider than the crop (WIN_GROUP): taps of the group's four columns are at most 3
// apart, and both pairs' selectors count from the window of the group's first column.
// .nearest: the two nearest columns.
struct PairTaps {
    uint4 c;
    uint32_t nearest;
};
enum { WIN_NONE = 0, WIN_PAIR = 1, WIN_GROUP = 2 };
__device__ __forceinline__ int windows(int rect_w, int out, const uint8_t* grey, int W) {
    if (rect_w > 2 * out || (W & 3) != 0 || W < 8 || (reinterpret_cast<size_t>(grey) & 3) != 0) return WIN_NONE;
    return rect_w <= out ? WIN_GROUP : WIN_PAIR;
}
__device__ __forceinline__ PairTaps make_pair_taps(int x, int w, int out, int i, int W, int win) {
    const uint2 t0 = make_tap(rect_coord_q16(x, w, out, min(2 * i, out - 1)), W);
    const uint2 t1 = make_tap(rect_coord_q16(x, w, out, min(2 * i + 1, out - 1)), W);
    PairTaps p;
    p.nearest = t0.y | (t1.y << 16);
    if (win == WIN_NONE) {
        p.c = make_uint4(t0.x, 0u, t1.x, 0u);
        return p;
    }
    const uint32_t first = win == WIN_GROUP && (i & 1) ? make_tap(rect_coord_q16(x, w, out, min(2 * i - 2, out - 1)), W).x
                                                       : t0.x;
    const uint32_t wb = min(first & 0xFFFCu, (uint32_t)W - 8u);
    auto sel = [&](uint32_t t) {
        const uint32_t o = (t & 0xFFFFu) - wb, od = o + ((t >> 16) & 1u);
        return o | (od << 4) | (o << 8);
    };
    auto wts = [](uint32_t t) { return (255u - (t >> 24)) | ((t >> 24) << 8) | (1u << 16); };
    p.c = make_uint4(sel(t0.x) | (wb << 16), wts(t0.x), sel(t1.x), wts(t1.x));
    return p;
}

// The taps of a crop row as offsets into the frame (H, W <= 65535): the two grey rows, the depth
// row, and the Q8 fraction.
__device__ __forceinline__ uint4 make_row_taps(int y, int h, int out, int v, int H, int W) {
    const uint2 t = make_tap(rect_coord_q16(y, h, out, v), H);
    const uint32_t ya = t.x & 0xFFFFu;
    return make_uint4(ya * (uint32_t)W, (ya + ((t.x >> 16) & 1u)) * (uint32_t)W, t.y * (uint32_t)W, t.x >> 24);
}

// Four neighbouring crop pixels from the taps of their two column pairs and of their row: grey in
// the bytes of gw, depth in the halves of d01 and d23.
__device__ __forceinline__ void sample_group(const uint8_t* gsrc, const uint16_t* dsrc, uint4 row,
                                             const PairTaps (&pair)[2], int win, uint32_t& gw, uint32_t& d01,
                                             uint32_t& d23) {
    const uint32_t fy = row.w;
    const uint8_t* g0 = gsrc + row.x;
    const uint8_t* g1 = gsrc + row.y;
    const uint16_t* drow = dsrc + row.z;
    uint32_t acc[4], dv[4];  // acc: the grey value in byte 2
    uint32_t a0 = 0, a1 = 0, b0 = 0, b1 = 0;
#pragma unroll
    for (int e2 = 0; e2 < 2; ++e2) {
        const uint4 c = pair[e2].c;
        if (win) {
            if (e2 == 0 || win == WIN_PAIR) {
                const uint32_t* w0 = reinterpret_cast<const uint32_t*>(g0 + (c.x >> 16));
                const uint32_t* w1 = reinterpret_cast<const uint32_t*>(g1 + (c.x >> 16));
                a0 = __ldg(w0), a1 = __ldg(w0 + 1), b0 = __ldg(w1), b1 = __ldg(w1 + 1);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const uint32_t h0 = __dp4a(__byte_perm(a0, a1, j ? c.z : c.x), j ? c.w : c.y, 0u);
                const uint32_t h1 = __dp4a(__byte_perm(b0, b1, j ? c.z : c.x), j ? c.w : c.y, 0u);
                acc[2 * e2 + j] = h0 * (256u - fy) + (h1 * fy + 32768u);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const uint32_t t = j ? c.z : c.x;
                const uint32_t xa = t & 0xFFFFu, dx = (t >> 16) & 1u, fx = t >> 24;
                const uint32_t h0 = (256u - fx) * __ldg(g0 + xa) + fx * __ldg(g0 + xa + dx);
                const uint32_t h1 = (256u - fx) * __ldg(g1 + xa) + fx * __ldg(g1 + xa + dx);
                acc[2 * e2 + j] = h0 * (256u - fy) + (h1 * fy + 32768u);
            }
        }
        dv[2 * e2] = __ldg(drow + (pair[e2].nearest & 0xFFFFu));
        dv[2 * e2 + 1] = __ldg(drow + (pair[e2].nearest >> 16));
    }
    gw = __byte_perm(__byte_perm(acc[0], acc[1], 0x0062u), __byte_perm(acc[2], acc[3], 0x0062u), 0x5410u);
    d01 = dv[0] | (dv[1] << 16);
    d23 = dv[2] | (dv[3] << 16);
}

}  // namespace rgbd
