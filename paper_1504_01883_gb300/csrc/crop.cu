// crop.cu -- A1 alone (rgbd_crop_affine; Section 2.1, Eq. 1): face rects resampled into crops that
// are written out, for callers that want the faces themselves.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "resample.cuh"

namespace rgbd {
namespace {

constexpr int kCropThreads = 256;

struct CropArgs {
    const uint8_t* grey;
    const uint16_t* depth;
    int n_frames, H, W;
    const rgbd_rect* rects;
    const int32_t* affine;
    int n, oh, ow;
    int ow4;        // groups of 4 columns
    int rows;       // crop rows per CTA
    int lanes_log2; // lanes of a warp on one row
    int narrow;     // the padding of a row's last group is a fifth of it or more
    int wide;       // 4-byte grey and 8-byte depth stores are aligned
    uint8_t* og;
    uint16_t* od;
    uint32_t* status;
};

__device__ __forceinline__ void store_group(const CropArgs& a, size_t o, int u, uint32_t gw, uint32_t d01,
                                            uint32_t d23) {
    if (a.wide) {
        *reinterpret_cast<uint32_t*>(a.og + o) = gw;
        *reinterpret_cast<uint2*>(a.od + o) = make_uint2(d01, d23);
        return;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (u + e < a.ow) {
            a.og[o + e] = (uint8_t)(gw >> (8 * e));
            a.od[o + e] = (uint16_t)((e < 2 ? d01 : d23) >> (16 * (e & 1)));
        }
}

// One CTA per (strip of crop rows, rect).  The taps of every column and of the strip's rows are
// computed once into shared memory (a 64-bit division each: one per pixel and axis is what bound
// this step before), and a thread makes 4 neighbouring pixels and stores them in two words.  For
// rects at most twice as wide as the crop the four grey taps of a column pair lie in one aligned
// 8-byte window of a source row, so a pair costs two 32-bit loads per row (for rects no wider than
// the crop the whole group does) and each horizontal interpolation is a byte permute and a 4-way
// byte dot product.  Bound by the gathers through L1,
// with HBM behind (frames in once, crops out once).  4096 rects of side 48..256 over 256 frames
// of 640x480 -> 128x128: 570 us with a thread and two divisions per pixel, 98 us now.
__global__ void __launch_bounds__(kCropThreads) crop_rect_kernel(const CropArgs a) {
    extern __shared__ __align__(16) unsigned char crop_smem[];
    uint4* cm = reinterpret_cast<uint4*>(crop_smem);                  // [2][ow4]: taps of a column pair
    uint32_t* nn = reinterpret_cast<uint32_t*>(cm + 2 * a.ow4);       // [2][ow4]: its nearest columns
    uint4* rm = reinterpret_cast<uint4*>(crop_smem + (((sizeof(uint4) + sizeof(uint32_t)) * 2 * (size_t)a.ow4 + 15) & ~size_t(15)));  // [rows]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int v0 = blockIdx.x * a.rows, v1 = min(a.oh, v0 + a.rows);
    const int lpr = 1 << a.lanes_log2, rpw = 32 >> a.lanes_log2;      // lanes per row, rows per warp
    const int ql = lane & (lpr - 1), vl = v0 + warp * rpw + (lane >> a.lanes_log2);
    const int vstep = (kCropThreads / 32) * rpw;
    for (int k = blockIdx.y; k < a.n; k += gridDim.y) {
        const rgbd_rect r = a.rects[k];
        const size_t crop0 = (size_t)k * a.oh * a.ow;
        const bool ok = r.frame >= 0 && r.frame < a.n_frames && r.w > 0 && r.h > 0;
        if (!ok) {
            for (int v = vl; v < v1; v += vstep)
                for (int q = ql; q < a.ow4; q += lpr)
                    store_group(a, crop0 + (size_t)v * a.ow + 4 * q, 4 * q, 0u, 0u, 0u);
            if (blockIdx.x == 0 && tid == 0) atomicOr(a.status, RGBD_STATUS_BAD_RECT);
            continue;
        }
        const uint8_t* gsrc = a.grey + (size_t)r.frame * a.H * a.W;
        const uint16_t* dsrc = a.depth + (size_t)r.frame * a.H * a.W;
        const int win = windows(r.w, a.ow, a.grey, a.W);
        __syncthreads();  // the taps of the rect before are no longer read
        for (int i = tid; i < 2 * a.ow4 + (v1 - v0); i += kCropThreads) {
            if (i < 2 * a.ow4) {
                const PairTaps p = make_pair_taps(r.x, r.w, a.ow, i, a.W, win);
                const int at = (i & 1) * a.ow4 + (i >> 1);
                cm[at] = p.c;
                nn[at] = p.nearest;
            } else {
                const int v = i - 2 * a.ow4;
                rm[v] = make_row_taps(r.y, r.h, a.oh, v0 + v, a.H, a.W);
            }
        }
        __syncthreads();
        // a loop per kind of window, rolled: 104 us when it was made so, against 107 us unrolled twice (113 us
        // with the kind tested inside), 114 us four times
        auto rows = [&](auto mode) {
            constexpr int M = decltype(mode)::value;
#pragma unroll 1
            for (int v = vl; v < v1; v += vstep) {
                const uint4 ry = rm[v - v0];
                for (int q = ql; q < a.ow4; q += lpr) {
                    const PairTaps pair[2] = {{cm[q], nn[q]}, {cm[a.ow4 + q], nn[a.ow4 + q]}};
                    uint32_t gw, d01, d23;
                    sample_group(gsrc, dsrc, ry, pair, M, gw, d01, d23);
                    store_group(a, crop0 + (size_t)v * a.ow + 4 * q, 4 * q, gw, d01, d23);
                }
            }
        };
        if (win == WIN_NONE && a.narrow) {
            // without windows a pixel costs its own loads, the padding's too: a thread per pixel on the same taps
            // (3000 rects of side 48..256 to 300x5: 53 us in groups, 26 us; to 300x9 66 and 35 us)
            for (int p = tid; p < (v1 - v0) * a.ow; p += kCropThreads) {
                const int v = p / a.ow, u = p - v * a.ow, at = ((u >> 1) & 1) * a.ow4 + (u >> 2);
                const uint4 c = cm[at], ry = rm[v];
                const uint32_t t = u & 1 ? c.z : c.x, near = u & 1 ? nn[at] >> 16 : nn[at] & 0xFFFFu;
                const uint32_t xa = t & 0xFFFFu, dx = (t >> 16) & 1u, fx = t >> 24, fy = ry.w;
                const uint32_t h0 = (256u - fx) * __ldg(gsrc + ry.x + xa) + fx * __ldg(gsrc + ry.x + xa + dx);
                const uint32_t h1 = (256u - fx) * __ldg(gsrc + ry.y + xa) + fx * __ldg(gsrc + ry.y + xa + dx);
                const size_t o = crop0 + (size_t)v0 * a.ow + p;
                a.og[o] = (uint8_t)((h0 * (256u - fy) + h1 * fy + 32768u) >> 16);
                a.od[o] = __ldg(dsrc + ry.z + near);
            }
        } else if (win == WIN_GROUP)
            rows(std::integral_constant<int, WIN_GROUP>{});
        else if (win == WIN_PAIR)
            rows(std::integral_constant<int, WIN_PAIR>{});
        else
            rows(std::integral_constant<int, WIN_NONE>{});
    }
}

// A general affine map: source points by 64-bit products per pixel, a thread per group of 4 columns.  ROWS (where a
// row is whole warps of groups): a warp per crop row, a strip of a.rows rows per CTA; else a crop's groups in a row,
// a.rows steps of 256 per CTA.  Either way neighbouring rows meet in a CTA's L1.  Bound by the products and the
// gathers.  600 maps to 128x128: 74 us a thread per pixel, 62 us now; to 100x100 (25 groups a row) 48 and 37 us (a warp
// per row there: 47 us; groups in a row at 512x512: 5 % slower).
template <bool ROWS>
__global__ void __launch_bounds__(kCropThreads) crop_affine_kernel(const CropArgs a) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lpr = 1 << a.lanes_log2;  // 32 for ROWS (as a constant: 40 maps to 512x512 in 56 us instead of 51)
    for (int k = blockIdx.y; k < a.n; k += gridDim.y) {
        const rgbd_rect r = a.rects[k];
        const bool ok = r.frame >= 0 && r.frame < a.n_frames && r.w > 0 && r.h > 0;
        if (!ok && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(a.status, RGBD_STATUS_BAD_RECT);
        int64_t m[6] = {0, 0, 0, 0, 0, 0};
        if (ok)
            for (int i = 0; i < 6; ++i) m[i] = __ldg(a.affine + 6 * (size_t)k + i);
        const uint8_t* gsrc = a.grey + (ok ? (size_t)r.frame * a.H * a.W : 0);
        const uint16_t* dsrc = a.depth + (ok ? (size_t)r.frame * a.H * a.W : 0);
        auto group = [&](int v, int q, int64_t xv, int64_t yv) {  // xv, yv: the row's share of the source point
            uint32_t gw = 0, d[2] = {0, 0};
            if (ok) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int u = 4 * q + e;
                    const uint2 tx = make_tap(m[0] * u + xv, a.W);
                    const uint2 ty = make_tap(m[3] * u + yv, a.H);
                    gw |= bilerp(gsrc, a.W, tx.x, ty.x) << (8 * e);
                    d[e >> 1] |= (uint32_t)__ldg(dsrc + (size_t)ty.y * a.W + tx.y) << (16 * (e & 1));
                }
            }
            store_group(a, ((size_t)k * a.oh + v) * a.ow + 4 * q, 4 * q, gw, d[0], d[1]);
        };
        if (ROWS) {
            const int v0 = blockIdx.x * a.rows, v1 = min(a.oh, v0 + a.rows);
            for (int v = v0 + warp; v < v1; v += kCropThreads / 32)
                for (int q = lane; q < a.ow4; q += lpr) group(v, q, m[1] * v + m[2], m[4] * v + m[5]);
        } else {
            const int i0 = blockIdx.x * a.rows * kCropThreads, i1 = min(a.oh * a.ow4, i0 + a.rows * kCropThreads);
            for (int i = i0 + threadIdx.x; i < i1; i += kCropThreads) {
                const int v = i / a.ow4;
                group(v, i - v * a.ow4, m[1] * v + m[2], m[4] * v + m[5]);
            }
        }
    }
}

// A thread per pixel, its coordinates computed for itself: no taps to make and share first.
template <bool AFFINE>
__global__ void __launch_bounds__(kCropThreads) crop_pixel_kernel(const CropArgs a) {
    const int p = blockIdx.x * kCropThreads + threadIdx.x, v = p / a.ow, u = p - v * a.ow;
    if (v >= a.oh) return;
    for (int k = blockIdx.y; k < a.n; k += gridDim.y) {
        const rgbd_rect r = a.rects[k];
        const size_t o = (size_t)k * a.oh * a.ow + p;
        uint32_t g = 0, d = 0;
        if (r.frame >= 0 && r.frame < a.n_frames && r.w > 0 && r.h > 0) {
            const int32_t* m = a.affine + 6 * (size_t)k;
            const int64_t x = AFFINE ? (int64_t)m[0] * u + (int64_t)m[1] * v + m[2] : rect_coord_q16(r.x, r.w, a.ow, u);
            const int64_t y = AFFINE ? (int64_t)m[3] * u + (int64_t)m[4] * v + m[5] : rect_coord_q16(r.y, r.h, a.oh, v);
            const uint2 tx = make_tap(x, a.W), ty = make_tap(y, a.H);
            const size_t base = (size_t)r.frame * a.H * a.W;
            g = bilerp(a.grey + base, a.W, tx.x, ty.x);
            d = __ldg(a.depth + base + (size_t)ty.y * a.W + tx.y);
        } else if (p == 0) {
            atomicOr(a.status, RGBD_STATUS_BAD_RECT);
        }
        a.og[o] = (uint8_t)g;
        a.od[o] = (uint16_t)d;
    }
}

}  // namespace

int launch_crop_affine(rgbd_ctx* ctx, const uint8_t* grey, const uint16_t* depth, int n_frames, int H, int W,
                       const rgbd_rect* rects, const int32_t* affine, int n, int out_h, int out_w, uint8_t* og,
                       uint16_t* od, cudaStream_t s) {
    CropArgs a;
    a.grey = grey, a.depth = depth, a.n_frames = n_frames, a.H = H, a.W = W, a.rects = rects, a.affine = affine;
    a.n = n, a.oh = out_h, a.ow = out_w, a.og = og, a.od = od, a.status = ctx->d_status;
    a.ow4 = (out_w + 3) / 4;
    a.narrow = 5 * out_w <= 16 * a.ow4;
    a.lanes_log2 = 0;
    while (a.lanes_log2 < 5 && (1 << a.lanes_log2) < a.ow4) ++a.lanes_log2;
    a.wide = out_w % 4 == 0 && (reinterpret_cast<uintptr_t>(og) & 3) == 0 && (reinterpret_cast<uintptr_t>(od) & 7) == 0;
    // Rows per CTA: a strip pays for the column taps (two divisions per 4 columns), so strips are as
    // tall as they can be while the grid still has some CTAs for every SM; at least one pass of the
    // CTA's warps over the strip.
    const int pass = (kCropThreads / 32) * (32 >> a.lanes_log2);
    const long long want = 6LL * ctx->props.sm_count;
    const long long strips = std::max(1LL, std::min((want + n - 1) / n, (long long)(out_h + pass - 1) / pass));
    a.rows = (int)((out_h + strips - 1) / strips);
    const dim3 grid((unsigned)((out_h + a.rows - 1) / a.rows), (unsigned)std::min(n, 65535));
    const size_t smem = (((sizeof(uint4) + sizeof(uint32_t)) * 2 * (size_t)a.ow4 + 15) & ~size_t(15)) +
                        sizeof(uint4) * (size_t)a.rows;
    // Few pixels are bound by the chain of steps before the first store, which is shorter with a thread per
    // pixel, while the chip has threads to spare: up to about 1000 pixels per SM (one 100x100 crop: 3.1 us
    // in strips, 2.4 us; 40 of 32x32: 3.8 and 2.6 us; 40 of 100x100: 3.8 and 5.5 us).  So are crops of a few
    // pixels, a CTA each in strips (3000 of 8x8: 10.1 and 4.9 us).  With an affine map there are no taps
    // to share, and groups gain less: they need more pixels (40 of 100x100: 5.3 and 5.1 us; 600: 37 and 45
    // us), and 4-byte stores or long rows (3000 of 33x33: 34 and 30 us; of 300x9: 72 and 68 us).
    const long long sms = ctx->props.sm_count, px = (long long)n * out_h * out_w;
    const bool pixels = affine ? px <= 3072 * sms || out_w < 12 || (out_w % 4 != 0 && out_w < 64 && px <= 32768 * sms)
                               : px <= 1024 * sms || out_h * out_w <= 256;
    if (pixels) {
        const dim3 cells((unsigned)((out_h * out_w + kCropThreads - 1) / kCropThreads), grid.y);
        if (affine)
            crop_pixel_kernel<true><<<cells, kCropThreads, 0, s>>>(a);
        else
            crop_pixel_kernel<false><<<cells, kCropThreads, 0, s>>>(a);
    } else if (affine) {
        if (a.ow4 % 32 == 0) {
            crop_affine_kernel<true><<<grid, kCropThreads, 0, s>>>(a);
        } else {
            const int steps = (out_h * a.ow4 + kCropThreads - 1) / kCropThreads;
            const int parts = (int)std::min((long long)steps, std::max((steps + 63) / 64LL, (16 * sms + n - 1) / n));
            a.rows = (steps + parts - 1) / parts;
            crop_affine_kernel<false><<<dim3((unsigned)((steps + a.rows - 1) / a.rows), grid.y), kCropThreads, 0, s>>>(a);
        }
    } else {
        // crops up to 4096 columns and rows: 41 KB of column taps and 66 KB of row taps at most
        constexpr size_t most = (sizeof(uint4) + sizeof(uint32_t)) * 2 * 1024 + sizeof(uint4) * 4096;
        if (smem > 48 * 1024) {
            const cudaError_t e =
                cudaFuncSetAttribute(crop_rect_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
            if (e != cudaSuccess) return cuda_error(e, "rgbd_crop_affine: smem attribute");
        }
        crop_rect_kernel<<<grid, kCropThreads, smem, s>>>(a);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "rgbd_crop_affine: launch");
    return RGBD_OK;
}

}  // namespace rgbd
