// roi.cu -- the depth-space region of a colour-detected face (Section 2.1): every depth pixel is
// mapped into the colour image (the camera mapping, here an exact integer calibration), the
// pixels landing inside the detected colour rect belong to the face, and the rect bounding them
// is the face region of the depth image.
#include <limits.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>

#include <algorithm>

#include "internal.h"

namespace rgbd {
namespace {

constexpr int kRoiThreads = 256;
// Windows of up to this many pixels are read in full: the scan from the edges is a chain of strips with a barrier
// each, which a window with few pixels in it goes through to the end (600 boxes of side 10..30: every pixel tested with a
// division 7.3 us full and 4.9 us nearly empty, from the edges 7.8 and 8.6 us, now 5.6 and 5.1 us).  At 8192 full windows of
// 60..80 a side would take 12.4 us instead of 8.2 us, nearly empty ones 9.7 us instead of 15.9.
constexpr int kRoiSmall = 4096;

// The mapping of one launch and one rect, for the per-pixel test.  T is int when every coordinate
// of the frame and of the colour image stays below 2^30 in Q16.16 (the host checks; any camera up
// to 16383 pixels wide), else long long.
//   X0 <= A + 256 q < X1 with q = parallax / d (integer quotient) holds exactly when
//   l <= q < h with l = ceil((X0 - A) / 256), h = ceil((X1 - A) / 256), and for q >= 0 that is
//   l d <= parallax < h d with l, h clamped to >= 0: two widening products instead of a division.
template <typename T>
struct RoiTest {
    T a0, a1, a2, a3, a4, a5;
    T X0, X1, Y0, Yn;  // Yn = Y1 - Y0
    uint32_t parallax, d_min, d_span;

    __device__ __forceinline__ bool hit(uint32_t d, int j, int i) const {
        if (d - d_min > d_span) return false;
        const T Y = a3 * j + a4 * i + a5;
        if (sizeof(T) == 4 ? (uint32_t)(Y - Y0) >= (uint32_t)Yn
                           : (unsigned long long)(Y - Y0) >= (unsigned long long)Yn)
            return false;
        const T A = a0 * j + a1 * i + a2;
        T l = (X0 - A + 255) >> 8, h = (X1 - A + 255) >> 8;
        l = l < 0 ? 0 : l;
        h = h < 0 ? 0 : h;
        if (sizeof(T) == 8) {  // parallax < 2^31, so a bound of 2^31 decides like any larger one
            const T top = (T)0x80000000u;
            l = l > top ? top : l;
            h = h > top ? top : h;
        }
        return (uint64_t)(uint32_t)l * d <= parallax && parallax < (uint64_t)(uint32_t)h * d;
    }

    // Whether row i can meet the box's rows between columns ja and jb (Y is linear in the column).
    __device__ __forceinline__ bool row_meets(int i, int ja, int jb) const {
        const T Ya = a3 * ja + a4 * i + a5 - Y0, Yb = a3 * jb + a4 * i + a5 - Y0;
        return !((Ya < 0 && Yb < 0) || (Ya >= Yn && Yb >= Yn));
    }

    // Depths lo .. lo + span outside which no pixel of column j, rows ra..rb, can pass hit();
    // false when there are none.
    __device__ __forceinline__ bool depths(int j, int ra, int rb, uint32_t& lo, uint32_t& span) const {
        const T Aa = a0 * j + a1 * ra + a2, Ab = a0 * j + a1 * rb + a2;
        const T top = (T)0x40000000;  // bounds that large (narrow: never) only widen the range
        T l = (X0 - (Aa > Ab ? Aa : Ab) + 255) >> 8, h = (X1 - (Aa < Ab ? Aa : Ab) + 255) >> 8;
        l = l < 0 ? 0 : (l > top ? top : l);
        if (h <= 0) return false;
        uint32_t a = d_min, b = d_min + d_span;
        if (h < top) a = max(a, parallax / (uint32_t)h + 1u);
        if (l > 0) b = min(b, parallax / (uint32_t)l);
        if (a > b) return false;
        lo = a, span = b - a;
        return true;
    }
};

// What every face of a launch shares: the range of p(d), and the inverse of the linear part (where
// there is none to speak of, the whole frame is scanned).
struct RoiWindow {
    long long p_lo, p_hi;
    float ia, ib, ic, id;
    int degenerate;
};

// One CTA per face.  The scan covers a window that holds every depth pixel which can map inside
// the rect: with p(d) = 256 (parallax / d) between p_lo (at d_max) and p_hi (at d_min), a pixel
// inside needs A = a0 j + a1 i + a2 in [X0 - p_hi, X1 - p_lo) and B = a3 j + a4 i + a5 in [Y0, Y1)
// (X0, X1, Y0, Y1 the rect clipped to the colour image, in Q16.16), a parallelogram in (j, i)
// whose corners bound the window (computed in float, widened by 2 pixels; the per-pixel test
// is exact, so the window only has to be large enough).
// Only the four extremes are wanted, so a larger window is scanned from its edges inwards: rows from
// the top and from the bottom until one holds a pixel, then, between those rows, the columns
// outside the extremes found so far.  A face fills its box, so this reads the margins (a few rows,
// and the columns that only a nearer surface could have reached) instead of the area.  What is left is a chain of few L2 or DRAM round trips, so
// each step issues all its loads first (two rows of the window per warp, 16 rows of a column).
// 4096 boxes over 256 frames of 640x480, faces of side 48..256: 640 us when every window pixel was
// tested with a division, 95 us with the scan from the edges, 84 us since rows that cannot meet the box
// are passed over, what all faces share comes from the host, and small windows are read in full.
template <typename T>
__global__ void __launch_bounds__(kRoiThreads) face_roi_kernel(const uint16_t* __restrict__ depth, int n_frames, int H,
                                                               int W, rgbd_calib c, RoiWindow wd,
                                                               const rgbd_rect* __restrict__ rects, int n,
                                                               rgbd_rect* __restrict__ out,
                                                               uint32_t* __restrict__ status) {
    constexpr int NW = kRoiThreads / 32;
    __shared__ int ext[4];  // least and largest row and column so far
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = blockIdx.x; k < n; k += gridDim.x) {
        const rgbd_rect r = rects[k];
        const bool bad = r.frame < 0 || r.frame >= n_frames || r.w <= 0 || r.h <= 0;
        const long long cx0 = max(0ll, (long long)r.x), cx1 = min((long long)c.colour_w, (long long)r.x + r.w);
        const long long cy0 = max(0ll, (long long)r.y), cy1 = min((long long)c.colour_h, (long long)r.y + r.h);
        if (bad && tid == 0) atomicOr(status, RGBD_STATUS_BAD_RECT);
        int j0 = 0, j1 = -1, i0 = 0, i1 = -1;  // empty
        if (!bad && cx0 < cx1 && cy0 < cy1) {
            if (wd.degenerate) {
                j1 = W - 1, i1 = H - 1;
            } else {
                const float A[2] = {(float)((T)(cx0 * 65536) - (T)wd.p_hi - c.a[2]),
                                    (float)((T)(cx1 * 65536) - (T)wd.p_lo - c.a[2])};
                const float Bv[2] = {(float)((T)(cy0 * 65536) - c.a[5]), (float)((T)(cy1 * 65536) - c.a[5])};
                float jmn = 3e38f, jmx = -3e38f, imn = 3e38f, imx = -3e38f;
#pragma unroll
                for (int u = 0; u < 2; ++u)
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const float jj = wd.ia * A[u] + wd.ib * Bv[v], ii = wd.ic * A[u] + wd.id * Bv[v];
                        jmn = fminf(jmn, jj), jmx = fmaxf(jmx, jj);
                        imn = fminf(imn, ii), imx = fmaxf(imx, ii);
                    }
                j0 = (int)fmaxf(0.f, floorf(jmn) - 2.f), j1 = (int)fminf((float)(W - 1), ceilf(jmx) + 2.f);
                i0 = (int)fmaxf(0.f, floorf(imn) - 2.f), i1 = (int)fminf((float)(H - 1), ceilf(imx) + 2.f);
            }
        }
        __syncthreads();  // the face before has read ext
        if (tid == 0) ext[0] = ext[2] = INT_MAX, ext[1] = ext[3] = -1;
        __syncthreads();
        if (j0 <= j1 && i0 <= i1) {
            const uint16_t* dp = depth + (size_t)r.frame * H * W;
            RoiTest<T> t;
            t.a0 = c.a[0], t.a1 = c.a[1], t.a2 = c.a[2], t.a3 = c.a[3], t.a4 = c.a[4], t.a5 = c.a[5];
            t.X0 = (T)(cx0 * 65536), t.X1 = (T)(cx1 * 65536);
            t.Y0 = (T)(cy0 * 65536), t.Yn = (T)((cy1 - cy0) * 65536);
            t.parallax = (uint32_t)c.parallax, t.d_min = (uint32_t)c.d_min, t.d_span = (uint32_t)(c.d_max - c.d_min);
            // a small window: every pixel once, 8 loads of a thread in flight
            const int ww = j1 - j0 + 1, area = ww * (i1 - i0 + 1);
            const bool small = area <= kRoiSmall;
            if (small) {
                const uint32_t inv = (uint32_t)((0x100000000ull + ww - 1) / ww);  // x / ww for x < 2^16 (ww > 1)
                int xl = INT_MAX, xh = -1, yl = INT_MAX, yh = -1;
#pragma unroll 1
                for (int x0 = tid; x0 < area; x0 += 8 * kRoiThreads) {
                    uint32_t d[8];
                    int row[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int x = x0 + u * kRoiThreads;
                        row[u] = ww > 1 ? (int)__umulhi((uint32_t)x, inv) : x;
                        d[u] = x < area ? __ldg(dp + (size_t)(i0 + row[u]) * W + j0 + (x - row[u] * ww)) : 0u;
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int i = i0 + row[u], j = j0 + (x0 + u * kRoiThreads - row[u] * ww);
                        if (d[u] && t.hit(d[u], j, i)) {
                            xl = min(xl, j), xh = max(xh, j);
                            yl = min(yl, i), yh = max(yh, i);
                        }
                    }
                }
                xl = __reduce_min_sync(0xFFFFFFFFu, xl), xh = __reduce_max_sync(0xFFFFFFFFu, xh);
                yl = __reduce_min_sync(0xFFFFFFFFu, yl), yh = __reduce_max_sync(0xFFFFFFFFu, yh);
                if (lane == 0 && xh >= 0) {
                    atomicMin(&ext[0], yl), atomicMax(&ext[1], yh);
                    atomicMin(&ext[2], xl), atomicMax(&ext[3], xh);
                }
                __syncthreads();
            }
            // rows, a strip of one per warp from the top and one from the bottom at a time
            bool top = !small, bottom = !small;
            for (int s0 = 0; s0 <= i1 - i0 && (top || bottom); s0 += NW) {
                if (top && bottom && 2 * s0 > i1 - i0) break;  // met in the middle: no pixel (600 of side 300..400: 82 -> 43 us)
                const int it = i0 + s0 + warp, ib = i1 - s0 - warp;
                // (a row that is above or below the box at both ends of the window cannot hold one)
                const bool dt = top && it <= i1 && t.row_meets(it, j0, j1);
                const bool db = bottom && ib >= i0 && t.row_meets(ib, j0, j1);
                int tl = INT_MAX, th = -1, bl = INT_MAX, bh = -1;  // columns with a pixel in the two rows
                for (int jb = j0; jb <= j1 && (dt || db); jb += 4 * 32) {
                    uint32_t d[2][4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int j = jb + 32 * u + lane;
                        d[0][u] = dt && j <= j1 ? __ldg(dp + (size_t)it * W + j) : 0u;
                        d[1][u] = db && j <= j1 ? __ldg(dp + (size_t)ib * W + j) : 0u;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int j = jb + 32 * u + lane;
                        if (d[0][u] && t.hit(d[0][u], j, it)) tl = min(tl, j), th = j;
                        if (d[1][u] && t.hit(d[1][u], j, ib)) bl = min(bl, j), bh = j;
                    }
                }
                const int lo = __reduce_min_sync(0xFFFFFFFFu, min(tl, bl));
                const int hi = __reduce_max_sync(0xFFFFFFFFu, max(th, bh));
                const bool t_any = __any_sync(0xFFFFFFFFu, th >= 0), b_any = __any_sync(0xFFFFFFFFu, bh >= 0);
                if (lane == 0 && hi >= 0) {
                    atomicMin(&ext[2], lo);
                    atomicMax(&ext[3], hi);
                    if (t_any) atomicMin(&ext[0], it);
                    if (b_any) atomicMax(&ext[1], ib);
                }
                __syncthreads();
                top = ext[0] == INT_MAX;
                bottom = ext[1] < 0;
                __syncthreads();  // everyone has read ext before the next strip changes it
            }
            if (!small && !top && !bottom) {
                // Columns outside the extremes found so far, 32 at a time (a lane stays on its
                // column) and 16 rows at once.  These columns are read in full, so a lane first
                // narrows the depths that could map inside on its column at all (A is linear in the
                // row, so its bounds over the rows are those at the ends) and tests exactly only
                // what passes.
                const int ymin = ext[0], ymax = ext[1], left = ext[2], right = ext[3];
                __syncthreads();
                int best_l = left, best_r = right;
#pragma unroll 1
                for (int q = 0; q < 2; ++q) {
#pragma unroll 1
                    for (int jb = 0; q ? j1 - jb > best_r : j0 + jb < best_l; jb += 32) {
                        const int j = q ? j1 - jb - lane : j0 + jb + lane;
                        uint32_t lo = 1, span = 0;
                        bool look = (q ? j > right : j < left) && t.depths(j, ymin, ymax, lo, span);
                        const uint16_t* p = dp + j;
#pragma unroll 1
                        for (int row = ymin + warp; row <= ymax; row += 16 * NW) {
                            uint32_t d[16];
#pragma unroll
                            for (int u = 0; u < 16; ++u)
                                d[u] = look && row + u * NW <= ymax ? __ldg(p + (size_t)(row + u * NW) * W) : 0u;
                            uint32_t pass = 0;
#pragma unroll
                            for (int u = 0; u < 16; ++u) pass |= (d[u] - lo <= span ? 1u : 0u) << u;
                            if (pass) {
                                bool found = false;
#pragma unroll
                                for (int u = 0; u < 16; ++u)
                                    if ((pass >> u) & 1u) found |= t.hit(d[u], j, row + u * NW);
                                if (found) {
                                    if (q) best_r = max(best_r, j);
                                    else best_l = min(best_l, j);
                                    look = false;
                                }
                            }
                        }
                        best_l = __reduce_min_sync(0xFFFFFFFFu, best_l);
                        best_r = __reduce_max_sync(0xFFFFFFFFu, best_r);
                    }
                }
                if (lane == 0) {
                    if (best_l < left) atomicMin(&ext[2], best_l);
                    if (best_r > right) atomicMax(&ext[3], best_r);
                }
                __syncthreads();
            }
        }
        if (tid == 0) {
            rgbd_rect o;
            o.frame = r.frame;
            if (!bad && ext[1] >= 0) {
                o.x = ext[2], o.y = ext[0], o.w = ext[3] - ext[2] + 1, o.h = ext[1] - ext[0] + 1;
            } else {
                o.x = o.y = o.w = o.h = 0;
            }
            out[k] = o;
        }
    }
}

}  // namespace
}  // namespace rgbd

using namespace rgbd;

extern "C" int rgbd_face_roi(rgbd_ctx* ctx, const uint16_t* depth, int n_frames, int H, int W, const rgbd_calib* calib,
                             const rgbd_rect* colour_rects, int n, rgbd_rect* depth_rects, void* stream) {
    rgbd::NvtxRange nvtx_range("rgbd_face_roi");
    if (!ctx) return set_error(RGBD_ERR_ARG, "rgbd_face_roi: ctx is NULL");
    if (!calib) return set_error(RGBD_ERR_ARG, "rgbd_face_roi: calib is NULL");
    if (n < 0 || n_frames <= 0 || H <= 0 || W <= 0)
        return set_error(RGBD_ERR_ARG, "rgbd_face_roi: n %d, frames %d, H %d, W %d", n, n_frames, H, W);
    const rgbd_calib c = *calib;
    if (c.d_min < 1 || c.d_max < c.d_min || c.parallax < 0 || c.colour_w <= 0 || c.colour_h <= 0)
        return set_error(RGBD_ERR_ARG, "rgbd_face_roi: calibration depth range %d..%d, parallax %d, colour %dx%d",
                         c.d_min, c.d_max, c.parallax, c.colour_w, c.colour_h);
    for (int i = 0; i < 6; ++i) {
        const int lim = (i == 2 || i == 5) ? (1 << 30) : (1 << 24);  // offsets, linear terms
        if (c.a[i] > lim || c.a[i] < -lim)
            return set_error(RGBD_ERR_ARG, "rgbd_face_roi: calibration entry a[%d] = %d out of range", i, c.a[i]);
    }
    if (n == 0) return RGBD_OK;
    if (!depth || !colour_rects || !depth_rects) return set_error(RGBD_ERR_ARG, "rgbd_face_roi: NULL pointer");
    DeviceGuard g(ctx->props.device);
    const int grid = std::min(n, ctx->props.sm_count * 8);
    // 32-bit coordinates when no point of the frame, and no edge of the colour image, reaches 2^30
    auto reach = [&](int a, int b, int o) {
        return std::llabs((long long)a) * W + std::llabs((long long)b) * H + std::llabs((long long)o);
    };
    const long long lim = 1ll << 30;
    RoiWindow wd;
    wd.p_lo = (long long)(c.parallax / c.d_max) * 256;
    wd.p_hi = (long long)(c.parallax / c.d_min) * 256;
    const double det = (double)c.a[0] * c.a[4] - (double)c.a[1] * c.a[3];
    wd.ia = (float)(c.a[4] / det), wd.ib = (float)(-c.a[1] / det);
    wd.ic = (float)(-c.a[3] / det), wd.id = (float)(c.a[0] / det);
    // A window is right to 2 pixels while single precision places its corners to 1; a mapping that
    // (nearly) collapses a direction has the whole frame scanned.
    const double a_max = 65536.0 * c.colour_w + (double)wd.p_hi + fabs((double)c.a[2]);
    const double b_max = 65536.0 * c.colour_h + fabs((double)c.a[5]);
    const double reach_px = std::max((fabs((double)c.a[4]) * a_max + fabs((double)c.a[1]) * b_max),
                                     (fabs((double)c.a[3]) * a_max + fabs((double)c.a[0]) * b_max));
    wd.degenerate = fabs(det) < 1.0 || 4.8e-7 * reach_px > fabs(det);  // 4 roundings of 2^-23
    const bool narrow = reach(c.a[0], c.a[1], c.a[2]) < lim && reach(c.a[3], c.a[4], c.a[5]) < lim &&
                        c.colour_w < 16384 && c.colour_h < 16384 && wd.p_hi < lim;
    auto kernel = narrow ? face_roi_kernel<int> : face_roi_kernel<long long>;
    kernel<<<grid, kRoiThreads, 0, (cudaStream_t)stream>>>(depth, n_frames, H, W, c, wd, colour_rects, n, depth_rects,
                                                           ctx->d_status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "rgbd_face_roi: launch");
    return RGBD_OK;
}
