// face256.cu -- Section 3's own descriptor: one 0-255 histogram of the raw LBP codes per face (crop
// up to 255 x 255; the paper uses 200 x 200), with the resample, median mask and codes of the
// fused kernel (lbp.cu) for crops of any size.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <algorithm>

#include "internal.h"
#include "lbp_codes.cuh"
#include "resample.cuh"

namespace rgbd {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int F256_THREADS = 1024;
constexpr int F256_COPIES = 32;  // histogram copies, one per lane

// Shared memory of a crop of side S: SW words of 4 pixels per row (the last one padded).
struct F256Layout {
    int SW, SP;                                       // words per row, with a border word on each side
    size_t region, cm, nn, rm, ctab, h1, h2, misc, bytes;  // byte offsets (the grey plane is at 0)
};
__host__ __device__ inline F256Layout f256_layout(int S) {
    F256Layout l;
    l.SW = (S + 3) / 4;
    l.SP = l.SW + 2;
    auto up = [](size_t b) { return (b + 15) & ~size_t(15); };
    l.region = up(4 * (size_t)(S + 2) * l.SP);
    // the depths (8 bytes a word of pixels); later the mask words and behind them the histograms
    const size_t items = (size_t)S * l.SW, after = items + 256 * F256_COPIES;
    l.cm = l.region + up(4 * (2 * items > after ? 2 * items : after));
    l.nn = l.cm + sizeof(uint4) * 2 * (size_t)l.SW;
    l.rm = up(l.nn + 4 * 2 * (size_t)l.SW);
    l.ctab = up(l.rm + sizeof(uint4) * (size_t)S);
    l.h1 = up(l.ctab + 8 * 65);
    l.h2 = l.h1 + 4 * 64;
    l.misc = l.h2 + 4 * 1024;
    l.bytes = l.misc + 4 * (32 + 4 + 32);
    return l;
}

// One CTA of 1024 threads per face, persistent over faces.  Everything works on words of 4
// neighbouring pixels, as in the fused kernel: the resample by 8-byte windows, a radix select of the
// median (coarse counts in registers, then 1 mm bins of one coarse bin), byte-SIMD compares on a
// grey plane whose border repeats the edge, a thread walking down its column of words.  The raw
// codes are counted with shared atomics on a copy per lane (a warp's lanes never meet in a bank).
// Bound by instruction issue and the latency of the phases (one CTA fills an SM's shared memory at
// 200 x 200).  576 faces of 200 x 200 from 640x480 frames: 313 us one pixel at a time with its
// divisions, serial scans by one lane and 8 histogram copies, 107 us now.
__global__ void __launch_bounds__(F256_THREADS, 1) lbp_face256_kernel(const LbpArgs a, uint32_t sw_inv) {
    const int S = a.crop;
    const F256Layout L = f256_layout(S);
    const int SW = L.SW, SP = L.SP, items = S * SW;
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* grey = reinterpret_cast<uint32_t*>(smem);
    uint2* dep = reinterpret_cast<uint2*>(smem + L.region);
    uint32_t* mask = reinterpret_cast<uint32_t*>(smem + L.region);  // over the depths
    uint32_t* hist = mask + items;                                  // [256][COPIES]
    uint4* cm = reinterpret_cast<uint4*>(smem + L.cm);
    uint32_t* nn = reinterpret_cast<uint32_t*>(smem + L.nn);
    uint4* rm = reinterpret_cast<uint4*>(smem + L.rm);
    unsigned long long* ctab = reinterpret_cast<unsigned long long*>(smem + L.ctab);
    uint32_t* h1 = reinterpret_cast<uint32_t*>(smem + L.h1);
    uint32_t* h2 = reinterpret_cast<uint32_t*>(smem + L.h2);
    uint32_t* wsum = reinterpret_cast<uint32_t*>(smem + L.misc);
    int* info = reinterpret_cast<int*>(wsum + 32);
    float* red = reinterpret_cast<float*>(info + 4);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool strict = !(a.flags & RGBD_LBP_GE);
    const bool nbr_ignore = (a.flags & RGBD_LBP_NBR_IGNORE_MASK) != 0;
    const bool masked_grey = strict && !nbr_ignore;
    const int x_dtype = a.x_out ? a.x_dtype : 0;
    const int npx = S - 4 * (SW - 1);  // pixels of a row's last word (1..4)
    const uint32_t last_bytes = npx == 4 ? 0xFFFFFFFFu : (1u << (8 * npx)) - 1u;
    for (int i = tid; i < 65; i += F256_THREADS) ctab[i] = i < 8 ? 1ull << (8 * i) : 0ull;

    for (int face = blockIdx.x; face < a.n; face += gridDim.x) {
        __syncthreads();  // the face before is done with shared memory
        bool ok = true, win = false;
        rgbd_rect r = {0, 0, 0, S, S};
        const uint8_t* gsrc = a.grey;
        const uint16_t* dsrc = a.depth;
        int64_t aff[6] = {0, 0, 0, 0, 0, 0};
        if (a.rects) {
            r = a.rects[face];
            ok = r.frame >= 0 && r.frame < a.n_frames && r.w > 0 && r.h > 0;
            if (!ok && tid == 0) atomicOr(a.status, RGBD_STATUS_BAD_RECT);
            if (ok) {
                gsrc += (size_t)r.frame * a.H * a.W;
                dsrc += (size_t)r.frame * a.H * a.W;
                if (a.affine) {
                    for (int i = 0; i < 6; ++i) aff[i] = a.affine[6 * (size_t)face + i];
                } else {
                    win = windows(r.w, S, a.grey, a.W) != WIN_NONE;  // (pairs: a window per group is 3 % slower here)
                    for (int i = tid; i < 2 * SW + S; i += F256_THREADS) {
                        if (i < 2 * SW) {
                            const PairTaps p = make_pair_taps(r.x, r.w, S, i, a.W, win ? WIN_PAIR : WIN_NONE);
                            const int at = (i & 1) * SW + (i >> 1);
                            cm[at] = p.c;
                            nn[at] = p.nearest;
                        } else {
                            rm[i - 2 * SW] = make_row_taps(r.y, r.h, S, i - 2 * SW, a.H, a.W);
                        }
                    }
                }
            }
        } else {
            gsrc += (size_t)face * S * S;
            dsrc += (size_t)face * S * S;
        }
        h2[tid] = 0;
        if (tid < 64) h1[tid] = 0;
        __syncthreads();

        // ---- resample; coarse depth histogram (keys (d - 1) >> 10, a hole wraps to 64) ----------
        unsigned long long cnt8 = 0;  // eight 8-bit counters; a thread has at most 64 depths
#pragma unroll 1
        for (int item = tid; item < items; item += F256_THREADS) {
            const int v = (int)__umulhi((uint32_t)item, sw_inv), q = item - v * SW;
            uint32_t gw = 0, d01 = 0, d23 = 0;
            if (ok) {
                if (a.rects && !a.affine) {
                    const PairTaps pair[2] = {{cm[q], nn[q]}, {cm[SW + q], nn[SW + q]}};
                    sample_group(gsrc, dsrc, rm[v], pair, win ? WIN_PAIR : WIN_NONE, gw, d01, d23);
                } else {
                    uint32_t dv[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int u = min(4 * q + e, S - 1);
                        if (!a.rects) {
                            gw |= (uint32_t)__ldg(gsrc + v * S + u) << (8 * e);
                            dv[e] = __ldg(dsrc + v * S + u);
                        } else {
                            const uint2 tx = make_tap(aff[0] * u + aff[1] * v + aff[2], a.W);
                            const uint2 ty = make_tap(aff[3] * u + aff[4] * v + aff[5], a.H);
                            gw |= bilerp(gsrc, a.W, tx.x, ty.x) << (8 * e);
                            dv[e] = __ldg(dsrc + (size_t)ty.y * a.W + tx.y);
                        }
                    }
                    d01 = dv[0] | (dv[1] << 16);
                    d23 = dv[2] | (dv[3] << 16);
                }
                if (q == SW - 1) {  // padding is a hole
                    d01 &= npx >= 2 ? 0xFFFFFFFFu : 0xFFFFu;
                    d23 &= npx == 4 ? 0xFFFFFFFFu : (npx == 3 ? 0xFFFFu : 0u);
                }
            }
            grey[(v + 1) * SP + q + 1] = gw;
            dep[item] = make_uint2(d01, d23);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t d = ((e < 2 ? d01 : d23) >> (16 * (e & 1))) & 0xFFFFu;
                const uint32_t key = min((d - 1u) >> 10, 64u);
                cnt8 += ctab[key];
                if (key - 8u < 56u) atomicAdd(&h1[key], 1u);
            }
        }
        {
            const unsigned long long ev = cnt8 & 0x00FF00FF00FF00FFull, od = (cnt8 >> 8) & 0x00FF00FF00FF00FFull;
            const uint32_t s02 = __reduce_add_sync(FULL, (uint32_t)ev), s46 = __reduce_add_sync(FULL, (uint32_t)(ev >> 32));
            const uint32_t s13 = __reduce_add_sync(FULL, (uint32_t)od), s57 = __reduce_add_sync(FULL, (uint32_t)(od >> 32));
            if (lane == 0) {
                const uint32_t c8[8] = {s02 & 0xFFFFu, s13 & 0xFFFFu, s02 >> 16, s13 >> 16,
                                        s46 & 0xFFFFu, s57 & 0xFFFFu, s46 >> 16, s57 >> 16};
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (c8[k]) atomicAdd(&h1[k], c8[k]);
            }
        }
        __syncthreads();

        // ---- lower median of the non-zero depths: its coarse bin, then its value in that bin ------
        if (warp == 0) {
            const uint32_t c0 = h1[2 * lane], c1 = h1[2 * lane + 1];
            uint32_t incl = c0 + c1;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t t = __shfl_up_sync(FULL, incl, off);
                if (lane >= off) incl += t;
            }
            const uint32_t total = __shfl_sync(FULL, incl, 31), k = total ? (total - 1) / 2 : 0;
            const uint32_t excl = incl - c0 - c1;
            if (total == 0) {
                if (lane == 0) info[0] = -1;
            } else if (k >= excl && k < incl) {
                const bool second = k >= excl + c0;
                info[0] = 2 * lane + (second ? 1 : 0);
                info[1] = (int)(k - excl - (second ? c0 : 0));
            }
        }
        __syncthreads();
        const int b1 = info[0];
        int med = -1;
        if (b1 >= 0) {
#pragma unroll 2
            for (int item = tid; item < items; item += F256_THREADS) {
                const uint2 dd = dep[item];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t d = (((e < 2 ? dd.x : dd.y) >> (16 * (e & 1))) & 0xFFFFu) - 1u;
                    if ((d >> 10) == (uint32_t)b1) atomicAdd(&h2[d & 1023u], 1u);
                }
            }
            __syncthreads();
            const uint32_t k1 = (uint32_t)info[1], c = h2[tid];
            uint32_t incl = c;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t t = __shfl_up_sync(FULL, incl, off);
                if (lane >= off) incl += t;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            uint32_t base = lane < warp ? wsum[lane] : 0u;  // the warps before this one
            base = __reduce_add_sync(FULL, base);
            const uint32_t excl = base + incl - c;
            if (k1 >= excl && k1 < excl + c) info[2] = b1 * 1024 + tid + 1;
            __syncthreads();
            med = info[2];
        }

        // a face without a depth (a bad rect, too) has no centre: its counts are the zeros in h2 (8 x 8: 6.2 us
        // through all phases, 4.8 us; 1000 of 50 x 50 42 and 29 us)
        uint32_t nvalid = 0;
        if (b1 >= 0) {
            // ---- depth mask; masked grey and the border of the grey plane ---------------------------
            const int mk = min(a.mask_mm, 65536);
            const int lo_i = max(med - mk + 1, 1);  // d != 0 && |d - med| < mask <=> d - lo < width, unsigned
            const uint32_t lo = (uint32_t)lo_i, width = (med >= 0 && med + mk > lo_i) ? (uint32_t)(med + mk - lo_i) : 0u;
            unsigned long long bits = 0;  // 4 per word of this thread, at most 16 words
            {
                int at = 0;
    #pragma unroll 1
                for (int item = tid; item < items; item += F256_THREADS, at += 4) {
                    const int v = (int)__umulhi((uint32_t)item, sw_inv), q = item - v * SW;
                    const uint2 dd = dep[item];
                    uint32_t m = 0;
    #pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint32_t d = ((e < 2 ? dd.x : dd.y) >> (16 * (e & 1))) & 0xFFFFu;
                        m |= (d - lo < width ? 1u : 0u) << e;
                    }
                    bits |= (unsigned long long)m << at;
                    uint32_t* gp = grey + (v + 1) * SP + q + 1;
                    uint32_t g = *gp;
                    // strict compares with masked neighbours: a grey of 0 never compares greater
                    if (masked_grey)
                        g &= ((m & 1u) * 0xFFu) | ((m & 2u) * 0x7F80u) | ((m & 4u) * 0x3FC000u) | ((m & 8u) * 0x1FE00000u);
                    if (q == SW - 1) {  // the pixel past the edge repeats the last one
                        g &= last_bytes;
                        const uint32_t edge = (g >> (8 * (npx - 1))) & 0xFFu;
                        if (npx < 4) g |= edge << (8 * npx);
                        gp[1] = edge;
                    }
                    *gp = g;
                    if (q == 0) gp[-1] = g << 24;
                    if (v == 0 || v == S - 1)
                        for (int side = 0; side < 2; ++side) {  // the border rows (both, for a crop of one row)
                            if (side == 0 ? v != 0 : v != S - 1) continue;
                            uint32_t* row = gp + (side == 0 ? -SP : SP);
                            row[0] = g;
                            if (q == 0) row[-1] = g << 24;
                            if (q == SW - 1) row[1] = gp[1];
                        }
                }
            }
            __syncthreads();  // the depths are no longer needed
            for (int item = tid; item < items; item += F256_THREADS, bits >>= 4) {
                const uint32_t m = (uint32_t)bits & 15u;
                mask[item] = ((m & 1u) << 7) | ((m & 2u) << 14) | ((m & 4u) << 21) | ((m & 8u) << 28);
            }
            for (int i = tid; i < 256 * F256_COPIES; i += F256_THREADS) hist[i] = 0;
            __syncthreads();

            // ---- codes and the 0-255 histogram: a thread walks down part of a column of words ---------
            {
                const int chunk = (int)__umulhi((uint32_t)tid, sw_inv), wc = tid - chunk * SW;
                const int chunks = F256_THREADS / SW, per = (S + chunks - 1) / chunks;
                const int r0 = chunk * per, r1 = chunk < chunks ? min(S, r0 + per) : 0;
                const bool le = wc == 0, re = wc == SW - 1;
                const uint32_t centres = (re ? last_bytes : 0xFFFFFFFFu) & 0x80808080u;
                uint32_t* my = hist + lane;
                auto row3g = [&](int row, uint32_t& Lw, uint32_t& M, uint32_t& R) {
                    const uint32_t* p = grey + (row + 1) * SP + wc + 1;
                    const uint32_t c0 = p[0];
                    Lw = __byte_perm(p[-1], c0, 0x6543);
                    M = c0;
                    R = __byte_perm(c0, p[1], 0x4321);
                };
                auto row3m = [&](int row, uint32_t& Lw, uint32_t& M, uint32_t& R) {  // masks, edges repeated
                    const uint32_t* p = mask + min(max(row, 0), S - 1) * SW + wc;
                    uint32_t c0 = p[0];
                    if (re && npx < 4) c0 |= ((c0 >> (8 * (npx - 1))) & 0xFFu) << (8 * npx);
                    Lw = __byte_perm(le ? c0 << 24 : p[-1], c0, 0x6543);
                    M = c0;
                    R = __byte_perm(c0, re ? c0 >> 24 : p[1], 0x4321);
                };
                auto count = [&](uint32_t code, uint32_t valid) {
    #pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if ((valid >> (8 * e + 7)) & 1u) atomicAdd(my + ((code >> (8 * e)) & 0xFFu) * F256_COPIES, 1u);
                };
                if (r0 < r1) {
                    uint32_t gUL, gUC, gUR, gCL, gCC, gCR, gDL, gDC, gDR;
                    row3g(r0 - 1, gUL, gUC, gUR);
                    row3g(r0, gCL, gCC, gCR);
                    if (masked_grey) {
    #pragma unroll 2
                        for (int i = r0; i < r1; ++i) {
                            row3g(i + 1, gDL, gDC, gDR);
                            const uint32_t cb = (gCC & 0x7F7F7F7Fu) + 0x01010101u;
                            const uint32_t code = (cmp_msb(gUL, gCC, cb) >> 7) | (cmp_msb(gUC, gCC, cb) >> 6) |
                                                  (cmp_msb(gUR, gCC, cb) >> 5) | (cmp_msb(gCR, gCC, cb) >> 4) |
                                                  (cmp_msb(gDR, gCC, cb) >> 3) | (cmp_msb(gDC, gCC, cb) >> 2) |
                                                  (cmp_msb(gDL, gCC, cb) >> 1) | cmp_msb(gCL, gCC, cb);
                            count(code, mask[i * SW + wc] & centres);
                            gUL = gCL; gUC = gCC; gUR = gCR; gCL = gDL; gCC = gDC; gCR = gDR;
                        }
                    } else {
                        const uint32_t any = nbr_ignore ? 0x80808080u : 0u;  // neighbours whatever their depth
                        uint32_t mUL, mUC, mUR, mCL, mCC, mCR, mDL, mDC, mDR;
                        row3m(r0 - 1, mUL, mUC, mUR);
                        row3m(r0, mCL, mCC, mCR);
    #pragma unroll 1
                        for (int i = r0; i < r1; ++i) {
                            row3g(i + 1, gDL, gDC, gDR);
                            row3m(i + 1, mDL, mDC, mDR);
                            const uint32_t cb = (gCC & 0x7F7F7F7Fu) + (strict ? 0x01010101u : 0u);
                            const uint32_t code = ((cmp_msb(gUL, gCC, cb) & (mUL | any)) >> 7) |
                                                  ((cmp_msb(gUC, gCC, cb) & (mUC | any)) >> 6) |
                                                  ((cmp_msb(gUR, gCC, cb) & (mUR | any)) >> 5) |
                                                  ((cmp_msb(gCR, gCC, cb) & (mCR | any)) >> 4) |
                                                  ((cmp_msb(gDR, gCC, cb) & (mDR | any)) >> 3) |
                                                  ((cmp_msb(gDC, gCC, cb) & (mDC | any)) >> 2) |
                                                  ((cmp_msb(gDL, gCC, cb) & (mDL | any)) >> 1) |
                                                  (cmp_msb(gCL, gCC, cb) & (mCL | any));
                            count(code, mCC & centres);
                            gUL = gCL; gUC = gCC; gUR = gCR; gCL = gDL; gCC = gDC; gCR = gDR;
                            mUL = mCL; mUC = mCC; mUR = mCR; mCL = mDL; mCC = mDC; mCR = mDR;
                        }
                    }
                }
            }
            __syncthreads();

            // ---- totals (four threads per bin, each 8 copies in an order that avoids bank conflicts) ----
            {
                const int bin = tid >> 2, part = tid & 3;
                uint32_t t = 0;
    #pragma unroll
                for (int i = 0; i < 8; ++i) t += hist[bin * F256_COPIES + part * 8 + ((i + bin) & 7)];
                t += __shfl_xor_sync(FULL, t, 1);
                t += __shfl_xor_sync(FULL, t, 2);
                if (part == 0) h2[bin] = t;
            }
            __syncthreads();
    #pragma unroll
            for (int i = 0; i < 8; ++i) nvalid += h2[lane + 32 * i];
            nvalid = __reduce_add_sync(FULL, nvalid);
        }

        // ---- counts, the normalised row and its squared norm ------------------------------------
        float sq = 0.f;
        const int len = x_dtype ? a.k_pad : 256;
        for (int j = tid; j < len; j += F256_THREADS) {
            const uint32_t h = j < 256 ? h2[j] : 0u;
            if (j < 256 && a.feats) a.feats[(size_t)face * 256 + j] = (uint16_t)h;
            if (x_dtype) {
                float x = (j < 256 && nvalid) ? (float)h / (float)nvalid : 0.f;
                if (a.x_centre && j < 256) x = __fsub_rn(x, a.x_centre[j]);
                const size_t idx = (size_t)face * a.k_pad + j;
                float qv = x;
                if (x_dtype == RGBD_DT_BF16) {
                    const __nv_bfloat16 b = __float2bfloat16_rn(x);
                    reinterpret_cast<uint16_t*>(a.x_out)[idx] = __bfloat16_as_ushort(b);
                    qv = __bfloat162float(b);
                } else if (x_dtype == RGBD_DT_BF16X3) {
                    const __nv_bfloat16 hi = __float2bfloat16_rn(x);
                    const __nv_bfloat16 lo16 = __float2bfloat16_rn(x - __bfloat162float(hi));
                    reinterpret_cast<uint16_t*>(a.x_out)[idx] = __bfloat16_as_ushort(hi);
                    reinterpret_cast<uint16_t*>(a.x_out)[idx + a.x_plane] = __bfloat16_as_ushort(lo16);
                    qv = __bfloat162float(hi) + __bfloat162float(lo16);
                } else if (x_dtype == RGBD_DT_FP8) {
                    const __nv_fp8_e4m3 b(x * a.x_scale);
                    reinterpret_cast<uint8_t*>(a.x_out)[idx] = b.__x;
                    qv = static_cast<float>(b) * (1.0f / a.x_scale);
                } else {
                    reinterpret_cast<float*>(a.x_out)[idx] = x;
                }
                sq = fmaf(qv, qv, sq);
            }
        }
        if (a.xsq) {
            for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(FULL, sq, off);
            if (lane == 0) red[warp] = sq;
            __syncthreads();
            if (tid == 0) {
                float t = 0.f;
                for (int w = 0; w < F256_THREADS / 32; ++w) t += red[w];
                a.xsq[face] = t;
            }
        }
    }
}

}  // namespace

int launch_face256(rgbd_ctx* ctx, const LbpArgs& a, cudaStream_t s) {
    const F256Layout l = f256_layout(a.crop);
    static const int most = (int)f256_layout(255).bytes;
    cudaError_t e = cudaFuncSetAttribute(lbp_face256_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return cuda_error(e, "lbp_fused_features: 0-255 histogram smem attribute");
    const int grid = std::min(a.n, ctx->props.sm_count);
    const uint32_t sw_inv = (uint32_t)((0x100000000ull + l.SW - 1) / l.SW);  // i / SW, exact for i < 2^16
    lbp_face256_kernel<<<grid, F256_THREADS, l.bytes, s>>>(a, sw_inv);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "lbp_fused_features: 0-255 histogram launch");
    return RGBD_OK;
}

}  // namespace rgbd
