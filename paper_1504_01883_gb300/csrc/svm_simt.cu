// svm_simt.cu -- A6/A7 with exact fp32 SIMT arithmetic (Section 2.5: the SVM decision function):
//   linear   S_c = w_c . x + b_c
//   RBF      S_c = sum_i a_ci exp(-gamma d_i^2) + b_c,  d_i^2 = |x|^2 + |sv_i|^2 - 2 x.sv_i
// For RBF the kernel value is split as exp(-gamma d^2) = 1 + E with E = expm1(-gamma d^2),
// so S_c = asum_c + sum_i a_ci E_i + b_c.  With gamma = 1/dim on per-cell normalised
// histograms gamma*d^2 is ~2e-4, and E keeps the information that 1 + E would round away.
//
// Two fp32 kernels produce per-split partial sums D_s[k][c] = sum_{i in split s} a_ci E_ki:
//   rbf_rows8_kernel   n <= 8 rows: partial products of K slices, all rows at once (the
//                      one-frame workload, bound by reading the SV matrix once); scored by the
//                      epilogue kernel of the tensor-core path's small batches;
//   rbf_f32_kernel     tiles of the fp32 product over (rows, SVs), E in the epilogue, then
//                      E x a^T per tile or slice of tiles.
// reduce_scores_kernel adds the splits, asum and the bias, and takes the argmax
// (reduce_scores_wide_kernel, reduce_scores_hoisted_kernel: the tensor-core splits, the row-independent
// sums shared by a block; a thread per output, and a warp per row for more than 1024 rows).
#include <algorithm>

#include "f32_tile.cuh"
#include "internal.h"

namespace rgbd {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

// ---------------------------------------------------------------------------------------
// Linear SVM: a CTA takes R rows and CG classes at a time, its threads split the columns.  One row
// is bound by latency (a 64 x 64 crop: 1 row of 3840, 5 classes), so every load of a pass is in
// flight at once; many rows are bound by reading the weights from L2, which R rows share, and, when
// rows are short, by the sums over the threads at the end of a pass.
// ---------------------------------------------------------------------------------------
template <int R, int T, int CG>
__global__ void __launch_bounds__(T) linear_kernel(const float* __restrict__ x, int n, int k_pad,
                                                             const float* __restrict__ w,
                                                             const float* __restrict__ bias, int C,
                                                             float* __restrict__ scores,
                                                             int32_t* __restrict__ labels) {
    constexpr int NW = T / 32;
    __shared__ float part[NW][R * CG];
    __shared__ float row_scores[R][256];  // C <= 256
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k4 = k_pad / 4;
    const int row0 = blockIdx.x * R;
    const float4* xr[R];
#pragma unroll
    for (int r = 0; r < R; ++r) xr[r] = reinterpret_cast<const float4*>(x + (size_t)min(row0 + r, n - 1) * k_pad);
    for (int c0 = 0; c0 < C; c0 += CG) {
        const float4* wr[CG];
#pragma unroll
        for (int c = 0; c < CG; ++c) wr[c] = reinterpret_cast<const float4*>(w + (size_t)min(c0 + c, C - 1) * k_pad);
        float acc[R * CG];
#pragma unroll
        for (int v = 0; v < R * CG; ++v) acc[v] = 0.f;
#pragma unroll 2
        for (int j = tid; j < k4; j += T) {
            float4 a[R];
#pragma unroll
            for (int r = 0; r < R; ++r) a[r] = __ldg(xr[r] + j);
#pragma unroll
            for (int c = 0; c < CG; ++c) {
                const float4 b = __ldg(wr[c] + j);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    float s = acc[r * CG + c];
                    s = fmaf(a[r].x, b.x, s);
                    s = fmaf(a[r].y, b.y, s);
                    s = fmaf(a[r].z, b.z, s);
                    acc[r * CG + c] = fmaf(a[r].w, b.w, s);
                }
            }
        }
        // Sums over the lanes: while several values are left, each half of the lanes keeps half of
        // them; then lanes that hold the same value add up.
        int held = 0;  // this lane's value once one is left
#pragma unroll
        for (int off = 16, m = R * CG; off > 0; off >>= 1) {
            if (m > 1) {
                m >>= 1;
                const bool upper = (lane & off) != 0;
#pragma unroll
                for (int v = 0; v < m; ++v) {
                    const float other = __shfl_xor_sync(FULL, upper ? acc[v] : acc[v + m], off);
                    acc[v] = (upper ? acc[v + m] : acc[v]) + other;
                }
                held += upper ? m : 0;
            } else {
                acc[0] += __shfl_xor_sync(FULL, acc[0], off);
            }
        }
        constexpr int SAME = 32 / (R * CG);  // lanes that hold the same value
        if (lane % SAME == 0) part[warp][held] = acc[0];
        __syncthreads();
        if (tid < R * CG) {
            float s = 0.f;
#pragma unroll
            for (int i = 0; i < NW; ++i) s += part[i][tid];
            const int r = tid / CG, c = c0 + tid % CG;
            if (c < C && row0 + r < n) {
                s += bias[c];
                scores[(size_t)(row0 + r) * C + c] = s;
                row_scores[r][c] = s;
            }
        }
        __syncthreads();
    }
    if (labels && warp < R && row0 + warp < n) {  // the first of the largest scores
        float best = row_scores[warp][0];
        int bi = 0;
        for (int c = lane; c < C; c += 32) {
            const float v = row_scores[warp][c];
            if (v > best) {
                best = v;
                bi = c;
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            const float ob = __shfl_xor_sync(FULL, best, off);
            const int oi = __shfl_xor_sync(FULL, bi, off);
            if (ob > best || (ob == best && oi < bi)) {
                best = ob;
                bi = oi;
            }
        }
        if (lane == 0) labels[row0 + warp] = bi;
    }
}

// ---------------------------------------------------------------------------------------
// RBF, n <= 8 rows: partial products of (K slice, SVs), bound by reading the SV matrix once.  A CTA
// keeps its slice of the rows in shared memory and its warps take two SVs at a time, all lanes
// along K with 8 steps of both SVs in flight (8 KB a warp); the sums of the lanes are halved over
// the values until a lane holds one.  launch_rows_epilogue adds the slices and scores.
// 4 rows x 512 SVs x 15104, 10 classes: 62 us for the products (a warp per SV, one load in flight
// per lane) and 58 us for one warp per row adding 512 partial sums; 11 us and 6 us now.
// ---------------------------------------------------------------------------------------
constexpr int kSlice = 2048;       // K per slice
constexpr int kRows8Threads = 256;

template <int MB>
__global__ void __launch_bounds__(kRows8Threads) rbf_rows8_kernel(const float* x, int n, int k_pad,
                                                                  const float* __restrict__ sv, int n_sv, int n_pad,
                                                                  int sv_per_cta, float* __restrict__ gpart,
                                                                  uint32_t* __restrict__ counter) {
    extern __shared__ __align__(16) float xs[];  // [MB][kSlice]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int k0 = blockIdx.x * kSlice, klen = min(kSlice, k_pad - k0);  // a multiple of 128
    // launched as a programmatic dependent of the kernel that makes the rows (asking L2 for the SVs
    // before this wait made no difference)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *counter = 0u;  // the epilogue counts on it
    for (int m = 0; m < MB; ++m)
        for (int k = 4 * tid; k < klen; k += 4 * kRows8Threads)
            *reinterpret_cast<float4*>(xs + m * kSlice + k) =
                __ldcg(reinterpret_cast<const float4*>(x + (size_t)min(m, n - 1) * k_pad + k0 + k));
    __syncthreads();
    const int i1 = min(n_sv, (int)(blockIdx.y + 1) * sv_per_cta);
    for (int i = blockIdx.y * sv_per_cta + 2 * warp; i < i1; i += 2 * (kRows8Threads / 32)) {
        const float* s0 = sv + (size_t)i * k_pad + k0 + 4 * lane;
        const float* s1 = sv + (size_t)min(i + 1, n_sv - 1) * k_pad + k0 + 4 * lane;
        float acc[2 * MB];
#pragma unroll
        for (int v = 0; v < 2 * MB; ++v) acc[v] = 0.f;
        for (int kb = 0; kb < klen; kb += 8 * 128) {
            float4 b[2][8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const bool in = kb + 128 * u < klen;
                b[0][u] = in ? __ldg(reinterpret_cast<const float4*>(s0 + kb + 128 * u)) : make_float4(0, 0, 0, 0);
                b[1][u] = in ? __ldg(reinterpret_cast<const float4*>(s1 + kb + 128 * u)) : make_float4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (kb + 128 * u >= klen) break;
#pragma unroll
                for (int m = 0; m < MB; ++m) {
                    const float4 a = *reinterpret_cast<const float4*>(xs + m * kSlice + kb + 128 * u + 4 * lane);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        float t = acc[q * MB + m];
                        t = fmaf(a.x, b[q][u].x, t);
                        t = fmaf(a.y, b[q][u].y, t);
                        t = fmaf(a.z, b[q][u].z, t);
                        acc[q * MB + m] = fmaf(a.w, b[q][u].w, t);
                    }
                }
            }
        }
        int held = 0;  // the value this lane holds in the end
#pragma unroll
        for (int off = 16, left = 2 * MB; off > 0; off >>= 1) {
            if (left > 1) {
                left >>= 1;
                const bool upper = (lane & off) != 0;
#pragma unroll
                for (int v = 0; v < left; ++v) {
                    const float other = __shfl_xor_sync(FULL, upper ? acc[v] : acc[v + left], off);
                    acc[v] = (upper ? acc[v + left] : acc[v]) + other;
                }
                held += upper ? left : 0;
            } else {
                acc[0] += __shfl_xor_sync(FULL, acc[0], off);
            }
        }
        const int q = held / MB, m = held % MB;
        if (lane % (32 / (2 * MB)) == 0 && m < n && i + q < i1)
            gpart[((size_t)blockIdx.x * n + m) * n_pad + i + q] = acc[0];
    }
}

// ---------------------------------------------------------------------------------------
// RBF, general n: the fp32 product of (rows, SVs) tile by tile (f32_tile.cuh), E = expm1(-gamma d^2)
// of a tile into shared memory, then part[slice][row][c] (+)= sum_i E[row][i] a[c][i], i ascending.
// Bound by the FMA pipes.  777 rows x 3001 SVs x 15104, 50 classes: 4.23 ms with a CTA per
// (row tile, split) in lock step with two barriers every 8 k, 1.45 ms now.
// ---------------------------------------------------------------------------------------
struct F32Score {
    const float* x;
    const float* xsq;
    int n, k_pad;
    const float* sv;
    const float* svsq;
    int n_sv, n_pad;
    const float* coef;
    int C;
    float gamma;
    int mt, nt, tps;  // row tiles, SV tiles, SV tiles per slice
    float* part;      // [slices][n][C]
    // ORDERED: chains and flags handed from CTA to CTA
    uint64_t* stash;  // [CTA][32][threads]
    uint32_t* failed;  // [row tile]
};

template <int BM>
struct F32ScoreSmem {
    union {
        typename F32Tile<BM, BM>::Smem stage;
        float E[BM][BM + 4];
    };
};

// One tile's E and its product with the coefficients; `add` to what the slice holds already.
template <int BM>
__device__ __forceinline__ void f32_score_tile(const F32Score& p, const F32Tile<BM, BM>& t, int mi, int ni, int slice,
                                               bool add, F32ScoreSmem<BM>& sm) {
    constexpr int NT = F32Tile<BM, BM>::NT, GROUPS = NT / BM;
    const int m0 = mi * BM, n0 = ni * BM;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int rl = t.m_of(i);
        const float xs = m0 + rl < p.n ? p.xsq[m0 + rl] : 0.f;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int cl = t.n_of(q);
            float e[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float d2 = fmaxf(xs + p.svsq[n0 + cl + h] - 2.f * t.get(i, q, h), 0.f);
                e[h] = expm1f(-p.gamma * d2);
            }
            *reinterpret_cast<float2*>(&sm.E[rl][cl]) = make_float2(e[0], e[1]);
        }
    }
    __syncthreads();
    // a thread = one row and four classes at a time; the coefficients are the same for a warp
    const int rl = threadIdx.x % BM, row = m0 + rl;
    for (int c0 = 4 * (threadIdx.x / BM); c0 < p.C; c0 += 4 * GROUPS) {
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        const float* a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = p.coef + (size_t)min(c0 + q, p.C - 1) * p.n_pad + n0;
#pragma unroll 4
        for (int i = 0; i < BM; i += 4) {
            const float4 e = *reinterpret_cast<const float4*>(&sm.E[rl][i]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 w = __ldg(reinterpret_cast<const float4*>(a[q] + i));
                s[q] = fmaf(e.x, w.x, s[q]);
                s[q] = fmaf(e.y, w.y, s[q]);
                s[q] = fmaf(e.z, w.z, s[q]);
                s[q] = fmaf(e.w, w.w, s[q]);
            }
        }
        if (row < p.n) {
            float* o = p.part + ((size_t)slice * p.n + row) * p.C + c0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (c0 + q < p.C) o[q] = add ? o[q] + s[q] : s[q];
        }
    }
}

// ORDERED: every SV tile is a slice of its own, and the tiles are spread evenly over one CTA per
// SM.  Otherwise CTA (row tile, slice) walks the SV tiles of its slice.
template <int BM, bool ORDERED>
__global__ void __launch_bounds__(F32Tile<BM, BM>::NT, 1) rbf_f32_kernel(const F32Score p, const F32HandOver ho) {
    using Tile = F32Tile<BM, BM>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    auto& sm = *reinterpret_cast<F32ScoreSmem<BM>*>(smem_raw);
    auto rows = [&](int mi, int ni) {
        return F32Rows{p.x + (size_t)mi * BM * p.k_pad, p.n - mi * BM, p.sv + (size_t)ni * BM * p.k_pad, p.n_sv - ni * BM};
    };
    if (ORDERED) {
        f32_ordered_tiles<Tile, true>(
            (long long)p.mt * p.nt, p.k_pad, ho, sm.stage,
            [&](long long i) { return rows((int)(i % p.mt), (int)(i / p.mt)); },
            [&](long long i, const Tile& t) {
                f32_score_tile<BM>(p, t, (int)(i % p.mt), (int)(i / p.mt), (int)(i / p.mt), false, sm);
            },
            [&](long long, const Tile& t) {
                uint64_t* out = p.stash + (size_t)blockIdx.x * 32 * Tile::NT + threadIdx.x;
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    __stcg(reinterpret_cast<unsigned long long*>(out + i * Tile::NT), t.acc[i >> 2][i & 3]);
            },
            [&](long long, Tile& t) {
                const uint64_t* in = p.stash + (size_t)(blockIdx.x - 1) * 32 * Tile::NT + threadIdx.x;
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    t.acc[i >> 2][i & 3] = __ldcg(reinterpret_cast<const unsigned long long*>(in + i * Tile::NT));
            },
            [&](long long i) { p.failed[i % p.mt] = 1u; });
    } else {
        const int mi = blockIdx.x, slice = blockIdx.y, t0 = slice * p.tps, t1 = min(p.nt, t0 + p.tps);
        for (int ni = t0; ni < t1; ++ni) {
            const F32Rows r = rows(mi, ni);
            Tile t;
            t.clear();
            t.template run<true>(r.a, r.na, r.b, r.nb, p.k_pad, 0, p.k_pad / Tile::KB, sm.stage);
            f32_score_tile<BM>(p, t, mi, ni, slice, ni > t0, sm);
        }
    }
}

// Most bytes of partial sums for which every SV tile keeps a slice of its own.
constexpr size_t kF32SliceBytes = (size_t)256 << 20;

// How a call of n rows is laid out, and the workspace it takes.
struct F32Plan {
    int bm, mt, nt, slices, tps;
    bool ordered;
    size_t off_stash, off_ready, bytes;  // (at off_ready: a word per CTA, then one per row tile)
};

F32Plan plan_f32(const rgbd_ctx* ctx, const rgbd_svm* m, int n) {
    F32Plan p;
    const int sms = ctx->props.sm_count;
    auto tiles = [&](int bm) {
        p.bm = bm;
        p.mt = (n + bm - 1) / bm;
        p.nt = (m->n_sv + bm - 1) / bm;
        return (long long)p.mt * p.nt;
    };
    // 128 x 128 tiles when there is one for every SM (57 TFLOP/s against 51 in 64 x 64 tiles),
    // spread evenly (1.45 ms against 2.0 ms in 64 x 64 tiles with a CTA each at 777 x 3001)
    // while a slice of partial sums per SV tile stays small; smaller tiles on more CTAs otherwise.
    const bool big = tiles(128) >= sms;
    if (!big) tiles(64);
    p.ordered = big && sizeof(float) * (size_t)p.nt * n * m->C <= kF32SliceBytes;
    p.tps = 1;
    if (!p.ordered) {
        // fewest waves of tiles on the SMs (64 x 64 tiles: four CTAs each), fewest slices on ties
        const long long slots = (long long)sms * (big ? 1 : 4);
        long long best = -1;
        for (int sp = 1; sp; sp = next_split(p.nt, sp)) {
            const int tps = (p.nt + sp - 1) / sp;
            const long long cost = (((long long)p.mt * sp + slots - 1) / slots) * tps;
            if (best < 0 || cost < best) best = cost, p.tps = tps;
        }
    }
    p.slices = (p.nt + p.tps - 1) / p.tps;
    p.off_stash = (sizeof(float) * (size_t)p.slices * n * m->C + 255) & ~size_t(255);
    p.off_ready = p.off_stash + (p.ordered ? sizeof(uint64_t) * 32 * F32Tile<128, 128>::NT * (size_t)sms : 0);
    p.bytes = p.off_ready + (p.ordered ? sizeof(uint32_t) * ((size_t)sms + p.mt) : 0);
    return p;
}

template <int BM, bool ORDERED>
cudaError_t launch_f32(const F32Score& p, const F32HandOver& ho, dim3 grid, cudaStream_t s) {
    const size_t smem = sizeof(F32ScoreSmem<BM>);
    const cudaError_t e =
        cudaFuncSetAttribute(rbf_f32_kernel<BM, ORDERED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    rbf_f32_kernel<BM, ORDERED><<<grid, F32Tile<BM, BM>::NT, smem, s>>>(p, ho);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------
// Final reduction: one warp per row.
//   ref == NULL:  S_c = asum_c + sum_s D_s[c] + b_c
//   ref != NULL:  the partial sums of split s are relative to a reference distance r_s
//                 (D_s = sum_i a_ci expm1(-gamma (d_i^2 - r_s))); with r* = r_0 and
//                 delta_s = expm1(-gamma (r_s - r*)):
//                 S_c = exp(-gamma r*) (asum_c + sum_s [D_s + delta_s (asum_{c,s} + D_s)]) + b_c
// ---------------------------------------------------------------------------------------
__global__ void reduce_scores_kernel(const float* __restrict__ part, const float* __restrict__ ref,
                                     int splits, int n, int C, int C_stride, const float* __restrict__ asum,
                                     const float* __restrict__ asum_tile, int tps, int nt,
                                     const float* __restrict__ bias, float gamma, float* __restrict__ scores,
                                     int32_t* __restrict__ labels, const uint32_t* __restrict__ failed,
                                     int fail_rows) {
    const int lane = threadIdx.x & 31;
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= n) return;
    if (failed && failed[row / fail_rows]) {
        for (int c = lane; c < C; c += 32) scores[(size_t)row * C + c] = 0.f;
        if (labels && lane == 0) labels[row] = 0;
        return;
    }
    float best = -INFINITY;
    int bi = 0x7FFFFFFF;
    const float rstar = ref ? ref[row] : 0.f;
    const float escale = ref ? expf(-gamma * rstar) : 1.f;
    for (int c = lane; c < C; c += 32) {
        float acc = 0.f;
        for (int s = 0; s < splits; ++s) {
            const float d = part[((size_t)s * n + row) * C_stride + c];
            if (ref) {
                float as = 0.f;  // sum of a_ci over the SVs of split s
                if (s > 0)
                    for (int t = s * tps; t < min(nt, (s + 1) * tps); ++t) as += asum_tile[(size_t)t * C_stride + c];
                const float delta = (s == 0) ? 0.f : expm1f(-gamma * (ref[(size_t)s * n + row] - rstar));
                acc += d + delta * (as + d);
            } else {
                acc += d;
            }
        }
        const float sc = escale * (asum[c] + acc) + bias[c];
        scores[(size_t)row * C + c] = sc;
        if (sc > best) {
            best = sc;
            bi = c;
        }
    }
    if (labels) {
        for (int off = 16; off > 0; off >>= 1) {
            const float ob = __shfl_xor_sync(FULL, best, off);
            const int oi = __shfl_xor_sync(FULL, bi, off);
            if (ob > best || (ob == best && oi < bi)) {
                best = ob;
                bi = oi;
            }
        }
        if (lane == 0) labels[row] = bi;
    }
}

// The same combination with the row-independent parts hoisted: a block of rows first sums, per
// split and class, the coefficients of the split's tiles (sum_{i in split s} a_ci) and, per row
// and split, delta_s = expm1(-gamma (r_s - r*)), into shared memory; then one warp per row adds
// the splits in the same order and with the same operations as reduce_scores_kernel, so the
// scores are bit-identical to it.  (reduce_scores_kernel repeats the tile sums per row and the
// expm1 per class, as a chain of dependent loads in every warp.)
__global__ void reduce_scores_hoisted_kernel(const float* __restrict__ part, const float* __restrict__ ref,
                                             int splits, int n, int C, int C_stride,
                                             const float* __restrict__ asum, const float* __restrict__ asum_tile,
                                             int tps, int nt, const float* __restrict__ bias, float gamma,
                                             float* __restrict__ scores, int32_t* __restrict__ labels) {
    extern __shared__ float sh[];
    const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* s_as = sh;                              // [splits][C]
    float* s_del = sh + (size_t)splits * C;        // [nw][splits]
    const int row = blockIdx.x * nw + warp;
    if (ref) {
        for (int i = threadIdx.x; i < splits * C; i += blockDim.x) {
            const int sp = i / C, c = i - sp * C;
            float as = 0.f;
            if (sp > 0)
                for (int t = sp * tps; t < min(nt, (sp + 1) * tps); ++t) as += asum_tile[(size_t)t * C_stride + c];
            s_as[i] = as;
        }
    }
    float escale = 1.f;
    if (ref && row < n) {
        const float rstar = ref[row];
        escale = expf(-gamma * rstar);
        for (int sp = lane; sp < splits; sp += 32)
            s_del[warp * splits + sp] = (sp == 0) ? 0.f : expm1f(-gamma * (ref[(size_t)sp * n + row] - rstar));
    }
    __syncthreads();
    if (row >= n) return;
    float best = -INFINITY;
    int bi = 0x7FFFFFFF;
    for (int c = lane; c < C; c += 32) {
        float acc = 0.f;
        for (int s = 0; s < splits; ++s) {
            const float d = part[((size_t)s * n + row) * C_stride + c];
            if (ref)
                acc += d + s_del[warp * splits + s] * (s_as[s * C + c] + d);
            else
                acc += d;
        }
        const float sc = escale * (asum[c] + acc) + bias[c];
        scores[(size_t)row * C + c] = sc;
        if (sc > best) {
            best = sc;
            bi = c;
        }
    }
    if (labels) {
        for (int off = 16; off > 0; off >>= 1) {
            const float ob = __shfl_xor_sync(FULL, best, off);
            const int oi = __shfl_xor_sync(FULL, bi, off);
            if (ob > best || (ob == best && oi < bi)) {
                best = ob;
                bi = oi;
            }
        }
        if (lane == 0) labels[row] = bi;
    }
}

// The same combination for splits with a reference distance, a thread per (row, class): a block
// first puts the coefficient sum of every split and class (over the split's tiles) and, per row and
// split, delta_s = expm1(-gamma (r_s - r*)) into shared memory, then every thread adds the splits in
// the same order and with the same operations as reduce_scores_kernel, 16 splits' loads at a time.
// Launched as a programmatic dependent of the tile kernel: its launch and the model's sums hide
// behind that kernel's last CTAs.  (In the last CTA of each row block instead, 32 splits x 128 rows x
// 64 classes on one SM took 54 us of a 118 us kernel.)
constexpr int kReduceThreads = 256;
__global__ void __launch_bounds__(kReduceThreads) reduce_scores_wide_kernel(
    const float* __restrict__ part, const float* __restrict__ ref, int splits, int n, int rows, int C, int C_stride,
    const float* __restrict__ asum, const float* __restrict__ asum_tile, int tps, int nt,
    const float* __restrict__ bias, float gamma, float* __restrict__ scores, int32_t* __restrict__ labels) {
    constexpr int CH = 16;
    extern __shared__ float sh[];
    float* s_as = sh;                                 // [splits][C]
    float* s_del = s_as + (size_t)splits * C;         // [rows][splits]
    float* s_sc = s_del + (size_t)rows * splits;      // [rows][C]
    const int tid = threadIdx.x, row0 = blockIdx.x * rows, here = min(rows, n - row0);
    // (the model's sums do not depend on the kernel before)
#pragma unroll 4
    for (int i = tid; i < splits * C; i += kReduceThreads) {
        const int sp = i / C, c = i - sp * C;
        float as = 0.f;
        if (sp > 0)
            for (int t = sp * tps; t < min(nt, (sp + 1) * tps); ++t) as += __ldg(asum_tile + (size_t)t * C_stride + c);
        s_as[i] = as;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int i = tid; i < here * splits; i += kReduceThreads) {
        const int k = i / splits, sp = i - k * splits;
        s_del[i] = sp == 0 ? 0.f
                           : expm1f(-gamma * (__ldcg(ref + (size_t)sp * n + row0 + k) - __ldcg(ref + row0 + k)));
    }
    __syncthreads();
    const size_t stride = (size_t)n * C_stride;
    for (int i = tid; i < here * C; i += kReduceThreads) {
        const int k = i / C, c = i - k * C;
        const float* pd = part + (size_t)(row0 + k) * C_stride + c;
        const float r0 = __ldcg(ref + row0 + k), as = __ldg(asum + c), bs = __ldg(bias + c);
        float acc = 0.f;
#pragma unroll 1
        for (int s0 = 0; s0 < splits; s0 += CH) {
            float d[CH];
#pragma unroll
            for (int j = 0; j < CH; ++j) d[j] = s0 + j < splits ? __ldcg(pd + (s0 + j) * stride) : 0.f;
#pragma unroll
            for (int j = 0; j < CH; ++j)
                if (s0 + j < splits) acc += d[j] + s_del[k * splits + s0 + j] * (s_as[(s0 + j) * C + c] + d[j]);
        }
        const float sc = expf(-gamma * r0) * (as + acc) + bs;
        scores[(size_t)(row0 + k) * C + c] = sc;
        s_sc[i] = sc;
    }
    if (!labels) return;
    __syncthreads();
    const int lane = tid & 31;
    for (int k = tid >> 5; k < here; k += kReduceThreads / 32) {
        float best = -INFINITY;
        int bi = 0x7FFFFFFF;
        for (int c = lane; c < C; c += 32) {
            const float v = s_sc[k * C + c];
            if (v > best) {
                best = v;
                bi = c;
            }
        }
        for (int off = 16; off > 0; off >>= 1) {
            const float ob = __shfl_xor_sync(FULL, best, off);
            const int oi = __shfl_xor_sync(FULL, bi, off);
            if (ob > best || (ob == best && oi < bi)) {
                best = ob;
                bi = oi;
            }
        }
        if (lane == 0) labels[row0 + k] = bi;
    }
}

}  // namespace

int launch_reduce_scores(const float* part, const float* ref, int splits, int n, int C, int C_stride,
                         const float* asum, const float* asum_tile, int tiles_per_split, int n_tiles,
                         const float* bias, float gamma, float* scores, int32_t* labels, cudaStream_t s,
                         const uint32_t* failed, int fail_rows) {
    // Up to 1024 rows (many splits each): a thread per output.  More rows have few splits and enough
    // warps at a row each (4096 rows, 4 splits, 64 classes: 7 us, against 9 a thread per output).
    // Four rows to a block at most, so that few classes do not leave the rows to few blocks (300 rows x 8192 SVs x
    // 944, 1 class: 53 us with 256 rows to a block, 27 us with four; 10 classes: 28.8 and 27.0 us).
    const int rows = std::max(1, std::min(4, kReduceThreads / C));
    const size_t sh_wide = sizeof(float) * ((size_t)splits * C + (size_t)rows * splits + (size_t)rows * C);
    constexpr int kRowsHoisted = 16;
    const size_t sh = sizeof(float) * ((size_t)splits * C + (size_t)kRowsHoisted * splits);
    cudaError_t e;
    if (ref && n <= 1024 && sh_wide <= 48 * 1024) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)((n + rows - 1) / rows), 1, 1);
        cfg.blockDim = dim3(kReduceThreads, 1, 1);
        cfg.dynamicSmemBytes = sh_wide;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, reduce_scores_wide_kernel, part, ref, splits, n, rows, C, C_stride, asum,
                               asum_tile, tiles_per_split, n_tiles, bias, gamma, scores, labels);
    } else if (ref && sh <= 32 * 1024) {
        reduce_scores_hoisted_kernel<<<(n + kRowsHoisted - 1) / kRowsHoisted, 32 * kRowsHoisted, sh, s>>>(
            part, ref, splits, n, C, C_stride, asum, asum_tile, tiles_per_split, n_tiles, bias, gamma, scores,
            labels);
        e = cudaGetLastError();
    } else {
        const int rows_per_block = 8;
        reduce_scores_kernel<<<(n + rows_per_block - 1) / rows_per_block, 32 * rows_per_block, 0, s>>>(
            part, ref, splits, n, C, C_stride, asum, asum_tile, tiles_per_split, n_tiles, bias, gamma, scores,
            labels, failed, fail_rows);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_error(e, "svm_score: reduce launch");
    return RGBD_OK;
}

int score_linear(rgbd_ctx* ctx, const rgbd_svm* m, const float* x, int n, float* scores,
                 int32_t* labels, cudaStream_t s) {
    // As many threads per row as let every row be resident at once: 16 warps up to a row per SM, 8 up to
    // four, 4 up to eight; more rows go four to a CTA.  Classes at a time: no more than there are, and few
    // where a CTA's registers would cost residents, but for up to 8 classes, which then take one pass.
    // Against a warp per class and row (columns x classes, rows: before -> now, us): 3840 x 5, 1: 7.2 -> 3.3;
    // 944 x 2, 20000: 25.5 -> 11; 944 x 64, 500: 19.9 -> 15.6 (30 with 16 warps), 2400: 56 -> 39 (210 with four
    // rows to 16 warps); 15104 x 64, 1: 156 -> 39, 500: 183 -> 90, 5000: 1529 -> 763.
    const int per_sm = (n + ctx->props.sm_count - 1) / ctx->props.sm_count, C = m->C;
    auto launch = [&](auto kernel, int rows, int threads) {
        kernel<<<(n + rows - 1) / rows, threads, 0, s>>>(x, n, m->k_pad, m->coef, m->bias, C, scores, labels);
    };
    if (per_sm > 8) {
        if (m->k_pad >= 12000 && C > 4)  // (4 warps, 4 classes at a time: 1.2 x as long)
            launch(linear_kernel<4, 256, 8>, 4, 256);
        else
            C <= 2 ? launch(linear_kernel<4, 128, 2>, 4, 128) : launch(linear_kernel<4, 128, 4>, 4, 128);
    } else if (per_sm > 4) {
        C <= 2             ? launch(linear_kernel<1, 128, 2>, 1, 128)
        : C > 4 && C <= 8 ? launch(linear_kernel<1, 128, 8>, 1, 128)
                           : launch(linear_kernel<1, 128, 4>, 1, 128);
    } else if (per_sm > 1) {
        C <= 2                  ? launch(linear_kernel<1, 256, 2>, 1, 256)
        : C > 4 && per_sm <= 2 ? launch(linear_kernel<1, 256, 8>, 1, 256)
                                : launch(linear_kernel<1, 256, 4>, 1, 256);
    } else {
        C <= 2   ? launch(linear_kernel<1, 512, 2>, 1, 512)
        : C <= 4 ? launch(linear_kernel<1, 512, 4>, 1, 512)
                 : launch(linear_kernel<1, 512, 8>, 1, 512);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "svm_score: linear launch");
    return RGBD_OK;
}

// Layout of a call of up to 8 rows: K slices, SVs per CTA, and the epilogue's scratch.
struct Rows8Plan {
    int kz, groups, sv_per_cta;
    size_t off_ref, off_cnt, off_gpart, bytes;
};

static Rows8Plan plan_rows8(const rgbd_ctx* ctx, const rgbd_svm* m, int n) {
    Rows8Plan p;
    const int nt = m->n_pad / kSvTile;
    p.kz = (m->k_pad + kSlice - 1) / kSlice;
    // two CTAs per SM (64 KB of rows and 16 KB x 8 warps in flight each), all in one wave
    const int most = std::max(1, 2 * ctx->props.sm_count / p.kz);
    const int groups = std::max(1, std::min(most, (m->n_sv + 15) / 16));
    p.sv_per_cta = ((m->n_sv + groups - 1) / groups + 15) / 16 * 16;  // 8 warps x 2 SVs
    p.groups = (m->n_sv + p.sv_per_cta - 1) / p.sv_per_cta;
    p.off_ref = (sizeof(float) * (size_t)nt * n * m->C_pad + 255) & ~size_t(255);
    p.off_cnt = (p.off_ref + sizeof(float) * (size_t)nt * n + 255) & ~size_t(255);
    p.off_gpart = p.off_cnt + 256;
    p.bytes = p.off_gpart + sizeof(float) * (size_t)p.kz * m->n_pad * n;
    return p;
}

template <int MB>
static cudaError_t launch_rows8(const Rows8Plan& p, const float* x, int n, const rgbd_svm* m, float* gpart,
                                uint32_t* counter, cudaStream_t s) {
    const size_t smem = sizeof(float) * MB * kSlice;
    const cudaError_t e =
        cudaFuncSetAttribute(rbf_rows8_kernel<MB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.kz, (unsigned)p.groups, 1);
    cfg.blockDim = dim3(kRows8Threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, rbf_rows8_kernel<MB>, x, n, m->k_pad, (const float*)m->sv, m->n_sv, m->n_pad,
                              p.sv_per_cta, gpart, counter);
}

// Up to 8 rows are bound by reading the SVs, more rows by the products (8 rows x 66000 SVs x 15104: 0.82 ms
// by K slices, 4.6 ms in tiles, which multiply whole row tiles).
static bool takes_rows8(int n) { return n <= 8; }

// The workspace score_rbf_f32 takes for n rows (the same arithmetic as its two paths).
size_t score_rbf_f32_bytes(rgbd_ctx* ctx, const rgbd_svm* m, int n) {
    if (takes_rows8(n)) return plan_rows8(ctx, m, n).bytes;
    return plan_f32(ctx, m, n).bytes;
}

int f32_slice_rows(const rgbd_svm* m) {
    const size_t nt = ((size_t)m->n_sv + 127) / 128;
    return (int)std::min<size_t>(kF32SliceBytes / (sizeof(float) * nt * m->C), 1u << 30);
}

int score_rbf_f32(rgbd_ctx* ctx, const rgbd_svm* m, const float* x, const float* xsq, int n,
                  float* scores, int32_t* labels, cudaStream_t s) {
    if (m->C > 128) return set_error(RGBD_ERR_UNSUPPORTED, "svm_score: fp32 RBF supports up to 128 classes");
    cudaError_t e;
    if (takes_rows8(n)) {
        const Rows8Plan pl = plan_rows8(ctx, m, n);
        int rc = ensure_workspace(ctx, pl.bytes, s);
        if (rc) return rc;
        char* ws = (char*)ctx->workspace;
        float* gpart = (float*)(ws + pl.off_gpart);
        uint32_t* counter = (uint32_t*)(ws + pl.off_cnt);
        e = n == 1   ? launch_rows8<1>(pl, x, n, m, gpart, counter, s)
            : n == 2 ? launch_rows8<2>(pl, x, n, m, gpart, counter, s)
            : n <= 4 ? launch_rows8<4>(pl, x, n, m, gpart, counter, s)
                     : launch_rows8<8>(pl, x, n, m, gpart, counter, s);
        if (e != cudaSuccess) return cuda_error(e, "svm_score: rbf small-n launch");
        return launch_rows_epilogue(m, gpart, pl.kz, n, xsq, 1.f, 0.f, (float*)ws, (float*)(ws + pl.off_ref), counter,
                                    scores, labels, s);
    }
    const F32Plan pl = plan_f32(ctx, m, n);
    int rc = ensure_workspace(ctx, pl.bytes, s);
    if (rc) return rc;
    char* ws = (char*)ctx->workspace;
    F32Score p;
    p.x = x, p.xsq = xsq, p.n = n, p.k_pad = m->k_pad, p.sv = (const float*)m->sv, p.svsq = m->sv_sq;
    p.n_sv = m->n_sv, p.n_pad = m->n_pad, p.coef = m->coef, p.C = m->C, p.gamma = m->gamma;
    p.mt = pl.mt, p.nt = pl.nt, p.tps = pl.tps, p.part = (float*)ws;
    p.stash = (uint64_t*)(ws + pl.off_stash);
    const int grid = ctx->props.sm_count;
    const F32HandOver ho = {(uint32_t*)(ws + pl.off_ready), ctx->d_status, ctx->handover_ns, ctx->drop_handover};
    p.failed = ho.ready + grid;
    if (pl.ordered) {
        e = cudaMemsetAsync(ho.ready, 0, sizeof(uint32_t) * ((size_t)grid + pl.mt), s);
        if (e != cudaSuccess) return cuda_error(e, "svm_score: tile hand-over reset");
        e = launch_f32<128, true>(p, ho, dim3((unsigned)grid), s);
    } else {
        const dim3 tiles((unsigned)pl.mt, (unsigned)pl.slices);
        e = pl.bm == 128 ? launch_f32<128, false>(p, ho, tiles, s) : launch_f32<64, false>(p, ho, tiles, s);
    }
    if (e != cudaSuccess) return cuda_error(e, "svm_score: rbf fp32 launch");
    return launch_reduce_scores(p.part, nullptr, pl.slices, n, m->C, m->C, m->asum, nullptr, 0, 0, m->bias, m->gamma,
                                scores, labels, s, pl.ordered ? p.failed : nullptr, pl.bm);
}

}  // namespace rgbd
