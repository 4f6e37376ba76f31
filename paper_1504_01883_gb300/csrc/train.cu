// train.cu -- one-vs-rest RBF SVM training on the GPU (Section 2.5 trains the classifier on the
// face database; the paper does it on the CPU).  The dual problem of every class is solved by
// sequential minimal optimisation with the maximal violating pair, on one kernel matrix that all
// classes share:
//   kernel_matrix_kernel  K_st = exp(-gamma max(0, |x_s|^2 + |x_t|^2 - 2 x_s . x_t)), fp32, one
//                         tile of the lower triangle per CTA, written twice;
//   smo_kernel            one CTA per class; the gradient stays in registers; each step selects the
//                         pair over the CTA, updates it, then moves the gradient with all threads.
#include <limits.h>
#include <stdint.h>

#include <algorithm>

#include "f32_tile.cuh"
#include "internal.h"

namespace rgbd {
namespace {

// K_st = exp(-gamma max(0, |x_s|^2 + |x_t|^2 - 2 x_s . x_t)) for s >= t by tiles of BM x BM, and its
// mirror image: the product, the sum of norms and so K itself are symmetric bit for bit, so half of
// the products do.  The tiles of the lower triangle are numbered row by row.  Bound by the FMA
// pipes.  4096 x 4096 rows of 15104: 20.4 ms as a full matrix with 4 x 4 outputs a thread,
// 4.5 ms now.
__device__ __forceinline__ void triangle_tile(long long idx, int& bi, int& bj) {
    long long r = (long long)((sqrt(8.0 * (double)idx + 1.0) - 1.0) * 0.5);
    while ((r + 1) * (r + 2) / 2 <= idx) ++r;  // the root is rounded: step to the exact row
    while (r * (r + 1) / 2 > idx) --r;
    bi = (int)r;
    bj = (int)(idx - r * (r + 1) / 2);
}

// ORDERED: tiles spread evenly over one CTA per SM (f32_ordered_tiles), else one tile per CTA.
template <int BM, bool VEC, bool ORDERED>
__global__ void __launch_bounds__(F32Tile<BM, BM>::NT, 1) kernel_matrix_kernel(const float* __restrict__ x,
                                                                          const float* __restrict__ xsq, int n,
                                                                          int k_pad, float gamma, long long tiles,
                                                                          float* K, F32HandOver ho, int32_t* failed,
                                                                          int n_classes) {
    using Tile = F32Tile<BM, BM>;
    extern __shared__ __align__(16) unsigned char km_smem[];
    auto& sm = *reinterpret_cast<typename Tile::Smem*>(km_smem);
    auto rows = [&](long long idx) {
        int bi, bj;
        triangle_tile(idx, bi, bj);
        return F32Rows{x + (size_t)bi * BM * k_pad, n - bi * BM, x + (size_t)bj * BM * k_pad, n - bj * BM};
    };
    auto finish = [&](long long idx, const Tile& tile) {
        int bi, bj;
        triangle_tile(idx, bi, bj);
        const int s0 = bi * BM, t0 = bj * BM;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int s = s0 + tile.m_of(i);
            if (s >= n) continue;
            const float xs = xsq[s];
#pragma unroll
            for (int p = 0; p < 4; ++p) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int t = t0 + tile.n_of(p) + h;
                    if (t >= n) continue;
                    const float d2 = fmaxf(xs + xsq[t] - 2.f * tile.get(i, p, h), 0.f);
                    const float k = (s == t) ? 1.f : expf(-gamma * d2);
                    K[(size_t)s * n + t] = k;
                    if (s0 != t0) K[(size_t)t * n + s] = k;
                }
            }
        }
    };
    if (ORDERED) {
        // a split tile's chains wait in its own place of K
        auto at = [&](long long idx, int i, int p, int h) -> float* {
            int bi, bj;
            triangle_tile(idx, bi, bj);
            Tile t;
            const int s = bi * BM + t.m_of(i), c = bj * BM + t.n_of(p) + h;
            return s < n && c < n ? K + (size_t)s * n + c : nullptr;
        };
        auto stash = [&](long long idx, const Tile& t) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (float* q = at(idx, i, p, h)) __stcg(q, t.get(i, p, h));
        };
        auto fetch = [&](long long idx, Tile& t) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const float *lo = at(idx, i, p, 0), *hi = at(idx, i, p, 1);
                    t.put(i, p, lo ? __ldcg(lo) : 0.f, hi ? __ldcg(hi) : 0.f);
                }
        };
        // every class hangs on every tile
        auto fail = [&](long long) {
            for (int c = 0; c < n_classes; ++c) failed[c] = 1;
        };
        f32_ordered_tiles<Tile, VEC>(tiles, k_pad, ho, sm, rows, finish, stash, fetch, fail);
    } else {
        const F32Rows r = rows(blockIdx.x);
        Tile t;
        t.clear();
        t.template run<VEC>(r.a, r.na, r.b, r.nb, k_pad, 0, (k_pad + Tile::KB - 1) / Tile::KB, sm);
        finish(blockIdx.x, t);
    }
}

// Order of floats as signed integers (and back): the largest value by an integer maximum.
__device__ __forceinline__ int float_key(float v) {
    const int b = __float_as_int(v);
    return b ^ ((b >> 31) & 0x7FFFFFFF);
}
__device__ __forceinline__ float key_float(int k) { return __int_as_float(k ^ ((k >> 31) & 0x7FFFFFFF)); }

// One CTA per class.  A step is a chain of latencies (select a pair, fetch its two rows of K, move,
// select again), so it holds one barrier: every thread keeps the values u_t = -y_t G_t of its EPT
// rows in registers with a bit each for "may move up / down", its warp selects by integer redux
// (largest or smallest value, then the lowest index), and the warps' candidates -- with alpha and
// y, which only the owner of a row keeps -- go to shared memory, where after the barrier every
// warp makes the same final selection and update for itself.  u_t += -lam (K_it - K_jt) is the
// gradient step G_t += y_t lam (K_it - K_jt) with the sign folded in, rounding alike.  K_ii = 1.
// 64 classes x 4096 rows, ~1500 steps each: 8.4 ms with three barriers and a serial selection by
// one thread per step, 1.86 ms now.
struct SmoPick {
    int key;
    uint32_t idx;  // ~0: none
    float alpha;
    int y;
};

// marked: iters[c] says whether K is incomplete (a tile's hand-over failed); the class gets zeros then.
template <int T, int EPT>
__global__ void __launch_bounds__(T, 1) smo_kernel(const float* __restrict__ K, int n,
                                                   const int32_t* __restrict__ labels, float cost, float eps,
                                                   int max_iter, float* __restrict__ coef, float* __restrict__ bias,
                                                   int32_t* iters, bool marked) {
    constexpr int NW = T / 32;
    constexpr uint32_t NONE = 0xFFFFFFFFu, FULL = 0xFFFFFFFFu;
    extern __shared__ float alpha[];  // [n], each entry touched by the thread that owns the row
    __shared__ __align__(16) SmoPick picks[2][2][NW];
    __shared__ float sums[32];
    __shared__ int counts[32];
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (marked && iters[c] != 0) {
        __syncthreads();  // everyone has read the mark
        for (int t = tid; t < n; t += T) coef[(size_t)c * n + t] = 0.f;
        if (tid == 0) bias[c] = 0.f, iters[c] = 0;
        return;
    }
    float u[EPT];
    uint32_t ypos = 0, up = 0, low = 0;  // a bit per row: y > 0, may move up, may move down
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        const int t = tid + e * T;
        u[e] = 0.f;
        if (t < n) {  // alpha = 0: y > 0 may move up, y < 0 down
            const bool pos = labels[t] == c;
            u[e] = pos ? 1.f : -1.f;
            alpha[t] = 0.f;
            ypos |= (uint32_t)pos << e;
            up |= (uint32_t)pos << e;
            low |= (uint32_t)!pos << e;
        }
    }
    int it = 0;
    float mu, ml;
    uint32_t iu, il;
    for (;; ++it) {
        int key[EPT], ku = INT_MIN, kl = INT_MAX;
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            key[e] = float_key(u[e]);
            if ((up >> e) & 1u) ku = max(ku, key[e]);
            if ((low >> e) & 1u) kl = min(kl, key[e]);
        }
        ku = __reduce_max_sync(FULL, ku);
        kl = __reduce_min_sync(FULL, kl);
        iu = il = NONE;
#pragma unroll
        for (int e = EPT - 1; e >= 0; --e) {
            if (((up >> e) & 1u) && key[e] == ku) iu = (uint32_t)(tid + e * T);
            if (((low >> e) & 1u) && key[e] == kl) il = (uint32_t)(tid + e * T);
        }
        const uint32_t wu = __reduce_min_sync(FULL, iu), wl = __reduce_min_sync(FULL, il);
        SmoPick* pk = &picks[it & 1][0][0];
        if (wu == NONE ? lane == 0 : iu == wu) {
            SmoPick q = {ku, wu, 0.f, 0};
            if (wu != NONE) q.alpha = alpha[wu], q.y = (ypos >> ((wu - tid) / T)) & 1u ? 1 : -1;
            pk[warp] = q;
        }
        if (wl == NONE ? lane == 0 : il == wl) {
            SmoPick q = {kl, wl, 0.f, 0};
            if (wl != NONE) q.alpha = alpha[wl], q.y = (ypos >> ((wl - tid) / T)) & 1u ? 1 : -1;
            pk[NW + warp] = q;
        }
        __syncthreads();
        // i = argmax over the rows that may move up, j = argmin over those that may move down
        SmoPick a = {INT_MIN, NONE, 0.f, 0}, b = {INT_MAX, NONE, 0.f, 0};
        if (lane < NW) {
            a = pk[lane];
            b = pk[NW + lane];
        }
        ku = __reduce_max_sync(FULL, a.idx == NONE ? INT_MIN : a.key);
        kl = __reduce_min_sync(FULL, b.idx == NONE ? INT_MAX : b.key);
        iu = __reduce_min_sync(FULL, a.key == ku ? a.idx : NONE);
        il = __reduce_min_sync(FULL, b.key == kl ? b.idx : NONE);
        mu = key_float(ku);
        ml = key_float(kl);
        if (iu == NONE || il == NONE || mu - ml <= eps || it >= max_iter) break;
        const float* Ki = K + (size_t)iu * n;
        const float* Kj = K + (size_t)il * n;
        const float kij = __ldg(Ki + il);
        float vi[EPT], vj[EPT];
#pragma unroll
        for (int e = 0; e < EPT; ++e) {
            const int t = tid + e * T;
            vi[e] = t < n ? __ldg(Ki + t) : 0.f;
            vj[e] = t < n ? __ldg(Kj + t) : 0.f;
        }
        const int sa = __ffs(__ballot_sync(FULL, a.idx == iu)) - 1, sb = __ffs(__ballot_sync(FULL, b.idx == il)) - 1;
        const float alpha_i = __shfl_sync(FULL, a.alpha, sa), alpha_j = __shfl_sync(FULL, b.alpha, sb);
        const int yi = __shfl_sync(FULL, a.y, sa), yj = __shfl_sync(FULL, b.y, sb);
        float eta = 1.f + 1.f - 2.f * kij;
        if (eta < 1e-12f) eta = 1e-12f;
        float lam = (mu - ml) / eta;
        const float lim_i = yi > 0 ? cost - alpha_i : alpha_i;
        const float lim_j = yj > 0 ? alpha_j : cost - alpha_j;
        const bool hit_i = lam >= lim_i, hit_j = lam >= lim_j;
        lam = fminf(lam, fminf(lim_i, lim_j));
        float ai = alpha_i + (float)yi * lam, aj = alpha_j - (float)yj * lam;
        ai = fminf(fmaxf(ai, 0.f), cost);
        aj = fminf(fmaxf(aj, 0.f), cost);
        if (hit_i && lam == lim_i) ai = yi > 0 ? cost : 0.f;  // snap the box edges exactly
        if (hit_j && lam == lim_j) aj = yj > 0 ? 0.f : cost;
        auto move = [&](uint32_t row, float al, int y) {  // by the thread that owns the row
            if ((int)(row % T) != tid) return;
            const uint32_t bit = 1u << (row / T);
            alpha[row] = al;
            const bool can_grow = al < cost, can_shrink = al > 0.f;
            up = (y > 0 ? can_grow : can_shrink) ? up | bit : up & ~bit;
            low = (y > 0 ? can_shrink : can_grow) ? low | bit : low & ~bit;
        };
        move(iu, ai, yi);
        move(il, aj, yj);
#pragma unroll
        for (int e = 0; e < EPT; ++e) u[e] = fmaf(-lam, vi[e] - vj[e], u[e]);
    }
    // bias: mean of -y G over the free vectors, else the midpoint of the last bounds.  In fp32 the
    // order counts: rows t, t + 1024, t + 2048, ... in a chain, 32 neighbouring chains by halves,
    // and those sums in order, whatever T is.
    constexpr int CH = EPT < 1024 / T ? EPT : 1024 / T;  // chains per thread
#pragma unroll
    for (int q = 0; q < CH; ++q) {
        float s = 0.f;
        int k = 0;
#pragma unroll
        for (int e = q; e < EPT; e += CH) {
            const int t = tid + e * T;
            if (t < n && alpha[t] > 0.f && alpha[t] < cost) {
                s += u[e];
                ++k;
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(FULL, s, off);
        k = __reduce_add_sync(FULL, k);
        if (lane == 0) sums[q * NW + warp] = s, counts[q * NW + warp] = k;
    }
    __syncthreads();
    if (tid == 0) {
        float s = 0.f;
        int k = 0;
        for (int w = 0; w < CH * NW; ++w) s += sums[w], k += counts[w];
        float b;
        if (k > 0)
            b = s / (float)k;
        else if (iu != NONE && il != NONE)
            b = 0.5f * (mu + ml);
        else if (iu != NONE)
            b = mu;
        else if (il != NONE)
            b = ml;
        else
            b = 0.f;
        bias[c] = b;
        iters[c] = it;
    }
#pragma unroll
    for (int e = 0; e < EPT; ++e) {
        const int t = tid + e * T;
        if (t < n) coef[(size_t)c * n + t] = ((ypos >> e) & 1u ? 1.f : -1.f) * alpha[t];
    }
}

template <int BM, bool VEC, bool ORDERED>
cudaError_t launch_kernel_matrix(int grid, const float* x, const float* xsq, int n, int k_pad, float gamma,
                                 long long tiles, float* K, const F32HandOver& ho, int32_t* failed, int n_classes,
                                 cudaStream_t s) {
    const size_t smem = sizeof(typename F32Tile<BM, BM>::Smem);
    kernel_matrix_kernel<BM, VEC, ORDERED>
        <<<grid, F32Tile<BM, BM>::NT, smem, s>>>(x, xsq, n, k_pad, gamma, tiles, K, ho, failed, n_classes);
    return cudaGetLastError();
}

template <int T, int EPT>
cudaError_t launch_smo(const float* K, int n, const int32_t* labels, int n_classes, float cost, float eps,
                       int max_iter, float* coef, float* bias, int32_t* iters, bool marked, cudaStream_t s) {
    const size_t smem = sizeof(float) * (size_t)n;
    const cudaError_t e = cudaFuncSetAttribute(smo_kernel<T, EPT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)sizeof(float) * T * EPT);
    if (e != cudaSuccess) return e;
    smo_kernel<T, EPT><<<n_classes, T, smem, s>>>(K, n, labels, cost, eps, max_iter, coef, bias, iters, marked);
    return cudaGetLastError();
}

}  // namespace
}  // namespace rgbd

using namespace rgbd;

extern "C" int svm_train_rbf(rgbd_ctx* ctx, const float* x, const float* xsq, int n, int k_pad, const int32_t* labels,
                             int n_classes, float gamma, float cost, float eps, int max_iter, float* coef, float* bias,
                             int32_t* iters, void* stream) {
    rgbd::NvtxRange nvtx_range("svm_train_rbf");
    if (!ctx) return set_error(RGBD_ERR_ARG, "svm_train_rbf: ctx is NULL");
    if (n < 2 || n > 16384 || k_pad <= 0 || n_classes < 1 || !(gamma > 0.f) || !(cost > 0.f) || !(eps > 0.f) ||
        max_iter < 0 || max_iter > 2000000)
        return set_error(RGBD_ERR_ARG,
                         "svm_train_rbf: n %d (2..16384), k_pad %d, classes %d, gamma %g, cost %g, eps %g, max_iter %d (0..2e6)",
                         n, k_pad, n_classes, gamma, cost, eps, max_iter);
    if (!x || !xsq || !labels || !coef || !bias || !iters) return set_error(RGBD_ERR_ARG, "svm_train_rbf: NULL pointer");
    DeviceGuard g(ctx->props.device);
    cudaStream_t s = (cudaStream_t)stream;
    // 128 x 128 tiles spread over one CTA per SM when there is at least one for each, smaller tiles
    // with a CTA each otherwise (a full 4096 x 4096 x 15104 product: 8.8 ms in 128 x 128
    // tiles, 9.3 ms in 64 x 64; 168 of the large tiles, 777 x 3001: 1.45 ms spread, 2.0 ms as small ones).
    const long long b128 = (n + 127) / 128, t128 = b128 * (b128 + 1) / 2;
    const bool ordered = t128 >= ctx->props.sm_count && n >= ctx->props.sm_count;
    const long long b64 = (n + 63) / 64;
    const long long tiles = ordered ? t128 : b64 * (b64 + 1) / 2;
    const int grid = ordered ? ctx->props.sm_count : (int)tiles;
    int rc = ensure_workspace(ctx, sizeof(float) * (size_t)n * n, s);
    if (rc) return rc;
    float* K = (float*)ctx->workspace;
    // the hand-over flags live in the coefficients until SMO writes them (n >= 2049 when ordered), the
    // marks of a failed one in the step counts
    const F32HandOver ho = {reinterpret_cast<uint32_t*>(coef), ctx->d_status, ctx->handover_ns, ctx->drop_handover};
    const bool vec = k_pad % 16 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    cudaError_t e = cudaSuccess;
    if (ordered) {
        e = cudaMemsetAsync(ho.ready, 0, sizeof(uint32_t) * (size_t)grid, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(iters, 0, sizeof(int32_t) * (size_t)n_classes, s);
        if (e != cudaSuccess) return cuda_error(e, "svm_train_rbf: tile hand-over reset");
        e = vec ? launch_kernel_matrix<128, true, true>(grid, x, xsq, n, k_pad, gamma, tiles, K, ho, iters, n_classes, s)
                : launch_kernel_matrix<128, false, true>(grid, x, xsq, n, k_pad, gamma, tiles, K, ho, iters, n_classes, s);
    } else {
        e = vec ? launch_kernel_matrix<64, true, false>(grid, x, xsq, n, k_pad, gamma, tiles, K, ho, iters, n_classes, s)
                : launch_kernel_matrix<64, false, false>(grid, x, xsq, n, k_pad, gamma, tiles, K, ho, iters, n_classes, s);
    }
    if (e != cudaSuccess) return cuda_error(e, "svm_train_rbf: kernel matrix launch");
    // Up to 16 rows per thread (they live in registers), and no more warps than that takes: the
    // selection and the barrier cost every warp the same, however few rows it holds (4096 rows:
    // 1.86 ms with 8 warps, 2.48 ms with 32).
#define RGBD_SMO(TV, EV) launch_smo<TV, EV>(K, n, labels, n_classes, cost, eps, max_iter, coef, bias, iters, ordered, s)
    e = n <= 256    ? RGBD_SMO(256, 1)
        : n <= 1024 ? RGBD_SMO(256, 4)
        : n <= 2048 ? RGBD_SMO(256, 8)
        : n <= 4096 ? RGBD_SMO(256, 16)
        : n <= 8192 ? RGBD_SMO(512, 16)
                    : RGBD_SMO(1024, 16);
#undef RGBD_SMO
    if (e != cudaSuccess) return cuda_error(e, "svm_train_rbf: SMO launch");
    return RGBD_OK;
}
