// train.cu -- one-vs-rest RBF SVM training on the GPU (Section 2.5 trains the classifier on the
// face database; the paper does it on the CPU).  The dual problem of every class is solved by
// sequential minimal optimisation with the maximal violating pair, on one kernel matrix that all
// classes share:
//   kernel_matrix_kernel  K_st = exp(-gamma max(0, |x_s|^2 + |x_t|^2 - 2 x_s . x_t)), fp32, one
//                         tile of the lower triangle per CTA, written twice;
//   smo_kernel            one CTA per class; alpha and the gradient G stay in shared memory; each
//                         step reduces the two selections over the CTA, updates the pair on one
//                         thread, then G_t += y_t lambda (K_it - K_jt) with all threads.
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
                                                                          float* K, uint32_t* ready,
                                                                          uint32_t* status) {
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
        f32_ordered_tiles<Tile, VEC>(tiles, k_pad, ready, status, sm, rows, finish, stash, fetch);
    } else {
        const F32Rows r = rows(blockIdx.x);
        Tile t;
        t.clear();
        t.template run<VEC>(r.a, r.na, r.b, r.nb, k_pad, 0, (k_pad + Tile::KB - 1) / Tile::KB, sm);
        finish(blockIdx.x, t);
    }
}

constexpr int SMO_THREADS = 1024;

// (value, index) pairs: the larger value wins (or the smaller, for the minimum), then the lower index
__device__ __forceinline__ void arg_better_max(float& v, int& i, float ov, int oi) {
    if (oi >= 0 && (i < 0 || ov > v || (ov == v && oi < i))) {
        v = ov;
        i = oi;
    }
}
__device__ __forceinline__ void arg_better_min(float& v, int& i, float ov, int oi) {
    if (oi >= 0 && (i < 0 || ov < v || (ov == v && oi < i))) {
        v = ov;
        i = oi;
    }
}

__global__ void __launch_bounds__(SMO_THREADS, 1) smo_kernel(const float* __restrict__ K, int n,
                                                            const int32_t* __restrict__ labels, float cost, float eps,
                                                            int max_iter, float* __restrict__ coef,
                                                            float* __restrict__ bias, int32_t* __restrict__ iters) {
    extern __shared__ float smo_smem[];
    float* alpha = smo_smem;
    float* G = smo_smem + n;
    int8_t* y = reinterpret_cast<int8_t*>(smo_smem + 2 * n);
    __shared__ float rv[2][32];
    __shared__ int ri[2][32];
    __shared__ int sel_i, sel_j, stop;
    __shared__ float sel_lam, sel_m, sel_M;
    const int c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int t = tid; t < n; t += SMO_THREADS) {
        y[t] = labels[t] == c ? 1 : -1;
        alpha[t] = 0.f;
        G[t] = -1.f;
    }
    __syncthreads();
    int it = 0;
    for (;;) {
        // selection: i = argmax over I_up of -y G, j = argmin over I_low of -y G
        float mu = 0.f, ml = 0.f;
        int iu = -1, il = -1;
        for (int t = tid; t < n; t += SMO_THREADS) {
            const float v = -(float)y[t] * G[t];
            const bool up = (y[t] > 0 && alpha[t] < cost) || (y[t] < 0 && alpha[t] > 0.f);
            const bool low = (y[t] > 0 && alpha[t] > 0.f) || (y[t] < 0 && alpha[t] < cost);
            if (up) arg_better_max(mu, iu, v, t);
            if (low) arg_better_min(ml, il, v, t);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            arg_better_max(mu, iu, __shfl_xor_sync(0xFFFFFFFFu, mu, off), __shfl_xor_sync(0xFFFFFFFFu, iu, off));
            arg_better_min(ml, il, __shfl_xor_sync(0xFFFFFFFFu, ml, off), __shfl_xor_sync(0xFFFFFFFFu, il, off));
        }
        if (lane == 0) {
            rv[0][warp] = mu, ri[0][warp] = iu;
            rv[1][warp] = ml, ri[1][warp] = il;
        }
        __syncthreads();
        if (tid == 0) {
            for (int w = 1; w < SMO_THREADS / 32; ++w) {
                arg_better_max(mu, iu, rv[0][w], ri[0][w]);
                arg_better_min(ml, il, rv[1][w], ri[1][w]);
            }
            sel_m = mu, sel_M = ml;
            sel_i = iu, sel_j = il;
            int st = iu < 0 || il < 0 || mu - ml <= eps || it >= max_iter;
            if (!st) {
                const float kii = K[(size_t)iu * n + iu], kjj = K[(size_t)il * n + il], kij = K[(size_t)iu * n + il];
                float eta = kii + kjj - 2.f * kij;
                if (eta < 1e-12f) eta = 1e-12f;
                float lam = (mu - ml) / eta;
                const float lim_i = y[iu] > 0 ? cost - alpha[iu] : alpha[iu];
                const float lim_j = y[il] > 0 ? alpha[il] : cost - alpha[il];
                const bool hit_i = lam >= lim_i, hit_j = lam >= lim_j;
                lam = fminf(lam, fminf(lim_i, lim_j));
                float ai = alpha[iu] + (float)y[iu] * lam, aj = alpha[il] - (float)y[il] * lam;
                ai = fminf(fmaxf(ai, 0.f), cost);
                aj = fminf(fmaxf(aj, 0.f), cost);
                if (hit_i && lam == lim_i) ai = y[iu] > 0 ? cost : 0.f;  // snap the box edges exactly
                if (hit_j && lam == lim_j) aj = y[il] > 0 ? 0.f : cost;
                alpha[iu] = ai;
                alpha[il] = aj;
                sel_lam = lam;
            }
            stop = st;
        }
        __syncthreads();
        if (stop) break;
        const float lam = sel_lam;
        const float* Ki = K + (size_t)sel_i * n;
        const float* Kj = K + (size_t)sel_j * n;
        for (int t = tid; t < n; t += SMO_THREADS) G[t] += (float)y[t] * lam * (Ki[t] - Kj[t]);
        ++it;
        __syncthreads();
    }
    // bias: mean of -y G over the free vectors, else the midpoint of the last bounds
    float sum = 0.f;
    int cnt = 0;
    for (int t = tid; t < n; t += SMO_THREADS)
        if (alpha[t] > 0.f && alpha[t] < cost) {
            sum += -(float)y[t] * G[t];
            ++cnt;
        }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
        cnt += __shfl_xor_sync(0xFFFFFFFFu, cnt, off);
    }
    __syncthreads();
    if (lane == 0) {
        rv[0][warp] = sum;
        ri[0][warp] = cnt;
    }
    __syncthreads();
    if (tid == 0) {
        float s = 0.f;
        int k = 0;
        for (int w = 0; w < SMO_THREADS / 32; ++w) s += rv[0][w], k += ri[0][w];
        float b;
        if (k > 0)
            b = s / (float)k;
        else if (sel_i >= 0 && sel_j >= 0)
            b = 0.5f * (sel_m + sel_M);
        else if (sel_i >= 0)
            b = sel_m;
        else if (sel_j >= 0)
            b = sel_M;
        else
            b = 0.f;
        bias[c] = b;
        iters[c] = it;
    }
    for (int t = tid; t < n; t += SMO_THREADS) coef[(size_t)c * n + t] = (float)y[t] * alpha[t];
}

template <int BM, bool VEC, bool ORDERED>
cudaError_t launch_kernel_matrix(int grid, const float* x, const float* xsq, int n, int k_pad, float gamma,
                                 long long tiles, float* K, uint32_t* ready, uint32_t* status, cudaStream_t s) {
    const size_t smem = sizeof(typename F32Tile<BM, BM>::Smem);
    kernel_matrix_kernel<BM, VEC, ORDERED>
        <<<grid, F32Tile<BM, BM>::NT, smem, s>>>(x, xsq, n, k_pad, gamma, tiles, K, ready, status);
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
    // the hand-over flags live in the coefficients until SMO writes them (n >= 2049 when ordered)
    uint32_t* ready = reinterpret_cast<uint32_t*>(coef);
    const bool vec = k_pad % 16 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
    cudaError_t e = cudaSuccess;
    if (ordered) {
        e = cudaMemsetAsync(ready, 0, sizeof(uint32_t) * (size_t)grid, s);
        if (e != cudaSuccess) return cuda_error(e, "svm_train_rbf: tile hand-over reset");
        e = vec ? launch_kernel_matrix<128, true, true>(grid, x, xsq, n, k_pad, gamma, tiles, K, ready, ctx->d_status, s)
                : launch_kernel_matrix<128, false, true>(grid, x, xsq, n, k_pad, gamma, tiles, K, ready, ctx->d_status, s);
    } else {
        e = vec ? launch_kernel_matrix<64, true, false>(grid, x, xsq, n, k_pad, gamma, tiles, K, ready, ctx->d_status, s)
                : launch_kernel_matrix<64, false, false>(grid, x, xsq, n, k_pad, gamma, tiles, K, ready, ctx->d_status, s);
    }
    if (e != cudaSuccess) return cuda_error(e, "svm_train_rbf: kernel matrix launch");
    const size_t smem = sizeof(float) * 2 * (size_t)n + (size_t)n;
    e = cudaFuncSetAttribute(smo_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(e, "svm_train_rbf: smem attribute");
    smo_kernel<<<n_classes, SMO_THREADS, smem, s>>>(K, n, labels, cost, eps, max_iter, coef, bias, iters);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "svm_train_rbf: SMO launch");
    return RGBD_OK;
}
