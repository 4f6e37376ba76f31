// rows.cu -- A5 alone: normalised rows from stored counts (Section 2.4's histograms per cell), and
// the row passes of model packing: quantisation, column means, centring.
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include <algorithm>

#include "internal.h"

namespace rgbd {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

// ---------------------------------------------------------------------------------------
// A5 alone: per-cell normalisation of count rows; one CTA per row.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ float store_x(void* out, int dtype, size_t idx, float x, float scale,
                                         size_t plane = 0) {
    if (dtype == RGBD_DT_BF16) {
        const __nv_bfloat16 q = __float2bfloat16_rn(x);
        reinterpret_cast<uint16_t*>(out)[idx] = __bfloat16_as_ushort(q);
        return __bfloat162float(q);
    } else if (dtype == RGBD_DT_BF16X3) {
        // hi = bf16(x), lo = bf16(x - hi): x = hi + lo to 2^-18 relative
        const __nv_bfloat16 hi = __float2bfloat16_rn(x);
        const float hf = __bfloat162float(hi);
        const __nv_bfloat16 lo = __float2bfloat16_rn(x - hf);
        reinterpret_cast<uint16_t*>(out)[idx] = __bfloat16_as_ushort(hi);
        reinterpret_cast<uint16_t*>(out)[idx + plane] = __bfloat16_as_ushort(lo);
        return hf + __bfloat162float(lo);
    } else if (dtype == RGBD_DT_FP8) {
        const __nv_fp8_e4m3 q(x * scale);
        reinterpret_cast<uint8_t*>(out)[idx] = q.__x;
        return static_cast<float>(q) * (1.0f / scale);
    }
    reinterpret_cast<float*>(out)[idx] = x;
    return x;
}

// Rows staged in shared memory: one CTA per row reads it once (16-byte asynchronous copies), sums
// its cells from shared memory (LPC lanes per cell, two counts per dot product), makes 8
// neighbouring outputs per thread step, stored in 16-byte words, and last sums the norm.  HBM
// bounds the row (each count read once, each value written once), instruction issue is close
// behind: a value's quotient takes 5 instructions and its norm 3.
//   h / t is q0 = h (1/t) followed by Markstein's correction q = fma(fma(-q0, t, h), 1/t, q0)
//   (P. Markstein, IBM J. Res. Dev. 34(1), 1990), with 1/t the correctly rounded reciprocal of the
//   cell's sum: the IEEE quotient whenever t is not all ones in its significand, and
//   t <= 256 * 65535 < 2^24 - 1.  A count becomes a float by its bits (2^23 + h) - 2^23, exactly.
//   The norm is summed as the general form below sums it (thread t adds the values t, t + 256, ... in
//   a chain), so a row's norm does not depend on the form: from the values of 16 or fewer bits left
//   in place of the counts, or from the row just written (which L2 still has).
// 8192 rows x 15104 to bf16: 412 us when every value was read twice in 2-byte loads and divided,
// 120 us when the chain's order was the order of the outputs too (31 instructions a value), 100 us
// with the norm in its own pass.
constexpr int kRowThreads = 256;

template <int DT, bool CENTRED>
__global__ void __launch_bounds__(kRowThreads) normalize_rows_kernel(
    const uint16_t* __restrict__ feats, int n, int dim, int nbins, uint32_t nbins_inv, int lpc_log2, int wide_in,
    void* x_out, int k_pad, float x_scale, float* __restrict__ xsq, float* row_max, size_t plane,
    const float* __restrict__ centre) {
    extern __shared__ __align__(16) unsigned char rows_smem[];
    const int cells = dim / nbins, dim8 = (dim + 7) & ~7;
    uint16_t* cnt = reinterpret_cast<uint16_t*>(rows_smem);                         // [dim8], zero past dim
    float2* inv = reinterpret_cast<float2*>(rows_smem + 2 * (size_t)dim8);          // [cells + 2]: t, 1 / t
    __shared__ float red[kRowThreads / 32];
    const int tid = threadIdx.x;
    const float back = DT == RGBD_DT_FP8 ? 1.0f / x_scale : 1.f;
    for (int row = blockIdx.x; row < n; row += gridDim.x) {
        const uint16_t* h = feats + (size_t)row * dim;
        __syncthreads();  // the row before is done with shared memory
        if (wide_in) {
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(cnt);
            for (int j = 8 * tid; j < dim; j += 8 * kRowThreads)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 2u * j), "l"(h + j) : "memory");
            asm volatile("cp.async.wait_all;" ::: "memory");
        } else {
            for (int j = tid; j < dim8; j += kRowThreads) cnt[j] = j < dim ? __ldg(h + j) : (uint16_t)0;
        }
        __syncthreads();
        // cell sums: LPC lanes per cell; the words of a cell's range, its odd ends apart
        const int lpc = 1 << lpc_log2;
        for (int i0 = 0; i0 < (cells << lpc_log2); i0 += kRowThreads) {  // whole warps: the sums shuffle
            const int i = i0 + tid, c = i >> lpc_log2, sub = i & (lpc - 1);
            uint32_t t = 0;
            if (c < cells) {
                int b = c * nbins, e = b + nbins;
                if (b & 1) {
                    if (sub == 0) t += cnt[b];
                    ++b;
                }
                if (e & 1) {
                    --e;
                    if (sub == 0) t += cnt[e];
                }
                const uint32_t* w = reinterpret_cast<const uint32_t*>(cnt);
                for (int k = (b >> 1) + sub; k < (e >> 1); k += lpc) t = __dp2a_lo(w[k], 0x0101u, t);
            }
            for (int off = lpc >> 1; off > 0; off >>= 1) t += __shfl_xor_sync(FULL, t, off);
            if (c < cells && sub == 0) {
                const float tf = (float)t;  // exact: below 2^24
                inv[c] = make_float2(tf, t ? __frcp_rn(tf) : 0.f);
            }
        }
        if (tid < 2) inv[cells + tid] = make_float2(0.f, 0.f);
        __syncthreads();
        float mx = 0.f;
        for (int j = 8 * tid; j < k_pad; j += 8 * kRowThreads) {
            float x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = 0.f;
            if (j < dim) {
                const uint4 hv = *reinterpret_cast<const uint4*>(cnt + j);
                const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w};
                const int c0 = (int)__umulhi((uint32_t)j, nbins_inv);  // j / nbins
                const int left = (c0 + 1) * nbins - j;                 // values before the next cell
                const float2 ca = inv[c0], cb = inv[c0 + 1];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float t = e < left ? ca.x : cb.x, r = e < left ? ca.y : cb.y;
                    const float hf = __uint_as_float(__byte_perm(hw[e >> 1], 0x4B000000u, e & 1 ? 0x7632 : 0x7610)) - 8388608.f;
                    const float q0 = __fmul_rn(hf, r);
                    x[e] = __fmaf_rn(__fmaf_rn(-q0, t, hf), r, q0);
                }
                if (CENTRED) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = j + e < dim ? __fsub_rn(x[e], __ldg(centre + j + e)) : 0.f;
                }
            }
            if (row_max) {
#pragma unroll
                for (int e = 0; e < 8; ++e) mx = fmaxf(mx, fabsf(x[e]));
            }
            const size_t at = (size_t)row * k_pad + j;
            if (DT == RGBD_DT_BF16 || DT == RGBD_DT_BF16X3) {
                uint32_t hi[4], lo[4];
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const __nv_bfloat162 b = __floats2bfloat162_rn(x[e], x[e + 1]);
                    hi[e >> 1] = *reinterpret_cast<const uint32_t*>(&b);
                    if (DT == RGBD_DT_BF16X3) {
                        const __nv_bfloat162 l = __floats2bfloat162_rn(x[e] - __low2float(b), x[e + 1] - __high2float(b));
                        lo[e >> 1] = *reinterpret_cast<const uint32_t*>(&l);
                    }
                }
                uint16_t* o = reinterpret_cast<uint16_t*>(x_out) + at;
                const uint4 hv = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<uint4*>(o) = hv;
                if (DT == RGBD_DT_BF16X3)
                    *reinterpret_cast<uint4*>(o + plane) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                else if (j < dim)
                    *reinterpret_cast<uint4*>(cnt + j) = hv;
            } else if (DT == RGBD_DT_FP8) {
                uint32_t c[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) c[e] = __nv_fp8_e4m3(x[e] * x_scale).__x;
                *reinterpret_cast<uint2*>(reinterpret_cast<uint8_t*>(x_out) + at) =
                    make_uint2(c[0] | (c[1] << 8) | (c[2] << 16) | (c[3] << 24),
                               c[4] | (c[5] << 8) | (c[6] << 16) | (c[7] << 24));
                if (j < dim)
                    *reinterpret_cast<uint4*>(cnt + j) = make_uint4(c[0] | (c[1] << 16), c[2] | (c[3] << 16),
                                                                   c[4] | (c[5] << 16), c[6] | (c[7] << 16));
            } else {
                float4* o = reinterpret_cast<float4*>(reinterpret_cast<float*>(x_out) + at);
                o[0] = make_float4(x[0], x[1], x[2], x[3]);
                o[1] = make_float4(x[4], x[5], x[6], x[7]);
            }
        }
        if (row_max) {
            for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, off));
            if (tid % 32 == 0) atomicMax(reinterpret_cast<int*>(row_max), __float_as_int(mx));  // mx >= 0
        }
        if (!xsq) continue;
        __syncthreads();  // the row's values are in place
        float sq = 0.f;
        const size_t at = (size_t)row * k_pad;
#pragma unroll 8
        for (int j = tid; j < dim; j += kRowThreads) {
            float v;
            if (DT == RGBD_DT_BF16) {
                v = __uint_as_float((uint32_t)cnt[j] << 16);
            } else if (DT == RGBD_DT_FP8) {
                __nv_fp8_e4m3 q;
                q.__x = (__nv_fp8_storage_t)cnt[j];
                v = static_cast<float>(q) * back;
            } else if (DT == RGBD_DT_BF16X3) {
                const uint16_t* o = reinterpret_cast<const uint16_t*>(x_out) + at + j;
                v = __uint_as_float((uint32_t)o[0] << 16) + __uint_as_float((uint32_t)o[plane] << 16);
            } else {
                v = reinterpret_cast<const float*>(x_out)[at + j];
            }
            sq = fmaf(v, v, sq);
        }
        for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(FULL, sq, off);
        if (tid % 32 == 0) red[tid / 32] = sq;
        __syncthreads();
        if (tid == 0) {
            float t = 0.f;
            for (int w = 0; w < kRowThreads / 32; ++w) t += red[w];
            xsq[row] = t;
        }
    }
}

// The general form: rows too long for shared memory, cells of fewer than 8 bins, unaligned output.
__global__ void normalize_kernel(const uint16_t* __restrict__ feats, int n, int dim, int nbins,
                                 int x_dtype, void* x_out, int k_pad, float x_scale, float* xsq,
                                 float* row_max, size_t plane, const float* __restrict__ centre) {
    extern __shared__ uint32_t nv[];  // [dim / nbins]
    __shared__ float red[2][32];
    const int cells = dim / nbins;
    for (int row = blockIdx.x; row < n; row += gridDim.x) {
        __syncthreads();
        const uint16_t* h = feats + (size_t)row * dim;
        for (int c = threadIdx.x; c < cells; c += blockDim.x) {
            uint32_t t = 0;
            for (int b = 0; b < nbins; ++b) t += h[c * nbins + b];
            nv[c] = t;
        }
        __syncthreads();
        float sq = 0.f, mx = 0.f;
        for (int j = threadIdx.x; j < k_pad; j += blockDim.x) {
            float x = 0.f;
            if (j < dim) {
                const uint32_t t = nv[j / nbins];
                x = t ? (float)h[j] / (float)t : 0.f;
                if (centre) x = __fsub_rn(x, centre[j]);
            }
            mx = fmaxf(mx, fabsf(x));
            const float q = store_x(x_out, x_dtype, (size_t)row * k_pad + j, x, x_scale, plane);
            sq = fmaf(q, q, sq);
        }
        for (int off = 16; off > 0; off >>= 1) {
            sq += __shfl_xor_sync(FULL, sq, off);
            mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, off));
        }
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (lane == 0) {
            red[0][warp] = sq;
            red[1][warp] = mx;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.f, m = 0.f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
                t += red[0][w];
                m = fmaxf(m, red[1][w]);
            }
            if (xsq) xsq[row] = t;
            if (row_max) atomicMax(reinterpret_cast<int*>(row_max), __float_as_int(m));  // m >= 0
        }
    }
}

// fp32 rows -> dtype rows (FP8 with `scale`), with squared norms of the stored values.
__global__ void quantize_kernel(const float* __restrict__ src, int n, int k_pad, int dtype, void* dst,
                                float scale, float* sq_out, size_t plane) {
    __shared__ float red[32];
    for (int row = blockIdx.x; row < n; row += gridDim.x) {
        __syncthreads();
        float sq = 0.f;
        for (int j = threadIdx.x; j < k_pad; j += blockDim.x) {
            const float q = store_x(dst, dtype, (size_t)row * k_pad + j, src[(size_t)row * k_pad + j], scale, plane);
            sq = fmaf(q, q, sq);
        }
        for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(FULL, sq, off);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sq;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
            if (sq_out) sq_out[row] = t;
        }
    }
}

// mu[j] = fp32(sum_i rows[i][j] / n), the sum in fp64 in row order (one thread per column, so
// the order and the result are fixed); mu[j] = 0 for j >= dim.
__global__ void column_mean_kernel(const float* __restrict__ rows, int n, int dim, int k_pad, float* __restrict__ mu) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= k_pad) return;
    double acc = 0.0;
    if (j < dim)
        for (int i = 0; i < n; ++i) acc += (double)rows[(size_t)i * k_pad + j];
    mu[j] = j < dim ? (float)(acc / (double)n) : 0.f;
}

// rows[i][j] -= mu[j] (fp32, round to nearest even); *absmax = max |result| (non-negative floats
// order like their bit patterns, so an integer max serves).
__global__ void centre_kernel(float* __restrict__ rows, int n, int k_pad, const float* __restrict__ mu,
                              float* absmax) {
    __shared__ float red[32];
    for (int row = blockIdx.x; row < n; row += gridDim.x) {
        float m = 0.f;
        for (int j = threadIdx.x; j < k_pad; j += blockDim.x) {
            const size_t idx = (size_t)row * k_pad + j;
            const float v = __fsub_rn(rows[idx], mu[j]);
            rows[idx] = v;
            m = fmaxf(m, fabsf(v));
        }
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, off));
        __syncthreads();
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, red[w]);
            atomicMax(reinterpret_cast<int*>(absmax), __float_as_int(m));
        }
    }
}

}  // namespace

int launch_normalize(const uint16_t* feats, int n, int dim, int nbins, int x_dtype, void* x_out,
                     int k_pad, float x_scale, float* xsq, float* row_max, cudaStream_t s, size_t plane,
                     const float* centre) {
    const int cells = dim / nbins;
    if (plane == 0) plane = (size_t)n * k_pad;
    cudaError_t e;
    // Staged rows: any row of up to 64 K counts (131 KB of the 227 KB of shared memory; the widest
    // rows of this library have 15104, 32 KB, six CTAs per SM) with at most one cell border in a
    // group of 8, written to a 16-byte aligned buffer (k_pad and the plane are multiples of 128).
    const size_t staged = 2 * (size_t)((dim + 7) & ~7) + sizeof(float2) * ((size_t)cells + 2);
    if (dim <= 65536 && nbins >= 8 && (reinterpret_cast<uintptr_t>(x_out) & 15) == 0 && (plane & 7) == 0) {
        int lpc = 0;  // lanes per cell: few cells (one 256-bin histogram per row) share the summing
        while (lpc < 5 && (cells << (lpc + 1)) <= kRowThreads) ++lpc;
        const uint32_t inv = (uint32_t)((0x100000000ull + nbins - 1) / nbins);  // j / nbins for j < 2^24
        const int wide = dim % 8 == 0 && (reinterpret_cast<uintptr_t>(feats) & 15) == 0;
        const bool centred = centre != nullptr;
        auto kernel = centred ? normalize_rows_kernel<RGBD_DT_F32, true> : normalize_rows_kernel<RGBD_DT_F32, false>;
        if (x_dtype == RGBD_DT_BF16)
            kernel = centred ? normalize_rows_kernel<RGBD_DT_BF16, true> : normalize_rows_kernel<RGBD_DT_BF16, false>;
        else if (x_dtype == RGBD_DT_FP8)
            kernel = centred ? normalize_rows_kernel<RGBD_DT_FP8, true> : normalize_rows_kernel<RGBD_DT_FP8, false>;
        else if (x_dtype == RGBD_DT_BF16X3)
            kernel = centred ? normalize_rows_kernel<RGBD_DT_BF16X3, true> : normalize_rows_kernel<RGBD_DT_BF16X3, false>;
        if (staged > 48 * 1024) {
            constexpr size_t most = 2 * (size_t)65536 + sizeof(float2) * (65536 / 8 + 2);
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
            if (e != cudaSuccess) return cuda_error(e, "lbp_normalize_features: smem attribute");
        }
        kernel<<<n, kRowThreads, staged, s>>>(feats, n, dim, nbins, inv, lpc, wide, x_out, k_pad, x_scale, xsq,
                                              row_max, plane, centre);
        e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_error(e, "lbp_normalize_features: launch");
        return RGBD_OK;
    }
    const size_t smem = sizeof(uint32_t) * (size_t)cells;
    if (smem > 48 * 1024) return set_error(RGBD_ERR_UNSUPPORTED, "normalize: %d cells", cells);
    const int grid = std::min(n, 8192);
    normalize_kernel<<<grid, 256, smem, s>>>(feats, n, dim, nbins, x_dtype, x_out, k_pad, x_scale,
                                             xsq, row_max, plane, centre);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "lbp_normalize_features: launch");
    return RGBD_OK;
}

int launch_quantize_f32(const float* src, int n, int k_pad, int x_dtype, void* dst, float scale,
                        float* sq, cudaStream_t s, size_t plane) {
    const int grid = std::min(n, 8192);
    if (plane == 0) plane = (size_t)n * k_pad;
    quantize_kernel<<<grid, 256, 0, s>>>(src, n, k_pad, x_dtype, dst, scale, sq, plane);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "quantize: launch");
    return RGBD_OK;
}

int launch_centre_rows(float* rows, int n, int dim, int k_pad, float* mu, float* absmax, cudaStream_t s) {
    column_mean_kernel<<<(k_pad + 255) / 256, 256, 0, s>>>(rows, n, dim, k_pad, mu);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "centre: mean launch");
    centre_kernel<<<std::min(n, 8192), 256, 0, s>>>(rows, n, k_pad, mu, absmax);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "centre: launch");
    return RGBD_OK;
}

}  // namespace rgbd
