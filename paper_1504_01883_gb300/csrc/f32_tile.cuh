// f32_tile.cuh -- the exact fp32 product G = A . B^T of two sets of rows, tile by tile, on the FMA
// pipes (no tensor core multiplies fp32): shared by the fp32 scoring path and the kernel matrix of
// training.  Every output is one chain acc = fma(a_k, b_k, acc) with k ascending from 0, whatever
// the tile and whoever computes which part of the chain, so results do not depend on the split.
#pragma once

#include <stdint.h>

#include "internal.h"

namespace rgbd {

__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// BM x BN outputs by (BM / 8)(BN / 8) threads, 16 values of k per stage.
// Bound by the fp32 FMA rate (128 a clock and SM).  A thread owns 8 x 8 outputs and issues packed
// FMAs (fma.rn.f32x2: two IEEE FMAs per instruction, each a chain of its own), which leaves issue
// slots free for the rest: per k four 16-byte shared loads, 8 moves that put an A value in both
// halves of a register pair, and 32 FMAs.  Rows come through registers (16 bytes of a row per load)
// and are stored transposed, two stages deep.  4096 x 4096 x 15104: 8.8 ms (57 TFLOP/s) in 128 x 128
// tiles, 9.3 ms in 64 x 64 tiles; 10.4 ms with A values doubled in shared memory instead of in
// registers (the loads then take 6 x 4 of the 64 cycles a k's FMAs take), 9.7 ms with scalar FMAs.
template <int BM, int BN>
struct F32Tile {
    static constexpr int KB = 16;
    static constexpr int NT = (BM / 8) * (BN / 8);
    static constexpr int WY = BM / 32;  // warps along m (a warp is 4 x 8 threads)
    static constexpr int QK = KB / 4;   // 16-byte loads per row and stage
    static constexpr int LA = BM * QK / NT, LB = BN * QK / NT;  // of them per thread
    static_assert(BM % 32 == 0 && BN % 64 == 0 && LA >= 1 && LB >= 1 && NT % QK == 0, "tile shape");
    struct Smem {
        float a[2][KB][BM + 4];
        float b[2][KB][BN + 4];
    };

    uint64_t acc[8][4];  // [m][pair of n]
    int ty, tx;

    __device__ __forceinline__ F32Tile() {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        ty = (warp % WY) * 4 + (lane >> 3);
        tx = (warp / WY) * 8 + (lane & 7);
    }
    // Row i (0..7) of this thread within the tile, and the first column of its pair p (0..3).
    __device__ __forceinline__ int m_of(int i) const { return (i >> 2) * (BM / 2) + ty * 4 + (i & 3); }
    __device__ __forceinline__ int n_of(int p) const { return (p >> 1) * (BN / 2) + tx * 4 + 2 * (p & 1); }
    __device__ __forceinline__ float get(int i, int p, int h) const {
        return __uint_as_float((uint32_t)(acc[i][p] >> (32 * h)));
    }
    __device__ __forceinline__ void put(int i, int p, float lo, float hi) {
        acc[i][p] = __float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
    }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[i][p] = 0ull;
    }

    // Continues every chain over the stages k0 .. k1 - 1 (of KB values) of rows of K values.
    // VEC: rows are 16-byte aligned and K a multiple of KB; else scalar loads, zero past K.
    // Rows past na (nb) repeat the last one: their outputs are not used.
    template <bool VEC>
    __device__ __forceinline__ void run(const float* __restrict__ a, int na, const float* __restrict__ b, int nb,
                                        int K, int k0, int k1, Smem& sm) {
        const int tid = threadIdx.x;
        const float *pa[LA], *pb[LB];
#pragma unroll
        for (int i = 0; i < LA; ++i) {
            const int e = tid + i * NT;
            pa[i] = a + (size_t)min(e / QK, na - 1) * K + 4 * (e % QK);
        }
#pragma unroll
        for (int i = 0; i < LB; ++i) {
            const int e = tid + i * NT;
            pb[i] = b + (size_t)min(e / QK, nb - 1) * K + 4 * (e % QK);
        }
        float4 ra[LA], rb[LB];
        auto fetch = [&](const float* p, int k) -> float4 {
            if (VEC) return __ldg(reinterpret_cast<const float4*>(p + k));
            const int left = K - k - 4 * (tid % QK);  // NT is a multiple of QK: every load's quad is tid's
            return make_float4(left > 0 ? __ldg(p + k) : 0.f, left > 1 ? __ldg(p + k + 1) : 0.f,
                               left > 2 ? __ldg(p + k + 2) : 0.f, left > 3 ? __ldg(p + k + 3) : 0.f);
        };
        auto load = [&](int kt) {
#pragma unroll
            for (int i = 0; i < LA; ++i) ra[i] = fetch(pa[i], kt * KB);
#pragma unroll
            for (int i = 0; i < LB; ++i) rb[i] = fetch(pb[i], kt * KB);
        };
        auto store = [&](int s) {
#pragma unroll
            for (int i = 0; i < LA; ++i) {
                const int e = tid + i * NT, r = e / QK, q = 4 * (e % QK);
                sm.a[s][q + 0][r] = ra[i].x;
                sm.a[s][q + 1][r] = ra[i].y;
                sm.a[s][q + 2][r] = ra[i].z;
                sm.a[s][q + 3][r] = ra[i].w;
            }
#pragma unroll
            for (int i = 0; i < LB; ++i) {
                const int e = tid + i * NT, r = e / QK, q = 4 * (e % QK);
                sm.b[s][q + 0][r] = rb[i].x;
                sm.b[s][q + 1][r] = rb[i].y;
                sm.b[s][q + 2][r] = rb[i].z;
                sm.b[s][q + 3][r] = rb[i].w;
            }
        };
        load(k0);
        __syncthreads();  // the stages may still be read by the piece before, or used by its epilogue
        store(0);
        __syncthreads();
        for (int kt = k0; kt < k1; ++kt) {
            const int cur = (kt - k0) & 1;
            if (kt + 1 < k1) load(kt + 1);
#pragma unroll
            for (int k = 0; k < KB; ++k) {
                float as[8];
                uint64_t av[8], bv[4];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const float4 v = *reinterpret_cast<const float4*>(&sm.a[cur][k][c * (BM / 2) + ty * 4]);
                    as[4 * c] = v.x, as[4 * c + 1] = v.y, as[4 * c + 2] = v.z, as[4 * c + 3] = v.w;
                    const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(&sm.b[cur][k][c * (BN / 2) + tx * 4]);
                    bv[2 * c] = w.x, bv[2 * c + 1] = w.y;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) asm("mov.b64 %0, {%1, %1};" : "=l"(av[i]) : "f"(as[i]));
#pragma unroll
                for (int i = 0; i < 8; ++i)
#pragma unroll
                    for (int p = 0; p < 4; ++p) fma2(acc[i][p], av[i], bv[p]);
            }
            if (kt + 1 < k1) store(cur ^ 1);
            __syncthreads();
        }
    }
};

// The rows of one tile.
struct F32Rows {
    const float* a;
    int na;
    const float* b;
    int nb;
};

// `tiles` tiles spread evenly over the CTAs of the grid, which must not be more than the tiles:
// CTA g takes the stages [U g / G, U (g + 1) / G) of all U = tiles x stages in a row, so a range
// begins inside a tile that the CTA before began and ends inside one that the CTA after ends.  It
// computes the beginning of that last tile first and leaves the chains with stash(tile index, t),
// then its whole tiles, and last the end of its first tile, whose beginning the CTA before computed
// first (taken up by fetch(tile index, t), thread by thread what stash left): as a
// range is at least one tile long, nobody waits for work that has not been done by then.  (A CTA
// waits only for one of a lower index, which the hardware starts before it; the wait is bounded all the
// same, and a tile whose wait runs out is not finished: fail(tile index), by one thread, lets the outputs
// that hang on it be zeroed.)  Without the split 168 tiles on 152 SMs take the time of two.
struct F32HandOver {
    uint32_t* ready;    // a word per CTA, zero before the launch
    uint32_t* status;   // RGBD_STATUS_WAIT_TIMEOUT when a wait runs out
    uint64_t limit_ns;
    int drop;           // a CTA that hands on nothing (for tests), or -1
};
template <class Tile, bool VEC, class Rows, class Finish, class Stash, class Fetch, class Fail>
__device__ __forceinline__ void f32_ordered_tiles(long long tiles, int K, const F32HandOver& ho,
                                                  typename Tile::Smem& sm, Rows rows, Finish finish, Stash stash,
                                                  Fetch fetch, Fail fail) {
    __shared__ int gave_up;
    const int stages = (K + Tile::KB - 1) / Tile::KB, tid = threadIdx.x;
    const long long U = tiles * stages;
    const long long u0 = U * blockIdx.x / gridDim.x, u1 = U * (blockIdx.x + 1) / gridDim.x;
    const long long first = u0 / stages, last = u1 / stages;  // the tiles in which the range begins and ends
    const int k0 = (int)(u0 - first * stages), k1 = (int)(u1 - last * stages);
    Tile t;
    if (k1 > 0) {
        const F32Rows r = rows(last);
        t.clear();
        t.template run<VEC>(r.a, r.na, r.b, r.nb, K, 0, k1, sm);
        stash(last, t);
        __threadfence();
        __syncthreads();
        if (tid == 0 && (int)blockIdx.x != ho.drop)
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ho.ready + blockIdx.x), "r"(1u) : "memory");
    }
    for (long long i = first + (k0 > 0); i < last; ++i) {
        const F32Rows r = rows(i);
        t.clear();
        t.template run<VEC>(r.a, r.na, r.b, r.nb, K, 0, stages, sm);
        finish(i, t);
    }
    if (k0 > 0) {
        const F32Rows r = rows(first);
        if (tid == 0) {
            uint64_t since = 0, now;
            uint32_t ok = 0;
            int failed = 0;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];"
                             : "=r"(ok)
                             : "l"(ho.ready + blockIdx.x - 1)
                             : "memory");
                if (ok) break;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (since == 0) since = now;
                if (now - since > ho.limit_ns) {
                    failed = 1;
                    atomicOr(ho.status, RGBD_STATUS_WAIT_TIMEOUT);
                    fail(first);
                    break;
                }
                __nanosleep(200);
            }
            gave_up = failed;
        }
        __syncthreads();
        if (gave_up) return;
        fetch(first, t);
        t.template run<VEC>(r.a, r.na, r.b, r.nb, K, k0, stages, sm);
        finish(first, t);
    }
}

}  // namespace rgbd
