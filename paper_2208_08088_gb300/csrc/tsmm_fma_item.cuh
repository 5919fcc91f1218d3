// One work item (128 rows x a k range) by plain fmas in the working precision: what the tensor-core kernels of regime
// (i) fall back to for values that their splits cannot carry.
#pragma once
#include "tsmm_device.cuh"
#include "tsmm_internal.h"

namespace tsmm {

constexpr int kFmaRows = 16;  // rows of packed B per stage

template <typename T, int HW>
struct FmaAcc {
    T v[HW];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int j = 0; j < HW; ++j) v[j] = T(0);
    }
    __device__ __forceinline__ void add(T x, const T *b, int cols) {
#pragma unroll
        for (int j = 0; j < HW; j += 16 / (int)sizeof(T))
            if (j < cols) {
                const Vec<T, 16 / (int)sizeof(T)> bv = ld_vec<T, 16 / (int)sizeof(T)>(b + j);
#pragma unroll
                for (int u = 0; u < 16 / (int)sizeof(T); ++u) v[j + u] = fma(x, bv.v[u], v[j + u]);
            }
    }
    __device__ __forceinline__ T get(int j) const { return v[j]; }
};
template <int HW>
struct FmaAcc<float, HW> {
    float2 v[HW / 2];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int j = 0; j < HW / 2; ++j) v[j] = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ void add(float x, const float *b, int cols) {
        const float2 x2 = make_float2(x, x);
#pragma unroll
        for (int j = 0; j < HW; j += 4)
            if (j < cols) {
                const float4 bv = *reinterpret_cast<const float4 *>(b + j);
                v[j / 2] = __ffma2_rn(x2, make_float2(bv.x, bv.y), v[j / 2]);
                v[j / 2 + 1] = __ffma2_rn(x2, make_float2(bv.z, bv.w), v[j / 2 + 1]);
            }
    }
    __device__ __forceinline__ float get(int j) const { return (j & 1) ? v[j / 2].y : v[j / 2].x; }
};

// out[0..HW) = columns [c0, c0 + HW) of row `row` of A[:, k0:k1] * B[k0:k1, :], for 256 threads (tid 0..255, named
// barrier 1) of two column halves x 128 rows.  Packed rows of B arrive by bulk copies into two stages of kFmaRows rows
// at sb (FP64 with HW = 8: 8 x 128 values more behind them), entries of A a stage ahead in registers; tot: room for HW x 256
// values.  Bound by the fma pipe (FP64) or about half of it (FP32).  fbar: two barriers, fresh.  A wait that runs out sets
// *abort_flag and the status.
template <typename T, int HW>
__device__ __forceinline__ void fma_item(const TallArgs &a, int64_t row, int64_t k0, int64_t k1, int c0, T *out, T *sb,
                                         T *tot, uint64_t *fbar, unsigned *abort_flag, int tid) {
    constexpr int CH = kFmaRows;
    const int np = a.np;
    const int cols = np - c0;
    const uint32_t bytes = (uint32_t)(CH * np * (int)sizeof(T));
    const T *Bp = static_cast<const T *>(a.Bp) + k0 * np;
    const int chunks = (int)((k1 - k0) / CH);
    const bool in = row < a.m;
    const T *Ap = static_cast<const T *>(a.A) + (in ? row : 0) + k0 * a.lda;
    const int64_t kk = a.k - k0;  // columns of A from k0 on
    if (tid == 0) {
        fence_proxy_async_smem();
        for (int c = 0; c < 2 && c < chunks; ++c) {
            mbar_arrive_expect_tx(&fbar[c], bytes);
            bulk_load(sb + c * CH * np, Bp + (int64_t)c * CH * np, bytes, &fbar[c], policy_evict_last());
        }
    }
    auto stage_wait = [&](int c) {
        if (!mbar_wait_bounded(&fbar[c & 1], (uint32_t)(c >> 1) & 1)) {
            atomicOr(a.status, kDevErrTimeout);
            atomicOr(abort_flag, 1u);
        }
    };
    // the stage is read by all, or given up by all: refill it
    auto stage_next = [&](int c) {
        const int b = c & 1;
        release_reads_to_async_copy();
        named_barrier(1, 256);
        if (*abort_flag != 0u) {
            // a copy in flight lands before the block may exit
            if (tid == 0 && c + 1 < chunks) mbar_wait_bounded(&fbar[b ^ 1], (uint32_t)((c + 1) >> 1) & 1);
            return false;
        }
        if (tid == 0 && c + 2 < chunks) {
            mbar_arrive_expect_tx(&fbar[b], bytes);
            bulk_load(sb + b * CH * np, Bp + (int64_t)(c + 2) * CH * np, bytes, &fbar[b], policy_evict_last());
        }
        return true;
    };
    // Chains of SEG (SEGN) stages, their sums added in `tot`: one chain over a whole item would be several times as long as
    // the fma kernels', whose blocks split k among warps and more splits (FP64, n = 64, k = 2048, uneven columns: error
    // 5.5e-16, theirs 3.7e-16, so 2.5e-16).  The totals sit in shared memory because registers for them spill (FP32,
    // n = 64: 5 times the time).
    tot += tid;
    // up to 8 columns of FP64 (np <= 8 = HW): the halves share the columns and split each stage's rows, and 16 sums a
    // thread (16 / np rows in turn) cover the FP64 pipe's latency, which one warp per scheduler with 8 sums does not (40 %)
    const int half = tid / 128;
    auto narrow = [&](auto np_tag) {
        constexpr int NPW = decltype(np_tag)::value, SETS = 16 / NPW < CH / 2 ? 16 / NPW : CH / 2;
        constexpr int SEGN = 4 * SETS;  // chains of 32 entries
        FmaAcc<T, NPW> acc[SETS];
#pragma unroll
        for (int q = 0; q < SETS; ++q) acc[q].zero();
        auto sum = [&](int j) {
            T t = acc[0].get(j);
#pragma unroll
            for (int q = 1; q < SETS; ++q) t += acc[q].get(j);
            return t;
        };
        T x[CH / 2];
        Ap += (int64_t)(half * (CH / 2)) * a.lda;
#pragma unroll
        for (int q = 0; q < CH / 2; ++q) x[q] = (in && half * (CH / 2) + q < kk) ? __ldg(Ap + (int64_t)q * a.lda) : T(0);
        for (int c = 0; c < chunks; ++c) {
            stage_wait(c);
            Ap += (int64_t)CH * a.lda;
            const T *bs = sb + (c & 1) * CH * NPW + half * (CH / 2) * NPW;
            const int64_t left = kk - (int64_t)(c + 1) * CH - half * (CH / 2);
#pragma unroll
            for (int q = 0; q < CH / 2; ++q) {
                acc[q % SETS].add(x[q], bs + q * NPW, NPW);
                x[q] = (in && c + 1 < chunks && q < left) ? __ldg(Ap + (int64_t)q * a.lda) : T(0);
            }
            if (c % SEGN == SEGN - 1) {
#pragma unroll
                for (int j = 0; j < NPW; ++j) tot[j * 256] = c < SEGN ? sum(j) : tot[j * 256] + sum(j);
#pragma unroll
                for (int q = 0; q < SETS; ++q) acc[q].zero();
            }
            if (!stage_next(c)) break;
        }
        T *ex = sb + 2 * CH * 16 + tid % 128;
        T s[NPW];
#pragma unroll
        for (int j = 0; j < NPW; ++j) {
            s[j] = chunks < SEGN ? sum(j) : tot[j * 256] + sum(j);
            if (half == 1) ex[j * 128] = s[j];
        }
        named_barrier(1, 256);
#pragma unroll
        for (int j = 0; j < HW; ++j) out[j] = T(0);
        if (half == 0) {
#pragma unroll
            for (int j = 0; j < NPW; ++j) out[j] = s[j] + ex[j * 128];
        }
    };
    if constexpr (sizeof(T) == 8 && HW == 8) {
        if (np == 2) return narrow(std::integral_constant<int, 2>{});
        if (np == 4) return narrow(std::integral_constant<int, 4>{});
        if (np == 8) return narrow(std::integral_constant<int, 8>{});
    }
    constexpr int SEG = sizeof(T) == 8 ? 2 : 8;
    FmaAcc<T, HW> acc;
    acc.zero();
    T x[CH];
#pragma unroll
    for (int q = 0; q < CH; ++q) x[q] = (in && q < kk) ? __ldg(Ap + (int64_t)q * a.lda) : T(0);
    for (int c = 0; c < chunks; ++c) {
        stage_wait(c);
        Ap += (int64_t)CH * a.lda;
        const T *bs = sb + (c & 1) * CH * np + c0;
        const int64_t left = kk - (int64_t)(c + 1) * CH;
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            acc.add(x[q], bs + q * np, cols);
            x[q] = (in && c + 1 < chunks && q < left) ? __ldg(Ap + (int64_t)q * a.lda) : T(0);
        }
        if (c % SEG == SEG - 1) {
#pragma unroll
            for (int j = 0; j < HW; ++j) {
                tot[j * 256] = c < SEG ? acc.get(j) : tot[j * 256] + acc.get(j);
                if (j % 4 == 3) asm volatile("" ::: "memory");  // few of them in registers at a time
            }
            acc.zero();
        }
        if (!stage_next(c)) break;
    }
#pragma unroll
    for (int j = 0; j < HW; ++j) out[j] = chunks < SEG ? acc.get(j) : tot[j * 256] + acc.get(j);
}

}  // namespace tsmm
