// Regime (i), FP32, n > 16, on the tensor cores at FP32 accuracy:
// C[m x n] = alpha * A[m x k] * B[k x n] + beta * C0.
//
// The FMA pipes cannot stream A at HBM speed for these widths (n = 64 needs 215 TFLOP/s, the pipes have 80).
// An FP32 value is the exact sum of three BF16 values (h + m + l, 8 significant bits each), so a product is the sum
// of nine BF16 products, each exact in FP32; the six largest are accumulated on the tensor cores in FP32:
//     l*h, h*l, m*m, m*h, h*m, then h*h
// (the three left out are below 2^-25 of |a||b|, under the rounding of one FP32 fma).  A chunk of 32 k-columns starts
// from a zero accumulator, smallest products first, so only the last two MMAs round at the size of the chunk's
// sum; the chunk sums are then added in FP32 registers, rounded to nearest.  A chain of k fmas becomes a chain of
// k/32 additions, and the error against exact products is smaller than the fma kernel's at every length.
//
// Measured, m = k = 32768, n = 64, calls back to back: 1.93 ms (fma kernel, 88 % of the FP32 pipe) -> 0.81 ms at 5.4
// TB/s (0.70 ms, 6.1 TB/s, at the clock of a single call); n = 32: 0.98 -> 0.68 ms; n = 20: 0.78 -> 0.68 ms.  Relative
// error (2-norm) against 64 bits 1.2e-6 -> 2.3e-7; k = 64: 1.4e-7 -> 6.3e-8.  Bound by HBM, then by power: the MMAs keep
// the tensor pipe 40 % busy, the issue slots 50 %.  Two blocks of one item each per SM so that one block's start and
// finish overlap the other's stream; four converter warps a block (eight spill at the registers left: 0.83 ms).  The MMA
// warp stays converged and elects the issuing lane: a loop under `lane == 0` keeps every descriptor in vector registers
// and took 100 cycles an MMA (0.80 -> 0.70 ms at n = 64).
//
// What the split cannot carry goes another way, by plain fmas before anything is stored, so that results follow IEEE fma
// arithmetic there: rows with an infinity, a NaN or an overflow (seen as a non-finite sum), and rows with a sum so small
// that what a piece or a piece's product loses below FP32's normal range could show in it.  Where the smallest nonzero
// |a| of the row times the smallest nonzero |b| of the item is at least 2^-100 nothing is lost; elsewhere the loss is below
// k 2^-126 (max|a| + max|b| + 8), with max|a| over chunks where B has entries below 2^-108, and a sum 2^26 times that is
// safe.  (The entries' sizes alone had decided: one entry of 1e-31 in B sent every row of its k range to the fmas; m = k =
// 8192, n = 64, such an entry in every item: 0.41 -> 0.064 ms, 0.060 without.)  Up to kRedoRows such rows of an item are
// recomputed on their own (redo_rows; one NaN row a slab: 0.41 -> 0.10 ms), more as a whole item (fma_item; all rows: 0.47
// ms, the fma kernel 0.15); so are products with k < kTcMinK.
//
// Block: one work item = one slab of 128 rows x one k range (the split-K scheme of the fma kernel, same workspace,
// counters and fixed summation order), 12 warps, two blocks per SM:
//   warps 0-3   converters: thread = row; FP32 A from shared memory, split, pieces to tensor memory (tcgen05.st)
//   warps 4-7   promoters: thread = row; chunk sums from tensor memory, added in registers; epilogue
//   warp 8      producer of A by tensor copies (U: of every fourth column, encode_a_rows)
//   warp 9      tensor-memory owner and MMA issuer;  warp 10  producer of packed B chunks
#pragma once
#include "tsmm_internal.h"
#include "tsmm_finish.cuh"
#include "tsmm_fma_item.cuh"
#include "tsmm_tc.cuh"

namespace tsmm {

constexpr int kRedoRows = 16;

// Rows i0 + list[0..count) of A[:, k0:k1] * B[k0:k1, :]: the four converter warps take every fourth 32 columns of k each, and
// leave their sums in out[warp][slot][W]; a lane takes two columns of four rows, A arrives 32 columns of k at a time, one a
// lane.  Chains of 32 columns, as short as the tensor cores' chunks.  Bound by L2 latency.
template <int W>
__device__ __forceinline__ void redo_rows(const TallArgs &a, int64_t i0, int64_t k0, int64_t k1, const unsigned char *list,
                                          int count, float *out, int warp, int lane) {
    constexpr int R = 4;
    const int np = a.np, c = 2 * lane;
    out += warp * (kRedoRows * W) + c;
#pragma unroll 1
    for (int first = 0; first < count; first += R) {
        const float *A[R];
#pragma unroll
        for (int q = 0; q < R; ++q)
            A[q] = static_cast<const float *>(a.A) + i0 + list[first + q < count ? first + q : first];
        float2 sum[R];
        float x[R], y[R];
        auto load = [&](int64_t p) {
#pragma unroll
            for (int q = 0; q < R; ++q) y[q] = p < a.k ? __ldg(A[q] + p * a.lda) : 0.f;
        };
#pragma unroll
        for (int q = 0; q < R; ++q) sum[q] = make_float2(0.f, 0.f);
        load(k0 + 32 * warp + lane);
#pragma unroll 1
        for (int64_t p = k0 + 32 * warp; p < k1; p += 128) {
            const float *B = static_cast<const float *>(a.Bp) + p * np + (c < np ? c : 0);
#pragma unroll
            for (int q = 0; q < R; ++q) x[q] = y[q];
            load(p + 128 + lane);
            float2 s[R];
#pragma unroll
            for (int q = 0; q < R; ++q) s[q] = make_float2(0.f, 0.f);
#pragma unroll 16
            for (int u = 0; u < 32; ++u) {
                const float2 b = __ldg(reinterpret_cast<const float2 *>(B + u * np));
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    const float v = __shfl_sync(0xffffffffu, x[q], u);
                    s[q] = __ffma2_rn(make_float2(v, v), b, s[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < R; ++q) sum[q] = __fadd2_rn(sum[q], s[q]);
        }
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (first + q < count && c < W) *reinterpret_cast<float2 *>(out + (first + q) * W) = sum[q];
    }
}

template <int W, bool U>
struct TallTcCfg {
    static constexpr int BM = kTcRows;
    static constexpr int KB = kTcKB;                          // k per chunk (one stage)
    static constexpr int A_STRIDE = U ? BM + 4 : BM;          // floats per column slot (U: column 4 c + q in slot 8 q + c)
    static constexpr int A_BYTES = KB * A_STRIDE * 4;
    static constexpr int PIECE = W * KB * 2;                  // one BF16 piece of a chunk of B
    static constexpr int B_BYTES = 3 * PIECE;
    static constexpr int SBO = KB / 8 * 128;
    static constexpr int BUDGET = 112 * 1024;                 // two blocks per SM
    static constexpr int SB = 3;
    static constexpr int SA_RAW = (BUDGET - SB * B_BYTES) / A_BYTES;
    static constexpr int SA = SA_RAW > 6 ? 6 : SA_RAW;
    static constexpr int OFF_B = SA * A_BYTES;
    static constexpr int OFF_BAR = OFF_B + SB * B_BYTES;
    static constexpr int NBAR = 2 * SA + 2 * SB + 8;
    static constexpr int OFF_THR = OFF_BAR + NBAR * 8 + 48;   // rows' least safe sums, then the list of unsafe rows
    static constexpr int SMEM = OFF_THR + BM * 4 + kRedoRows;
    static constexpr int THREADS = 384;
    static constexpr int COL_A = 2 * W;                       // TMEM: 2 accumulators, then 2 x 3 pieces of 16 columns
    static constexpr int TMEM_COLS = 256;
    static_assert(SA >= 3, "A ring");
    static_assert(COL_A + 96 <= TMEM_COLS, "tensor memory");
    static_assert(2 * (SMEM + 1024) <= 228 * 1024, "two blocks per SM");
    static constexpr int OFF_F = BM * (W / 2) * 4;            // fallback, over the A ring: exchange, rows of B, totals
    static constexpr int OFF_T = OFF_F + 2 * kFmaRows * W * 4;
    static_assert(OFF_T + 256 * (W / 2) * 4 <= SA * A_BYTES && 4 * kRedoRows * W * 4 <= OFF_F, "fallback");
};

template <int W, bool U>
__device__ __forceinline__ void tall_tc_block(const CUtensorMap *tmA, const TallArgs &a, int64_t slab, int split) {
    using Cfg = TallTcCfg<W, U>;
    constexpr int SA = Cfg::SA, SB = Cfg::SB, KB = Cfg::KB, BM = Cfg::BM;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + Cfg::OFF_BAR);
    uint64_t *afull = bar;             // [SA] FP32 A landed
    uint64_t *aempty = afull + SA;     // [SA] converters have read it
    uint64_t *bfull = aempty + SA;     // [SB] B chunk landed
    uint64_t *bempty = bfull + SB;     // [SB] the MMAs have read it
    uint64_t *conv = bempty + SB;      // [2] pieces of A in tensor memory
    uint64_t *mdone = conv + 2;        // [2] the chunk's MMAs are complete
    uint64_t *drained = mdone + 2;     // [2] accumulator read
    uint64_t *fbar = drained + 2;      // [2] fallback: rows of B landed
    unsigned *tslot = reinterpret_cast<unsigned *>(bar + Cfg::NBAR);
    unsigned *flag = tslot + 1;
    unsigned *abort_flag = tslot + 2;
    unsigned *unsafe = tslot + 3;      // rows to recompute
    unsigned *doubt = tslot + 4;       // some row has entries small enough to ask its sums
    float *thr = reinterpret_cast<float *>(smem + Cfg::OFF_THR);
    unsigned char *list = smem + Cfg::OFF_THR + BM * 4;

    const int warp = threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    const int64_t k0 = (int64_t)split * a.kchunk;
    const int64_t k1 = (k0 + a.kchunk < a.kp) ? k0 + a.kchunk : a.kp;
    const int iters = (int)((k1 - k0) / KB);
    const int64_t i0 = slab * BM;

    if (threadIdx.x == 0) {
        if (!U || a.arows != 0) prefetch_tmap(tmA);
        for (int s = 0; s < SA; ++s) {
            mbar_init(&afull[s], 1);
            mbar_init(&aempty[s], 4);
        }
        for (int s = 0; s < SB; ++s) {
            mbar_init(&bfull[s], 1);
            mbar_init(&bempty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&conv[b], 4);
            mbar_init(&mdone[b], 1);
            mbar_init(&drained[b], 4);
            mbar_init(&fbar[b], 1);
        }
        *abort_flag = 0u;
        *unsafe = a.k < kTcMinK ? kRedoRows + 1u : 0u;
        *doubt = 0u;
        fence_mbar_init();
    }
    if (warp == 9) tc_alloc(tslot, Cfg::TMEM_COLS);
    tcf_before();
    __syncthreads();
    tcf_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);  // uniform: MMA operands stay in uniform registers

    if (warp >= 8) {
        reg_dec<40>();
        if (warp == 8) {
            // ------------------------------------------------ A
            const uint64_t pol = policy_evict_first();
            bool ok = true;
            int it = 0;
            if constexpr (!U) {
                if (lane == 0) {
                    for (; it < iters; ++it) {
                        const int s = it % SA;
                        if (it >= SA && !mbar_wait_bounded(&aempty[s], (uint32_t)((it / SA) & 1) ^ 1)) {
                            ok = false;
                            break;
                        }
                        mbar_arrive_expect_tx(&afull[s], Cfg::A_BYTES);
                        tma_load_2d(smem + s * Cfg::A_BYTES, tmA, (int32_t)i0, (int32_t)(k0 + (int64_t)it * KB),
                                    &afull[s], pol);
                    }
                }
            } else {
                // Chunks within the map's rows: one tensor copy per q (one bulk copy per column, which the copy engine
                // takes every 36 cycles an SM, bounded these shapes: m =
                // 32765, n = 64, k = 32768: 1.00 -> 0.72 ms, m = 141591, n = 39, k = 1607: 231 -> 169 us).
                // Other chunks: lane = column, one bulk copy of the aligned span around its rows (column_span_bytes);
                // columns beyond k are zero-filled.
                const int rows = (int)((a.m - i0 < BM) ? a.m - i0 : BM);
                const int abase = (int)((reinterpret_cast<uintptr_t>(a.A) / 4) & 3);
                const int ldv = (int)((uint64_t)a.lda & 3);
                for (; it < iters; ++it) {
                    const int s = it % SA;
                    if (it >= SA) {
                        const bool got = mbar_wait_bounded(&aempty[s], (uint32_t)((it / SA) & 1) ^ 1);
                        if (!__all_sync(0xffffffffu, got)) {
                            ok = false;
                            break;
                        }
                    }
                    const int64_t pc = k0 + (int64_t)it * KB;
                    if (pc + KB <= 4 * a.arows) {
                        if (lane == 0) {
                            mbar_arrive_expect_tx(&afull[s], Cfg::A_BYTES);
                            for (int q = 0; q < 4; ++q)
                                tma_load_2d(smem + s * Cfg::A_BYTES + q * (kARowsBox * Cfg::A_STRIDE * 4), tmA,
                                            (int32_t)((abase + q * a.lda + i0) & ~(int64_t)3), (int32_t)(pc / 4), &afull[s], pol);
                        }
                        continue;
                    }
                    const int64_t p = pc + lane;
                    float *slot = reinterpret_cast<float *>(smem + s * Cfg::A_BYTES) + ((lane & 3) * 8 + lane / 4) * Cfg::A_STRIDE;
                    const int d = (abase + (int)(p & 3) * ldv) & 3;
                    const uint32_t bytes = p < a.k ? column_span_bytes<float>(rows, d) : 0u;
                    if (p >= a.k) {
                        for (int r = 0; r < Cfg::A_STRIDE; r += 4)
                            *reinterpret_cast<uint4 *>(slot + r) = make_uint4(0, 0, 0, 0);
                        fence_proxy_async_smem();
                    }
                    const uint32_t sum = __reduce_add_sync(0xffffffffu, bytes);
                    __syncwarp();
                    if (lane == 0) mbar_arrive_expect_tx(&afull[s], sum);
                    __syncwarp();
                    if (bytes != 0u)
                        bulk_load(slot, static_cast<const float *>(a.A) + i0 + p * a.lda - d, bytes, &afull[s], pol);
                }
            }
            if (!ok) {
                if (lane == 0) atomicOr(a.status, kDevErrTimeout);
                // copies in flight land before the block may exit
                for (int q = it > SA ? it - SA : 0; q < it; ++q) mbar_wait_bounded(&afull[q % SA], (uint32_t)((q / SA) & 1));
            }
        } else if (warp == 10) {
            // ------------------------------------------------ B
            if (lane == 0) {
                const uint64_t pol = policy_evict_last();
                const unsigned char *Bt = static_cast<const unsigned char *>(a.Bt) + (k0 / KB) * Cfg::B_BYTES;
                int it = 0;
                bool ok = true;
                for (; it < iters; ++it, Bt += Cfg::B_BYTES) {
                    const int s = it % SB;
                    if (it >= SB && !mbar_wait_bounded(&bempty[s], (uint32_t)((it / SB) & 1) ^ 1)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&bfull[s], Cfg::B_BYTES);
                    bulk_load(smem + Cfg::OFF_B + s * Cfg::B_BYTES, Bt, Cfg::B_BYTES, &bfull[s], pol);
                }
                if (!ok) {
                    atomicOr(a.status, kDevErrTimeout);
                    for (int q = it > SB ? it - SB : 0; q < it; ++q)
                        mbar_wait_bounded(&bfull[q % SB], (uint32_t)((q / SB) & 1));
                }
            }
        } else if (warp == 9) {
            // ------------------------------------------------ MMAs
            // the whole warp walks the loop (uniform operands), one elected lane issues
            constexpr uint32_t idesc = tc_idesc_bf16(BM, W);
            const uint64_t bdesc = tc_desc(smem_addr(smem + Cfg::OFF_B), Cfg::SBO);
            bool ok = true;
            int it = 0, s = 0;
            uint32_t sph = 0;
            for (; it < iters; ++it) {
                const int b = it & 1;
                const uint32_t par = (uint32_t)(it >> 1) & 1;
                ok = mbar_wait_bounded(&bfull[s], sph) && mbar_wait_bounded(&conv[b], par) &&
                     (it < 2 || mbar_wait_bounded(&drained[b], par ^ 1));
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tcf_after();
                if (elect_one()) {
                    const uint32_t d = tmem + b * W;
                    const uint32_t at = tmem + Cfg::COL_A + b * 48;
                    const uint64_t bd = bdesc + (uint64_t)(s * (Cfg::B_BYTES / 16));
                    // (piece of A, piece of B), smallest products first
                    constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
                    for (int q = 0; q < 6; ++q)
#pragma unroll
                        for (int ks = 0; ks < KB / 16; ++ks)
                            tc_mma_ts(d, at + PA[q] * 16 + ks * 8, bd + (uint64_t)((PB[q] * Cfg::PIECE + ks * 256) / 16),
                                      idesc, (q | ks) != 0);
                    tc_commit(&bempty[s]);
                    tc_commit(&mdone[b]);
                }
                __syncwarp();
                if (++s == SB) {
                    s = 0;
                    sph ^= 1;
                }
            }
            if (!ok && lane == 0) {
                atomicOr(a.status, kDevErrTimeout);
                atomicOr(abort_flag, 1u);
            }
            // nothing may still write tensor memory when it is freed (the last chunks' MMAs)
            for (int q = it > 2 ? it - 2 : 0; q < it; ++q) mbar_wait_bounded(&mdone[q & 1], (uint32_t)(q >> 1) & 1);
            __syncwarp();
            tcf_before();
            named_barrier(2, 160);  // with the promoters: every accumulator is read
            tcf_after();
            tc_dealloc(tmem, Cfg::TMEM_COLS);
        }
        return;
    }

    const int r = threadIdx.x % 128;
    const int64_t row = i0 + r;
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    constexpr int HW = W / 2;
    float *ex = reinterpret_cast<float *>(smem);  // fallback: the converters' half of the columns
    const float alpha = static_cast<float>(a.alpha);
    const float beta = static_cast<float>(a.beta);
    const int n = (int)a.n;
    const int64_t mpad = a.slabs * BM;
    float *ws = static_cast<float *>(a.ws) + i0 + r;
    // C = alpha*v + beta*C0 for G columns from c0 of this thread's row, the C0 loads issued ahead of the stores
    auto store = [&](int c0, const float *v, auto g_tag) {
        constexpr int G = decltype(g_tag)::value;
        if (row >= a.m) return;
        float *c = static_cast<float *>(a.C) + row + (int64_t)c0 * a.ldc;
        float old[G];
#pragma unroll
        for (int j = 0; j < G; ++j) old[j] = (beta != 0.f && c0 + j < n) ? c[(int64_t)j * a.ldc] : 0.f;
#pragma unroll
        for (int j = 0; j < G; ++j)
            if (c0 + j < n) {
                float o = alpha * v[j];
                if (beta != 0.f) o = fmaf(beta, old[j], o);
                c[(int64_t)j * a.ldc] = o;
            }
    };
    // split-K: take an arrival ticket; the last arriver finishes, all 256 threads of it
    auto finish = [&]() {
        named_barrier(1, 256);
        if (threadIdx.x == 0) *flag = atomicAdd(a.tickets + slab, 1u) == (unsigned)(a.splits - 1) ? 1u : 0u;
        named_barrier(1, 256);
        if (*flag == 0u) return;
        __threadfence();
        tc_finish<float, 256>(a, i0, threadIdx.x);
        if (threadIdx.x == 0) a.tickets[slab] = 0u;  // ready for the next launch on this stream
    };
    if (warp < 4) {
        // ---------------------------------------------------- converters
        reg_dec<72>();
        float bmin = __uint_as_float(0x7f800000u);
        {
            const float *bm = a.bmin + k0 / KB;
            for (int c = lane; c < iters; c += 32) bmin = fminf(bmin, __ldg(bm + c));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) bmin = fminf(bmin, __shfl_xor_sync(0xffffffffu, bmin, o));
        }
        // U: offsets within 16 bytes of the columns 0..3 mod 4 of a chunk
        const int abase = (int)((reinterpret_cast<uintptr_t>(a.A) / 4) & 3);
        const int ldv = (int)((uint64_t)a.lda & 3);
        uint32_t amin = 0xffffffffu;  // smallest 2|x| - 1 over the nonzero x (bit patterns)
        bool ok = true;
        for (int it = 0; it < iters; ++it) {
            const int s = it % SA, b = it & 1;
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&afull[s], (uint32_t)((it / SA) & 1)))) {
                ok = false;
                break;
            }
            const float *src = reinterpret_cast<const float *>(smem + s * Cfg::A_BYTES) + r;
#pragma unroll
            for (int h = 0; h < KB / 16; ++h) {
                float x[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const int col = h * 16 + q;
                    x[q] = U ? src[((col & 3) * 8 + col / 4) * Cfg::A_STRIDE + ((abase + (q & 3) * ldv) & 3)] : src[col * BM];
                }
                uint32_t ph[8], pm[8], pl[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    amin = min(amin, __float_as_uint(x[2 * q]) * 2u - 1u);
                    amin = min(amin, __float_as_uint(x[2 * q + 1]) * 2u - 1u);
                    split3_bf16x2(x[2 * q], x[2 * q + 1], ph[q], pm[q], pl[q]);
                }
                if (h == 0) {
                    // the pieces' place is free once the MMAs of two chunks ago are done
                    if (it >= 2)
                        ok = __all_sync(0xffffffffu, mbar_wait_bounded(&mdone[b], ((uint32_t)(it >> 1) & 1) ^ 1));
                    tcf_after();
                } else {
                    release_reads_to_async_copy();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&aempty[s]);
                }
                const uint32_t t = tlane + Cfg::COL_A + b * 48 + h * 8;
                tc_st8(t, ph);
                tc_st8(t + 16, pm);
                tc_st8(t + 32, pl);
            }
            if (!ok) break;
            tc_wait_st();
            tcf_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&conv[b]);
        }
        if (!ok && lane == 0) {
            atomicOr(a.status, kDevErrTimeout);
            atomicOr(abort_flag, 1u);
        }
        const float amn = amin == 0xffffffffu ? __uint_as_float(0x7f800000u) : __uint_as_float((amin + 1u) >> 1);
        constexpr float kTiny = 7.8886091e-31f;  // 2^-100
        float least = 0.f;
        const bool small = row < a.m && !(amn >= kTiny && bmin >= kTiny && amn * bmin >= kTiny);
        if (__any_sync(0xffffffffu, small)) {
            // largest |b|, and |a| in the chunks of k where pieces of B may be lost (tracked in the loop above, 2 % of it)
            const float *bm = a.bmin + k0 / KB;
            float ax = 0.f, bx = 0.f;
            for (int c = 0; c < iters; ++c) {
                bx = fmaxf(bx, __ldg(bm + a.kp / KB + c));
                if (__ldg(bm + c) < 3.0814879e-33f) {  // 2^-108
                    const float *Ar = static_cast<const float *>(a.A) + (row < a.m ? row : 0);
                    const int64_t p = k0 + (int64_t)c * KB;
                    float y[KB];
#pragma unroll
                    for (int q = 0; q < KB; ++q) y[q] = p + q < a.k ? __ldg(Ar + (p + q) * a.lda) : 0.f;
#pragma unroll
                    for (int q = 0; q < KB; ++q) ax = fmaxf(ax, fabsf(y[q]));
                }
            }
            if (small) least = (float)(k1 - k0) * 1.5777218e-30f * (ax + bx + 4.f);  // 2^-99
            *doubt = 1u;
        }
        thr[r] = least;
        // every converter and promoter warp gets here (bounded waits); the flags are read between barriers
        named_barrier(1, 256);
        named_barrier(1, 256);
        const bool stop = *abort_flag != 0u;
        const unsigned redo = *unsafe;
        if (stop) return;  // tile not written; the host sees TSMM_ERR_TIMEOUT
        if (redo > kRedoRows) {
            float part[HW];
            fma_item<float, HW>(a, row, k0, k1, 0, part, reinterpret_cast<float *>(smem + Cfg::OFF_F),
                                reinterpret_cast<float *>(smem + Cfg::OFF_T), fbar, abort_flag, threadIdx.x);
            if (*abort_flag != 0u) return;
#pragma unroll
            for (int j = 0; j < HW; ++j) ex[j * BM + r] = part[j];
            named_barrier(1, 256);
        } else if (redo != 0u) {
            redo_rows<W>(a, i0, k0, k1, list, (int)redo, ex, warp, lane);
            named_barrier(1, 256);
        }
        if (a.splits > 1) finish();
        return;
    }

    // -------------------------------------------------------- promoters
        reg_inc<120>();
        float acc[W];
#pragma unroll
        for (int j = 0; j < W; ++j) acc[j] = 0.f;
        bool ok = true;
        for (int it = 0; it < iters; ++it) {
            const int b = it & 1;
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&mdone[b], (uint32_t)(it >> 1) & 1))) {
                ok = false;
                break;
            }
            tcf_after();
#pragma unroll
            for (int c = 0; c < W; c += 16) {
                uint32_t v[16];
                tc_ld16(tlane + b * W + c, v);
                if (c + 16 == W) {
                    tcf_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&drained[b]);
                }
#pragma unroll
                for (int j = 0; j < 16; j += 2) {
                    const float2 t = __fadd2_rn(make_float2(acc[c + j], acc[c + j + 1]),
                                                make_float2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])));
                    acc[c + j] = t.x;
                    acc[c + j + 1] = t.y;
                }
            }
        }
        if (!ok && lane == 0) {
            atomicOr(a.status, kDevErrTimeout);
            atomicOr(abort_flag, 1u);
        }
        tcf_before();
        named_barrier(2, 160);
        float z = 0.f;  // 0 unless a sum is infinite or NaN
#pragma unroll
        for (int j = 0; j < W; ++j) z = fmaf(acc[j], 0.f, z);
    named_barrier(1, 256);
    bool bad = z != 0.f;
    if (*doubt != 0u) {
        const float least = thr[r];
#pragma unroll
        for (int j = 0; j < W; ++j) bad |= j < n && fabsf(acc[j]) < least;
    }
    unsigned slot = kRedoRows;
    if (bad && row < a.m) {
        slot = atomicAdd(unsafe, 1u);
        if (slot < kRedoRows) list[slot] = (unsigned char)r;
    }
    named_barrier(1, 256);
    const bool stop = *abort_flag != 0u;
    const unsigned redo = *unsafe;
    if (stop) return;
    if (redo > kRedoRows) {
        fma_item<float, HW>(a, row, k0, k1, HW, acc + HW, reinterpret_cast<float *>(smem + Cfg::OFF_F),
                            reinterpret_cast<float *>(smem + Cfg::OFF_T), fbar, abort_flag, threadIdx.x);
        if (*abort_flag != 0u) return;
        named_barrier(1, 256);
#pragma unroll
        for (int j = 0; j < HW; ++j) acc[j] = ex[j * BM + r];
    } else if (redo != 0u) {
        named_barrier(1, 256);
        if (slot < kRedoRows) {
#pragma unroll
            for (int j = 0; j < W; ++j) {
                const float *e = ex + slot * W + j;
                acc[j] = e[0] + e[kRedoRows * W] + e[2 * kRedoRows * W] + e[3 * kRedoRows * W];
            }
        }
    }
    if (a.splits == 1) {
#pragma unroll
        for (int c = 0; c < W; c += 8) store(c, acc + c, std::integral_constant<int, 8>{});
        return;
    }
#pragma unroll
    for (int j = 0; j < W; ++j)
        if (j < n) ws[((int64_t)split * a.np + j) * mpad] = acc[j];
    __threadfence();
    finish();
}

template <int W, bool U>
__global__ void __launch_bounds__(TallTcCfg<W, U>::THREADS, 2) tall_tc_kernel(const __grid_constant__ CUtensorMap tmA, const TallArgs a) {
    tall_tc_block<W, U>(&tmA, a, blockIdx.x, (int)blockIdx.y);
}

}  // namespace tsmm
