// Regime (ii), FP32, k > 32, on the tensor cores at FP32 accuracy: C[m x n] = alpha * A[m x k] * B[k x n] + beta * C0.
//
// The FMA pipe bounded these shapes (m = n = 16384, k = 64 / 128, beta = 1: 0.567 / 1.063 ms, 0.755 / 0.806 of its
// peak) where the m x n output stream alone takes 0.32 ms; here 0.353 / 0.366 ms (0.381 under sustained load).  As in regime (i) (tsmm_tall_tc.cuh) every entry is the exact
// sum of three BF16 values h + m + l and the six largest products are accumulated in FP32: here the five small ones
// (l*h, h*l, m*m, m*h, h*m) in one accumulator and h*h in another, added at the end, so that only the k/16 MMAs of h*h
// round at the size of the sum.  What the split cannot carry (tsmm_tall_tc.cuh: non-finite sums, and sums too small for
// the entries that make them up) is recomputed per output row of a tile with plain fmas.
//
// Persistent blocks, one per SM, walk equal shares of the tiles (128 rows x 64 columns), an item per m-tile, 16 warps:
//   warps 0-3   converters: the item's A tile, FP32 in shared memory -> its pieces in tensor memory (read by every tile)
//   warp 4      producer: A by tensor copies, packed pieces of B (64 k x 64 columns, 24 KB) through a ring
//   warp 5      tensor-memory owner and MMA issuer, two pairs of accumulators
//   warps 6-13  epilogue: two per TMEM lane quarter, 32 columns (one sub-tile) each
//   warp 14     C0 loader;  warp 15  storer: sub-tiles of 128 x 32 live in one of CS slots from C0's arrival to C's store
// (without TMA for C: C0 by 4-byte cp.async, C by plain stores).
#include <cstring>

#include "tsmm_internal.h"
#include "tsmm_tc.cuh"

namespace tsmm {

namespace {

constexpr int kKB = 64;                      // k per chunk
constexpr int kNT = kRankNT;                 // 64 columns per tile
constexpr int kSUB = 32;                     // columns per sub-tile
constexpr int kPIECE = kNT * kKB * 2;        // one BF16 piece of a chunk of B
constexpr int kBCHUNK = 3 * kPIECE;

template <int KC>  // 64-column k chunks: 1 (k <= 64) or 2
struct RankTcCfg {
    static constexpr int BM = 128;
    static constexpr int A_BYTES = KC * kKB * BM * 4;
    static constexpr int NB = 4;                       // B chunk buffers
    static constexpr int CS = KC == 1 ? 6 : 4;         // C slots; even, so that a slot always serves the same half
    static constexpr int SLOT = BM * kSUB * 4;
    static constexpr int OFF_E = 512;                  // smallest and largest exponents of A's rows, 4 items x 128 x 2 bytes
    static constexpr int OFF_A = OFF_E + 4 * BM * 2;
    static constexpr int OFF_B = OFF_A + A_BYTES;
    static constexpr int OFF_C = OFF_B + NB * kBCHUNK;
    static constexpr int SMEM = OFF_C + CS * SLOT;
    static constexpr int NBAR = 2 + 4 + 2 * NB + 4 + 3 * CS;
    // tensor memory: 2 x (h*h, the rest) of 64 columns, then the pieces of A: 3 x 32 columns per chunk, twice if KC == 1
    static constexpr int COL_A = 4 * kNT, A_COLS = KC * 96, A_BUFS = KC == 1 ? 2 : 1;
    static constexpr int TMEM_COLS = 512;
    static constexpr int THREADS = 512;
    static_assert(NBAR * 8 + 16 <= OFF_E, "barrier area");
    static_assert(COL_A + A_BUFS * A_COLS <= TMEM_COLS, "tensor memory");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ void store_2d(const void *tmap, const void *src, int32_t x, int32_t y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                     reinterpret_cast<uint64_t>(tmap)),
                 "r"(x), "r"(y), "r"(smem_addr(src))
                 : "memory");
}

__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity));
}

// v[jj] = row `lane` of A times column jj of B (packed, kNT to a row) by plain fmas, for the lanes in `rows`.  Not inlined: its
// registers would spill the epilogue's.
__noinline__ __device__ void redo_rows(const float *A, int64_t lda, int64_t k, const float *Bp, unsigned rows, float *v) {
    const int lane = threadIdx.x % 32;
    if (__popc(rows) <= 8) {
        // few rows: one by one, lane = column, A 32 columns of k at a time
        for (; rows != 0u; rows &= rows - 1u) {
            const int src = __ffs((int)rows) - 1;
            float s = 0.f;
#pragma unroll 1
            for (int64_t p = 0; p < k; p += 32) {
                const float x = p + lane < k ? __ldg(A + src + (p + lane) * lda) : 0.f;
                const int left = (int)min((int64_t)32, k - p);
#pragma unroll 16
                for (int u = 0; u < 32; ++u) {
                    const float b = u < left ? __ldg(Bp + (p + u) * kNT + lane) : 0.f;
                    s = fmaf(__shfl_sync(0xffffffffu, x, u), b, s);
                }
            }
            for (int jj = 0; jj < 32; ++jj) {
                const float o = __shfl_sync(0xffffffffu, s, jj);
                if (lane == src) v[jj] = o;
            }
        }
        return;
    }
    const bool mine = rows >> lane & 1u;
    float2 s[16];
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) s[jj] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int64_t p = 0; p < k; ++p) {
        const float x = mine ? __ldg(A + lane + p * lda) : 0.f;
        const float2 x2 = make_float2(x, x);
#pragma unroll
        for (int jj = 0; jj < 16; jj += 2) {
            const float4 b = __ldg(reinterpret_cast<const float4 *>(Bp + p * kNT + 2 * jj));
            s[jj] = __ffma2_rn(x2, make_float2(b.x, b.y), s[jj]);
            s[jj + 1] = __ffma2_rn(x2, make_float2(b.z, b.w), s[jj + 1]);
        }
    }
#pragma unroll
    for (int jj = 0; jj < 32; ++jj)
        if (mine) v[jj] = jj & 1 ? s[jj / 2].y : s[jj / 2].x;
}

}  // namespace

// Pieces of B: block (tile, chunk), per column j and k kk of a piece at (j/8)*1024 + (kk/8)*128 + (j%8)*16 + (kk%8)*2,
// and the smallest and the largest 2|b| - 1 (bits) over the chunk's nonzero entries (0 for the largest of none).
__global__ void __launch_bounds__(256) pack_b_rank_tc_kernel(const float *__restrict__ B, int64_t k, int64_t n, int64_t ldb,
                                                             unsigned char *__restrict__ dst, uint2 *__restrict__ brange) {
    __shared__ uint32_t smin, smax;
    if (threadIdx.x == 0) smin = 0xffffffffu, smax = 0u;
    __syncthreads();
    const int64_t at = (int64_t)blockIdx.x * gridDim.y + blockIdx.y;
    unsigned char *chunk = dst + at * kBCHUNK;
    uint32_t mn = 0xffffffffu, mx = 0u;
    for (int e = threadIdx.x; e < kNT * kKB / 2; e += 256) {
        const int j = e / (kKB / 2), kk = e % (kKB / 2) * 2;
        const int64_t col = (int64_t)blockIdx.x * kNT + j, p = (int64_t)blockIdx.y * kKB + kk;
        const float x0 = (col < n && p < k) ? B[p + col * ldb] : 0.f;
        const float x1 = (col < n && p + 1 < k) ? B[p + 1 + col * ldb] : 0.f;
        mn = min(mn, min(__float_as_uint(x0) * 2u - 1u, __float_as_uint(x1) * 2u - 1u));
        mx = max(mx, max(__float_as_uint(x0) * 2u, __float_as_uint(x1) * 2u));
        uint32_t h, m, l;
        split3_bf16x2(x0, x1, h, m, l);
        unsigned char *q = chunk + (j / 8) * 1024 + (kk / 8) * 128 + (j % 8) * 16 + (kk % 8) * 2;
        *reinterpret_cast<uint32_t *>(q) = h;
        *reinterpret_cast<uint32_t *>(q + kPIECE) = m;
        *reinterpret_cast<uint32_t *>(q + 2 * kPIECE) = l;
    }
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (threadIdx.x % 32 == 0) atomicMin(&smin, mn), atomicMax(&smax, mx);
    __syncthreads();
    if (threadIdx.x == 0) brange[at] = make_uint2(smin, smax == 0u ? 0u : smax - 1u);
}

template <int KC>
__global__ void __launch_bounds__(512, 1)
    rankk_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmC, const RankArgs a,
                    unsigned *status, int c_tma) {
    using Cfg = RankTcCfg<KC>;
    constexpr int NB = Cfg::NB, CS = Cfg::CS, BM = Cfg::BM;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);
    uint64_t *a_full = bar;             // FP32 A tile landed
    uint64_t *a_empty = bar + 1;        // converters have read it
    uint64_t *a_conv = bar + 2;         // [2] pieces of A in tensor memory
    uint64_t *a_done = a_conv + 2;      // [2] the item's MMAs are complete
    uint64_t *b_full = a_done + 2;      // [NB]
    uint64_t *b_empty = b_full + NB;    // [NB]
    uint64_t *tfull = b_empty + NB;     // [2]
    uint64_t *tempty = tfull + 2;       // [2]
    uint64_t *c_full = tempty + 2;      // [CS] C0 landed in the slot
    uint64_t *c_store = c_full + CS;    // [CS] results written to it
    uint64_t *c_empty = c_store + CS;   // [CS] slot free
    unsigned *tslot = reinterpret_cast<unsigned *>(bar + Cfg::NBAR);
    uchar2 *rowexp = reinterpret_cast<uchar2 *>(smem + Cfg::OFF_E);  // [4][BM]
    float *cslots = reinterpret_cast<float *>(smem + Cfg::OFF_C);

    const int warp = threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    const int64_t ntiles = (a.n + kNT - 1) / kNT;
    const int64_t total = (a.m + BM - 1) / BM * ntiles;
    const int64_t first = total * blockIdx.x / gridDim.x, last = total * (blockIdx.x + 1) / gridDim.x;
    const bool use_c0 = a.beta != 0.0;
    const int ksteps = (int)((a.k + 15) / 16);

    if (threadIdx.x == 0) {
        prefetch_tmap(&tmA);
        if (c_tma) prefetch_tmap(&tmC);
        mbar_init(a_full, 1);
        mbar_init(a_empty, 4);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&a_conv[b], 4);
            mbar_init(&a_done[b], 1);
            mbar_init(&tfull[b], 2);  // the MMAs' completion and the issuer's own arrival, which orders rowexp before it
            mbar_init(&tempty[b], 8);
        }
        for (int b = 0; b < NB; ++b) {
            mbar_init(&b_full[b], 1);
            mbar_init(&b_empty[b], 1);
        }
        for (int s = 0; s < CS; ++s) {
            mbar_init(&c_full[s], c_tma ? 1 : 32);
            mbar_init(&c_store[s], 4);
            mbar_init(&c_empty[s], c_tma ? 1 : 4);
        }
        fence_mbar_init();
    }
    if (warp == 5) tc_alloc(tslot, Cfg::TMEM_COLS);
    tcf_before();
    __syncthreads();
    tcf_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);

    // items of this block, its share of the tiles cut at the m-tiles: f(item's running number, m-tile, first and last
    // n-tile) until it returns false
    auto items = [&](auto &&f) {
        int j = 0;
        for (int64_t at = first; at < last; ++j) {
            int64_t mt, t0;
            udivmod(at, ntiles, mt, t0);
            const int64_t t1 = t0 + (last - at) < ntiles ? t0 + (last - at) : ntiles;
            if (!f(j, mt, t0, t1)) return false;
            at += t1 - t0;
        }
        return true;
    };

    if (warp == 4) {
        // ------------------------------------------------ producer: A and B
        if (lane == 0) {
            const uint64_t pol = policy_evict_last();  // both are read again by other items
            const unsigned char *Bt = static_cast<const unsigned char *>(a.Bt);
            int64_t gq = 0;
            int na = 0;
            const bool ok = items([&](int j, int64_t mt, int64_t t0, int64_t t1) {
                if (j >= 1 && !mbar_wait_bounded(a_empty, (uint32_t)(j - 1) & 1)) return false;
                mbar_arrive_expect_tx(a_full, Cfg::A_BYTES);
                ++na;
                for (int box = 0; box < 2 * KC; ++box)
                    tma_load_2d(smem + Cfg::OFF_A + box * (BM * 32 * 4), &tmA, (int32_t)(mt * BM), box * 32, a_full, pol);
                for (int64_t t = t0; t < t1; ++t)
                    for (int c = 0; c < KC; ++c, ++gq) {
                        const int sb = (int)(gq % NB);
                        if (gq >= NB && !mbar_wait_bounded(&b_empty[sb], (uint32_t)((gq / NB) & 1) ^ 1)) return false;
                        mbar_arrive_expect_tx(&b_full[sb], kBCHUNK);
                        bulk_load(smem + Cfg::OFF_B + sb * kBCHUNK, Bt + (t * KC + c) * kBCHUNK, kBCHUNK, &b_full[sb], pol);
                    }
                return true;
            });
            if (!ok) atomicOr(status, kDevErrTimeout);
            // copies still in flight land before the block may exit
            if (na >= 1) mbar_wait_bounded(a_full, (uint32_t)((na - 1) & 1));
            for (int64_t q = gq > NB ? gq - NB : 0; q < gq; ++q)
                mbar_wait_bounded(&b_full[q % NB], (uint32_t)((q / NB) & 1));
        }
        return;
    }

    if (warp == 14) {
        // ------------------------------------------------ C0 loader
        if (!use_c0) return;
        const uint64_t pol = policy_evict_first();
        const float *C = static_cast<const float *>(a.C);
        int64_t q = 0;  // sub-tiles issued
        const bool ok = items([&](int, int64_t mt, int64_t t0, int64_t t1) {
            for (int64_t col0 = t0 * kNT; col0 < t1 * kNT; col0 += kSUB, ++q) {
                const int st = (int)(q % CS);
                if (q >= CS && !warp_wait(&c_empty[st], (uint32_t)((q / CS) & 1) ^ 1)) return false;
                float *slot = cslots + st * (BM * kSUB);
                if (c_tma) {
                    if (lane == 0) {
                        mbar_arrive_expect_tx(&c_full[st], Cfg::SLOT);
                        tma_load_2d(slot, &tmC, (int32_t)(mt * BM), (int32_t)col0, &c_full[st], pol);
                    }
                } else {
                    // rows lane + 32 rr of every column, walking one column pointer by ldc
                    const int64_t i0 = mt * BM;
                    const float *colp = C + i0 + lane + col0 * a.ldc;
                    float *dst = slot + lane;
                    for (int c = 0; c < kSUB; ++c, colp += a.ldc, dst += BM) {
                        const bool cin = col0 + c < a.n;
#pragma unroll
                        for (int rr = 0; rr < BM / 32; ++rr) {
                            const bool in = cin && i0 + lane + 32 * rr < a.m;
                            cp_async_elem(dst + 32 * rr, in ? colp + 32 * rr : C, in, 4);
                        }
                    }
                    cp_async_arrive_noinc(&c_full[st]);
                }
            }
            return true;
        });
        if (!ok && lane == 0) atomicOr(status, kDevErrTimeout);
        if (!c_tma) asm volatile("cp.async.wait_all;" ::: "memory");
        if (lane == 0)
            for (int64_t r = q > CS ? q - CS : 0; r < q; ++r) mbar_wait_bounded(&c_full[r % CS], (uint32_t)((r / CS) & 1));
        return;
    }

    if (warp == 15) {
        // ------------------------------------------------ storer (TMA): a slot is freed once its store has read it
        if (!c_tma || lane != 0) return;
        int64_t q = 0;
        const bool ok = items([&](int, int64_t mt, int64_t t0, int64_t t1) {
            for (int64_t col0 = t0 * kNT; col0 < t1 * kNT; col0 += kSUB, ++q) {
                const int st = (int)(q % CS);
                if (!mbar_wait_bounded(&c_store[st], (uint32_t)((q / CS) & 1))) return false;
                if (col0 < a.n)  // boxes wholly past the last column are not issued
                    store_2d(&tmC, cslots + st * (BM * kSUB), (int32_t)(mt * BM), (int32_t)col0);
                // one group a sub-tile, stored or not: the wait below counts groups, and "all but the newest" has to mean
                // every sub-tile before this one
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                // with C0 to prefetch into few slots, a slot is freed as early as possible; else the newest store stays in flight
                if (CS == 4 && use_c0) {
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                    mbar_arrive(&c_empty[st]);
                } else if (q >= 1) {
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    mbar_arrive(&c_empty[(q - 1) % CS]);
                }
            }
            return true;
        });
        if (!ok) atomicOr(status, kDevErrTimeout);
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        return;
    }

    if (warp == 5) {
        // ------------------------------------------------ MMAs, from one elected lane
        if (elect_one()) {
            constexpr uint32_t idesc = tc_idesc_bf16(BM, kNT);
            const uint64_t bdesc = tc_desc(smem_addr(smem + Cfg::OFF_B), 1024);
            const uint32_t blo = (uint32_t)bdesc, bhi = (uint32_t)(bdesc >> 32);
            int64_t gq = 0;
            int g = 0, nj = 0;
            const bool ok = items([&](int j, int64_t, int64_t t0, int64_t t1) {
                const int ab = Cfg::A_BUFS == 2 ? j & 1 : 0;
                if (!mbar_wait_bounded(&a_conv[j & 1], (uint32_t)(j >> 1) & 1)) return false;
                tcf_after();
                for (int64_t t = t0; t < t1; ++t, ++g) {
                    const int tb = g & 1;
                    if (g >= 2 && !mbar_wait_bounded(&tempty[tb], (uint32_t)((g >> 1) & 1) ^ 1)) return false;
                    const uint32_t dh = tmem + tb * (2 * kNT), dl = dh + kNT;
#pragma unroll 1
                    for (int c = 0; c < KC; ++c, ++gq) {
                        const int sb = (int)(gq % NB);
                        if (!mbar_wait_bounded(&b_full[sb], (uint32_t)((gq / NB) & 1))) return false;
                        tcf_after();
                        const uint32_t at = tmem + Cfg::COL_A + ab * Cfg::A_COLS + c * 96;
                        const uint32_t bd = blo + sb * (kBCHUNK / 16);
                        static_for<0, kKB / 16>([&](auto ks_tag) {
                            constexpr int ks = decltype(ks_tag)::value;
                            if (c * (kKB / 16) + ks < ksteps) {
                                constexpr int PA[5] = {2, 0, 1, 1, 0}, PB[5] = {0, 2, 1, 0, 1};
                                static_for<0, 5>([&](auto q_tag) {
                                    constexpr int q = decltype(q_tag)::value;
                                    const uint32_t af = at + PA[q] * 32 + ks * 8, bf = bd + (PB[q] * kPIECE + ks * 256) / 16;
                                    if (ks == 0 && q == 0 && c == 0) tc_mma_ts2<false>(dl, af, bf, bhi, idesc);
                                    else tc_mma_ts2<true>(dl, af, bf, bhi, idesc);
                                });
                                if (ks == 0 && c == 0) tc_mma_ts2<false>(dh, at + ks * 8, bd + ks * 16, bhi, idesc);
                                else tc_mma_ts2<true>(dh, at + ks * 8, bd + ks * 16, bhi, idesc);
                            }
                        });
                        tc_commit(&b_empty[sb]);
                    }
                    mbar_arrive(&tfull[tb]);
                    tc_commit(&tfull[tb]);
                }
                tc_commit(&a_done[j & 1]);
                nj = j + 1;
                return true;
            });
            if (!ok) {
                atomicOr(status, kDevErrTimeout);
                tc_commit(&a_done[nj & 1]);  // the MMAs of the item given up
                ++nj;
            }
            // nothing may still write tensor memory when it is freed
            for (int q = nj > 2 ? nj - 2 : 0; q < nj; ++q) mbar_wait_bounded(&a_done[q & 1], (uint32_t)(q >> 1) & 1);
        }
        __syncwarp();
        tcf_before();
        named_barrier(2, 288);  // warps 5..13
        tcf_after();
        tc_dealloc(tmem, Cfg::TMEM_COLS);
        return;
    }

    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    if (warp < 4) {
        // ------------------------------------------------ converters: thread = row
        const int r = threadIdx.x;
        const bool ok = items([&](int j, int64_t, int64_t, int64_t) {
            if (!warp_wait(a_full, (uint32_t)(j & 1))) return false;
            // the pieces' place: the MMAs of the item that last used it are complete
            if (j >= Cfg::A_BUFS && !warp_wait(&a_done[(j - Cfg::A_BUFS) & 1], (uint32_t)((j - Cfg::A_BUFS) >> 1) & 1)) return false;
            tcf_after();
            const float *src = reinterpret_cast<const float *>(smem + Cfg::OFF_A) + r;
            const uint32_t at = tlane + Cfg::COL_A + (Cfg::A_BUFS == 2 ? j & 1 : 0) * Cfg::A_COLS;
            uint32_t mn = 0xffffffffu, mx = 0u;
#pragma unroll 1
            for (int ks = 0; ks < ksteps; ++ks) {
                float x[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) x[q] = src[(ks * 16 + q) * BM];
                uint32_t ph[8], pm[8], pl[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    mn = min(mn, __float_as_uint(x[2 * q]) * 2u - 1u);
                    mn = min(mn, __float_as_uint(x[2 * q + 1]) * 2u - 1u);
                    mx = max(mx, max(__float_as_uint(x[2 * q]) * 2u, __float_as_uint(x[2 * q + 1]) * 2u));
                    split3_bf16x2(x[2 * q], x[2 * q + 1], ph[q], pm[q], pl[q]);
                }
                const uint32_t t = at + (ks / 4) * 96 + (ks % 4) * 8;
                tc_st8(t, ph);
                tc_st8(t + 32, pm);
                tc_st8(t + 64, pl);
            }
            // exponent fields of the smallest nonzero entry (255: none) and of the largest
            rowexp[(j & 3) * BM + r] = make_uchar2(mn == 0xffffffffu ? 255 : (unsigned char)((mn + 1u) >> 24),
                                                   (unsigned char)(mx >> 24));
            release_reads_to_async_copy();
            tc_wait_st();
            tcf_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(a_empty);
                mbar_arrive(&a_conv[j & 1]);
            }
            return true;
        });
        if (!ok && lane == 0) atomicOr(status, kDevErrTimeout);
        return;
    }

    // ---------------------------------------------------- epilogue (warps 6-13); each warp gives up on its own
    const int half = (warp - 6) / 4;
    const int r = (warp & 3) * 32 + lane;
    const float alpha = static_cast<float>(a.alpha), beta = static_cast<float>(a.beta);
    float *C = static_cast<float *>(a.C);
    int64_t q = half;  // this warp's sub-tile in the ring
    int g = 0;
    const bool ok = items([&](int j, int64_t mt, int64_t t0, int64_t t1) {
        const int64_t i = mt * BM + r;
        for (int64_t t = t0; t < t1; ++t, ++g, q += 2) {
            const int tb = g & 1;
            uint2 br = __ldg(a.brange + t * KC);
            if (KC == 2) {
                const uint2 b1 = __ldg(a.brange + t * KC + 1);
                br.x = min(br.x, b1.x);
                br.y = max(br.y, b1.y);
            }
            if (!warp_wait(&tfull[tb], (uint32_t)((g >> 1) & 1))) return false;
            tcf_after();
            uint32_t vh[32], vl[32];
            tc_ld32(tlane + tb * (2 * kNT) + half * 32, vh);
            tc_ld32(tlane + tb * (2 * kNT) + kNT + half * 32, vl);
            const uchar2 ea = rowexp[(j & 3) * BM + r];
            tcf_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[tb]);
            float v[32];
            float z = 0.f;  // 0 unless a sum is infinite or NaN
#pragma unroll
            for (int jj = 0; jj < 32; ++jj) {
                v[jj] = __uint_as_float(vh[jj]) + __uint_as_float(vl[jj]);
                z = fmaf(v[jj], 0.f, z);
            }
            const int eb = br.x == 0xffffffffu ? 255 : (int)((br.x + 1u) >> 24);
            const bool small = ea.x < 27 || eb < 27 || ea.x + eb < 2 * 127 - 100;
            if (__any_sync(0xffffffffu, i < a.m && (z != 0.f || small))) {
                bool redo = z != 0.f;
                // Entries so small that a piece or a product may have left FP32's normal range: the loss is below
                // k 2^-126 (max|a| + max|b| + 8), k <= 128, and a sum is safe from 2^26 times that on (2^(e - 217) here).
                if (small) {
                    const int e = max(130, max((int)ea.y, (int)((br.y + 1u) >> 24)));
                    const float least = __uint_as_float((uint32_t)min(255, e - 90) << 23);
                    const int cols = (int)min((int64_t)32, a.n - (t * kNT + half * 32));
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) redo |= jj < cols && fabsf(v[jj]) < least;
                }
                redo = redo && i < a.m;
                const unsigned rows = __ballot_sync(0xffffffffu, redo);
                if (rows != 0u) {
                    float w[32];
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) w[jj] = v[jj];
                    redo_rows(static_cast<const float *>(a.A) + mt * BM + (warp & 3) * 32, a.lda, a.k,
                              static_cast<const float *>(a.Bp) + t * a.kp * kNT + half * 32, rows, w);
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj) v[jj] = w[jj];
                }
            }
            const int st = (int)(q % CS);
            const uint32_t par = (uint32_t)((q / CS) & 1);
            float *slot = cslots + st * (BM * kSUB) + r;  // column 0, own row
            if (use_c0 ? !warp_wait(&c_full[st], par) : (c_tma && q >= CS && !warp_wait(&c_empty[st], par ^ 1))) return false;
#pragma unroll
            for (int jj = 0; jj < 32; ++jj) {
                v[jj] *= alpha;
                if (use_c0) v[jj] = fmaf(beta, slot[jj * BM], v[jj]);
            }
            if (c_tma) {
#pragma unroll
                for (int jj = 0; jj < 32; ++jj) slot[jj * BM] = v[jj];
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&c_store[st]);
            } else {
                if (use_c0) {
                    release_reads_to_async_copy();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&c_empty[st]);
                }
                const int64_t jb = t * kNT + half * 32;
                if (i < a.m) {
#pragma unroll
                    for (int jj = 0; jj < 32; ++jj)
                        if (jb + jj < a.n) C[i + (jb + jj) * a.ldc] = v[jj];
                }
            }
        }
        return true;
    });
    if (!ok && lane == 0) atomicOr(status, kDevErrTimeout);
    tcf_before();
    named_barrier(2, 288);  // with warp 5, before it frees tensor memory
}

size_t rank_tc_bytes(int64_t k, int64_t ntiles) {
    return (size_t)ntiles * (size_t)(k <= kKB ? 1 : 2) * (kBCHUNK + sizeof(uint2));
}

cudaError_t launch_pack_b_rank_tc(int64_t k, int64_t n, const float *B, int64_t ldb, int64_t ntiles, void *dst, cudaStream_t s) {
    const int kc = k <= kKB ? 1 : 2;
    unsigned char *d = static_cast<unsigned char *>(dst);
    pack_b_rank_tc_kernel<<<dim3((unsigned)ntiles, (unsigned)kc), 256, 0, s>>>(
        B, k, n, ldb, d, reinterpret_cast<uint2 *>(d + ntiles * kc * kBCHUNK));
    return cudaGetLastError();
}

template <int KC>
static cudaError_t launch_rank_tc_t(const CUtensorMap *tmA, const CUtensorMap *tmC, RankArgs a, unsigned *status,
                                    cudaStream_t s) {
    using Cfg = RankTcCfg<KC>;
    const cudaError_t e = ensure_smem_limit(reinterpret_cast<const void *>(rankk_tc_kernel<KC>), Cfg::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t ntiles = (a.n + kNT - 1) / kNT, tiles = (a.m + Cfg::BM - 1) / Cfg::BM * ntiles;
    const int64_t slots = a.num_sms > 0 ? a.num_sms : 1;
    const unsigned grid = (unsigned)(tiles < slots ? tiles : slots);
    if (grid == 0) return cudaSuccess;
    a.brange = reinterpret_cast<const uint2 *>(static_cast<const unsigned char *>(a.Bt) + ntiles * KC * kBCHUNK);
    CUtensorMap none;
    std::memset(&none, 0, sizeof(none));
    rankk_tc_kernel<KC><<<grid, Cfg::THREADS, Cfg::SMEM, s>>>(*tmA, tmC ? *tmC : none, a, status, tmC ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_rankk_tc(const CUtensorMap *tmA, const CUtensorMap *tmC, const RankArgs &a, unsigned *status,
                            cudaStream_t s) {
    return a.k <= kKB ? launch_rank_tc_t<1>(tmA, tmC, a, status, s) : launch_rank_tc_t<2>(tmA, tmC, a, status, s);
}

}  // namespace tsmm
