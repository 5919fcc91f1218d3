// Regime (ii), FP64, on the tensor cores at FP64 accuracy: C[m x n] = alpha * A[m x k] * B[k x n] + beta * C0.
//
// The FP64 pipe has 4 flop per clock and SM and bounded these shapes (m = n = 16384, k = 32, beta = 1: 14.0 ms, where C in
// and out takes 0.64 ms).  As in regime (i) (tsmm_tall_tc64.cuh) every row of A and column of B is written in fixed point
// over a power of two above its largest entry, here cut into eight signed digits of 8 bits each (63 bits), and the 36
// products of digits i + j <= 7 are summed exactly, one FP32 accumulator per order, over at most 32 columns of k
// (8 * 32 * 2^14 = 2^22).  The orders are combined in a 64-bit integer per output, over the whole k, and rounded to a
// double by integer operations; what is left to the FP64 pipe is alpha * v + beta * C0.
//
// Measured, m = n = 16384, beta = 1: k = 4: 1.97 -> 0.93 ms, k = 32: 14.0 -> 0.93 ms, k = 64: 28.1 -> 1.28 ms, k = 128: 55.7 ->
// 2.79 ms; without TMA for C (m = 16383) 14.5 -> 1.15 ms; relative error at k = 32: 2.1e-16 -> 7.4e-17.  Bound by the
// epilogue's instructions (75 an output at k <= 32, issued in 54 % of the cycles).  What made it so: the integers out of the
// accumulators by bits alone (they start at 1.5 * 2^23, one more MMA a chunk; 104 instructions an output and 1.35 ms
// without), equal shares of the tiles per block, loads of accumulators and of C0 ahead of their use (1.03 -> 0.97 ms),
// no comparisons of doubles per tile (they take the FP64 pipe like an output: 1.03 -> 0.93 ms), no spills (k = 64: 1.69 ->
// 1.28 ms).
//
// Errors, relative to S = 2^E 2^F (the row's and the column's power): 2^-62 k of the cut, 2^-61.2 k of the orders above 7,
// 2^-(55+SH) per 32 columns of k of order 7's rounding.  The library's bound 4 k 2^-53 sum|a||b|, less three roundings, holds
// where sum|a||b| is at least 0.0041 S (k >= 4); the epilogue proves that per output from the top 7 bits of the entries,
// usually of the eight columns of k that are largest in B's tile.  Outputs where it cannot (and rows or columns with infinities, NaNs or entries
// beyond 2^+-400) are recomputed with FP64 fmas: row by row where a warp has few such rows (rows of B scaled by
// 10^+-3, k = 8, m = 8192: 2.97 ms with all rows, 1.06 ms so; fma kernel 1.86 ms).
//
// Persistent blocks, one per SM, walk equal shares of the tiles (128 rows x 16 columns), an item per m-tile, 24 warps:
//   warps 0-3   converters: thread = row of the item's A, from global memory; digits of the first 64 columns to tensor
//               memory, of columns 64..127 to shared memory
//   warp 4      producer of B's digits (32 k x 16 columns, 8.5 KB a chunk)
//   warp 5      tensor-memory owner and MMA issuer: digit i of A times digits 0..7-i of B, N = 16 (8 - i), into the
//               adjacent accumulators of orders i..7; two sets of accumulators
//   warp 6      C0 loader;  warp 7  storer: tiles of C live in one of CS slots from C0's arrival to C's store
//   warps 8-23  epilogue: two sets for tiles of either parity, thread = row and 8 columns
#include <climits>
#include <cstring>

#include "tsmm_digits64.cuh"

namespace tsmm {

namespace {

constexpr int kKC = 32;                          // k per chunk: what an accumulator holds exactly
constexpr int kNT = kRank64Sub;                  // 16 columns per tile
constexpr int kND = 8;                           // digits
constexpr int kBCHUNK = kND * kNT * kKC * 2;     // digits of a chunk of B
constexpr int kG1 = kNT * 8 + 16 + kNT * 2;      // a tile's record: RankB64::g1
constexpr int kG1W = kNT * 8, kG1F = kNT * 8 + 16;
constexpr int kG2 = kNT * kKC;                   // guard bytes of a chunk
constexpr int kCONST = 128 * 16 * 2;             // operand that starts the accumulators
constexpr int kNeed = 72;                        // 0.0044 * 2^14

struct RankB64 {
    const unsigned char *digits;  // [tile of 16][chunk of 32 k][kBCHUNK]
    const unsigned char *g2;      // guard bytes: [tile][chunk][16][32]
    // [tile]: guard bytes [16][8] of its two largest groups of four rows, at kG1W the groups' numbers, at kG1F the scales
    // of the columns as 16-bit integers
    const unsigned char *g1;
};

template <int KH>  // chunks of k: 1, 2, or 3 and 4
struct RankTc64Cfg {
    static constexpr int BM = 128;
    static constexpr int NB = KH == 4 ? 3 : 4;              // chunks of B in flight
    static constexpr int CS = KH == 4 ? 2 : 8;              // C slots; even, so that a slot always serves tiles of one parity
    static constexpr int RING = KH == 1 ? 4 : 2;            // items whose scales and guard bytes are kept
    static constexpr int SH = KH == 1 ? 3 : KH == 2 ? 2 : 1;  // unit of the sums: 2^-SH of the order-5 products
    static constexpr int A_BUFS = KH == 1 ? 2 : 1;
    static constexpr int COL_A = 2 * kND * kNT, A_COLS = (KH == 1 ? 2 : 4) * kND * 8;
    static constexpr int SLOT = BM * kNT * 8;
    static constexpr int ADIG = BM * kKC * 2;               // one digit of a chunk of A in shared memory
    static constexpr int OFF_E = 512;
    static constexpr int OFF_G = OFF_E + RING * BM * 4;     // guard bytes of A: [RING][KH * 8 words][BM]
    static constexpr int OFF_K = (OFF_G + RING * KH * 8 * BM * 4 + 1023) / 1024 * 1024;
    static constexpr int OFF_B = OFF_K + kCONST;
    static constexpr int OFF_C = OFF_B + NB * kBCHUNK;
    static constexpr int OFF_A = OFF_C + CS * SLOT;
    static constexpr int SMEM = OFF_A + (KH == 4 ? 2 * kND * ADIG : 0);
    static constexpr int NBAR = 4 + 2 * NB + 6 + 3 * CS;
    static constexpr int THREADS = 768;                     // 80 registers each at launch, dealt out again by role:
    static constexpr int VREG = 72, MREG = 48, EREG = 88;
    static_assert(128 * VREG + 128 * MREG + 512 * EREG <= THREADS * 80, "register split");
    static_assert(NBAR * 8 + 16 <= OFF_E, "barrier area");
    static_assert(COL_A + A_BUFS * A_COLS <= 512, "tensor memory");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ void store_2d(const void *tmap, const void *src, int32_t x, int32_t y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];\n\t"
                 "cp.async.bulk.commit_group;" ::"l"(reinterpret_cast<uint64_t>(tmap)),
                 "r"(x), "r"(y), "r"(smem_addr(src))
                 : "memory");
}

__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity) {
    return __all_sync(0xffffffffu, mbar_wait_bounded(bar, parity));
}

__device__ __forceinline__ void tc_st4(uint32_t taddr, const uint32_t *r) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
                 "r"(r[3])
                 : "memory");
}

// Two columns of each of the eight orders' accumulators: started, and waited for (the values pass through the wait, so no
// use can move above it).
__device__ __forceinline__ void ld_orders(uint32_t taddr, uint32_t (&d)[kND][2]) {
#pragma unroll
    for (int i = 0; i < kND; ++i)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];"
                     : "=r"(d[i][0]), "=r"(d[i][1])
                     : "r"(taddr + i * kNT)
                     : "memory");
}
__device__ __forceinline__ void ld_wait(uint32_t (&d)[kND][2]) {
#pragma unroll
    for (int i = 0; i < kND; i += 4)
        asm volatile("tcgen05.wait::ld.sync.aligned;"
                     : "+r"(d[i][0]), "+r"(d[i][1]), "+r"(d[i + 1][0]), "+r"(d[i + 1][1]), "+r"(d[i + 2][0]),
                       "+r"(d[i + 2][1]), "+r"(d[i + 3][0]), "+r"(d[i + 3][1])::"memory");
}

// Scale of a row or column from its largest exponent field: kTc64Emin if it is zero, -1 if the digits do not serve it.
__device__ __forceinline__ int scale_of(int e, bool nonzero) {
    return e > kTc64Emin && e <= kTc64Emax ? e : nonzero ? -1 : kTc64Emin;
}

// T * 2^(x + 32 - 1023), rounded to nearest, for eight sums below 2^62
__device__ __forceinline__ void to_doubles(const int64_t (&T)[8], const int (&x)[8], double (&v)[8]) {
    uint32_t low = 0xffffffffu;
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) low = min(low, (uint32_t)((T[jj] ^ (T[jj] >> 63)) >> 32));
    if (__all_sync(0xffffffffu, low != 0u)) {
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
            const int64_t s = T[jj] >> 63;
            const uint64_t u = (uint64_t)((T[jj] ^ s) - s);
            uint32_t pos;  // of the leading bit, in the high word
            asm("bfind.u32 %0, %1;" : "=r"(pos) : "r"((uint32_t)(u >> 32)));
            const uint32_t sh = 30u - pos;
            const uint64_t w = (((uint64_t)__funnelshift_l((uint32_t)u, (uint32_t)(u >> 32), sh) << 32 | (uint32_t)u << sh) +
                                0x200u) >> 10;  // the leading bit counts into the exponent
            const uint32_t hi = (uint32_t)(w >> 32) + ((uint32_t)(x[jj] + 31 + (int)pos) << 20);
            v[jj] = __hiloint2double((int)(hi | ((uint32_t)(s >> 32) & 0x80000000u)), (int)(uint32_t)w);
        }
    } else {
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
            const int64_t s = T[jj] >> 63;
            uint64_t u = (uint64_t)((T[jj] ^ s) - s);
            const bool zero = u == 0ull;
            const int lz = __clzll((long long)u);
            u = ((u << ((lz - 1) & 63)) + 0x200u) >> 10;
            const uint32_t hi = (uint32_t)(u >> 32) + ((uint32_t)(x[jj] + 62 - lz) << 20);
            v[jj] = zero ? 0.0 : __hiloint2double((int)(hi | ((uint32_t)(s >> 32) & 0x80000000u)), (int)(uint32_t)u);
        }
    }
}

}  // namespace

// Block = tile of 16 columns: scales, then per chunk of 32 k the digits (digit i, column j, k kk at
// (2 i + j/8)*512 + (kk/8)*128 + (j%8)*16 + (kk%8)*2) and the guard's bytes [16][32]; then of the
// two groups of four rows that are largest over the tile, [16][8].
__global__ void __launch_bounds__(256) pack_b_rank_tc64_kernel(const double *__restrict__ B, int64_t k, int64_t n, int64_t ldb,
                                                               int nch, unsigned char *__restrict__ g1,
                                                               unsigned char *__restrict__ g2,
                                                               unsigned char *__restrict__ dst) {
    __shared__ int sF[kNT];
    __shared__ unsigned sum[kRankMaxK / 4];
    if (threadIdx.x < kRankMaxK / 4) sum[threadIdx.x] = 0u;
    {
        const int j = threadIdx.x / 16;
        const int64_t col = (int64_t)blockIdx.x * kNT + j;
        int e = 0;
        unsigned nz = 0u;
        if (col < n)
            for (int64_t p = threadIdx.x % 16; p < k; p += 16) {
                const double x = B[p + col * ldb];
                e = max(e, (__double2hiint(x) >> 20) & 0x7ff);
                nz |= x != 0.0 ? 1u : 0u;
            }
#pragma unroll
        for (int o = 8; o > 0; o /= 2) {
            e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
            nz |= __shfl_xor_sync(0xffffffffu, nz, o);
        }
        if (threadIdx.x % 16 == 0) sF[j] = scale_of(e, nz != 0u);
    }
    __syncthreads();
    for (int c = 0; c < nch; ++c) {
        unsigned char *chunk = dst + ((int64_t)blockIdx.x * nch + c) * kBCHUNK;
        const int j = threadIdx.x / 16, kk = threadIdx.x % 16 * 2;
        const int64_t col = (int64_t)blockIdx.x * kNT + j, p = (int64_t)c * kKC + kk;
        const double *q = B + p + col * ldb;
        uint32_t d[kND];
        uint32_t g = tc64_digits8(p < k && col < n ? q[0] : 0.0, p + 1 < k && col < n ? q[1] : 0.0, max(sF[j], kTc64Emin), d);
        if (sF[j] < 0) g = 0u;
#pragma unroll
        for (int i = 0; i < kND; ++i)
            *reinterpret_cast<uint32_t *>(chunk + (2 * i + j / 8) * 512 + (kk / 8) * 128 + (j % 8) * 16 + (kk % 8) * 2) = d[i];
        *reinterpret_cast<uint16_t *>(g2 + ((int64_t)blockIdx.x * nch + c) * kG2 + j * kKC + kk) = (uint16_t)g;
        atomicAdd(&sum[p / 4], (g & 0xffu) + (g >> 8));
    }
    __syncthreads();
    // the two largest groups, the earliest of equals
    unsigned w[2] = {0u, 1u};
    if (threadIdx.x < 32) {
        for (int u = 0; u < 2; ++u) {
            const unsigned mine = sum[threadIdx.x] << 5 | (31u - threadIdx.x);
            w[u] = 31u - (__reduce_max_sync(0xffffffffu, threadIdx.x < nch * 8 && (u == 0 || threadIdx.x != w[0]) ? mine : 0u) & 31u);
        }
        unsigned char *q = g1 + (int64_t)blockIdx.x * kG1;
        const int j = threadIdx.x / 2;
        const unsigned c = w[threadIdx.x % 2] / 8, at = w[threadIdx.x % 2] % 8;
        // (nothing is to be shown for a zero column)
        reinterpret_cast<uint32_t *>(q)[threadIdx.x] =
            sF[j] == kTc64Emin ? 0x7f7f7f7fu
                               : *reinterpret_cast<const uint32_t *>(g2 + ((int64_t)blockIdx.x * nch + c) * kG2 + j * kKC + at * 4);
        if (threadIdx.x < 2) reinterpret_cast<uint32_t *>(q + kG1W)[threadIdx.x] = w[threadIdx.x];
        if (threadIdx.x < kNT) reinterpret_cast<int16_t *>(q + kG1F)[threadIdx.x] = (int16_t)sF[threadIdx.x];
    }
}

template <int KH>
__global__ void __launch_bounds__(RankTc64Cfg<KH>::THREADS, 1)
    rankk_tc64_kernel(const __grid_constant__ CUtensorMap tmC, const RankArgs a, const RankB64 b64, int nch_arg,
                      unsigned *status, int mode) {
    using Cfg = RankTc64Cfg<KH>;
    constexpr int NB = Cfg::NB, CS = Cfg::CS, BM = Cfg::BM, RING = Cfg::RING, A_BUFS = Cfg::A_BUFS, SH = Cfg::SH;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);
    uint64_t *a_conv = bar;             // [2] digits of A in place
    uint64_t *a_done = a_conv + 2;      // [2] the item's MMAs are complete
    uint64_t *b_full = a_done + 2;      // [NB]
    uint64_t *b_empty = b_full + NB;    // [NB]
    uint64_t *tfull = b_empty + NB;     // [2][2] by parity of the tile (each epilogue set sees every phase), by accumulators
    uint64_t *tempty = tfull + 4;       // [2]
    uint64_t *c_full = tempty + 2;      // [CS] C0 landed in the slot
    uint64_t *c_store = c_full + CS;    // [CS] results written to it
    uint64_t *c_empty = c_store + CS;   // [CS] slot free
    unsigned *tslot = reinterpret_cast<unsigned *>(bar + Cfg::NBAR);
    int *rowE = reinterpret_cast<int *>(smem + Cfg::OFF_E);              // [RING][BM]
    uint32_t *guardA = reinterpret_cast<uint32_t *>(smem + Cfg::OFF_G);  // [RING][KH * 8][BM]
    double *cslots = reinterpret_cast<double *>(smem + Cfg::OFF_C);

    const int warp = threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    const int nch = KH == 1 ? 1 : nch_arg;  // chunks of k
    const int64_t ntiles = (a.n + kNT - 1) / kNT;
    const int64_t total = (a.m + BM - 1) / BM * ntiles;
    const int64_t first = total * blockIdx.x / gridDim.x, last = total * (blockIdx.x + 1) / gridDim.x;
    // from the host: a comparison of doubles takes the FP64 pipe as long as an output does, and would be repeated
    const bool use_c0 = (mode & 1) != 0, scaled = (mode & 2) != 0, c_tma = (mode & 4) != 0;
    const int ksteps = (int)((a.k + 15) / 16);

    if (threadIdx.x == 0) {
        if (c_tma) prefetch_tmap(&tmC);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&a_conv[b], 4);
            mbar_init(&a_done[b], 1);
            mbar_init(&tfull[b], 2);  // the MMAs' completion and the issuer's own arrival, which orders A's scales before it
            mbar_init(&tfull[b + 2], 2);
            mbar_init(&tempty[b], 8);
        }
        for (int b = 0; b < NB; ++b) {
            mbar_init(&b_full[b], 1);
            mbar_init(&b_empty[b], 1);
        }
        for (int s = 0; s < CS; ++s) {
            mbar_init(&c_full[s], c_tma ? 1 : 32);
            mbar_init(&c_store[s], 8);
            mbar_init(&c_empty[s], c_tma ? 1 : 8);
        }
        fence_mbar_init();
    }
    // three entries of 2048 a row: times itself 1.5 * 2^23, so that an accumulator's low bits are an integer
    if (threadIdx.x < kCONST / 16) {
        const bool on = (threadIdx.x / 8) % 2 == 0;
        *reinterpret_cast<uint4 *>(smem + Cfg::OFF_K + threadIdx.x * 16) =
            make_uint4(on ? 0x68006800u : 0u, on ? 0x00006800u : 0u, 0u, 0u);
    }
    fence_proxy_async_smem();
    if (warp == 5) tc_alloc(tslot, 512);
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
        // ------------------------------------------------ producer of B
        reg_dec<Cfg::MREG>();
        if (lane == 0) {
            const uint64_t pol = policy_evict_last();  // read again by other items
            const unsigned char *Bt = b64.digits;
            int64_t gq = 0;
            const bool ok = items([&](int, int64_t, int64_t t0, int64_t t1) {
                for (int64_t c = t0 * nch; c < t1 * nch; ++c, ++gq) {
                    const int sb = (int)(gq % NB);
                    if (gq >= NB && !mbar_wait_bounded(&b_empty[sb], (uint32_t)((gq / NB) & 1) ^ 1)) return false;
                    mbar_arrive_expect_tx(&b_full[sb], kBCHUNK);
                    bulk_load(smem + Cfg::OFF_B + sb * kBCHUNK, Bt + c * kBCHUNK, kBCHUNK, &b_full[sb], pol);
                }
                return true;
            });
            if (!ok) atomicOr(status, kDevErrTimeout);
            // copies still in flight land before the block may exit
            for (int64_t q = gq > NB ? gq - NB : 0; q < gq; ++q)
                mbar_wait_bounded(&b_full[q % NB], (uint32_t)((q / NB) & 1));
        }
        return;
    }

    if (warp == 6) {
        // ------------------------------------------------ C0 loader
        reg_dec<Cfg::MREG>();
        if (!use_c0) return;
        const uint64_t pol = policy_evict_first();
        const double *C = static_cast<const double *>(a.C);
        int64_t q = 0;  // tiles issued
        const bool ok = items([&](int, int64_t mt, int64_t t0, int64_t t1) {
            for (int64_t t = t0; t < t1; ++t, ++q) {
                const int st = (int)(q % CS);
                if (q >= CS && !warp_wait(&c_empty[st], (uint32_t)((q / CS) & 1) ^ 1)) return false;
                double *slot = cslots + st * (BM * kNT);
                if (c_tma) {
                    if (lane == 0) {
                        mbar_arrive_expect_tx(&c_full[st], Cfg::SLOT);
                        tma_load_2d(slot, &tmC, (int32_t)(mt * BM), (int32_t)(t * kNT), &c_full[st], pol);
                    }
                } else {
                    // rows lane + 32 rr of every column, walking one column pointer by ldc
                    const int64_t i0 = mt * BM;
                    const double *colp = C + i0 + lane + t * kNT * a.ldc;
                    double *dst = slot + lane;
                    for (int c = 0; c < kNT; ++c, colp += a.ldc, dst += BM) {
                        const bool cin = t * kNT + c < a.n;
#pragma unroll
                        for (int rr = 0; rr < BM / 32; ++rr) {
                            const bool in = cin && i0 + lane + 32 * rr < a.m;
                            cp_async_elem(dst + 32 * rr, in ? colp + 32 * rr : C, in, 8);
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

    if (warp == 7) {
        // ------------------------------------------------ storer (TMA): a slot is freed once its store has read it
        reg_dec<Cfg::MREG>();
        if (!c_tma || lane != 0) return;
        int64_t q = 0;
        const bool ok = items([&](int, int64_t mt, int64_t t0, int64_t t1) {
            for (int64_t t = t0; t < t1; ++t, ++q) {
                const int st = (int)(q % CS);
                if (!mbar_wait_bounded(&c_store[st], (uint32_t)((q / CS) & 1))) return false;
                store_2d(&tmC, cslots + st * (BM * kNT), (int32_t)(mt * BM), (int32_t)(t * kNT));
                if (CS == 2) {
                    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                    mbar_arrive(&c_empty[st]);
                } else if (q >= 1) {  // the newest store stays in flight
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
        reg_dec<Cfg::MREG>();
        if (elect_one()) {
            const uint64_t bdesc = tc_desc(smem_addr(smem + Cfg::OFF_B), 512);
            const uint64_t adesc = tc_desc(smem_addr(smem + Cfg::OFF_A), 512);
            const uint64_t kdesc = tc_desc(smem_addr(smem + Cfg::OFF_K), 256);
            const uint32_t blo = (uint32_t)bdesc, bhi = (uint32_t)(bdesc >> 32);
            int64_t g = 0;
            int nj = 0, par = 0;
            const bool ok = items([&](int j, int64_t, int64_t t0, int64_t t1) {
                const int ab = A_BUFS == 2 ? j & 1 : 0;
                if (!mbar_wait_bounded(&a_conv[j & 1], (uint32_t)(j >> 1) & 1)) return false;
                tcf_after();
                for (int64_t t = t0; t < t1; ++t, par ^= 1) {
#pragma unroll 1
                    for (int c = 0; c < nch; ++c, ++g) {
                        const int tb = (int)(g & 1), sb = (int)(g % NB);
                        if (g >= 2 && !mbar_wait_bounded(&tempty[tb], (uint32_t)((g >> 1) & 1) ^ 1)) return false;
                        if (!mbar_wait_bounded(&b_full[sb], (uint32_t)((g / NB) & 1))) return false;
                        tcf_after();
                        const uint32_t d0 = tmem + tb * (kND * kNT);
                        const uint32_t bd = blo + sb * (kBCHUNK / 16);
                        tc_mma_ss(d0, kdesc, kdesc, tc_idesc_f16(BM, kNT * kND), 0);
#pragma unroll
                        for (int ks = 0; ks < 2; ++ks) {
                            if (2 * c + ks >= ksteps) break;
                            const uint32_t at = tmem + Cfg::COL_A + ab * Cfg::A_COLS + (2 * c + ks) * (kND * 8);
                            const uint32_t bf = bd + ks * 16;
                            static_for<0, kND>([&](auto i_tag) {
                                constexpr int i = decltype(i_tag)::value;
                                constexpr uint32_t idesc = tc_idesc_f16(BM, kNT * (kND - i));
                                if (KH < 4 || c < 2) {
                                    tc_mma_ts2<true>(d0 + i * kNT, at + i * 8, bf, bhi, idesc);
                                } else {
                                    tc_mma_ss(d0 + i * kNT, adesc + (((c - 2) * kND + i) * Cfg::ADIG + ks * 256) / 16,
                                              (uint64_t)bhi << 32 | bf, idesc, 1);
                                }
                            });
                        }
                        tc_commit(&b_empty[sb]);
                        mbar_arrive(&tfull[2 * par + tb]);
                        tc_commit(&tfull[2 * par + tb]);
                    }
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
        named_barrier(2, 544);  // warps 5 and 8..23
        tcf_after();
        tc_dealloc(tmem, 512);
        return;
    }

    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    if (warp < 4) {
        // ------------------------------------------------ converters
        reg_dec<Cfg::VREG>();
        const int r = threadIdx.x;
        const bool ok = items([&](int j, int64_t mt, int64_t, int64_t) {
            // the digits' place: the MMAs of the item that last used it are complete (and the epilogue is done with the
            // scales and guard bytes of RING items ago: an accumulator of that item was reused since)
            if (j >= A_BUFS && !warp_wait(&a_done[(j - A_BUFS) & 1], (uint32_t)((j - A_BUFS) >> 1) & 1)) return false;
            tcf_after();
            const int64_t i = mt * BM + r;
            const double *src = static_cast<const double *>(a.A) + (i < a.m ? i : 0);
            auto at = [&](int p) { return p < a.k && i < a.m ? __ldg(src + p * a.lda) : 0.0; };
            int e = 0;
            bool nz = false;
#pragma unroll 1
            for (int p = 0; p < a.k; p += 16) {
                double x[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) x[q] = at(p + q);
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    e = max(e, (__double2hiint(x[q]) >> 20) & 0x7ff);
                    nz |= x[q] != 0.0;
                }
            }
            const int E = scale_of(e, nz);
            rowE[(j % RING) * BM + r] = E;
            uint32_t *gw = guardA + (j % RING) * (KH * 8 * BM) + r;
            const uint32_t td = tlane + Cfg::COL_A + (A_BUFS == 2 ? j & 1 : 0) * Cfg::A_COLS;
            for (int p = 0; p < nch * kKC; p += 8) {
                uint32_t d[kND][4], gb[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t dd[kND];
                    gb[q] = tc64_digits8(at(p + 2 * q), at(p + 2 * q + 1), max(E, kTc64Emin), dd);
#pragma unroll
                    for (int u = 0; u < kND; ++u) d[u][q] = dd[u];
                }
                gw[(p / 4) * BM] = E < 0 ? 0u : gb[0] | gb[1] << 16;
                gw[(p / 4 + 1) * BM] = E < 0 ? 0u : gb[2] | gb[3] << 16;
                if (KH < 4 || p < 64) {
                    const uint32_t tp = td + (p / 16) * (kND * 8) + (p % 16) / 2;
#pragma unroll
                    for (int u = 0; u < kND; ++u) tc_st4(tp + u * 8, d[u]);
                } else {
                    unsigned char *sp = smem + Cfg::OFF_A + (p / kKC - 2) * (kND * Cfg::ADIG) + (r / 8) * 512 +
                                        (p % kKC / 8) * 128 + (r % 8) * 16;
#pragma unroll
                    for (int u = 0; u < kND; ++u)
                        *reinterpret_cast<uint4 *>(sp + u * Cfg::ADIG) = make_uint4(d[u][0], d[u][1], d[u][2], d[u][3]);
                }
            }
            if (KH == 4) fence_proxy_async_smem();  // the MMAs read shared memory through the async proxy
            tc_wait_st();
            tcf_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&a_conv[j & 1]);
            return true;
        });
        if (!ok && lane == 0) atomicOr(status, kDevErrTimeout);
        return;
    }

    // ---------------------------------------------------- epilogue (warps 8-23); each warp gives up on its own
    reg_inc<Cfg::EREG>();
    const int par = (warp - 8) / 8, half = (warp / 4) & 1;
    const int r = (warp & 3) * 32 + lane;
    const double alpha = a.alpha, beta = a.beta;
    double *C = static_cast<double *>(a.C);
    int q = 0, g = 0;      // tiles and chunks of this block
    uint32_t phases = 0u;  // of this set's two tfull barriers
    const bool ok = items([&](int j, int64_t mt, int64_t t0, int64_t t1) {
        const int64_t i = mt * BM + r;
        const uint32_t *ga = guardA + (j % RING) * (KH * 8 * BM) + r;
        for (int64_t t = t0; t < t1; ++t, ++q, g += nch) {
            if ((q & 1) != par) continue;
            const int64_t j0 = t * kNT + half * 8;  // first column
            uint4 fs;  // scales of the eight columns, 16 bits each
            int64_t T[8];
            uint32_t redo = 0u;
            bool proven = false;
            int E = 0;
#pragma unroll
            for (int c = 0; c < KH; ++c) {
                if (c >= nch) break;
                const int tb = (g + c) & 1;
                uint4 gb[4];  // two columns each
                uint2 gw;
                if (c == 0) {
                    const unsigned char *g1 = b64.g1 + t * kG1;
#pragma unroll
                    for (int u = 0; u < 4; ++u) gb[u] = __ldg(reinterpret_cast<const uint4 *>(g1) + half * 4 + u);
                    gw = __ldg(reinterpret_cast<const uint2 *>(g1 + kG1W));
                    fs = __ldg(reinterpret_cast<const uint4 *>(g1 + kG1F) + half);
                }
                if (!warp_wait(&tfull[2 * par + tb], phases >> tb & 1u)) return false;
                phases ^= 1u << tb;
                tcf_after();
                const uint32_t acc = tlane + tb * (kND * kNT) + half * 8;
                uint32_t d[2][kND][2];
                ld_orders(acc, d[0]);  // on its way during the guard, as the next two columns are while two are combined
                if (c == 0) {
                    // guard: sum of products of top digits, here of eight columns of k
                    E = rowE[(j % RING) * BM + r];
                    const uint32_t w0 = ga[gw.x * BM], w1 = ga[gw.y * BM];
                    uint32_t low = 0xffffffffu;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        low = min(low, __dp4a(w0, gb[u].x, __dp4a(w1, gb[u].y, 0u)));
                        low = min(low, __dp4a(w0, gb[u].z, __dp4a(w1, gb[u].w, 0u)));
                    }
                    proven = __all_sync(0xffffffffu, low >= (uint32_t)kNeed || i >= a.m);
                }
                if (c == nch - 1 && !proven) {
                    // of all columns of k, and which outputs need the fmas (four at a time, for few registers)
#pragma unroll 1
                    for (int q4 = 0; q4 < 8; q4 += 4) {
                        const unsigned char *gc = b64.g2 + t * nch * kG2 + (half * 8 + q4) * kKC;
                        uint32_t gs[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
                        for (int w = 0; w < nch * 8; w += 4) {
                            const uint32_t *wa = ga + w * BM;
#pragma unroll
                            for (int jj = 0; jj < 4; ++jj) {
                                const uint4 b = __ldg(reinterpret_cast<const uint4 *>(gc + w / 8 * kG2 + w % 8 * 4 + jj * kKC));
                                gs[jj] = __dp4a(wa[0], b.x, __dp4a(wa[BM], b.y, __dp4a(wa[2 * BM], b.z, __dp4a(wa[3 * BM], b.w, gs[jj]))));
                            }
                        }
                        const uint32_t fp[2] = {q4 ? fs.z : fs.x, q4 ? fs.w : fs.y};
                        const int f[4] = {(int16_t)fp[0], (int)fp[0] >> 16, (int16_t)fp[1], (int)fp[1] >> 16};
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj)
                            if (E < 0 || f[jj] < 0 || (gs[jj] < (uint32_t)kNeed && E != kTc64Emin && f[jj] != kTc64Emin))
                                redo |= 1u << (q4 + jj);
                    }
                    if (i >= a.m) redo = 0u;
                }
                // An accumulator reads kM23 + order sum; a pair of orders 2 u, 2 u + 1 then is kPair plus a sum below
                // 2^30, modulo 2^32.  The constants leave the sum in one 64-bit addend.
                constexpr uint32_t kPair = 0x8b400000u;  // 0x4b400000 * 257
                constexpr uint64_t kOff = 0ull - ((uint64_t)kPair << (32 + SH)) - ((uint64_t)kPair << (16 + SH)) -
                                          ((uint64_t)kPair << SH) - (uint64_t)(kPair >> (16 - SH));
                static_assert(kPair % (1u << (16 - SH)) == 0u, "the rounding commutes with the offset");
                static_assert((kOff & 0xffffffffull) <= 0xffffffffull - (0xffffffffu >> (16 - SH)), "no carry");
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    ld_wait(d[h & 1]);
                    if (h < 3) {
                        ld_orders(acc + 2 * h + 2, d[(h + 1) & 1]);
                    } else {
                        tcf_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&tempty[tb]);
                    }
#pragma unroll
                    for (int jj = 0; jj < 2; ++jj) {
                        uint32_t pr[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) pr[u] = d[h & 1][2 * u][jj] * 256u + d[h & 1][2 * u + 1][jj];
                        const uint32_t low = ((pr[3] + (1u << (15 - SH))) >> (16 - SH)) + (uint32_t)kOff;
                        uint64_t x = (uint64_t)pr[2] * (1u << SH) + ((kOff & 0xffffffff00000000ull) | low);
                        x += (uint64_t)pr[1] * (1u << (16 + SH));
                        x += (uint64_t)(pr[0] << SH) << 32;
                        T[2 * h + jj] = (int64_t)(KH == 1 || c == 0 ? x : x + (uint64_t)T[2 * h + jj]);
                    }
                    // formed before the next but one is read (registers)
                    asm volatile("" : "+l"(T[2 * h]), "+l"(T[2 * h + 1]));
                }
            }
            const int st = q % CS;
            const uint32_t ph = (uint32_t)((q / CS) & 1);
            double *slot = cslots + st * (BM * kNT) + half * (8 * BM) + r;  // first column, own row
            if (use_c0 ? !warp_wait(&c_full[st], ph) : (c_tma && q >= CS && !warp_wait(&c_empty[st], ph ^ 1))) return false;
            if (uint32_t rows = __ballot_sync(0xffffffffu, redo != 0u)) {
                // FP64 fmas from the packed panel, in place before the other outputs
                const double *Bp = static_cast<const double *>(a.Bp) + (j0 / kRankNT) * a.kp * kRankNT + j0 % kRankNT;
                auto put = [&](int row, int jj, double o) {
                    double *p = slot - r + row + jj * BM;
                    o *= alpha;
                    if (use_c0) o = fma(beta, *p, o);
                    if (c_tma) *p = o;
                    else if (j0 + jj < a.n) C[mt * BM + row + (j0 + jj) * a.ldc] = o;
                };
                if (__popc(rows) <= 8) {
                    // few rows: one by one, lane = column and quarter of k
                    for (; rows != 0u; rows &= rows - 1u) {
                        const int src = __ffs((int)rows) - 1, jj = lane / 4;
                        const int row = (warp & 3) * 32 + src;
                        const double *Ap = static_cast<const double *>(a.A) + mt * BM + row;
                        double s = 0.0;
#pragma unroll 4
                        for (int p = lane % 4; p < a.k; p += 4) s = fma(__ldg(Ap + p * a.lda), __ldg(Bp + p * kRankNT + jj), s);
                        s += __shfl_xor_sync(0xffffffffu, s, 1);
                        s += __shfl_xor_sync(0xffffffffu, s, 2);
                        if ((__shfl_sync(0xffffffffu, redo, src) >> jj & 1u) && lane % 4 == 0) put(row, jj, s);
                    }
                } else {
                    const double *Ap = static_cast<const double *>(a.A) + (i < a.m ? i : 0);
#pragma unroll 1
                    for (int q4 = 0; q4 < 8; q4 += 4) {
                        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
                        for (int p = 0; p < (int)a.k; ++p) {
                            const double xa = __ldg(Ap + p * a.lda);
                            const double2 b0 = __ldg(reinterpret_cast<const double2 *>(Bp + p * kRankNT + q4));
                            const double2 b1 = __ldg(reinterpret_cast<const double2 *>(Bp + p * kRankNT + q4 + 2));
                            s[0] = fma(xa, b0.x, s[0]);
                            s[1] = fma(xa, b0.y, s[1]);
                            s[2] = fma(xa, b1.x, s[2]);
                            s[3] = fma(xa, b1.y, s[3]);
                        }
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj)
                            if (redo >> (q4 + jj) & 1u) put(r, q4 + jj, s[jj]);
                    }
                }
                __syncwarp();
            }
            double old[8];
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) old[jj] = use_c0 ? slot[jj * BM] : 0.0;
            int x[8];
            double v[8];
#pragma unroll
            for (int jj = 0; jj < 8; jj += 2) {
                const uint32_t fp = jj < 2 ? fs.x : jj < 4 ? fs.y : jj < 6 ? fs.z : fs.w;
                x[jj] = E + (int16_t)fp - 1075 - SH;
                x[jj + 1] = E + ((int)fp >> 16) - 1075 - SH;
            }
            to_doubles(T, x, v);
            if (scaled) {
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) v[jj] *= alpha;
            }
            if (use_c0) {
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) v[jj] = fma(beta, old[jj], v[jj]);
            }
            if (c_tma) {
#pragma unroll
                for (int jj = 0; jj < 8; ++jj)
                    if (!(redo >> jj & 1u)) slot[jj * BM] = v[jj];
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&c_store[st]);
            } else {
                if (use_c0) {
                    release_reads_to_async_copy();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&c_empty[st]);
                }
                if (i < a.m) {
#pragma unroll
                    for (int jj = 0; jj < 8; ++jj)
                        if (j0 + jj < a.n && !(redo >> jj & 1u)) C[i + (j0 + jj) * a.ldc] = v[jj];
                }
            }
        }
        return true;
    });
    if (!ok && lane == 0) atomicOr(status, kDevErrTimeout);
    tcf_before();
    named_barrier(2, 544);  // with warp 5, before it frees tensor memory
}

// Behind the packed panel: the digits, the guard's bytes and the tiles' records.
static RankB64 layout(const void *base, int64_t k, int64_t ntiles) {
    const int64_t tiles = ntiles * (kRankNT / kNT), nch = (k + kKC - 1) / kKC;
    RankB64 b;
    b.digits = static_cast<const unsigned char *>(base);
    b.g2 = b.digits + tiles * nch * kBCHUNK;
    b.g1 = b.g2 + tiles * nch * kG2;
    return b;
}

size_t rank_tc64_bytes(int64_t k, int64_t ntiles) {
    const int64_t nch = (k + kKC - 1) / kKC;
    return (size_t)(ntiles * (kRankNT / kNT) * (nch * (kBCHUNK + kG2) + kG1));
}

cudaError_t launch_pack_b_rank_tc64(int64_t k, int64_t n, const double *B, int64_t ldb, int64_t ntiles, void *dst,
                                    cudaStream_t s) {
    const RankB64 b = layout(dst, k, ntiles);
    pack_b_rank_tc64_kernel<<<(unsigned)(ntiles * (kRankNT / kNT)), 256, 0, s>>>(
        B, k, n, ldb, (int)((k + kKC - 1) / kKC), const_cast<unsigned char *>(b.g1),
        const_cast<unsigned char *>(b.g2), static_cast<unsigned char *>(dst));
    return cudaGetLastError();
}

template <int KH>
static cudaError_t launch_rank_tc64_t(const CUtensorMap *tmC, const RankArgs &a, unsigned *status, cudaStream_t s) {
    using Cfg = RankTc64Cfg<KH>;
    const cudaError_t e = ensure_smem_limit(reinterpret_cast<const void *>(rankk_tc64_kernel<KH>), Cfg::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (a.m + Cfg::BM - 1) / Cfg::BM * ((a.n + kNT - 1) / kNT);
    const int64_t slots = a.num_sms > 0 ? a.num_sms : 1;
    const unsigned grid = (unsigned)(tiles < slots ? tiles : slots);
    if (grid == 0) return cudaSuccess;
    CUtensorMap none;
    std::memset(&none, 0, sizeof(none));
    rankk_tc64_kernel<KH><<<grid, Cfg::THREADS, Cfg::SMEM, s>>>(tmC ? *tmC : none, a,
                                                                layout(a.Bt, a.k, (a.n + kRankNT - 1) / kRankNT),
                                                                (int)((a.k + kKC - 1) / kKC), status,
                                                                (a.beta != 0.0 ? 1 : 0) | (a.alpha != 1.0 ? 2 : 0) | (tmC ? 4 : 0));
    return cudaGetLastError();
}

cudaError_t launch_rankk_tc64(const CUtensorMap *tmC, const RankArgs &a, unsigned *status, cudaStream_t s) {
    if (a.k <= kKC) return launch_rank_tc64_t<1>(tmC, a, status, s);
    if (a.k <= 2 * kKC) return launch_rank_tc64_t<2>(tmC, a, status, s);
    return launch_rank_tc64_t<4>(tmC, a, status, s);
}

}  // namespace tsmm
