// Regime (i), FP64, on the tensor cores at FP64 accuracy: C[m x n] = alpha * A[m x k] * B[k x n] + beta * C0.
//
// The FP64 pipe has 4 flop per clock and SM; the FP16 tensor pipe has two thousand times that.  Every row of A (per
// work item) and every column of B is written in fixed point over a common power of two, A as X = trunc(|x| 2^(55-E)) in
// seven signed digits of 8 bits, x = +-sum_i d_i 2^(48-8i) with d in [-128, 128], B with 63 bits in eight.  FP16 holds a
// digit exactly.  The product of digit i of A with digit j of B has weight 2^-8(i+j); the products of one order i + j are
// summed on the tensor cores in an FP32 accumulator of their own.  Over at most 128 columns of k such a sum stays below
// 7 * 128 * 2^14 < 2^24, so it is an exact integer; it is then added to a 96-bit integer in registers.
// (Splitting a product into exactly accumulated slices: Ozaki, Ogita, Oishi, Rump, Numer. Algorithms 2012.)
//   W <= 48: the 35 products of orders 0..7, eight accumulators.
//   W = 64: tensor memory holds seven.  The 28 products of orders 0..6, where order 6 takes, in place of digit j of B,
//     FP16(d_j + 2^-8 d_(j+1)): its 11 bits bring in order 7 but for 2^-4 of it at no further product (order 7 as products
//     of its own: 4.09 ms at n = 64 against 3.56; without it, at 3.43 ms, B's rows scaled by 10^U[-3,3] had an
//     error of 1.3e-15 to 1.7e-15 where the fma kernel's is 3.9e-16 to 5.5e-16).
// Errors, per term and relative to 2^E 2^F (the powers above the row's and the column's largest entry): 2^-55 of the cut of
// A, 2^-60 of the orders left out.  Per group of up to 128 columns the sums are rounded to a multiple of 2^-58, and again
// where the row's scale grows (to a multiple of 2^-54, n = 64 took 3.48 ms but had twice the error on uneven rows).  An
// entry much smaller than its row's or column's largest is thus held with fewer bits than FP64 has: the error is that of
// the row's and column's scale, not of each product's own, and the guard below bounds what that may cost.
//
// Measured, m = k = 32768, calls back to back: n = 64: 111.6 -> 3.55 ms (FP64 pipe 98 % busy before; now 40 TFLOP/s FP64,
// 2.4 TB/s), n = 48: 3.25 ms, n = 32: 55.7 -> 2.48 ms, n = 4: 7.0 -> 2.00 ms (4.3 TB/s); relative error against compensated
// sums, k = 2048 and 8192: uniform entries 2.8e-16 to 5.5e-16 -> 1.2e-16 to 1.9e-16, rows of B scaled by 10^U[-3,3] 3.0e-16
// to 5.5e-16 -> 1.3e-16 to 1.8e-16, columns of A scaled by 2^U[-2,2] and rows of B by the inverse 2.8e-16 to 5.5e-16 ->
// 2.0e-16 to 2.4e-16.
// Bound by issue: a step of 16 columns costs the converters about 2000 warp instructions (HBM alone would leave 710
// cycles a step, the MMAs take 900 at n = 64, 330 at n <= 16), and at n = 64 by the drains of the accumulators, which
// tensor memory cannot hold twice there (seven conversions to integers an output had made a drain 4400 cycles, and
// 3.64 ms; two of them are magic additions).  Two sets of converters, so that one's waits overlap the
// other's work (n = 4: 2.60 -> 2.31 ms); two sets of digits where they fit (n = 4: 2.22 -> 2.03 ms); a single elected MMA
// lane (n = 64: 3.97 -> 3.64 ms).
//
// Scale.  E is kept per row and only grows: a chunk with a larger entry closes the current group of chunks (their
// sums are drained at the old scale) and the 96-bit sums are shifted once.
//
// Guard.  The library's bound asks for an error below 4 k 2^-53 sum|a||b|, so the split may be used where an item's
// sum|a||b| is at least 0.07 (W = 64: 0.31) * 2^E 2^F times its share of k; the promoters prove that at the start of the
// item from the top digits of its first columns (16, and up to 512 while those do not suffice): sum of products of 7-bit
// digits >= 1200 (5120) times the share.  Where it cannot be proven (a sparse or
// steeply scaled A or B), and for rows or columns with infinities, NaNs or entries beyond 2^+-400, the block computes
// its item with FP64 fmas from global memory, which is bound by the FP64 pipe as the fma kernel is.
//
// Block: one work item (slab of 128 rows x one k range, the split-K scheme of the fma kernel), 20 warps, one per SM:
//   warps 0-7    converters: thread = row; steps of 16 columns, warps 0-3 the even ones, 4-7 the odd ones (a row's
//                scale passes from step to step); digits to tensor memory
//   warps 8-15   promoters: thread = row and half of the columns; guard, exact sums, epilogue
//   warp 16 producer of A (U: tensor copies of every other column, encode_a_rows);  warp 17 tensor memory and MMAs;
//   warp 18 producer of the digits of B
#pragma once
#include "tsmm_internal.h"
#include "tsmm_finish.cuh"
#include "tsmm_digits64.cuh"
#include "tsmm_fma_item.cuh"

namespace tsmm {

template <int W, bool U>
struct TallTc64Cfg {
    static constexpr int BM = kTcRows;
    static constexpr int KB = kTc64KB;                        // k per step
    static constexpr int GROUP = 128 / KB;                    // steps per exact group, at most
    static constexpr int A_STRIDE = U ? BM + 2 : BM;          // doubles per column slot (U: column 2 c + q in slot 8 q + c)
    static constexpr int A_BYTES = KB * A_STRIDE * 8;
    static constexpr int ND = tc64_accumulators(W);
    static constexpr int B_BYTES = tc64_rows(W) * W * KB * 2;  // the digits of a step of B, digit-major
    static constexpr int SA = W == 64 ? 5 : 8, SB = 4;
    static constexpr int OFF_B = SA * A_BYTES;
    static constexpr int OFF_E = OFF_B + SB * B_BYTES;        // row scales of the last ERING steps
    // the guard's digits of B (kTc64Windows windows), later the fallback's rows of B
    // the promoters read a group's scales once it is complete, when converters may have begun the 4th step after its last
    // (DB; 3rd otherwise), with two sets of accumulators a group later
    static constexpr int ERING = W == 16 ? 16 : 8;
    static constexpr int OFF_F = OFF_E + ERING * BM * 4;
    static constexpr int F_BYTES = W == 16 ? 2 * kFmaRows * W * 8 + 8 * BM * 8 : kTc64Windows * 64 * W;
    static_assert(F_BYTES >= 2 * kFmaRows * W * 8, "fallback rows");
    static constexpr int OFF_BAR = OFF_F + F_BYTES;
    static constexpr int NBAR = 2 * SA + 2 * SB + 18;
    static constexpr int OFF_Z = OFF_BAR + NBAR * 8 + 96;     // rows taken as zero
    static constexpr int SMEM = OFF_Z + BM;
    static constexpr int THREADS = 640;                       // 96 registers each at launch, dealt out again by role:
    static constexpr int CREG = W == 64 ? 72 : 80, PREG = W == 64 ? 144 : W == 48 ? 128 : 112;
    static constexpr int MREG = W == 64 ? 48 : W == 48 ? 64 : 96;
    static constexpr int CB = W == 64 ? 4 : 8;                // columns a promoter drains at a time
    static constexpr int SH = 4;                              // unit of the sums: 2^-SH of the order-5 products
    // tensor memory: ND accumulators of W columns, then the digits of a step of A, 8 columns each: 3-6 (X), 0-2 (Y).
    // DB: two sets of digits, by step parity; else one, whose X and Y parts are refilled in turn
    static constexpr bool DB = W <= 48;
    static constexpr bool DDB = W == 16;                      // two sets of accumulators, by group parity
    static constexpr int COL_X = (DDB ? 2 : 1) * ND * W, COL_Y = COL_X + 32, COL_SET = DB ? 56 : 0;
    static constexpr int TMEM_COLS = 512;
    static_assert(256 * CREG + 256 * PREG + 128 * MREG <= THREADS * 96, "register split");
    static_assert(COL_Y + 24 + COL_SET <= TMEM_COLS, "tensor memory");
    static_assert(kTc64Windows * 64 * W <= F_BYTES, "guard windows");
    static_assert(256 * (W / 2) * 8 <= SA * A_BYTES, "fallback totals");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

template <int W, bool U>
__device__ __forceinline__ void tall_tc64_block(const CUtensorMap *tmA, const TallArgs &a, int64_t slab, int split) {
    using Cfg = TallTc64Cfg<W, U>;
    constexpr int SA = Cfg::SA, SB = Cfg::SB, KB = Cfg::KB, BM = Cfg::BM;
    extern __shared__ __align__(1024) unsigned char smem[];
    int *rowE = reinterpret_cast<int *>(smem + Cfg::OFF_E);  // [ERING][BM]
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + Cfg::OFF_BAR);
    uint64_t *afull = bar;             // [SA] A landed
    uint64_t *aempty = afull + SA;     // [SA] converters have read it
    uint64_t *bfull = aempty + SA;     // [SB]
    uint64_t *bempty = bfull + SB;     // [SB]
    uint64_t *convx = bempty + SB;     // [2] DB: a step's digits in tensor memory, by step parity; else [0] digits 3-6
    uint64_t *convy = convx + 2;       // digits 0-2 (not DB)
    uint64_t *xdone = convy + 1;       // [2] the MMAs reading digits 3-6 are complete (not DB; by step parity: the sets
    uint64_t *ydone = xdone + 2;       // of converters may be two steps apart); [2] a step's MMAs are complete
    uint64_t *gdone = ydone + 2;       // [2] a group's MMAs are complete, its last step's slot is in gslot
    uint64_t *drained = gdone + 2;     // [2] a group's accumulators are read, by group parity
    uint64_t *scale = drained + 2;     // [4] a step's row scales published, by quarter of the rows
    uint64_t *verdict = scale + 4;     // the guard's answer is in `unsafe`
    uint64_t *fbar = verdict + 1;      // [2] fallback: rows of B landed
    uint64_t *gbar = fbar + 2;         // the guard's digits of B landed
    unsigned *tslot = reinterpret_cast<unsigned *>(bar + Cfg::NBAR);
    unsigned *flag = tslot + 1;
    unsigned *abort_flag = tslot + 2;
    unsigned *unsafe = tslot + 3;
    unsigned *gslot = tslot + 4;       // [2] step of rowE that holds a group's scales
    unsigned char *zrow = smem + Cfg::OFF_Z;  // [BM] no nonzero entry in the guard's columns: zero unless the converters see one
    volatile unsigned *gnew = tslot + 8;  // [4] steps: a byte per quarter of the rows, set where scales grew: a new group

    const int warp = threadIdx.x / 32;
    const int lane = threadIdx.x % 32;
    const int64_t k0 = (int64_t)split * a.kchunk;
    const int64_t k1 = (k0 + a.kchunk < a.kp) ? k0 + a.kchunk : a.kp;
    const int64_t i0 = slab * BM;
    const TcB64 *tb = static_cast<const TcB64 *>(a.Bt);
    const int iters = (int)((k1 - k0) / KB);

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
        mbar_init(convy, 4);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&convx[b], 4);
            mbar_init(&xdone[b], 1);
            mbar_init(&ydone[b], 1);
        }
        mbar_init(&gdone[0], 2);
        mbar_init(&gdone[1], 2);
        mbar_init(&drained[0], 8);
        mbar_init(&drained[1], 8);
        for (int q = 0; q < 4; ++q) mbar_init(&scale[q], 1);
        mbar_init(verdict, 8);
        mbar_init(&fbar[0], 1);
        mbar_init(&fbar[1], 1);
        mbar_init(gbar, 1);
        *abort_flag = 0u;
        *unsafe = 0u;
        fence_mbar_init();
    }
    if (threadIdx.x < BM / 4) reinterpret_cast<unsigned *>(zrow)[threadIdx.x] = 0u;
    if (warp == 17) tc_alloc(tslot, Cfg::TMEM_COLS);
    tcf_before();
    __syncthreads();
    tcf_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);  // uniform: MMA operands stay in uniform registers

    // the guard's answer: false where the item is left to the fmas
    auto go = [&]() { return mbar_wait_bounded(verdict, 0) && *reinterpret_cast<volatile unsigned *>(unsafe) == 0u; };

    if (warp >= 16) {
        reg_dec<Cfg::MREG>();
        if (warp == 16) {
            // ------------------------------------------------ A
            const uint64_t pol = policy_evict_first();
            bool ok = true;
            int it = 0;
            if constexpr (!U) {
                if (lane == 0) {
                    for (; it < iters; ++it) {
                        const int s = it % SA;
                        if (it == SA && !go()) break;
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
                // Chunks within the map's rows: one tensor copy per q (tsmm_tall_tc.cuh; m = 32767, n = 4, k = 32768:
                // 2.14 ms here).
                // Other chunks: lane = column, one bulk copy of the aligned span around its rows (column_span_bytes);
                // columns beyond k are zero-filled.
                const int rows = (int)((a.m - i0 < BM) ? a.m - i0 : BM);
                const int abase = (int)((reinterpret_cast<uintptr_t>(a.A) / 8) & 1);
                const int ldv = (int)((uint64_t)a.lda & 1);
                for (; it < iters; ++it) {
                    const int s = it % SA;
                    if (it == SA && !__all_sync(0xffffffffu, go())) break;
                    if (it >= SA) {
                        const bool got = mbar_wait_bounded(&aempty[s], (uint32_t)((it / SA) & 1) ^ 1);
                        if (!__all_sync(0xffffffffu, got)) {
                            ok = false;
                            break;
                        }
                    }
                    const int64_t pc = k0 + (int64_t)it * KB;
                    if (pc + KB <= 2 * a.arows) {
                        if (lane == 0) {
                            mbar_arrive_expect_tx(&afull[s], Cfg::A_BYTES);
                            for (int q = 0; q < 2; ++q)
                                tma_load_2d(smem + s * Cfg::A_BYTES + q * (kARowsBox * Cfg::A_STRIDE * 8), tmA,
                                            (int32_t)((abase + q * a.lda + i0) & ~(int64_t)1), (int32_t)(pc / 2), &afull[s], pol);
                        }
                        continue;
                    }
                    const int64_t p = pc + lane;
                    double *slot = reinterpret_cast<double *>(smem + s * Cfg::A_BYTES) + ((lane & 1) * 8 + lane / 2) * Cfg::A_STRIDE;
                    const int d = (abase + (int)(p & 1) * ldv) & 1;
                    const bool mine = lane < KB;
                    const uint32_t bytes = mine && p < a.k ? column_span_bytes<double>(rows, d) : 0u;
                    if (mine && p >= a.k) {
                        for (int r = 0; r < Cfg::A_STRIDE; r += 2)
                            *reinterpret_cast<uint4 *>(slot + r) = make_uint4(0, 0, 0, 0);
                        fence_proxy_async_smem();
                    }
                    const uint32_t sum = __reduce_add_sync(0xffffffffu, bytes);
                    __syncwarp();
                    if (lane == 0) mbar_arrive_expect_tx(&afull[s], sum);
                    __syncwarp();
                    if (bytes != 0u)
                        bulk_load(slot, static_cast<const double *>(a.A) + i0 + p * a.lda - d, bytes, &afull[s], pol);
                }
            }
            if (!ok && lane == 0) atomicOr(a.status, kDevErrTimeout);
            if (!ok || !go()) {
                // nobody waits for the copies in flight: they land before the block may exit
                for (int q = it > SA ? it - SA : 0; q < it; ++q) mbar_wait_bounded(&afull[q % SA], (uint32_t)((q / SA) & 1));
            }
        } else if (warp == 18) {
            // ------------------------------------------------ B
            if (lane == 0) {
                const uint64_t pol = policy_evict_last();
                const unsigned char *src = static_cast<const unsigned char *>(a.Bt) + kTc64Head;
                const int64_t wins = (a.k + 63) / 64 - k0 / 64;
                const uint32_t gbytes = (uint32_t)(wins < kTc64Windows ? wins : kTc64Windows) * (64 * W);
                mbar_arrive_expect_tx(gbar, gbytes);
                bulk_load(smem + Cfg::OFF_F, src + (a.k + 63) / 64 * 4 * Cfg::B_BYTES + k0 * W, gbytes, gbar, pol);
                src += (k0 / KB) * Cfg::B_BYTES;
                int it = 0;
                bool ok = true;
                for (; it < iters; ++it, src += Cfg::B_BYTES) {
                    const int s = it % SB;
                    if (it == SB && !go()) break;
                    if (it >= SB && !mbar_wait_bounded(&bempty[s], (uint32_t)((it / SB) & 1) ^ 1)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(&bfull[s], Cfg::B_BYTES);
                    bulk_load(smem + Cfg::OFF_B + s * Cfg::B_BYTES, src, Cfg::B_BYTES, &bfull[s], pol);
                }
                if (!ok) atomicOr(a.status, kDevErrTimeout);
                if (!ok || !go()) {
                    for (int q = it > SB ? it - SB : 0; q < it; ++q)
                        mbar_wait_bounded(&bfull[q % SB], (uint32_t)((q / SB) & 1));
                }
            }
        } else if (warp == 17) {
            // ------------------------------------------------ MMAs: digit i of A times digit j of B into accumulator i + j.
            // One elected lane walks the loop, unrolled over the ring: its operands stay in uniform registers and it needs
            // few issue slots in competition with the converters of its scheduler.  28 (W = 64) or 35 MMAs of N = W: alone they take 9
            // cycles each at W = 16 and 32 (the tensor pipe's rate) at W = 64, and wider ones no less in sum
            if (elect_one()) {
                constexpr uint32_t idesc = tc_idesc_f16(BM, W);
                const uint64_t bdesc = tc_desc(smem_addr(smem + Cfg::OFF_B), 256);
                const uint32_t blo = (uint32_t)bdesc, bhi = (uint32_t)(bdesc >> 32);
                bool ok = true;
                int it = 0, cnt = 0, g = 0;
                uint32_t ring = 0;  // the rings' phase: it / 4
                uint32_t acc = tmem;
                const int steps = go() ? iters : 0;
                // digits [I0, I1) of A, of the step in stage u; an accumulator's first product of a group (digit 3 of A for
                // orders 3-6, 0 for 0-2) overwrites it
                auto mmas = [&](auto u_tag, auto i0_tag, auto i1_tag, auto fresh_tag) {
                    constexpr int u = decltype(u_tag)::value, I0 = decltype(i0_tag)::value, I1 = decltype(i1_tag)::value;
                    constexpr bool fresh = decltype(fresh_tag)::value;
                    const uint32_t bd = blo + u * (Cfg::B_BYTES / 16);
                    const uint32_t set = tmem + (u & 1) * Cfg::COL_SET;
                    static_for<I0, I1>([&](auto i_tag) {
                        constexpr int i = decltype(i_tag)::value;
                        static_for<0, Cfg::ND - i>([&](auto j_tag) {
                            constexpr int j = decltype(j_tag)::value;
                            constexpr int row = Cfg::ND == 7 && i + j == 6 ? 6 + j : j;
                            const uint32_t at = set + (i >= 3 ? Cfg::COL_X + (i - 3) * 8 : Cfg::COL_Y + i * 8);
                            tc_mma_ts2<!(fresh && (i == 3 || (i == 0 && j < 3)))>(acc + (uint32_t)((i + j) * W), at,
                                                                                  bd + row * (W * 2), bhi, idesc);
                        });
                    });
                };
                const auto c0 = std::integral_constant<int, 0>{};
                const auto c3 = std::integral_constant<int, 3>{};
                const auto c7 = std::integral_constant<int, 7>{};
                auto step = [&](auto u_tag) {
                    constexpr int u = decltype(u_tag)::value;  // it mod 4
                    if (!mbar_wait_bounded(&bfull[u], ring & 1)) return false;
                    if (!mbar_wait_bounded(&convx[Cfg::DB ? u & 1 : 0], Cfg::DB ? (uint32_t)(it >> 1) & 1 : u & 1)) return false;
                    tcf_after();
                    bool fresh = it == 0;
                    if (it > 0 && (cnt == Cfg::GROUP || gnew[u] != 0u)) {
                        // the group ends with the previous step
                        gslot[g & 1] = (unsigned)(it - 1) & (Cfg::ERING - 1);
                        mbar_arrive(&gdone[g & 1]);
                        tc_commit(&gdone[g & 1]);
                        // the accumulators of the group to come: the last group's, or (DDB) the one's before it
                        const int q = Cfg::DDB ? g - 1 : g;
                        if (q >= 0 && !mbar_wait_bounded(&drained[q & 1], (uint32_t)(q >> 1) & 1)) return false;
                        tcf_after();
                        fresh = true;
                        cnt = 0;
                        ++g;
                        acc = tmem + (Cfg::DDB ? (uint32_t)(g & 1) * (Cfg::ND * W) : 0u);
                    }
                    ++cnt;
                    if (fresh) mmas(u_tag, c3, c7, std::true_type{});
                    else mmas(u_tag, c3, c7, std::false_type{});
                    if constexpr (!Cfg::DB) {
                        tc_commit(&xdone[u & 1]);
                        if (!mbar_wait_bounded(convy, u & 1)) return false;
                    }
                    if constexpr (!Cfg::DB) tcf_after();
                    if (fresh) mmas(u_tag, c0, c3, std::true_type{});
                    else mmas(u_tag, c0, c3, std::false_type{});
                    tc_commit(&ydone[u & 1]);
                    tc_commit(&bempty[u]);
                    ++it;
                    return true;
                };
                while (it < steps) {
                    ok = step(std::integral_constant<int, 0>{}) && (it == steps || step(std::integral_constant<int, 1>{})) &&
                         (it == steps || step(std::integral_constant<int, 2>{})) &&
                         (it == steps || step(std::integral_constant<int, 3>{}));
                    if (!ok) break;
                    ++ring;
                }
                if (ok && steps > 0) {
                    gslot[g & 1] = 64u | ((unsigned)(it - 1) & (Cfg::ERING - 1));  // 64: the last group
                    mbar_arrive(&gdone[g & 1]);
                    tc_commit(&gdone[g & 1]);
                }
                if (!ok) {
                    atomicOr(a.status, kDevErrTimeout);
                    atomicOr(abort_flag, 1u);
                }
                // nothing may still write tensor memory when it is freed
                for (int q = it > 2 ? it - 2 : 0; q < it; ++q) mbar_wait_bounded(&ydone[q & 1], (uint32_t)(q >> 1) & 1);
            }
            __syncwarp();
            tcf_before();
            named_barrier(2, 288);  // with the promoters: every accumulator is read
            tcf_after();
            tc_dealloc(tmem, Cfg::TMEM_COLS);
        }
        return;
    }

    const int r = threadIdx.x % BM;
    const int64_t row = i0 + r;
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    // split-K: take an arrival ticket; the last arriver finishes, its converters and promoters
    auto finish = [&]() {
        named_barrier(3, 512);
        if (threadIdx.x == 0)  // an item given up in its fallback takes no ticket
            *flag = *abort_flag == 0u && atomicAdd(a.tickets + slab, 1u) == (unsigned)(a.splits - 1) ? 1u : 0u;
        named_barrier(3, 512);
        if (*flag == 0u) return;
        __threadfence();
        tc_finish<double, 512>(a, i0, threadIdx.x);
        if (threadIdx.x == 0) a.tickets[slab] = 0u;  // ready for the next launch on this stream
    };
    if (warp < 8) {
        // ---------------------------------------------------- converters
        reg_dec<Cfg::CREG>();
        const int abase = (int)((reinterpret_cast<uintptr_t>(a.A) / 8) & 1);
        const int ldv = (int)((uint64_t)a.lda & 1);
        const uint32_t vmask = row < a.m ? 0xffffffffu : 0u;  // rows beyond m count as zeros
        uint64_t *sbar = &scale[warp & 3];
        // for rows taken as zero: the bits of their entries (W = 16: while no scale has counted any, which costs n = 4 1 %;
        // without that branch 1.4 %, above W = 16 the branch costs more)
        uint32_t seen_lo = 0u, seen_hi = 0u;
        bool ok = true;
        const int steps = __all_sync(0xffffffffu, go()) ? iters : 0;
        for (int it = warp / 4; it < steps; it += 2) {
            const int s = it % SA;
            const uint32_t ppar = (uint32_t)(it - 1) & 1, dpar = (uint32_t)((it - 1) >> 1) & 1;  // of the step before
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&afull[s], (uint32_t)((it / SA) & 1)))) {
                ok = false;
                break;
            }
            const double *src = reinterpret_cast<const double *>(smem + s * Cfg::A_BYTES) + r;
            uint32_t hi[KB], lo[KB];
            int mx = 0;
#pragma unroll
            for (int q = 0; q < KB; ++q) {
                const double x = U ? src[((q & 1) * 8 + q / 2) * Cfg::A_STRIDE + ((abase + (q & 1) * ldv) & 1)] : src[q * BM];
                hi[q] = (uint32_t)__double2hiint(x);
                lo[q] = (uint32_t)__double2loint(x);
                if (U) hi[q] &= vmask;
            }
            release_reads_to_async_copy();
            __syncwarp();
            if (lane == 0) mbar_arrive(&aempty[s]);
#pragma unroll
            for (int q = 0; q < KB; q += 2) {
                mx = __vimax3_s32(mx, (int)tc64_abs(hi[q]), (int)tc64_abs(hi[q + 1]));
                if constexpr (W > 16) {
                    seen_lo |= lo[q] | lo[q + 1];
                    seen_hi |= hi[q] | hi[q + 1];
                }
            }
            mx >>= 20;
            // the row's scale after the step before, and after this one
            int E = kTc64Emin;
            if (it > 0) {
                if (!__all_sync(0xffffffffu, mbar_wait_bounded(sbar, ppar))) {
                    ok = false;
                    break;
                }
                E = rowE[((it - 1) & (Cfg::ERING - 1)) * BM + r];
            }
            const bool grown = __any_sync(0xffffffffu, mx > E);  // a larger entry: a new group starts
            E = max(E, mx);
            rowE[(it & (Cfg::ERING - 1)) * BM + r] = E;
            if (lane == 0)
                reinterpret_cast<volatile unsigned char *>(gnew)[(it & 3) * 4 + (warp & 3)] = grown ? 1 : 0;
            __syncwarp();
            if (lane == 0) mbar_arrive(sbar);
            if constexpr (W == 16) {
                if (E == kTc64Emin) {
#pragma unroll
                    for (int q = 0; q < KB; ++q) seen_lo |= hi[q] << 1 | lo[q];
                }
            }
            uint32_t sgn[KB / 2];
#pragma unroll
            for (int q = 0; q < KB; q += 2) sgn[q / 2] = tc64_sign2(hi[q], hi[q + 1]);
#pragma unroll
            for (int q = 0; q < KB; ++q) {
                const uint64_t y = tc64_fixed(hi[q], lo[q], tc64_shift(tc64_abs(hi[q]), E));
                hi[q] = (uint32_t)(y >> 32);
                lo[q] = (uint32_t)y;
            }
            // their place is free: DB, the MMAs of two steps ago are done; else those of the last step, part by part
            const uint32_t set = tlane + (it & 1) * Cfg::COL_SET;
            if (Cfg::DB ? (it >= 2 && !__all_sync(0xffffffffu, mbar_wait_bounded(&ydone[it & 1], (uint32_t)((it - 2) >> 1) & 1)))
                        : (it >= 1 && !__all_sync(0xffffffffu, mbar_wait_bounded(&xdone[ppar], dpar)))) {
                ok = false;
                break;
            }
            tcf_after();
            // digits 3-6: the low words
#pragma unroll
            for (int b = 0; b < 2; ++b) {  // bytes 2b, 2b + 1: digits 6 - 2b, 5 - 2b
                uint32_t d0[8], d1[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const uint32_t c = hfma2(sgn[q], kH1152, 0u);
                    tc64_digits2(lo[2 * q], lo[2 * q + 1], b ? 0x7362 : 0x5140, sgn[q], c, c, d0[q], d1[q]);
                }
                tc_st8(set + Cfg::COL_X + (3 - 2 * b) * 8, d0);
                tc_st8(set + Cfg::COL_X + (2 - 2 * b) * 8, d1);
            }
            if constexpr (!Cfg::DB) {
                tc_wait_st();
                tcf_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(convx);
                if (it >= 1 && !__all_sync(0xffffffffu, mbar_wait_bounded(&ydone[ppar], dpar))) {
                    ok = false;
                    break;
                }
                tcf_after();
            }
            // digits 0-2: the high words
            {
                uint32_t d1[8], d2[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const uint32_t c = hfma2(sgn[q], kH1152, 0u);
                    tc64_digits2(hi[2 * q], hi[2 * q + 1], 0x5140, sgn[q], c, c, d2[q], d1[q]);
                }
                tc_st8(set + Cfg::COL_Y + 8, d1);
                tc_st8(set + Cfg::COL_Y + 16, d2);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    d1[q] = hfma2(prmt(prmt(hi[2 * q], hi[2 * q + 1], 0x7362), 0x64646464u, 0x4140), sgn[q],
                                  hfma2(sgn[q], kH1024, 0u));
                tc_st8(set + Cfg::COL_Y, d1);
            }
            tc_wait_st();
            tcf_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(Cfg::DB ? &convx[it & 1] : convy);
        }
        if (!ok && lane == 0) {
            atomicOr(a.status, kDevErrTimeout);
            atomicOr(abort_flag, 1u);
        }
        if (zrow[r] != 0 && (seen_hi << 1 | seen_lo) != 0u) *unsafe = 1u;
        named_barrier(1, 512);  // the promoters read the last scales after it
        if (*abort_flag != 0u || a.splits == 1) return;
        finish();
        return;
    }

    // -------------------------------------------------------- promoters
    reg_inc<Cfg::PREG>();
    constexpr int HW = W / 2;
    const int half = (warp - 8) / 4;
    const int c0 = half * HW;
    const int n = (int)a.n;
    bool ok = true;

    // guard: a lower bound of sum|a||b| over the row, column by column, in units of 2^-14 2^E0 2^F
    // The item's share of the bound, 4 k 2^-53 of its own sum|a||b|, against its error, k_item 2^-54.9 (2^-52.7) 2^E 2^F:
    const int need = (int)((k1 - k0) * tc64_guard(W) / a.k) + 1;
    int E0 = 0, bound = 0x7fffffff;
    const unsigned bad_b = tb->bad;  // a column of B that the digits cannot hold
    uint32_t fzero = 0u;             // columns that do not count: zero, or beyond n
#pragma unroll
    for (int j = 0; j < HW; ++j) fzero |= (c0 + j >= n || tb->F[c0 + j] == kTc64Emin ? 1u : 0u) << j;
    {
        uint32_t sum[HW];
#pragma unroll
        for (int j = 0; j < HW; ++j) sum[j] = 0u;
        const uint32_t *ap = static_cast<const uint32_t *>(a.A) + 2 * (row < a.m ? row : 0) + 1;
        uint32_t h[16];  // high words of 16 entries of the row, a block ahead
        auto load = [&](int64_t p) {
#pragma unroll
            for (int q = 0; q < 16; ++q) h[q] = p + q < a.k ? __ldg(ap + 2 * (p + q) * a.lda) & 0x7fffffffu : 0u;
        };
        load(k0);
        ok = __all_sync(0xffffffffu, mbar_wait_bounded(gbar, 0));
#pragma unroll 1
        for (int q16 = 0; q16 < kTc64Windows * 4 && k0 + 16 * q16 < k1; ++q16) {
            if (E0 == 0) {  // the first block with a nonzero entry
#pragma unroll
                for (int q = 0; q < 16; ++q) E0 = max(E0, (int)(h[q] >> 20));
            }
            uint32_t da[4];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const int e = (int)(h[q] >> 20), sft = max(0, E0 - e);
                const uint32_t dig = (e > 0 && sft < 7) ? (((h[q] & 0xfffffu) | 0x100000u) >> 14) >> sft : 0u;
                da[q / 4] = q % 4 == 0 ? dig : da[q / 4] | dig << (8 * (q % 4));
            }
            load(k0 + 16 * (q16 + 1));
            const unsigned char *bw = smem + Cfg::OFF_F + (q16 / 4) * (W * 64) + c0 * 64 + (q16 % 4) * 16;
#pragma unroll
            for (int j = 0; j < HW; ++j) {
                const uint4 b = *reinterpret_cast<const uint4 *>(bw + j * 64);
                sum[j] = __dp4a(da[0], b.x, sum[j]);
                sum[j] = __dp4a(da[1], b.y, sum[j]);
                sum[j] = __dp4a(da[2], b.z, sum[j]);
                sum[j] = __dp4a(da[3], b.w, sum[j]);
            }
            bound = 0x7fffffff;
#pragma unroll
            for (int j = 0; j < HW; ++j)
                if (!(fzero >> j & 1u)) bound = min(bound, (int)sum[j]);
            if (row >= a.m) bound = 0x7fffffff;
            if (__all_sync(0xffffffffu, bound >= 4 * need)) break;
            // no more than half of what is needed in sight: given up (a block of columns takes about a microsecond)
            if (q16 >= 3 && __any_sync(0xffffffffu, (int64_t)bound * min(kTc64Windows * 4, (int)((k1 - k0) / 16)) <
                                                        (int64_t)(need / 2) * (q16 + 1)))
                break;
        }
        release_reads_to_async_copy();  // the fallback's copies may follow
        if (bound < need) {
            // Too small: fmas, unless the row is zero throughout, which the converters know at the end (a scan of the row
            // here held the block up for 0.4 us a column: m = k = 16384, n = 4 with one zero row in every slab 6.58 ms, 0.55
            // so, 0.53 without; every other row zero 0.58).
            if (E0 == 0) zrow[r] = 1;
            else *unsafe = 1u;
            bound = 0x7fffffff, E0 = kTc64Emax;
        }
        if ((E0 < kTc64Emin && row < a.m && bound != 0x7fffffff) || bad_b != 0u) *unsafe = 1u;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(verdict);
    const bool started = __all_sync(0xffffffffu, ok && go());

    // sums of 96 bits per output
    int64_t vh[HW];
    uint32_t vl[HW];
#pragma unroll
    for (int j = 0; j < HW; ++j) vh[j] = 0, vl[j] = 0u;
    int E = kTc64Emin;
    for (int g = 0; started; ++g) {
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&gdone[g & 1], (uint32_t)(g >> 1) & 1))) {
            ok = false;
            break;
        }
        tcf_after();
        const unsigned slot = *reinterpret_cast<volatile unsigned *>(&gslot[g & 1]);
        const int Eg = rowE[(slot & 63u) * BM + r];
        const int sft = Eg - E;
        E = Eg;
        if (__any_sync(0xffffffffu, sft > 0) && g > 0) {
#pragma unroll
            for (int j = 0; j < HW; ++j) {
                int64_t h = vh[j];
                uint32_t l = vl[j];
                int t = sft > 95 ? 95 : sft;
                for (; t >= 32; t -= 32) {
                    l = (uint32_t)h;
                    h >>= 32;
                }
                if (t > 0) {
                    // to nearest, ties to even: rows grow at different steps, so an item's sums may be shifted many times
                    const uint32_t b = ((1u << (t - 1)) - 1u) + (l >> t & 1u);
                    l += b;
                    h += l < b ? 1 : 0;
                    l = (l >> t) | ((uint32_t)h << (32 - t));
                    h >>= t;
                }
                vh[j] = h;
                vl[j] = l;
            }
        }
        // V += 2^SH (2^40 D0 + 2^32 D1 + 2^24 D2 + 2^16 D3 + 2^8 D4 + D5 + 2^-8 D6 + 2^-16 D7).
        // (W = 64: without D7, which sits in D6), its lowest part rounded to nearest.  A conversion to integers takes the
        // XU pipe 8 cycles, so D0 and D1, which stay within 2^22, take a magic addition.
        constexpr int CB = Cfg::CB, SH = Cfg::SH;
        constexpr uint32_t kM23 = 0x4b400000u;  // 1.5 * 2^23
        const uint32_t acc0 = tlane + (Cfg::DDB ? (uint32_t)(g & 1) * (Cfg::ND * W) : 0u) + c0;
#pragma unroll
        for (int c = 0; c < HW; c += CB) {
            uint32_t d[Cfg::ND][CB];
            tc_ldn<Cfg::ND, CB>(acc0 + c, W, d);
            if (c + CB == HW) {
                tcf_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&drained[g & 1]);
            }
#pragma unroll
            for (int j = 0; j < CB; ++j) {
                float t = __uint_as_float(d[6][j]);
                if constexpr (Cfg::ND == 8) t = fmaf(__uint_as_float(d[7][j]), 0.00390625f, t);
                t = fmaf(t, 0.00390625f, __uint_as_float(d[5][j]));
                int64_t L = (int64_t)(uint64_t)vl[c + j];
                L += __float2int_rn(t * (float)(1 << SH));
                L += (int64_t)__float2int_rn(__uint_as_float(d[4][j])) * (1 << (8 + SH));
                L += (int64_t)__float2int_rn(__uint_as_float(d[3][j])) * (1 << (16 + SH));
                L += (int64_t)__float2int_rn(__uint_as_float(d[2][j])) * (1 << (24 + SH));
                vl[c + j] = (uint32_t)L;
                const uint32_t h = __float_as_uint(__uint_as_float(d[0][j]) + __uint_as_float(kM23)) * 256u +
                                   __float_as_uint(__uint_as_float(d[1][j]) + __uint_as_float(kM23)) - kM23 * 257u;
                if constexpr (W == 64) {  // in place: 64-bit temporaries spill here (and in-place costs 1 % below)
                    vh[c + j] += L >> 32;
                    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(vh[c + j]) : "r"((int)h), "n"(1 << SH));
                } else {
                    vh[c + j] += (int64_t)(int)h * (1 << SH) + (L >> 32);
                }
            }
        }
        if (slot & 64u) break;
    }
    if (!ok && lane == 0) {
        atomicOr(a.status, kDevErrTimeout);
        atomicOr(abort_flag, 1u);
    }
    if (started && row < a.m) {
        // infinities and NaNs, rows wholly below the scales, rows taken as zero that are not, and a row that grew after its
        // guard columns
        const int sft = E - E0;
        if (E > kTc64Emax || (E == kTc64Emin && bound != 0x7fffffff) || (E != kTc64Emin && zrow[r] != 0) ||
            (bound != 0x7fffffff && (sft > 30 || (bound >> max(sft, 0)) < need)))
            *unsafe = 1u;
    }
    tcf_before();
    named_barrier(2, 288);
    named_barrier(1, 512);
    const bool stop = *abort_flag != 0u, redo = *unsafe != 0u;
    if (stop) return;  // tile not written; the host sees TSMM_ERR_TIMEOUT
    double acc[HW];
    if (redo) {
        // its totals lie over the ring of A, where the copies issued ahead of the verdict may still be on their way
        for (int q = 0; !started && q < SA && q < iters; ++q)
            if (!mbar_wait_bounded(&afull[q], 0)) {
                atomicOr(a.status, kDevErrTimeout);
                atomicOr(abort_flag, 1u);
            }
        fma_item<double, HW>(a, row, k0, k1, c0, acc, reinterpret_cast<double *>(smem + Cfg::OFF_F),
                             reinterpret_cast<double *>(smem), fbar, abort_flag, threadIdx.x - 256);
        if (*abort_flag != 0u) {
            if (a.splits > 1) finish();  // the converters wait there
            return;
        }
    } else {
        // |x| = X 2^(E-1077) with digits of weight 2^(48-8i); an order-5 product has weight 2^56 and the sums' unit 2^-SH of it.
        // They stay below 2^55 * 2^32.  The upper 64 bits of the
        // magnitude are rounded to a double, whose exponent and sign are then set by integer operations (FP64
        // arithmetic on 128 x W values would take longer than a group of MMAs)
#pragma unroll
        for (int j = 0; j < HW; ++j) {
            const int F = c0 + j < n ? tb->F[c0 + j] : kTc64Emin;
            uint64_t h = (uint64_t)vh[j];
            uint32_t l = vl[j];
            const uint32_t sg = (uint32_t)(h >> 32) & 0x80000000u;
            if (sg) {
                l = 0u - l;
                h = ~h + (l == 0u ? 1ull : 0ull);
            }
            const int sh = max(0, 32 - __clzll((long long)h));
            const uint64_t u = h << (32 - sh) | l >> sh;
            const double d = __ull2double_rn(u);
            const uint32_t hw = (uint32_t)__double2hiint(d) + (uint32_t)((sh + E + F - 2154 + 56 - Cfg::SH) * 1048576);
            acc[j] = u == 0ull ? 0.0 : __hiloint2double((int)(hw | sg), __double2loint(d));
        }
    }

    const double alpha = a.alpha, beta = a.beta;
    // C = alpha*v + beta*C0 for G columns from cc of this thread's row, the C0 loads issued ahead of the stores
    auto store = [&](int cc, const double *v, auto g_tag) {
        constexpr int G = decltype(g_tag)::value;
        if (row >= a.m) return;
        double *c = static_cast<double *>(a.C) + row + (int64_t)cc * a.ldc;
        double old[G];
#pragma unroll
        for (int j = 0; j < G; ++j) old[j] = (beta != 0.0 && cc + j < n) ? c[(int64_t)j * a.ldc] : 0.0;
#pragma unroll
        for (int j = 0; j < G; ++j)
            if (cc + j < n) {
                double o = alpha * v[j];
                if (beta != 0.0) o = fma(beta, old[j], o);
                c[(int64_t)j * a.ldc] = o;
            }
    };
    if (a.splits == 1) {
#pragma unroll
        for (int c = 0; c < HW; c += 8) store(c0 + c, acc + c, std::integral_constant<int, 8>{});
        return;
    }
    const int64_t mpad = a.slabs * BM;
    double *ws = static_cast<double *>(a.ws) + i0 + r;
#pragma unroll
    for (int j = 0; j < HW; ++j)
        if (c0 + j < n) ws[((int64_t)split * a.np + c0 + j) * mpad] = acc[j];
    __threadfence();
    finish();
}

template <int W, bool U>
__global__ void __launch_bounds__(TallTc64Cfg<W, U>::THREADS, 1)
    tall_tc64_kernel(const __grid_constant__ CUtensorMap tmA, const TallArgs a) {
    tall_tc64_block<W, U>(&tmA, a, blockIdx.x, (int)blockIdx.y);
}

}  // namespace tsmm
