// Internal (host-side) declarations shared by the library's translation units.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>
#include <mutex>
#include <set>
#include <utility>

#include "../../include/tsmm.h"

namespace tsmm {

// ---- tiling constants shared by planner, packer and kernels -------------------
// Regime (i): A columns per pipeline stage; packed B rows are padded to it.
constexpr int kTallBKS = 32;
// Regime (i): consumer warps per thread block (the producer warp is extra).
constexpr int kTallConsumerWarps = 4;
// Regime (ii): packed B tile width (columns) and k granule.
constexpr int kRankNT = 64;
constexpr int kRankKGran = 8;
constexpr int kRankMaxK = 128;
constexpr int kTallMaxN = 64;

inline size_t dtype_size(tsmm_dtype d) { return d == TSMM_F64 ? 8 : 4; }

// Smallest power of two >= n.
inline int pow2_ceil(int64_t n) {
    int np = 1;
    while (np < n) np <<= 1;
    return np;
}

// Padded column count of the regime-(i) kernel that serves n columns: one of
// 1, 2, 4, 8, 16, 24, 32, 48, 64 (the FMA-bound widths 24 and 48 save a
// quarter of the padded work for n in 17..24 and 33..48).
inline int tall_np(int64_t n) {
    if (n > 16 && n <= 24) return 24;
    if (n > 32 && n <= 48) return 48;
    return pow2_ceil(n);
}

// Rows per thread block (m-slab) of the regime-(i) kernel.  FP32 widths up to
// 32 take 256 rows: the consumer warps then split the slab by rows more and the
// stage's k columns less (widths 24 and 32: each warp reads whole 32-column
// stages instead of two warps splitting every stage, one stage wait per 16
// k-steps -- n = 24: 0.83 -> 0.79 ms, n = 32: 1.01 -> 0.98 ms at m = k = 32768;
// widths up to 16: 4 -> 2 warps per stage, 0.5-1.5 % faster; width 48 with
// its 8 x 12 tiles likewise).  The FP32 width 64 takes 128 (its warps already
// own whole stages), FP64 64.
constexpr int tall_block_rows(bool f64, int np) { return f64 ? 64 : (np == 64 ? 128 : 256); }
inline int tall_bm(tsmm_dtype d, int np) { return tall_block_rows(d == TSMM_F64, np); }

// Thread blocks of the regime-(i) TMA kernel resident per SM (its shared-memory
// ring is sized for this): 3 for the FMA-bound FP32 widths 32 and 64 (8 x 8
// tiles fit 136 registers), else 2 (the width 48's 8 x 12 tiles need ~160).
constexpr int tall_resident_blocks(bool f64, int np) { return (!f64 && (np == 32 || np == 64)) ? 3 : 2; }

// Whether the FP32 kernels up to 16 columns cut their chains of fmas (TallTotal): at width 16, whose registers then spill, where A
// has less than the 64 MB from which the split-K planner fills whole waves as it always did (m = 33868, n = 12, k = 1162: 36.9
// us without, 38.9 with); below it the planner's splits are fewer than they were, their chains longer.
__host__ __device__ constexpr bool tall_cut(int np, int64_t m, int64_t k) { return np < 16 || (double)m * (double)k * 4.0 < 64.0e6; }

// FP32 regime (i) with n > 16 runs on the tensor cores (tsmm_tall_tc.cuh): slabs of kTcRows rows, k in chunks of
// kTcKB, MMA width n rounded up to 16.  The line lies at 16 because up to there the fma kernel streams A at the copy
// rate (n = 16: 0.64 ms at m = k = 32768), above it does not (n = 20: 0.78 ms against 0.68); m and k need no line
// (m = 2048, n = 32, k = 2048: 85 us against 25; m = 100000, n = 64, k = 64: 25 us both).
constexpr int kTcRows = 128;
constexpr int kTcKB = kTallBKS;
// ... below which its blocks compute their items with fmas: an accumulator is cut, not rounded, which over a few terms costs
// more than a chain of fmas rounds (relative error, n = 64, positive entries: k = 1: 4.5e-8 against 2.5e-8, up to 0.84 of
// the library's bound; k = 8: 5.7e-8 against 4.7e-8; k = 12: 4.1e-8 against 5.2e-8; k = 16: 5.9e-8 against 6.3e-8).
constexpr int kTcMinK = 16;
inline int64_t tc_width(int64_t n) { return (n + 15) / 16 * 16; }
inline bool tc_pack(tsmm_dtype d, int regime, int precision, int64_t n, int64_t k) {
    return d == TSMM_F32 && regime == 1 && precision == 0 && n > 16 && k > 0;
}

// FP64 regime (i) on the tensor cores (tsmm_tall_tc64.cuh): steps of kTc64KB columns of k, MMA width per digit.  n = 1 stays
// with the fma kernel (1.75 ms at m = k = 32768; any n <= 16 takes 1.98 here); k from 256 on, where the truncation of the
// digits is below the fma chain's rounding (k = 256: 6.6e-17 against 3.9e-16) and the start of a block pays (m = 20000,
// n = 30, k = 256: 406 us against 54).
constexpr int kTc64KB = 16;
constexpr int kTc64Emin = 1023 - 400, kTc64Emax = 1023 + 400;  // range of the scales (exponent fields)
constexpr int kTc64Windows = 8;
__host__ __device__ constexpr int tc64_guard(int w) { return w <= 48 ? 1200 : 5120; }
inline int64_t tc64_width(int64_t n) { return (n + 15) / 16 * 16; }
// Accumulators per width: one for each of eight orders of products where tensor memory holds eight, else seven.  Rows (of
// `width` columns) of a packed step of B: its eight digits; or digits 0..5, then digits 0..6 each with the top of the next.
__host__ __device__ constexpr int tc64_accumulators(int w) { return w <= 48 ? 8 : 7; }
__host__ __device__ constexpr int tc64_rows(int w) { return w <= 48 ? 8 : 13; }
// k up to 2^20 keeps the sums' high words below 2^51.
inline bool tc64_pack(tsmm_dtype d, int regime, int64_t n, int64_t k) {
    return d == TSMM_F64 && regime == 1 && n > 1 && k >= 256 && k <= (1 << 20);
}
// ... and for at least 64 us of the FP64 pipe: below that a block's start and end weigh as much, and an item that its
// guard leaves to the fmas has too few blocks beside it (m = 1533, n = 7, k = 605, uneven rows: 28 us, 62 with digits).
inline bool tc64_plan(tsmm_dtype d, int regime, int64_t m, int64_t n, int64_t k) {
    return tc64_pack(d, regime, n, k) && (double)m * (double)tall_np(n) * (double)k >= 4.0e7;
}
// Head of the packed digits of B, in device memory, kTc64Head bytes.  Behind it, for k rounded up to 64: per step of
// kTc64KB rows tc64_rows x width columns, FP16, K-major; then per 64 rows width columns x 64 bytes, the top 7 bits of
// |b| at the column's scale.
struct TcB64 {
    unsigned bad;               // a nonzero column beyond the scales' range, an infinity or a NaN
    int F[kTallMaxN];           // scale of each column (kTc64Emin: zero column)
};
constexpr int kTc64Head = 512;
static_assert(sizeof(TcB64) <= kTc64Head, "head");

// Load form of the regime (i) kernel for an A that a tensor map cannot describe
// (its bulk/element-copy kernel): for FP32 widths of 16 and more with A's base
// 16-byte aligned, lda mod 4 -- every column's offset within 16 bytes is then
// fixed by its index mod 4, and the kernel is compiled for it -- else -1
// (offsets computed at run time).
inline int async_load_variant(bool f32, int np, const void *A, int64_t lda) {
    if (!f32 || np < 16 || reinterpret_cast<uintptr_t>(A) % 16 != 0) return -1;
    return (int)((uint64_t)lda & 3u);
}

// Regime of a (k, n) pair: 1 = tall (n <= 64), 2 = rank-k (k <= 128), 0 = unsupported.
inline int regime_of(int64_t k, int64_t n) {
    if (n <= kTallMaxN) return 1;
    if (k <= kRankMaxK) return 2;
    return 0;
}

inline int64_t round_up(int64_t x, int64_t g) { return (x + g - 1) / g * g; }

// Raises a kernel's dynamic shared-memory limit to `bytes` once per (kernel,
// device); thread-safe (the server thread and callers' threads launch alike).
inline cudaError_t ensure_smem_limit(const void *kernel, int bytes) {
    static std::mutex mu;
    static std::set<std::pair<const void *, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({kernel, dev})) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.insert({kernel, dev});
    return e;
}

}  // namespace tsmm

struct tsmm_packed_b_s {
    tsmm_dtype dtype;
    int precision;   // tsmm_precision
    int64_t k, n;
    int64_t kp;      // padded rows
    int64_t w;       // tile width (columns)
    int64_t ntiles;  // number of column tiles
    int regime;
    int device;
    void *data;      // device storage, kp * w * ntiles elements
    size_t bytes;
    // tensor-core form behind it in the same allocation (nullptr: none): per 32-row chunk of k three BF16 pieces of
    // tc_width(n) columns, then one float per chunk, the smallest nonzero |B| in it, and one more, the largest
    void *tc_data;
    float *tc_min;
};

struct tsmm_plan_s {
    int64_t m, n, k;
    tsmm_dtype dtype;
    int precision;   // tsmm_precision
    int regime;
    int device;
    int num_sms;
    // regime (i)
    int np;          // padded n
    int bm;          // rows per thread block
    int64_t slabs;   // ceil(m / bm)
    int splits;      // k splits (S)
    int64_t kchunk;  // packed-B rows per split (multiple of kTallBKS)
    int64_t kp;      // padded k
    bool tc;         // runs the tensor-core kernel
    // regime (ii)
    int64_t mtiles, ntiles;
    // device scratch owned by the plan
    void *workspace;           // splits * np * slabs * bm elements (regime (i), splits > 1)
    size_t workspace_bytes;
    unsigned *tickets;         // one arrival counter per slab
    unsigned *status;          // device error word
    // one-entry caches of the TMA descriptors for A and (regime (ii)) C
    const void *tmap_ptr;
    int64_t tmap_lda;
    bool tmap_tc;              // the tensor-core kernel's map (the fma kernel's has other boxes)
    CUtensorMap tmap;
    int64_t arows;             // tmap is encode_a_rows' with so many rows (tensor-core kernels, unaligned A)
    const void *tmapc_ptr;
    int64_t tmapc_ldc;
    int tmapc_cols;
    CUtensorMap tmapc;
};

namespace tsmm {

struct TallArgs {
    int64_t m, n, k, lda, ldc;
    const void *A;
    const void *Bp;     // packed B, kp x np row-major
    void *C;
    double alpha, beta;
    void *ws;
    unsigned *tickets;
    unsigned *status;
    int splits;
    int64_t kchunk, kp, slabs;
    int np;             // row length of Bp, and of the workspace's partial tiles
    const void *Bt;     // tensor-core form of B and its chunks' smallest nonzero magnitudes
    const float *bmin;
    // tensor-core kernels, A not aligned for a tensor map of its columns: rows of the map of encode_a_rows, 0 without one
    int64_t arows;
};

// Launchers (return cudaSuccess or the launch error).  `tma` selects the
// TMA-pipelined kernel (tmap must describe A) or the plain-load kernel.
cudaError_t launch_tall_f32(bool tma, int np, const CUtensorMap *tmap, const TallArgs &a,
                            cudaStream_t s);
cudaError_t launch_tall_f64(bool tma, int np, const CUtensorMap *tmap, const TallArgs &a,
                            cudaStream_t s);

// An A whose column stride is not a multiple of 16 bytes: R = 16 / element size columns together have such a stride, so a
// map over A's aligned base whose row c spans columns R c .. R c + R - 1 describes it; column R c + q starts in row c at
// element q * lda + (the base's offset), and a box that begins at the 16-byte boundary below covers eight such columns.
// Rows of the map: k / R (the columns left are moved one by one); 0 where its coordinates would not fit.
constexpr int kARowsBox = 8;
int64_t encode_a_rows(CUtensorMap *map, tsmm_dtype dtype, const void *A, int64_t m, int64_t k, int64_t lda);

// The tensor-core kernels; unaligned: tmap is encode_a_rows' (unused if a.arows == 0).
cudaError_t launch_tall_tc64(const CUtensorMap &tmap, bool unaligned, const TallArgs &a, cudaStream_t s);
cudaError_t launch_tall_tc(const CUtensorMap &tmap, bool unaligned, const TallArgs &a, cudaStream_t s);

struct RankArgs {
    int64_t m, n, k, lda, ldc, kp;
    const void *A;
    const void *Bp;  // packed B, ntiles x (kp x kRankNT)
    void *C;
    double alpha, beta;
    int num_sms;     // persistent grid size = resident blocks x SMs
    const void *Bt;         // tensor-core form of B, and the smallest and largest magnitudes in its chunks
    const uint2 *brange;
};
// tmA: tensor map of A (box bm x 32) or nullptr for the plain-load kernel;
// The FP32 regime (ii) kernel for k in kRankWideMinK..32 streams k in chunks of kRankWideKC, so its A
// tensor map's box is bm x kRankWideKC; every other kernel's is bm x kTallBKS.  From kRankTcMinK on the
// tensor cores serve it (tsmm_rankk_tc.cu; tmC with a box of bm x kRankTcSub): at m = n = 16384, beta = 1,
// the wide kernel in chunks of 32 took 0.414 / 0.566 / 1.063 ms at k = 40 / 64 / 128, they take 0.365 / 0.355 /
// 0.369; at k = 32 the wide kernel's 0.35 is already the output stream's.
constexpr int kRankWideMinK = 17;
constexpr int kRankWideKC = 16;
constexpr int kRankTcMinK = 33;
constexpr int kRankTcSub = 32;
inline bool rank_tc(tsmm_dtype d, int regime, int precision, int64_t k) {
    return d == TSMM_F32 && regime == 2 && precision == 0 && k >= kRankTcMinK;
}
inline bool rank_wide(tsmm_dtype d, int regime, int precision, int64_t k) {
    return d == TSMM_F32 && regime == 2 && precision != TSMM_PREC_BF16X3 && k >= kRankWideMinK && k < kRankTcMinK;
}
inline int a_box_k(tsmm_dtype d, int regime, int precision, int64_t k, bool tc) {
    if (tc && d == TSMM_F64) return kTc64KB;
    return rank_wide(d, regime, precision, k) ? kRankWideKC : kTallBKS;
}
size_t rank_tc_bytes(int64_t k, int64_t ntiles);
cudaError_t launch_pack_b_rank_tc(int64_t k, int64_t n, const float *B, int64_t ldb, int64_t ntiles, void *dst, cudaStream_t s);
cudaError_t launch_rankk_tc(const CUtensorMap *tmA, const CUtensorMap *tmC, const RankArgs &a, unsigned *status,
                            cudaStream_t s);
// FP64 from k = kRank64TcMinK on (tsmm_rankk_tc64.cu; A read by element, tmC with a box of kTcRows x kRank64Sub): at
// k = 4, m = n = 16384, beta = 1 the fma kernel took 1.97 ms (FP64 pipe), this one 0.93 at any k <= 32; below 4 the error
// bound leaves no room for the digits.
constexpr int kRank64TcMinK = 4;
constexpr int kRank64Sub = 16;
inline bool rank_tc64(tsmm_dtype d, int regime, int precision, int64_t k) {
    return d == TSMM_F64 && regime == 2 && precision == 0 && k >= kRank64TcMinK;
}
size_t rank_tc64_bytes(int64_t k, int64_t ntiles);
cudaError_t launch_pack_b_rank_tc64(int64_t k, int64_t n, const double *B, int64_t ldb, int64_t ntiles, void *dst,
                                    cudaStream_t s);
cudaError_t launch_rankk_tc64(const CUtensorMap *tmC, const RankArgs &a, unsigned *status, cudaStream_t s);
// tmC: tensor map of C (box bm x kRankNT) when C meets the TMA rules, else nullptr.
cudaError_t launch_rankk(tsmm_dtype dt, const CUtensorMap *tmA, const CUtensorMap *tmC,
                         const RankArgs &a, unsigned *status, cudaStream_t s);

// Plan construction with an optional forced split count (0 = planner's choice).
tsmm_status create_plan(int64_t m, int64_t n, int64_t k, tsmm_dtype dtype, int forced_splits,
                        tsmm_plan_t *out, int precision = 0);

// Plan fields without any device allocation: every member except workspace,
// tickets and status, plus the ticket bytes the plan needs; split-K workspaces
// are capped at max_workspace bytes.  (Used by create_plan and the server.)
tsmm_status plan_layout(int64_t m, int64_t n, int64_t k, tsmm_dtype dtype, int forced_splits,
                        int precision, int dev, int sms, int64_t max_workspace, tsmm_plan_s *p,
                        size_t *ticket_bytes_out);

// BF16x3 precision mode (tsmm_bf16x3.cu): k granule of its packed B and plan.
constexpr int kX3KB = 64;
inline int x3_np(int64_t n) {
    const int np = pow2_ceil(n);  // an MMA N of 16, 32 or 64
    return np < 16 ? 16 : np;
}
cudaError_t launch_tall_bf16x3(int np, const CUtensorMap *tmap, const TallArgs &a, int num_sms,
                               cudaStream_t s);
cudaError_t launch_pack_b_bf16x3(int64_t k, int64_t n, const void *B, int64_t ldb, void *dst, int np,
                                 int64_t nchunks, int64_t ntiles, cudaStream_t s);
// Regime (ii) in the BF16x3 mode: tile width of its packed B, and the kernel.
// tmC: tensor map of C (box 128 x kX3RankSub) when C meets the TMA rules
// (C0 loads and C stores by TMA), else nullptr (C0 by 4-byte cp.async, C by
// plain stores).
constexpr int kX3RankNT = 128;
constexpr int kX3RankSub = 32;
cudaError_t launch_rankk_bf16x3(const CUtensorMap *tmA, const CUtensorMap *tmC, const RankArgs &a,
                                unsigned *status, cudaStream_t s);

// Process-wide plan cache (tsmm_tune.cu): tuned split counts keyed by
// (dtype, m, n, k, SM count).  Lookup returns 0 when absent.
int plan_cache_lookup(tsmm_dtype dtype, int64_t m, int64_t n, int64_t k, int sms);
void plan_cache_store(tsmm_dtype dtype, int64_t m, int64_t n, int64_t k, int sms, int splits);

// tsmm_execute_grouped (tsmm_group_api.cu), for the server.
tsmm_status execute_grouped(const tsmm_group_item *items, int count, tsmm_stream_t stream);

// Costs of a regime (i) kernel for the choice of its split-K factor, in us: a block's stage of k alone on its SM, its
// bytes, a block's start and end, and the last block's sum over S partial tiles, f0 + c * S.
struct SplitCosts {
    int resident;     // blocks per SM
    double stage, stage2, bytes, block, f0, c;  // stage2: a stage where the SM has another block
    double waves_from;  // bytes of A from which whole waves of stages count at one price (0: never)
    double share;       // of a slab's sum over the partials, what it takes from the other blocks of a full wave
};
SplitCosts split_costs(tsmm_dtype dt, int np, bool tc, int64_t n);
int choose_splits(const SplitCosts &k, int64_t slabs, int64_t kstages, int num_sms, int64_t max_splits);

cudaError_t launch_pack_b(tsmm_dtype dt, int64_t k, int64_t n, const void *B, int64_t ldb,
                          void *dst, int64_t kp, int64_t w, int64_t ntiles, cudaStream_t s);
// One launch writes the regime (i) panel and its tensor-core form.
cudaError_t launch_pack_b_tc(int64_t k, int64_t n, const float *B, int64_t ldb, float *panel, int64_t kp, int np,
                             void *tc_data, float *tc_min, cudaStream_t s);
// The digits of B behind the panel (tsmm_tall_tc64.cu): bytes of the whole block, and the launches that fill it.
size_t tc64_bytes(int64_t k, int64_t n);
cudaError_t launch_pack_b_tc64(int64_t k, int64_t n, const double *B, int64_t ldb, void *dst, cudaStream_t s);
cudaError_t launch_scale(tsmm_dtype dt, int64_t m, int64_t n, double beta, void *C, int64_t ldc,
                         cudaStream_t s);
cudaError_t launch_copy_columns(tsmm_dtype dt, const void *src, int64_t lds, int64_t m, int64_t k, void *dst,
                                int64_t ldd, cudaStream_t s);

}  // namespace tsmm
