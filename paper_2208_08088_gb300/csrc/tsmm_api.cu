// The C ABI (include/tsmm.h): argument checking, the planner, packed-B and
// plan lifetimes, and kernel dispatch.  No entry point throws or aborts.
#include <cudaTypedefs.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>
#include <new>

#include "tsmm_device.cuh"
#include "tsmm_internal.h"

using namespace tsmm;

namespace {

constexpr int kVersion = 100;  // 0.1.0

// Resolved once: the driver's tensor-map encoder (no -lcuda link needed).
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
    std::call_once(g_encode_once, [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                             cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    });
    return g_encode;
}

bool valid_dtype(tsmm_dtype d) { return d == TSMM_F32 || d == TSMM_F64; }

bool valid_precision(tsmm_precision p, tsmm_dtype d) {
    return p == TSMM_PREC_NATIVE || p == TSMM_PREC_FMA || (p == TSMM_PREC_BF16X3 && d == TSMM_F32);
}

bool aligned(const void *p, size_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; }

thread_local const char *g_last_cuda_error = "no error";

tsmm_status cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return TSMM_OK;
    g_last_cuda_error = cudaGetErrorString(e);  // static string owned by the runtime
    if (e == cudaErrorMemoryAllocation) return TSMM_ERR_OUT_OF_MEMORY;
    return TSMM_ERR_CUDA;
}

int current_device() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return -1;
    return dev;
}

// C may be read by TMA: 16-byte aligned base and column stride, sizes in range.
bool c_tma_ok(const void *C_dev, int64_t ldc, int64_t n, size_t es) {
    return aligned(C_dev, 16) && ((ldc * (int64_t)es) % 16 == 0) && n < INT_MAX &&
           (ldc * (int64_t)es) < (1LL << 40) && encoder() != nullptr;
}

// (Re)encode the plan's cached tensor map of C (box rows x cols) when C's address
// or stride or the kernel (its columns) changed since the last execute.
tsmm_status encode_tmapc(tsmm_plan_t p, void *C_dev, int64_t m, int64_t n, int64_t ldc, size_t es,
                         int rows, int cols) {
    if (p->tmapc_ptr == C_dev && p->tmapc_ldc == ldc && p->tmapc_cols == cols) return TSMM_OK;
    const cuuint64_t gdim[2] = {(cuuint64_t)m, (cuuint64_t)n};
    const cuuint64_t gstride[1] = {(cuuint64_t)(ldc * (int64_t)es)};
    const cuuint32_t box[2] = {(cuuint32_t)rows, (cuuint32_t)cols};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = encoder()(&p->tmapc,
                           p->dtype == TSMM_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                                : CU_TENSOR_MAP_DATA_TYPE_FLOAT64,
                           2, C_dev, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        p->tmapc_ptr = nullptr;
        return TSMM_ERR_CUDA;
    }
    p->tmapc_ptr = C_dev;
    p->tmapc_ldc = ldc;
    p->tmapc_cols = cols;
    return TSMM_OK;
}

}  // namespace

namespace tsmm {

int64_t encode_a_rows(CUtensorMap *map, tsmm_dtype dtype, const void *A, int64_t m, int64_t k, int64_t lda) {
    const int64_t es = (int64_t)dtype_size(dtype), R = 16 / es;
    const int64_t off = (int64_t)(reinterpret_cast<uintptr_t>(A) % 16) / es;
    // ends with the last column's last element: no byte behind it is read
    const int64_t width = off + (R - 1) * lda + m, rows = std::min<int64_t>(k / R, INT_MAX / 2);
    if (rows < 1 || lda > INT_MAX / 8 || encoder() == nullptr) return 0;
    const cuuint64_t gdim[2] = {(cuuint64_t)width, (cuuint64_t)rows};
    const cuuint64_t gstride[1] = {(cuuint64_t)(R * lda * es)};
    const cuuint32_t box[2] = {(cuuint32_t)(kTcRows + R), (cuuint32_t)kARowsBox};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = encoder()(map, dtype == TSMM_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64,
                                 2, const_cast<char *>(static_cast<const char *>(A)) - off * es, gdim, gstride, box, estr,
                                 CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? rows : 0;
}

// Costs fitted to sweeps of S on GB300 (m 1000..32768, k 500..32768, every kernel; CUDA graphs of 20 calls).  The sum
// over the partials is the last block's alone and costs as much per split as one to four stages, which a model of
// waves and stages alone does not see: m = k = 2048, n = 16: 32 splits 23.8 us, 16 16.0, 8 14.5; m = 1024, n = 64,
// k = 8192: 37 splits 35.5 us, 16 24.1.
SplitCosts split_costs(tsmm_dtype dt, int np, bool tc, int64_t n) {
    SplitCosts k{};
    if (tc && dt == TSMM_F32) {
        const double w = (double)tc_width(n);
        k = {2, 0.45, 0.67, kTcRows * kTcKB * 4.0, 3.0, 2.5, 0.35 + 0.00625 * w, 1.0e9};
    } else if (tc) {
        const double w = (double)tc64_width(n);
        k = {1, 1.8 + 0.036 * w, 1.8 + 0.036 * w, kTcRows * 64 * 8.0, 5.0 + 0.12 * w, 2.7 + 0.4 * w, 0.1 + 0.03 * w, 0.0};
    } else if (dt == TSMM_F32) {
        const double stage = 0.28 + 0.0015 * np * np;
        k = {tall_resident_blocks(false, np), stage, stage, tall_block_rows(false, np) * 128.0, 2.5,
             0.5 + 0.1 * np, 0.03 + 0.031 * np, 64.0e6};
    } else if (np == 1) {
        k = {tall_resident_blocks(true, np), 0.66, 0.66, tall_block_rows(true, np) * 256.0, 2.5, 0.55, 0.035, 64.0e6};
    } else {
        // bound by the FP64 pipe, which two blocks share and the sums over the partials take too: m = 1500, n = 64, k = 250:
        // 4 splits 91 us, 8 104; m = 20000, n = 64, k = 64: 1 split 209 us, 2 215
        k = {tall_resident_blocks(true, np), 0.54 * np, 1.08 * np, tall_block_rows(true, np) * 256.0, 2.5, 0.19 * np,
             0.04 * np, 64.0e6, 0.5};
    }
    return k;
}

// Split-K choice for regime (i): the S of the least modelled time; the smallest wins ties, which also keeps the
// workspace small.  Blocks run `resident` to an SM; a stage costs what it does alone, or its share of HBM (7 TB/s) if
// that is more; a last wave that is not full runs at its own share.  From waves_from bytes of A on, whole waves of
// stages count at one price: there a block's start and the sum over the partials no longer matter, and HBM's rate needs
// every SM's full count of blocks (m = k = 32768, n = 16: S = 7 takes 611 us and S = 2 667; n = 64 on the tensor cores:
// 805 and, at S = 1, 852; but m = 30000, n = 48, k = 3000: S = 5 78 us and S = 1 65).
// Where that switch lies: n = 16 below 64 MB 22.3 us by block costs and 25.9 by waves (48 MB), 24.5 / 26.7 (67), above it 47.4 /
// 35.7 (134), 81.0 / 55.4 (268).  On the tensor cores the two differ in 29 % of shapes above 1 GB; of 25 such, block costs
// were faster in 23, by 1 to 3 % in most and 15 to 19 % where k is short (m = 167068, n = 50, k = 2380: S = 1 262 us, S = 2
// 310), and 9 % slower in one.  The switch stays for the chains of chunk sums, which more splits keep short.
int choose_splits(const SplitCosts &k, int64_t slabs, int64_t kstages, int num_sms, int64_t max_splits) {
    const int64_t resident = (int64_t)k.resident * num_sms;
    const double bw = 7.0e6;  // bytes per us
    const bool waves_only = k.waves_from > 0.0 && (double)slabs * (double)kstages * k.bytes >= k.waves_from;
    auto stage = [&](int64_t blocks) {
        return std::max(blocks <= num_sms ? k.stage : k.stage2, (double)blocks * k.bytes / bw);
    };
    int64_t best_s = 1;
    double best_t = -1.0;
    const int64_t s_max = std::max<int64_t>(1, std::min<int64_t>(kstages, max_splits));
    for (int64_t s = 1; s <= s_max; ++s) {
        const int64_t blocks = slabs * s, per = (kstages + s - 1) / s;
        const int64_t full = blocks / resident, rem = blocks % resident;
        const double finish = s > 1 ? k.f0 + k.c * (double)s : 0.0;
        double t;
        if (waves_only) {
            const int64_t waves = full + (rem ? 1 : 0);
            t = (double)waves * ((double)per + 4.0) * stage(resident) + finish;
        } else {
            t = (double)full * ((double)per * stage(resident) + k.block + k.share * finish) +
                (rem ? (double)per * stage(rem) + k.block : 0.0) + finish;
        }
        if (best_t < 0 || t < best_t * (1.0 - 1e-9)) {
            best_t = t;
            best_s = s;
        }
    }
    return (int)best_s;
}

}  // namespace tsmm

extern "C" {

const char *tsmm_status_string(tsmm_status status) {
    switch (status) {
        case TSMM_OK: return "TSMM_OK";
        case TSMM_ERR_INVALID_ARG: return "TSMM_ERR_INVALID_ARG";
        case TSMM_ERR_UNSUPPORTED_SHAPE: return "TSMM_ERR_UNSUPPORTED_SHAPE";
        case TSMM_ERR_MISMATCH: return "TSMM_ERR_MISMATCH";
        case TSMM_ERR_MISALIGNED: return "TSMM_ERR_MISALIGNED";
        case TSMM_ERR_OUT_OF_MEMORY: return "TSMM_ERR_OUT_OF_MEMORY";
        case TSMM_ERR_CUDA: return "TSMM_ERR_CUDA";
        case TSMM_ERR_TIMEOUT: return "TSMM_ERR_TIMEOUT";
    }
    return "TSMM_ERR_UNKNOWN";
}

int tsmm_version(void) { return kVersion; }

const char *tsmm_last_cuda_error(void) { return g_last_cuda_error; }

tsmm_status tsmm_pack_b(tsmm_dtype dtype, int64_t k, int64_t n, const void *B_dev, int64_t ldb,
                        tsmm_stream_t stream, tsmm_packed_b *out) {
    return tsmm_pack_b_ex(dtype, TSMM_PREC_NATIVE, k, n, B_dev, ldb, stream, out);
}

tsmm_status tsmm_pack_b_ex(tsmm_dtype dtype, tsmm_precision precision, int64_t k, int64_t n,
                           const void *B_dev, int64_t ldb, tsmm_stream_t stream, tsmm_packed_b *out) {
    if (!out || !valid_dtype(dtype) || k < 0 || n < 0) return TSMM_ERR_INVALID_ARG;
    if (!valid_precision(precision, dtype)) return TSMM_ERR_INVALID_ARG;
    if (ldb < std::max<int64_t>(1, k)) return TSMM_ERR_INVALID_ARG;
    if (k > 0 && n > 0 && !B_dev) return TSMM_ERR_INVALID_ARG;
    const size_t es = dtype_size(dtype);
    if (B_dev && !aligned(B_dev, es)) return TSMM_ERR_MISALIGNED;
    const int regime = regime_of(k, n);
    if (regime == 0) return TSMM_ERR_UNSUPPORTED_SHAPE;
    const int dev = current_device();
    if (dev < 0) return TSMM_ERR_CUDA;

    tsmm_packed_b pb = new (std::nothrow) tsmm_packed_b_s();
    if (!pb) return TSMM_ERR_OUT_OF_MEMORY;
    pb->dtype = dtype;
    pb->precision = precision;
    pb->k = k;
    pb->n = n;
    pb->regime = regime;
    pb->device = dev;
    if (precision == TSMM_PREC_BF16X3) {
        pb->kp = round_up(k, kX3KB);
        pb->w = regime == 1 ? x3_np(n) : kX3RankNT;
        pb->ntiles = regime == 1 ? 1 : (n + kX3RankNT - 1) / kX3RankNT;
    } else if (regime == 1) {
        pb->kp = round_up(k, kTallBKS);
        pb->w = tall_np(n);
        pb->ntiles = 1;
    } else {
        pb->kp = round_up(k, kRankKGran);
        pb->w = kRankNT;
        pb->ntiles = (n + kRankNT - 1) / kRankNT;
    }
    // BF16x3: a hi and a lo BF16 copy of every element
    pb->bytes = precision == TSMM_PREC_BF16X3 ? (size_t)(pb->kp * pb->w * pb->ntiles) * 2 * 2
                                              : (size_t)(pb->kp * pb->w * pb->ntiles) * es;
    pb->data = nullptr;
    pb->tc_data = nullptr;
    pb->tc_min = nullptr;
    if (pb->bytes > 0) {
        bool tc = tc_pack(dtype, regime, precision, n, k);
        const size_t off = (size_t)round_up((int64_t)pb->bytes, 256);
        const size_t pieces = (size_t)pb->kp * (size_t)tc_width(n) * 6;
        bool tc64 = precision == TSMM_PREC_NATIVE && tc64_pack(dtype, regime, n, k);
        bool rtc = rank_tc(dtype, regime, precision, k), rtc64 = rank_tc64(dtype, regime, precision, k);
        const size_t more = tc      ? pieces + (size_t)(pb->kp / kTcKB) * 2 * sizeof(float)
                            : tc64  ? tc64_bytes(k, n)
                            : rtc   ? rank_tc_bytes(k, pb->ntiles)
                            : rtc64 ? rank_tc64_bytes(k, pb->ntiles)
                                    : 0;
        cudaError_t e = cudaMalloc(&pb->data, more ? off + more : pb->bytes);
        if (e != cudaSuccess && more) {  // the panel alone serves the fma kernels
            cudaGetLastError();
            tc = tc64 = rtc = rtc64 = false;
            e = cudaMalloc(&pb->data, pb->bytes);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            delete pb;
            return cuda_status(e);
        }
        if (tc) {
            pb->tc_data = static_cast<char *>(pb->data) + off;
            pb->tc_min = reinterpret_cast<float *>(static_cast<char *>(pb->data) + off + pieces);
        }
        e = tc ? launch_pack_b_tc(k, n, static_cast<const float *>(B_dev), ldb, static_cast<float *>(pb->data), pb->kp,
                                  (int)pb->w, pb->tc_data, pb->tc_min, static_cast<cudaStream_t>(stream))
            : precision == TSMM_PREC_BF16X3
                ? launch_pack_b_bf16x3(k, n, B_dev, ldb, pb->data, (int)pb->w, pb->kp / kX3KB,
                                       pb->ntiles, static_cast<cudaStream_t>(stream))
                : launch_pack_b(dtype, k, n, B_dev, ldb, pb->data, pb->kp, pb->w, pb->ntiles,
                                static_cast<cudaStream_t>(stream));
        if (e == cudaSuccess && rtc) {
            pb->tc_data = static_cast<char *>(pb->data) + off;
            e = launch_pack_b_rank_tc(k, n, static_cast<const float *>(B_dev), ldb, pb->ntiles, pb->tc_data,
                                      static_cast<cudaStream_t>(stream));
        }
        if (e == cudaSuccess && rtc64) {
            pb->tc_data = static_cast<char *>(pb->data) + off;
            e = launch_pack_b_rank_tc64(k, n, static_cast<const double *>(B_dev), ldb, pb->ntiles, pb->tc_data,
                                        static_cast<cudaStream_t>(stream));
        }
        if (e == cudaSuccess && tc64) {
            pb->tc_data = static_cast<char *>(pb->data) + off;
            e = launch_pack_b_tc64(k, n, static_cast<const double *>(B_dev), ldb, pb->tc_data,
                                   static_cast<cudaStream_t>(stream));
        }
        if (e != cudaSuccess) {
            cudaFree(pb->data);
            delete pb;
            return cuda_status(e);
        }
    }
    *out = pb;
    return TSMM_OK;
}

tsmm_status tsmm_packed_b_destroy(tsmm_packed_b pb) {
    if (!pb) return TSMM_OK;
    tsmm_status st = TSMM_OK;
    if (pb->data) st = cuda_status(cudaFree(pb->data));
    delete pb;
    return st;
}

tsmm_status tsmm_packed_b_info(tsmm_packed_b pb, tsmm_dtype *dtype, int64_t *k, int64_t *n,
                               int64_t *kp, int64_t *w, int64_t *ntiles, const void **data_dev,
                               size_t *bytes) {
    if (!pb) return TSMM_ERR_INVALID_ARG;
    if (dtype) *dtype = pb->dtype;
    if (k) *k = pb->k;
    if (n) *n = pb->n;
    if (kp) *kp = pb->kp;
    if (w) *w = pb->w;
    if (ntiles) *ntiles = pb->ntiles;
    if (data_dev) *data_dev = pb->data;
    if (bytes) *bytes = pb->bytes;
    return TSMM_OK;
}

tsmm_status tsmm_packed_b_read(tsmm_packed_b pb, void *host_dst, size_t bytes) {
    if (!pb || bytes < pb->bytes || (pb->bytes > 0 && !host_dst)) return TSMM_ERR_INVALID_ARG;
    if (pb->bytes == 0) return TSMM_OK;
    if (cudaDeviceSynchronize() != cudaSuccess) return TSMM_ERR_CUDA;
    return cuda_status(cudaMemcpy(host_dst, pb->data, pb->bytes, cudaMemcpyDeviceToHost));
}

tsmm_status tsmm_plan(int64_t m, int64_t n, int64_t k, tsmm_dtype dtype, tsmm_plan_t *out) {
    return tsmm_plan_ex(m, n, k, dtype, TSMM_PREC_NATIVE, out);
}

tsmm_status tsmm_plan_ex(int64_t m, int64_t n, int64_t k, tsmm_dtype dtype, tsmm_precision precision,
                         tsmm_plan_t *out) {
    if (!out || !valid_dtype(dtype) || m < 0 || n < 0 || k < 0) return TSMM_ERR_INVALID_ARG;
    if (!valid_precision(precision, dtype)) return TSMM_ERR_INVALID_ARG;
    int dev = current_device();
    int sms = 0;
    if (dev >= 0 && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        sms = 0;
    // a tuned choice recorded in the plan cache wins over the heuristic (native precision)
    const int cached = precision == TSMM_PREC_NATIVE ? plan_cache_lookup(dtype, m, n, k, sms) : 0;
    return create_plan(m, n, k, dtype, cached, out, precision);
}

}  // extern "C"

namespace tsmm {

tsmm_status create_plan(int64_t m, int64_t n, int64_t k, tsmm_dtype dtype, int forced_splits,
                        tsmm_plan_t *out, int precision) {
    if (!out || !valid_dtype(dtype) || m < 0 || n < 0 || k < 0) return TSMM_ERR_INVALID_ARG;
    const int regime = regime_of(k, n);
    if (regime == 0) return TSMM_ERR_UNSUPPORTED_SHAPE;  // before any device query
    const int dev = current_device();
    if (dev < 0) return TSMM_ERR_CUDA;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return TSMM_ERR_CUDA;

    tsmm_plan_t p = new (std::nothrow) tsmm_plan_s();
    if (!p) return TSMM_ERR_OUT_OF_MEMORY;
    size_t ticket_bytes = 0;
    tsmm_status st = plan_layout(m, n, k, dtype, forced_splits, precision, dev, sms, 512LL << 20, p,
                                 &ticket_bytes);
    if (st != TSMM_OK) {
        delete p;
        return st;
    }
    cudaError_t e = cudaSuccess;
    if (p->workspace_bytes) e = cudaMalloc(&p->workspace, p->workspace_bytes);
    if (e == cudaSuccess && ticket_bytes) {
        e = cudaMalloc(reinterpret_cast<void **>(&p->tickets), ticket_bytes);
        if (e == cudaSuccess) e = cudaMemset(p->tickets, 0, ticket_bytes);
    }
    if (e == cudaSuccess) {
        e = cudaMalloc(reinterpret_cast<void **>(&p->status), sizeof(unsigned));
        if (e == cudaSuccess) e = cudaMemset(p->status, 0, sizeof(unsigned));
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        if (p->workspace) cudaFree(p->workspace);
        if (p->tickets) cudaFree(p->tickets);
        if (p->status) cudaFree(p->status);
        delete p;
        return cuda_status(e);
    }
    *out = p;
    return TSMM_OK;
}

tsmm_status plan_layout(int64_t m, int64_t n, int64_t k, tsmm_dtype dtype, int forced_splits,
                        int precision, int dev, int sms, int64_t max_workspace, tsmm_plan_s *p,
                        size_t *ticket_bytes_out) {
    if (!valid_dtype(dtype) || m < 0 || n < 0 || k < 0) return TSMM_ERR_INVALID_ARG;
    const int regime = regime_of(k, n);
    if (regime == 0) return TSMM_ERR_UNSUPPORTED_SHAPE;
    std::memset(static_cast<void *>(p), 0, sizeof(*p));
    p->m = m;
    p->n = n;
    p->k = k;
    p->dtype = dtype;
    p->precision = precision;
    p->regime = regime;
    p->device = dev;
    p->num_sms = sms;
    const size_t es = dtype_size(dtype);
    size_t ticket_bytes = 0;
    if (precision == TSMM_PREC_BF16X3 && regime == 2) {
        // 128 x 128 output tiles, k (<= 128) in one or two 64-column chunks
        p->kp = round_up(k, kX3KB);
        p->bm = 128;
        p->np = kX3RankNT;
        p->splits = 1;
        p->mtiles = (m + p->bm - 1) / p->bm;
        p->ntiles = (n + kX3RankNT - 1) / kX3RankNT;
    } else if (precision == TSMM_PREC_BF16X3) {
        // one 128-row slab per block, k in 64-column chunks, one block per SM
        p->np = x3_np(n);
        p->bm = 128;
        p->kp = round_up(k, kX3KB);
        p->slabs = (m + p->bm - 1) / p->bm;
        const int64_t kstages = p->kp / kX3KB;
        const int64_t per_split = (int64_t)p->np * p->slabs * p->bm * (int64_t)es;
        int64_t max_splits = 65535;
        if (per_split > 0) max_splits = std::min<int64_t>(max_splits, max_workspace / per_split);
        // whole waves of equal stages, a block's start and end worth four of them
        const SplitCosts x3_costs{1, 1.0, 1.0, 0.0, 4.0, 0.0, 0.0, 0.0};
        int s = (kstages > 0 && p->slabs > 0)
                    ? choose_splits(x3_costs, p->slabs, kstages, sms, max_splits)
                    : 1;
        if (forced_splits > 0)
            s = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)forced_splits, kstages, max_splits}));
        const int64_t chunk_stages = kstages > 0 ? (kstages + s - 1) / s : 1;
        p->kchunk = chunk_stages * kX3KB;
        p->splits = kstages > 0 ? (int)((kstages + chunk_stages - 1) / chunk_stages) : 1;
        if (p->splits > 1) {
            p->workspace_bytes = (size_t)p->splits * (size_t)per_split;
            ticket_bytes = (size_t)p->slabs * sizeof(unsigned);
        }
    } else if (regime == 1) {
        p->np = tall_np(n);
        p->tc = tc_pack(dtype, regime, precision, n, k) ||
                (precision == TSMM_PREC_NATIVE && tc64_plan(dtype, regime, m, n, k));
        // k split in stages of kTallBKS columns; the FP64 guard looks at aligned windows of 64
        const int64_t stage = p->tc && dtype == TSMM_F64 ? 64 : kTallBKS;
        p->bm = p->tc ? kTcRows : tall_bm(dtype, p->np);
        p->kp = round_up(k, kTallBKS);
        p->slabs = (m + p->bm - 1) / p->bm;
        const int64_t kstages = (p->kp + stage - 1) / stage;
        // keep the workspace within max_workspace and the grid's y extent legal
        const int64_t per_split = (int64_t)p->np * p->slabs * p->bm * (int64_t)es;
        int64_t max_splits = 65535;
        if (per_split > 0) max_splits = std::min<int64_t>(max_splits, max_workspace / per_split);
        int s = (kstages > 0 && p->slabs > 0)
                    ? choose_splits(split_costs(dtype, p->np, p->tc, n), p->slabs, kstages, sms, max_splits)
                    : 1;
        if (forced_splits > 0)
            s = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)forced_splits, kstages, max_splits}));
        const int64_t chunk_stages = kstages > 0 ? (kstages + s - 1) / s : 1;
        p->kchunk = chunk_stages * stage;
        p->splits = kstages > 0 ? (int)((kstages + chunk_stages - 1) / chunk_stages) : 1;
        if (p->splits > 1) {
            p->workspace_bytes = (size_t)p->splits * (size_t)per_split;
            ticket_bytes = (size_t)p->slabs * sizeof(unsigned);
        }
    } else {
        p->kp = round_up(k, kRankKGran);
        p->bm = dtype == TSMM_F64 ? 64 : 128;
        p->np = kRankNT;
        p->splits = 1;
        p->mtiles = (m + p->bm - 1) / p->bm;
        p->ntiles = (n + kRankNT - 1) / kRankNT;
    }
    if (ticket_bytes_out) *ticket_bytes_out = ticket_bytes;
    return TSMM_OK;
}

}  // namespace tsmm

extern "C" {

tsmm_status tsmm_plan_destroy(tsmm_plan_t p) {
    if (!p) return TSMM_OK;
    tsmm_status st = TSMM_OK;
    if (p->workspace && cudaFree(p->workspace) != cudaSuccess) st = TSMM_ERR_CUDA;
    if (p->tickets && cudaFree(p->tickets) != cudaSuccess) st = TSMM_ERR_CUDA;
    if (p->status && cudaFree(p->status) != cudaSuccess) st = TSMM_ERR_CUDA;
    delete p;
    return st;
}

tsmm_status tsmm_plan_info(tsmm_plan_t p, int *regime, int *np, int *bm, int *splits,
                           size_t *workspace_bytes) {
    if (!p) return TSMM_ERR_INVALID_ARG;
    if (regime) *regime = p->regime;
    if (np) *np = p->np;
    if (bm) *bm = p->bm;
    if (splits) *splits = p->splits;
    if (workspace_bytes) *workspace_bytes = p->workspace_bytes;
    return TSMM_OK;
}

int tsmm_plan_launches_per_execute(tsmm_plan_t p) {
    if (!p) return 0;
    return (p->m == 0 || p->n == 0) ? 0 : 1;
}

tsmm_status tsmm_execute(tsmm_plan_t p, double alpha, const void *A_dev, int64_t lda,
                         tsmm_packed_b pb, double beta, void *C_dev, int64_t ldc,
                         tsmm_stream_t stream) {
    if (!p || !pb) return TSMM_ERR_INVALID_ARG;
    if (pb->dtype != p->dtype || pb->k != p->k || pb->n != p->n || pb->device != p->device ||
        pb->precision != p->precision)
        return TSMM_ERR_MISMATCH;
    if (current_device() != p->device) return TSMM_ERR_MISMATCH;
    const int64_t m = p->m, n = p->n, k = p->k;
    if (lda < std::max<int64_t>(1, m) || ldc < std::max<int64_t>(1, m)) return TSMM_ERR_INVALID_ARG;
    if (m == 0 || n == 0) return TSMM_OK;
    const bool use_ab = (alpha != 0.0) && (k > 0);
    if (!C_dev || (use_ab && !A_dev)) return TSMM_ERR_INVALID_ARG;
    const size_t es = dtype_size(p->dtype);
    if (!aligned(C_dev, es) || (use_ab && !aligned(A_dev, es))) return TSMM_ERR_MISALIGNED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (p->dtype == TSMM_F32 && static_cast<float>(alpha) == 0.0f && alpha != 0.0) {
        // alpha underflows to zero in float: behave as alpha == 0
        return cuda_status(launch_scale(p->dtype, m, n, beta, C_dev, ldc, s));
    }
    if (!use_ab) return cuda_status(launch_scale(p->dtype, m, n, beta, C_dev, ldc, s));

    TallArgs a;
    a.m = m;
    a.n = n;
    a.k = k;
    a.lda = lda;
    a.ldc = ldc;
    a.A = A_dev;
    a.Bp = pb->data;
    a.C = C_dev;
    a.alpha = alpha;
    a.beta = beta;
    a.ws = p->workspace;
    a.tickets = p->tickets;
    a.status = p->status;
    a.splits = p->splits;
    a.kchunk = p->kchunk;
    a.kp = p->kp;
    a.slabs = p->slabs;
    a.np = p->np;
    a.Bt = pb->tc_data;
    a.bmin = pb->tc_min;
    a.arows = 0;

    // A tensor-core plan whose B was packed without its tensor-core form (for lack of memory), or too short in k for it: the
    // fma kernel on its own slabs, in one split, which needs no workspace.  (The blocks' own fma path, which grouped launches
    // with few columns take, gives the same bits there; m = 100000, n = 64, k = 8: 12 us, 50 on that path.)
    const bool tc = p->tc && pb->tc_data && !(p->dtype == TSMM_F32 && k < kTcMinK);
    const bool fma = p->tc && !tc;
    const int bm = fma ? tall_bm(p->dtype, p->np) : p->bm;
    if (fma) {
        a.slabs = (m + bm - 1) / bm;
        a.splits = 1;
        a.kchunk = a.kp;
    }

    const bool tma = aligned(A_dev, 16) && ((lda * (int64_t)es) % 16 == 0) && m < INT_MAX &&
                     k < INT_MAX && (lda * (int64_t)es) < (1LL << 40) && encoder() != nullptr;
    if (tma && (p->tmap_ptr != A_dev || p->tmap_lda != lda || p->tmap_tc != tc)) {
        // box: bm rows x 32 columns (the regime (i) stage and the regime (ii) k chunk)
        const cuuint64_t gdim[2] = {(cuuint64_t)m, (cuuint64_t)k};
        const cuuint64_t gstride[1] = {(cuuint64_t)(lda * (int64_t)es)};
        const cuuint32_t box[2] = {(cuuint32_t)bm,
                                   (cuuint32_t)a_box_k(p->dtype, p->regime, p->precision, p->k, tc)};
        const cuuint32_t estr[2] = {1, 1};
        CUresult r = encoder()(&p->tmap,
                               p->dtype == TSMM_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                                    : CU_TENSOR_MAP_DATA_TYPE_FLOAT64,
                               2, const_cast<void *>(A_dev), gdim, gstride, box, estr,
                               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                               CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            p->tmap_ptr = nullptr;
            return TSMM_ERR_CUDA;
        }
        p->tmap_ptr = A_dev;
        p->tmap_lda = lda;
        p->tmap_tc = tc;
    }
    if (p->precision == TSMM_PREC_BF16X3) {
        if (p->regime == 2) {
            RankArgs ra;
            ra.m = m;
            ra.n = n;
            ra.k = k;
            ra.lda = lda;
            ra.ldc = ldc;
            ra.kp = pb->kp;
            ra.A = A_dev;
            ra.Bp = pb->data;
            ra.Bt = nullptr;
            ra.brange = nullptr;
            ra.C = C_dev;
            ra.alpha = alpha;
            ra.beta = beta;
            ra.num_sms = p->num_sms;
            // C0 loads and C stores go through TMA when C allows it (any beta)
            const bool tmc = c_tma_ok(C_dev, ldc, n, es);
            if (tmc) {
                const tsmm_status st = encode_tmapc(p, C_dev, m, n, ldc, es, p->bm, kX3RankSub);
                if (st != TSMM_OK) return st;
            }
            // an A that a tensor map cannot describe is moved column by column
            return cuda_status(
                launch_rankk_bf16x3(tma ? &p->tmap : nullptr, tmc ? &p->tmapc : nullptr, ra, p->status, s));
        }
        // regime (i): an A that a tensor map cannot describe is moved column by column
        return cuda_status(launch_tall_bf16x3(p->np, tma ? &p->tmap : nullptr, a, p->num_sms, s));
    }
    if (p->regime == 2) {
        RankArgs ra;
        ra.m = m;
        ra.n = n;
        ra.k = k;
        ra.lda = lda;
        ra.ldc = ldc;
        ra.kp = pb->kp;
        ra.A = A_dev;
        ra.Bp = pb->data;
        ra.Bt = pb->tc_data;
        ra.brange = nullptr;
        ra.C = C_dev;
        ra.alpha = alpha;
        ra.beta = beta;
        ra.num_sms = p->num_sms;
        if (pb->tc_data && rank_tc64(p->dtype, p->regime, p->precision, k)) {
            const bool tmc = m < INT_MAX && c_tma_ok(C_dev, ldc, n, es);
            if (tmc) {
                const tsmm_status st = encode_tmapc(p, C_dev, m, n, ldc, es, kTcRows, kRank64Sub);
                if (st != TSMM_OK) return st;
            }
            return cuda_status(launch_rankk_tc64(tmc ? &p->tmapc : nullptr, ra, p->status, s));
        }
        // An A that a tensor map cannot describe is small here (k <= 128 columns
        // against an m x n output): it is copied into an aligned scratch buffer
        // from the stream's memory pool (released on the stream after the
        // kernel) so that the tensor-copy kernels run; only if that allocation
        // fails does the plain-load kernel read it directly.
        void *scratch = nullptr;
        CUtensorMap tm_scratch;
        bool tma_a = tma;
        if (!tma && encoder() != nullptr && m < INT_MAX && k <= 65535) {
            const int64_t v = 16 / (int64_t)es;
            const int64_t ldd = (m + v - 1) / v * v;
            const size_t bytes = (size_t)ldd * (size_t)k * es;
            if (bytes <= (size_t(1) << 32) && cudaMallocAsync(&scratch, bytes, s) == cudaSuccess) {
                const cuuint64_t gdim[2] = {(cuuint64_t)m, (cuuint64_t)k};
                const cuuint64_t gstride[1] = {(cuuint64_t)(ldd * (int64_t)es)};
                const cuuint32_t box[2] = {(cuuint32_t)p->bm,
                                           (cuuint32_t)a_box_k(p->dtype, p->regime, p->precision, p->k, p->tc)};
                const cuuint32_t estr[2] = {1, 1};
                const cudaError_t ce = launch_copy_columns(p->dtype, A_dev, lda, m, k, scratch, ldd, s);
                if (ce == cudaSuccess &&
                    encoder()(&tm_scratch,
                              p->dtype == TSMM_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64,
                              2, scratch, gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS) {
                    tma_a = true;
                    ra.A = scratch;
                    ra.lda = ldd;
                } else {
                    cudaFreeAsync(scratch, s);
                    scratch = nullptr;
                    if (ce != cudaSuccess) return cuda_status(ce);
                }
            } else {
                cudaGetLastError();  // no scratch: the plain-load kernel
                scratch = nullptr;
            }
        }
        const bool rtc = tma_a && pb->tc_data && rank_tc(p->dtype, p->regime, p->precision, k);
        // C tiles by TMA (C0 prefetch; C0 and C in the FP32 k > 32 kernel): the
        // same 16-byte rules for C
        const bool tmc = tma_a && c_tma_ok(C_dev, ldc, n, es);
        if (tmc) {
            const tsmm_status st = encode_tmapc(p, C_dev, m, n, ldc, es, p->bm, rtc ? kRankTcSub : kRankNT);
            if (st != TSMM_OK) {
                if (scratch) cudaFreeAsync(scratch, s);
                return st;
            }
        }
        // (without the tensor cores, by choice or a B packed without its form for lack of memory, FP32 is left to the
        // plain-load kernel here: the fma kernels' tensor copies serve k < kRankTcMinK)
        const bool plain = !rtc && p->dtype == TSMM_F32 && k >= kRankTcMinK;
        const CUtensorMap *ta = tma_a && !plain ? (scratch ? &tm_scratch : &p->tmap) : nullptr;
        const CUtensorMap *tc = tmc && !plain ? &p->tmapc : nullptr;
        const cudaError_t e = rtc ? launch_rankk_tc(ta, tc, ra, p->status, s)
                                  : launch_rankk(p->dtype, ta, tc, ra, p->status, s);
        if (scratch) cudaFreeAsync(scratch, s);  // after the kernel, in stream order
        return cuda_status(e);
    }
    if (tc && !tma) {
        if (p->tmap_ptr != A_dev || p->tmap_lda != lda || p->tmap_tc != tc) {
            p->arows = encode_a_rows(&p->tmap, p->dtype, A_dev, m, k, lda);
            p->tmap_ptr = A_dev;
            p->tmap_lda = lda;
            p->tmap_tc = tc;
        }
        a.arows = p->arows;
    }
    if (tc && p->dtype == TSMM_F64) return cuda_status(launch_tall_tc64(p->tmap, !tma, a, s));
    if (tc) return cuda_status(launch_tall_tc(p->tmap, !tma, a, s));
    cudaError_t e = p->dtype == TSMM_F32 ? launch_tall_f32(tma, p->np, &p->tmap, a, s)
                                         : launch_tall_f64(tma, p->np, &p->tmap, a, s);
    return cuda_status(e);
}

tsmm_status tsmm_plan_check(tsmm_plan_t p) {
    if (!p) return TSMM_ERR_INVALID_ARG;
    if (cudaDeviceSynchronize() != cudaSuccess) return TSMM_ERR_CUDA;
    unsigned word = 0;
    if (cudaMemcpy(&word, p->status, sizeof(word), cudaMemcpyDeviceToHost) != cudaSuccess)
        return TSMM_ERR_CUDA;
    if (word == 0) return TSMM_OK;
    // clear the record and the split-K arrival counters a failed launch may have left
    cudaMemset(p->status, 0, sizeof(unsigned));
    if (p->tickets) cudaMemset(p->tickets, 0, (size_t)p->slabs * sizeof(unsigned));
    cudaDeviceSynchronize();
    return (word & kDevErrTimeout) ? TSMM_ERR_TIMEOUT : TSMM_ERR_CUDA;
}

}  // extern "C"
