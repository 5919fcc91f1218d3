// Packing, instantiations and launch of the FP64 tensor-core regime (i) kernel.
#include "tsmm_group.cuh"
#include "tsmm_tall_tc64.cuh"

namespace tsmm {

// Scale of column blockIdx.x: its largest exponent field.
__global__ void __launch_bounds__(256) pack_b_tc64_scale_kernel(const double *__restrict__ B, int64_t k, int64_t ldb,
                                                                TcB64 *__restrict__ head) {
    __shared__ int mx;
    __shared__ unsigned any;
    if (threadIdx.x == 0) mx = 0, any = 0u;
    __syncthreads();
    const double *col = B + (int64_t)blockIdx.x * ldb;
    int e = 0;
    bool nz = false;
    for (int64_t p = threadIdx.x; p < k; p += 256) {
        const double x = col[p];
        e = max(e, (__double2hiint(x) >> 20) & 0x7ff);
        nz |= x != 0.0;
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (threadIdx.x % 32 == 0) atomicMax(&mx, e);
    if (nz) any = 1u;
    __syncthreads();
    if (threadIdx.x == 0) {
        const bool in = mx > kTc64Emin && mx <= kTc64Emax;
        head->F[blockIdx.x] = in ? mx : kTc64Emin;
        if (any && !in) atomicOr(&head->bad, 1u);
    }
}

// Digits and guard bytes: block = one step of kTc64KB rows, thread = column and pair of rows.
__global__ void pack_b_tc64_kernel(const double *__restrict__ B, int64_t k, int64_t n, int64_t ldb, int w,
                                   unsigned char *__restrict__ base) {
    const TcB64 *head = reinterpret_cast<const TcB64 *>(base);
    const int64_t off_guard = kTc64Head + (int64_t)gridDim.x * (tc64_rows(w) * w * kTc64KB * 2);
    unsigned char *dst = base + kTc64Head + blockIdx.x * (int64_t)(tc64_rows(w) * w * kTc64KB * 2);
    for (int e = threadIdx.x; e < w * (kTc64KB / 2); e += blockDim.x) {
        const int kk = e % (kTc64KB / 2) * 2, j = e / (kTc64KB / 2);
        const int64_t p = (int64_t)blockIdx.x * kTc64KB + kk;
        const double *q = B + p + (int64_t)j * ldb;
        uint32_t d[8];  // A has seven
        const uint32_t g = tc64_digits8(p < k && j < n ? q[0] : 0.0, p + 1 < k && j < n ? q[1] : 0.0,
                                        j < n ? head->F[j] : kTc64Emin, d);
        // digit-major rows (digit i, column j) of 16 k: 8-row groups of 256 bytes
#pragma unroll
        for (int i = 0; i < 13; ++i) {
            const int rw = i * w + j;
            if (i >= tc64_rows(w)) break;
            uint32_t v = d[i & 7];
            if (tc64_rows(w) == 13 && i >= 6) v = hfma2(d[i - 5], 0x1c001c00u, d[i - 6]);  // d[i-6] + 2^-8 d[i-5], rounded
            *reinterpret_cast<uint32_t *>(dst + (rw / 8) * 256 + (kk / 8) * 128 + (rw % 8) * 16 + (kk % 8) * 2) = v;
        }
        *reinterpret_cast<uint16_t *>(base + off_guard + (p / 64) * (w * 64) + j * 64 + p % 64) = (uint16_t)g;
    }
}

size_t tc64_bytes(int64_t k, int64_t n) {
    const int64_t w = tc64_width(n), steps = round_up(k, 64) / kTc64KB;
    return (size_t)(kTc64Head + steps * tc64_rows((int)w) * w * kTc64KB * 2 + round_up(k, 64) * w);
}

cudaError_t launch_pack_b_tc64(int64_t k, int64_t n, const double *B, int64_t ldb, void *dst, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(dst, 0, sizeof(TcB64), s);
    if (e != cudaSuccess) return e;
    pack_b_tc64_scale_kernel<<<(unsigned)n, 256, 0, s>>>(B, k, ldb, static_cast<TcB64 *>(dst));
    pack_b_tc64_kernel<<<(unsigned)(round_up(k, 64) / kTc64KB), 256, 0, s>>>(B, k, n, ldb, (int)tc64_width(n),
                                                                           static_cast<unsigned char *>(dst));
    return cudaGetLastError();
}

template <int W, bool U>
static cudaError_t launch_tall_tc64_t(const CUtensorMap &tmap, const TallArgs &a, cudaStream_t s) {
    using Cfg = TallTc64Cfg<W, U>;
    const cudaError_t e = ensure_smem_limit(reinterpret_cast<const void *>(tall_tc64_kernel<W, U>), Cfg::SMEM);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)a.slabs, (unsigned)a.splits);
    tall_tc64_kernel<W, U><<<grid, Cfg::THREADS, Cfg::SMEM, s>>>(tmap, a);
    return cudaGetLastError();
}

cudaError_t launch_tall_tc64(const CUtensorMap &tmap, bool u, const TallArgs &a, cudaStream_t s) {
    switch (tc64_width(a.n)) {
        case 16: return u ? launch_tall_tc64_t<16, true>(tmap, a, s) : launch_tall_tc64_t<16, false>(tmap, a, s);
        case 32: return u ? launch_tall_tc64_t<32, true>(tmap, a, s) : launch_tall_tc64_t<32, false>(tmap, a, s);
        case 48: return u ? launch_tall_tc64_t<48, true>(tmap, a, s) : launch_tall_tc64_t<48, false>(tmap, a, s);
        case 64: return u ? launch_tall_tc64_t<64, true>(tmap, a, s) : launch_tall_tc64_t<64, false>(tmap, a, s);
        default: return cudaErrorInvalidValue;
    }
}

// Many problems of one MMA width in one launch, one block per work item (tsmm_group.cuh).
template <int W, bool U>
__global__ void __launch_bounds__(TallTc64Cfg<W, U>::THREADS, 1)
    tall_tc64_grouped_kernel(const __grid_constant__ GroupParams gp) {
    const int64_t item = blockIdx.x;
    const int p = group_find(gp, item);
    const TallArgs &a = gp.p[p].a;
    int64_t slab, split;
    udivmod(item - gp.p[p].item_begin, a.splits, slab, split);
    tall_tc64_block<W, U>(&gp.p[p].tmA, a, slab, (int)split);
}

template <int W, bool U>
static cudaError_t launch_grouped_tc64_t(const GroupParams &gp, cudaStream_t s) {
    using Cfg = TallTc64Cfg<W, U>;
    const cudaError_t e = ensure_smem_limit(reinterpret_cast<const void *>(tall_tc64_grouped_kernel<W, U>), Cfg::SMEM);
    if (e != cudaSuccess) return e;
    if (gp.total_items <= 0) return cudaSuccess;
    if (gp.total_items > INT_MAX) return cudaErrorInvalidValue;
    tall_tc64_grouped_kernel<W, U><<<(unsigned)gp.total_items, Cfg::THREADS, Cfg::SMEM, s>>>(gp);
    return cudaGetLastError();
}

cudaError_t launch_grouped_tc64(int width, bool unaligned, const GroupParams &gp, cudaStream_t s) {
    switch (width) {
        case 16: return unaligned ? launch_grouped_tc64_t<16, true>(gp, s) : launch_grouped_tc64_t<16, false>(gp, s);
        case 32: return unaligned ? launch_grouped_tc64_t<32, true>(gp, s) : launch_grouped_tc64_t<32, false>(gp, s);
        case 48: return unaligned ? launch_grouped_tc64_t<48, true>(gp, s) : launch_grouped_tc64_t<48, false>(gp, s);
        case 64: return unaligned ? launch_grouped_tc64_t<64, true>(gp, s) : launch_grouped_tc64_t<64, false>(gp, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tsmm
