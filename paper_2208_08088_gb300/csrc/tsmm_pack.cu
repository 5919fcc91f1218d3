// PACKB of Algorithm 1 (bit-preserving re-layout of B into column tiles of
// row-major panels), and the alpha == 0 / k == 0 path C = beta * C0.
#include "tsmm_device.cuh"
#include "tsmm_internal.h"
#include "tsmm_tc.cuh"

namespace tsmm {

// One thread per packed element.  dst tile t: kp x w row-major at t*kp*w;
// element (p, jj) <- B[p + (t*w + jj)*ldb], or +0 outside the k x n matrix.
// Consecutive threads write consecutive packed elements (coalesced stores);
// the gather from column-major B is served by L1/L2 (B is small and read once).
template <typename T>
__global__ void pack_b_kernel(const T *__restrict__ B, int64_t k, int64_t n, int64_t ldb,
                              T *__restrict__ dst, int64_t kp, int64_t w, int64_t total) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = e / (kp * w);
        const int64_t rem = e - t * kp * w;
        const int64_t p = rem / w;
        const int64_t j = t * w + (rem - p * w);
        dst[e] = (p < k && j < n) ? B[p + j * ldb] : T(0);
    }
}

// The regime (i) panel and its tensor-core form (tsmm_tall_tc.cuh) in one pass: block c takes the 32 rows of chunk c
// (lanes along k, so B is read coalesced), writes the panel rows, the three BF16 pieces of every element at
// (j/8)*512 + (kk/8)*128 + (j%8)*16 + (kk%8)*2 of its piece, and the chunk's smallest nonzero
// magnitude (behind all chunks': its largest).
__global__ void __launch_bounds__(256) pack_b_tc_kernel(const float *__restrict__ B, int64_t k, int64_t n, int64_t ldb,
                                                        float *__restrict__ panel, int np, int w,
                                                        unsigned char *__restrict__ pieces, float *__restrict__ cmin) {
    __shared__ float t[kTcKB][kTallMaxN + 1];
    __shared__ uint32_t smin, smax;
    const int64_t p0 = (int64_t)blockIdx.x * kTcKB;
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    if (threadIdx.x == 0) smin = 0xffffffffu, smax = 0u;
    __syncthreads();
    uint32_t mn = 0xffffffffu, mx = 0u;
    for (int j = warp; j < kTallMaxN; j += 8) {
        const float x = (p0 + lane < k && j < n) ? B[p0 + lane + (int64_t)j * ldb] : 0.f;
        t[lane][j] = x;
        mn = min(mn, __float_as_uint(x) * 2u - 1u);
        mx = max(mx, __float_as_uint(x) & 0x7fffffffu);
    }
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) atomicMin(&smin, mn), atomicMax(&smax, mx);
    __syncthreads();
    for (int e = threadIdx.x; e < kTcKB * np; e += 256) panel[p0 * np + e] = t[e / np][e % np];
    unsigned char *dst = pieces + (int64_t)blockIdx.x * (w * kTcKB * 6);
    const int piece = w * kTcKB * 2;
    for (int e = threadIdx.x; e < w * (kTcKB / 2); e += 256) {
        const int j = e / (kTcKB / 2), kk = e % (kTcKB / 2) * 2;
        uint32_t h, m, l;
        split3_bf16x2(t[kk][j], t[kk + 1][j], h, m, l);
        unsigned char *q = dst + (j / 8) * (kTcKB / 8 * 128) + (kk / 8) * 128 + (j % 8) * 16 + (kk % 8) * 2;
        *reinterpret_cast<uint32_t *>(q) = h;
        *reinterpret_cast<uint32_t *>(q + piece) = m;
        *reinterpret_cast<uint32_t *>(q + 2 * piece) = l;
    }
    if (threadIdx.x == 0) {
        cmin[blockIdx.x] = smin == 0xffffffffu ? __uint_as_float(0x7f800000u) : __uint_as_float((smin + 1u) >> 1);
        cmin[gridDim.x + blockIdx.x] = __uint_as_float(smax);
    }
}

// C = beta * C0 (beta != 0) or C = 0 (beta == 0, C0 not read).
template <typename T>
__global__ void scale_kernel(int64_t m, int64_t n, T beta, T *__restrict__ C, int64_t ldc) {
    const int64_t total = m * n;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = e / m;
        const int64_t i = e - j * m;
        T *c = C + i + j * ldc;
        *c = (beta != T(0)) ? beta * *c : T(0);
    }
}

// dst[i + p*ldd] = src[i + p*lds] for i < m, p < k (blockIdx.y = p): a
// column-major copy into another leading dimension.  Regime (ii) uses it to give
// an A that a tensor map cannot describe an aligned copy that one can.
template <typename T>
__global__ void copy_columns_kernel(const T *__restrict__ src, int64_t lds, int64_t m, T *__restrict__ dst,
                                    int64_t ldd) {
    const T *sc = src + (int64_t)blockIdx.y * lds;
    T *dc = dst + (int64_t)blockIdx.y * ldd;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        dc[i] = sc[i];
}

static unsigned grid_for(int64_t total, int threads) {
    int64_t blocks = (total + threads - 1) / threads;
    if (blocks > 152 * 64) blocks = 152 * 64;
    if (blocks < 1) blocks = 1;
    return (unsigned)blocks;
}

cudaError_t launch_pack_b(tsmm_dtype dt, int64_t k, int64_t n, const void *B, int64_t ldb,
                          void *dst, int64_t kp, int64_t w, int64_t ntiles, cudaStream_t s) {
    const int64_t total = kp * w * ntiles;
    if (total == 0) return cudaSuccess;
    const int threads = 256;
    if (dt == TSMM_F32)
        pack_b_kernel<float><<<grid_for(total, threads), threads, 0, s>>>(
            static_cast<const float *>(B), k, n, ldb, static_cast<float *>(dst), kp, w, total);
    else
        pack_b_kernel<double><<<grid_for(total, threads), threads, 0, s>>>(
            static_cast<const double *>(B), k, n, ldb, static_cast<double *>(dst), kp, w, total);
    return cudaGetLastError();
}

cudaError_t launch_pack_b_tc(int64_t k, int64_t n, const float *B, int64_t ldb, float *panel, int64_t kp, int np,
                             void *tc_data, float *tc_min, cudaStream_t s) {
    if (kp == 0) return cudaSuccess;
    pack_b_tc_kernel<<<(unsigned)(kp / kTcKB), 256, 0, s>>>(B, k, n, ldb, panel, np, (int)tc_width(n),
                                                            static_cast<unsigned char *>(tc_data), tc_min);
    return cudaGetLastError();
}

cudaError_t launch_copy_columns(tsmm_dtype dt, const void *src, int64_t lds, int64_t m, int64_t k, void *dst,
                                int64_t ldd, cudaStream_t s) {
    if (m == 0 || k == 0) return cudaSuccess;
    if (k > 65535) return cudaErrorInvalidValue;
    const int threads = 256;
    int64_t bx = (m + threads - 1) / threads;
    if (bx > 64) bx = 64;
    const dim3 grid((unsigned)bx, (unsigned)k);
    if (dt == TSMM_F32)
        copy_columns_kernel<float><<<grid, threads, 0, s>>>(static_cast<const float *>(src), lds, m,
                                                            static_cast<float *>(dst), ldd);
    else
        copy_columns_kernel<double><<<grid, threads, 0, s>>>(static_cast<const double *>(src), lds, m,
                                                             static_cast<double *>(dst), ldd);
    return cudaGetLastError();
}

cudaError_t launch_scale(tsmm_dtype dt, int64_t m, int64_t n, double beta, void *C, int64_t ldc,
                         cudaStream_t s) {
    const int64_t total = m * n;
    if (total == 0) return cudaSuccess;
    const int threads = 256;
    if (dt == TSMM_F32)
        scale_kernel<float><<<grid_for(total, threads), threads, 0, s>>>(
            m, n, static_cast<float>(beta), static_cast<float *>(C), ldc);
    else
        scale_kernel<double><<<grid_for(total, threads), threads, 0, s>>>(
            m, n, beta, static_cast<double *>(C), ldc);
    return cudaGetLastError();
}

}  // namespace tsmm
