// Instantiations and launches of the tensor-core regime (i) kernel, single and grouped.
#include "tsmm_group.cuh"
#include "tsmm_tall_tc.cuh"

namespace tsmm {

template <int W, bool U>
static cudaError_t launch_tall_tc_t(const CUtensorMap &tmap, const TallArgs &a, cudaStream_t s) {
    using Cfg = TallTcCfg<W, U>;
    const cudaError_t e = ensure_smem_limit(reinterpret_cast<const void *>(tall_tc_kernel<W, U>), Cfg::SMEM);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)a.slabs, (unsigned)a.splits);
    tall_tc_kernel<W, U><<<grid, Cfg::THREADS, Cfg::SMEM, s>>>(tmap, a);
    return cudaGetLastError();
}

cudaError_t launch_tall_tc(const CUtensorMap &tmap, bool u, const TallArgs &a, cudaStream_t s) {
    switch (tc_width(a.n)) {
        case 32: return u ? launch_tall_tc_t<32, true>(tmap, a, s) : launch_tall_tc_t<32, false>(tmap, a, s);
        case 48: return u ? launch_tall_tc_t<48, true>(tmap, a, s) : launch_tall_tc_t<48, false>(tmap, a, s);
        case 64: return u ? launch_tall_tc_t<64, true>(tmap, a, s) : launch_tall_tc_t<64, false>(tmap, a, s);
        default: return cudaErrorInvalidValue;
    }
}

// Many problems of one MMA width in one launch, one block per work item (tsmm_group.cuh).
template <int W, bool U>
__global__ void __launch_bounds__(TallTcCfg<W, U>::THREADS, 2)
    tall_tc_grouped_kernel(const __grid_constant__ GroupParams gp) {
    const int64_t item = blockIdx.x;
    const int p = group_find(gp, item);
    const TallArgs &a = gp.p[p].a;
    int64_t slab, split;
    udivmod(item - gp.p[p].item_begin, a.splits, slab, split);
    tall_tc_block<W, U>(&gp.p[p].tmA, a, slab, (int)split);
}

template <int W, bool U>
static cudaError_t launch_grouped_tc_t(const GroupParams &gp, cudaStream_t s) {
    using Cfg = TallTcCfg<W, U>;
    const cudaError_t e = ensure_smem_limit(reinterpret_cast<const void *>(tall_tc_grouped_kernel<W, U>), Cfg::SMEM);
    if (e != cudaSuccess) return e;
    if (gp.total_items <= 0) return cudaSuccess;
    if (gp.total_items > INT_MAX) return cudaErrorInvalidValue;
    tall_tc_grouped_kernel<W, U><<<(unsigned)gp.total_items, Cfg::THREADS, Cfg::SMEM, s>>>(gp);
    return cudaGetLastError();
}

cudaError_t launch_grouped_tc(int width, bool unaligned, const GroupParams &gp, cudaStream_t s) {
    switch (width) {
        case 32: return unaligned ? launch_grouped_tc_t<32, true>(gp, s) : launch_grouped_tc_t<32, false>(gp, s);
        case 48: return unaligned ? launch_grouped_tc_t<48, true>(gp, s) : launch_grouped_tc_t<48, false>(gp, s);
        case 64: return unaligned ? launch_grouped_tc_t<64, true>(gp, s) : launch_grouped_tc_t<64, false>(gp, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace tsmm
