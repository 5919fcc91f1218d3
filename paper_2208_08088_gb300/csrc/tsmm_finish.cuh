// The split-K finish of the tensor-core regime (i) kernels: the last block of a slab adds the S partial tiles.
#pragma once
#include "tsmm_device.cuh"
#include "tsmm_internal.h"

namespace tsmm {

// C = alpha * sum + beta * C0 over the slab's rows [i0, i0 + kTcRows), the partials summed in the fixed order
// s = 0..S-1.  Thread t of THREADS takes 16 bytes of rows of one column at a time; the loads of 8 splits are in flight
// together, since the sum is otherwise a chain of L2 latencies.
template <typename T, int THREADS>
__device__ __forceinline__ void tc_finish(const TallArgs &a, int64_t i0, int t) {
    constexpr int V = 16 / (int)sizeof(T), PER = kTcRows / V;
    const T alpha = static_cast<T>(a.alpha), beta = static_cast<T>(a.beta);
    const int64_t mpad = a.slabs * kTcRows, step = (int64_t)a.np * mpad;
    const T *ws = static_cast<const T *>(a.ws) + i0;
    for (int v = t; v < (int)a.n * PER; v += THREADS) {
        const int j = v / PER, r = v % PER * V;
        const int64_t rows = a.m - (i0 + r);
        if (rows <= 0) continue;
        const T *src = ws + (int64_t)j * mpad + r;
        Vec<T, V> s;
#pragma unroll
        for (int u = 0; u < V; ++u) s.v[u] = T(0);
        sum_partials(s, src, step, a.splits);
        T *c = static_cast<T *>(a.C) + i0 + r + (int64_t)j * a.ldc;
        if (rows >= V && reinterpret_cast<uintptr_t>(c) % 16 == 0) {
            Vec<T, V> o;
            if (beta != T(0)) o = ld_vec<T, V>(c);
#pragma unroll
            for (int u = 0; u < V; ++u) {
                const T x = alpha * s.v[u];
                o.v[u] = beta != T(0) ? fma(beta, o.v[u], x) : x;
            }
            st_vec<T, V>(c, o);
        } else {
#pragma unroll
            for (int u = 0; u < V; ++u)
                if (u < rows) {
                    const T x = alpha * s.v[u];
                    c[u] = beta != T(0) ? fma(beta, c[u], x) : x;
                }
        }
    }
}

}  // namespace tsmm
