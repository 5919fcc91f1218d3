// Signed 8-bit digits of FP64 values as FP16 pairs, and the accumulator reads, of the FP64 tensor-core kernels.
#pragma once
#include "tsmm_internal.h"
#include "tsmm_tc.cuh"

namespace tsmm {

// CB (4 or 8) columns at each of N places, `step` apart, of this thread's lane.
template <int N, int CB>
__device__ __forceinline__ void tc_ldn(uint32_t taddr, uint32_t step, uint32_t (*r)[CB]) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        if constexpr (CB == 8)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(r[i][0]), "=r"(r[i][1]), "=r"(r[i][2]), "=r"(r[i][3]), "=r"(r[i][4]), "=r"(r[i][5]),
                           "=r"(r[i][6]), "=r"(r[i][7])
                         : "r"(taddr + i * step)
                         : "memory");
        else
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(r[i][0]), "=r"(r[i][1]), "=r"(r[i][2]), "=r"(r[i][3])
                         : "r"(taddr + i * step)
                         : "memory");
    }
    // the values pass through the wait, so no use can move above it
#pragma unroll
    for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < CB; j += 4)
            asm volatile("tcgen05.wait::ld.sync.aligned;"
                         : "+r"(r[i][j]), "+r"(r[i][j + 1]), "+r"(r[i][j + 2]), "+r"(r[i][j + 3])::"memory");
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
__device__ __forceinline__ uint32_t hfma2(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

// |x|'s high word with a bit set below the exponent field, so that tc64_shift is exact for powers of two.
__device__ __forceinline__ uint32_t tc64_abs(uint32_t hi) { return (hi & 0x7fffffffu) | 1u; }
// E - (exponent field): -(ah * 4096 >> 32) = -(field) - 1 in one multiply-add, off the ALU that the rest keeps busy.
__device__ __forceinline__ int tc64_shift(uint32_t ah, int E) {
    int s;
    asm("mad.hi.s32 %0, %1, %2, %3;" : "=r"(s) : "r"(ah), "r"(-4096), "r"(E + 1));
    return s;
}
// Fixed point of |x| (hi, lo: its words) under the shift s >= 0 of its exponent field to the scale, with 0x80 added to
// the six low bytes (digits 1..6 are then byte - 128, digit 0 is byte 6).
__device__ __forceinline__ uint64_t tc64_fixed(uint32_t hi, uint32_t lo, int s) {
    uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 2;
    asm("shr.b64 %0, %0, %1;" : "+l"(m) : "r"(s));  // a count above 63 gives 0
    return m + 0x0000808080808080ull;
}
// A pair's signs as FP16 +-1.
__device__ __forceinline__ uint32_t tc64_sign2(uint32_t hi0, uint32_t hi1) {
    return (prmt(hi0, hi1, 0x7030) & 0x80008000u) | 0x3c003c00u;
}
constexpr uint32_t kH1152 = 0xe480e480u;  // FP16 -1152, twice
constexpr uint32_t kH1024 = 0xe400e400u;  // FP16 -1024, twice
// Digits b and b + 1 (bytes of the words y0, y1 of a pair) as FP16 pairs: FP16 0x6400 | byte is 1024 + byte.
__device__ __forceinline__ void tc64_digits2(uint32_t y0, uint32_t y1, uint32_t sel, uint32_t sgn, uint32_t c0,
                                             uint32_t c1, uint32_t &d0, uint32_t &d1) {
    const uint32_t p = prmt(y0, y1, sel);
    d0 = hfma2(prmt(p, 0x64646464u, 0x4140), sgn, c0);
    d1 = hfma2(prmt(p, 0x64646464u, 0x4342), sgn, c1);
}
// Eight digits of a pair (x0, x1) under the scale F (exponent field of the largest entry): 63 bits below it, 0x80 added
// to the seven low bytes.  Returns the pair's top 7 bits of magnitude as bytes.
__device__ __forceinline__ uint32_t tc64_digits8(double x0, double x1, int F, uint32_t (&d)[8]) {
    uint32_t y0[2], y1[2], g = 0u;
    const uint32_t hi[2] = {(uint32_t)__double2hiint(x0), (uint32_t)__double2hiint(x1)};
    const uint32_t lo[2] = {(uint32_t)__double2loint(x0), (uint32_t)__double2loint(x1)};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int s = tc64_shift(tc64_abs(hi[u]), F);
        uint64_t m = ((uint64_t)((hi[u] & 0xfffffu) | 0x100000u) << 32 | lo[u]) << 10;
        m = s > 63 ? 0ull : m >> (s < 0 ? 0 : s);
        g |= (uint32_t)(m >> 56) << (8 * u);
        const uint64_t y = m + 0x0080808080808080ull;
        y0[u] = (uint32_t)y;
        y1[u] = (uint32_t)(y >> 32);
    }
    const uint32_t sgn = tc64_sign2(hi[0], hi[1]);
    const uint32_t c = hfma2(sgn, kH1152, 0u);
    tc64_digits2(y0[0], y0[1], 0x5140, sgn, c, c, d[7], d[6]);
    tc64_digits2(y0[0], y0[1], 0x7362, sgn, c, c, d[5], d[4]);
    tc64_digits2(y1[0], y1[1], 0x5140, sgn, c, c, d[3], d[2]);
    tc64_digits2(y1[0], y1[1], 0x7362, sgn, c, hfma2(sgn, kH1024, 0u), d[1], d[0]);
    return g;
}

}  // namespace tsmm
