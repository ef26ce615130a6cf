// umma_shape.cuh -- which tcgen05.mma a product of N columns takes, shared by the
// GEMM and a host-side check (plain C++, no CUDA needed).
//
// kind::f16 exists for 128 rows and one CTA with N a multiple of 16, and for 256
// rows and a pair of CTAs (cta_group::2) with N a multiple of 32, up to 256.  A
// product of 16 more columns than such a multiple takes a pair's MMA of 16 further
// columns: its B rows past N lie outside the tensor map and read as zero, its
// columns past N stay in tensor memory.
#pragma once

#ifndef __CUDACC__
#ifndef __host__
#define __host__
#endif
#ifndef __device__
#define __device__
#endif
#ifndef __forceinline__
#define __forceinline__ inline
#endif
#endif

// columns above which a pair of CTAs takes a tile: it costs a launch 2 us (cluster
// barriers) and pays where B's traffic counts (16000 x 32000: N 256 220 -> 203
// us, 192 205 -> 196, 128 189 -> 183; 6016 x 12032 x 128 in a solve 31.8 -> 33.5)
constexpr int UM_PAIR_N = 128;

// CTAs per tile of a product of n columns
__host__ __device__ __forceinline__ constexpr int umma_ctas(int n) { return n > UM_PAIR_N ? 2 : 1; }
// columns of its MMA
__host__ __device__ __forceinline__ constexpr int umma_cols(int n) {
    return umma_ctas(n) == 2 ? (n + 31) / 32 * 32 : n;
}
// B rows that each CTA of the tile loads (its box of the tensor map)
__host__ __device__ __forceinline__ constexpr int umma_b_rows(int n) { return umma_cols(n) / umma_ctas(n); }
// tensor-memory columns of one accumulator
__host__ __device__ __forceinline__ constexpr int umma_acc_cols(int n) {
    int c = 32;
    while (c < umma_cols(n)) c *= 2;
    return c;
}
