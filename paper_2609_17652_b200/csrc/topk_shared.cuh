// Order-preserving integer image of the fp32 score, shared by the top-k kernels.
#pragma once
#include "fathom_common.cuh"

__device__ __forceinline__ uint32_t ordered_key(float f) {
  uint32_t u = __float_as_uint(f);
  if ((u << 1) == 0u) u = 0u;                                // -0 -> +0
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// fp32 value whose ordered key is `key` (the inverse of ordered_key for non-NaN patterns)
__device__ __forceinline__ float key_to_float(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key);
}
// Lower edge of a histogram bin as a score: the bins below -inf's (no finite score lies there) stand for "every score",
// a bin past the last for "none" (a comparison with NaN is false).
__device__ __forceinline__ float edge_of_bin(uint32_t bin) {
  return bin >= FATHOM_TOPK_BINS ? __uint_as_float(0x7fc00000u) : (bin <= 7u ? -INFINITY : key_to_float(bin << 20));
}

struct Forced { long long sink_end, local_begin; };          // eligible tokens: sink_end <= i < local_begin

// Rows that a cluster of CTAs can hold in registers (topk_resident.cu)
constexpr long long FATHOM_TOPK_RESIDENT_MAX = 131072;
int fathom_topk_resident_ctas(long long n, int Hq, uint32_t want);          // CTAs per head
int fathom_launch_topk_resident(fathom_ctx* ctx, const float* scores, long long n, long long score_stride, int Hq, int k, Forced F,
                                uint32_t want, int32_t* idx, cudaStream_t st);
