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

// ---- histograms in shared memory whose bins are also counted together, SUPER at a time, so that one warp finds a rank
constexpr int COARSE = 4096;
constexpr int SUPER = 32;

// Coarse bin of a score (monotone, -0 with +0) and its lower edge.  Magnitudes from 2^-16 to 2^16 have 32 bins per octave, the others
// four: with the same eight everywhere (the 12 leading key bits) a head whose threshold fell to the upper end of a bin had twice
// the candidates it wanted.
constexpr uint32_t MAG_LO = 111u << 23, MAG_HI = 143u << 23, MID0 = MAG_LO >> 21, HIGH0 = MID0 + ((MAG_HI - MAG_LO) >> 18);
constexpr uint32_t ZERO_BIN = 1920;
static_assert(HIGH0 + ((0x7f800000u - MAG_HI) >> 21) < ZERO_BIN && 2 * ZERO_BIN <= COARSE, "bins of both signs");
__device__ __forceinline__ uint32_t coarse_bin(float f) {
  const uint32_t u = __float_as_uint(f) & 0x7fffffffu;
  const uint32_t m = u < MAG_LO ? u >> 21 : (u < MAG_HI ? MID0 + ((u - MAG_LO) >> 18) : HIGH0 + ((u - MAG_HI) >> 21));
  return f < 0.0f ? ZERO_BIN - 1u - m : ZERO_BIN + m;
}
__device__ __forceinline__ float coarse_edge(uint32_t bin) {
  auto smallest = [](uint32_t m) {                            // magnitude bits
    return m < MID0 ? m << 21 : (m < HIGH0 ? MAG_LO + ((m - MID0) << 18) : MAG_HI + ((m - HIGH0) << 21));
  };
  if (bin >= ZERO_BIN) return __uint_as_float(smallest(bin - ZERO_BIN));
  const uint32_t u = smallest(ZERO_BIN - bin) - 1u;           // the largest magnitude of the bin
  return u >= 0x7f800000u ? -INFINITY : __uint_as_float(u | 0x80000000u);
}

// One warp: the largest bin whose suffix count reaches `rank` (> 0), the count above it and its own, in every lane.  If there are
// fewer than `rank`: bin 0 with everything.
template <int BINS>
__device__ __forceinline__ void search_bins(const uint32_t* bins, const uint32_t* super, uint32_t rank, uint32_t& bin, uint32_t& above, uint32_t& count) {
  constexpr int PER = BINS / SUPER / 32;                      // lane l owns super bins BINS / SUPER - 1 - PER l .. descending
  const int lane = threadIdx.x & 31;
  uint32_t c[PER], local = 0u;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    c[u] = super[BINS / SUPER - 1 - PER * lane - u];
    local += c[u];
  }
  auto inclusive = [&](uint32_t x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    return x;
  };
  uint32_t incl = inclusive(local);
  const unsigned reach = __ballot_sync(0xffffffffu, incl >= rank);
  if (reach == 0u) {
    bin = above = 0u;
    count = __shfl_sync(0xffffffffu, incl, 31);
    return;
  }
  uint32_t run = incl - local;
  int u = 0;
#pragma unroll
  for (int x = 0; x < PER - 1; ++x)
    if (u == x && run + c[x] < rank) { run += c[x]; u = x + 1; }
  const int from = __ffs(reach) - 1;
  run = __shfl_sync(0xffffffffu, run, from);
  u = __shfl_sync(0xffffffffu, u, from);
  const int first = (BINS / SUPER - 1 - PER * from - u) * SUPER;
  const uint32_t mine = bins[first + SUPER - 1 - lane];
  incl = run + inclusive(mine);
  const int at = __ffs(__ballot_sync(0xffffffffu, incl >= rank)) - 1;
  bin = (uint32_t)(first + SUPER - 1 - at);
  count = __shfl_sync(0xffffffffu, mine, at);
  above = __shfl_sync(0xffffffffu, incl, at) - count;
}

struct Forced { long long sink_end, local_begin; };          // eligible tokens: sink_end <= i < local_begin

// Rows that a cluster of CTAs can hold in registers (topk_resident.cu)
constexpr long long FATHOM_TOPK_RESIDENT_MAX = 131072;
int fathom_topk_resident_ctas(long long n, int Hq);           // CTAs per head
int fathom_launch_topk_resident(fathom_ctx* ctx, const float* scores, long long n, long long score_stride, int Hq, int k, Forced F,
                                uint32_t want, int32_t* idx, cudaStream_t st);
