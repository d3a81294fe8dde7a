// fathom_alloc_depth: per-plan read depths (Sec. 3.3, Eq. 3 and Eq. 4; fixed-channel rule of Sec. 2).
//
// Eq. 4 at the smallest water line that fits the budget grants exactly the min(B, 4d) candidate planes
// (channel j, plane m = 1..4) with the largest priority g_j 4^-m, so a candidate is granted when fewer than
// B others rank before it (ties: lower channel, then lower plane).  The importances are formed in fp64 with explicit
// round-to-nearest intrinsics and no fused multiply-add, so the ranking is identical on every machine; no logarithm is evaluated.
//
// Two channels are compared once for all their planes: non-negative doubles order like their bit patterns, dividing by 4 takes 2^53 off
// the pattern, so with D = pattern(g_i) - pattern(g_j) the planes of i that rank before (j, m) are those up to m + floor(D / 2^53)
// (D - 1 where j wins ties).  (Products and sums of squares of fp32 numbers are far from fp64's subnormals, so the quarters are exact.)
// Infinite and NaN importances rank before all finite ones, by their patterns and then by channel, all planes of a channel together (their
// quarters are no smaller).
// A warp per channel j, four channels i per lane, the four planes' counts summed by two warp reductions of packed halves.
// Eight CTAs serve a plan, 16 channels each; every CTA computes all 128 importances (thread = channel).  The kernel is a latency chain: it
// compared each of the 512 candidates with all others before, eight threads per candidate (back to back: one plan 2.9 -> 1.4 us, 8 plans 3.1 -> 1.6, 32 plans 6.8 -> 2.0).
#include "fathom_common.cuh"

namespace {

constexpr int CTAS_PER_PLAN = 8;
constexpr int AD_CHANNELS = FATHOM_D / CTAS_PER_PLAN;        // 16 channels ranked per CTA, a warp each
constexpr int AD_THREADS = 32 * AD_CHANNELS;                 // 512
constexpr long long FIRST_NONFINITE = 928LL << 52;           // where the patterns of infinity and NaN are moved to

// Bit pattern without its sign.  (The sign is taken off an integer in which the compiler does not see a double: it would make that a floating-point
// absolute value, which leaves a NaN its sign.)
__device__ __forceinline__ long long magnitude(double x) {
  long long b;
  asm("mov.b64 %0, %1;" : "=l"(b) : "d"(x));
  return b & 0x7fffffffffffffffLL;
}

__global__ void __launch_bounds__(AD_THREADS)
alloc_depth_kernel(const float* q, const float* var, int mode, int budget,
                   int heads_per_plan, int G, uint8_t* __restrict__ depth) {
  __shared__ long long order[FATHOM_D];                       // bit patterns of the (non-negative) importances
  FATHOM_PDL_WAIT();
  FATHOM_PDL_RELEASE();                                       // the scan that follows may become resident now
  const int plan = blockIdx.x / CTAS_PER_PLAN, part = blockIdx.x % CTAS_PER_PLAN;
  const int tid = threadIdx.x;
  const int h0 = plan * heads_per_plan;
  const int kv = h0 / G;
  uint8_t* out = depth + (size_t)plan * FATHOM_D;

  if (mode == FATHOM_DEPTH_UNIFORM) {
    if (part == 0 && tid < FATHOM_D) out[tid] = (uint8_t)min(max(budget, 0), FATHOM_NPLANES);
    return;
  }

  if (tid < FATHOM_D) {                                       // thread = channel
    const int j = tid;
    double acc = 0.0;
    const float* qj = q + (size_t)h0 * FATHOM_D + j;
    auto add_heads = [&](auto term) {                         // ascending order; up to four loads in flight
      int h = 0;
      for (; h + 4 <= heads_per_plan; h += 4) {
        float x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = qj[(h + u) * FATHOM_D];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = __dadd_rn(acc, term((double)x[u]));
      }
      for (; h < heads_per_plan; ++h) acc = __dadd_rn(acc, term((double)qj[h * FATHOM_D]));
    };
    if (mode == FATHOM_DEPTH_WATERFILL) {
      const float v = var[(size_t)kv * FATHOM_D + j];
      add_heads([](double x) { return __dmul_rn(x, x); });    // Eq. 3
      const long long g = magnitude(__dmul_rn(acc, (double)v));
      // Patterns of the products of finite fp32 numbers have exponents from 576 to 1420; 512 less, they leave room for channels of no
      // importance below: so far apart that all planes of one rank before all planes of the next.  The other patterns are moved to where
      // no plane of a finite channel comes near them and no difference overflows
      const long long low = -((long long)(j + 1) << 55), nonfinite = 2047LL << 52;
      order[j] = g == 0 ? low : (g < nonfinite ? g - (512LL << 52) : g - nonfinite + FIRST_NONFINITE);
    } else {                                                  // fixed top-r channels by sum_h |q_j|
      add_heads([](double x) { return fabs(x); });
      order[j] = magnitude(acc);
    }
  }
  __syncthreads();

  const int lane = tid & 31, j = part * AD_CHANNELS + (tid >> 5);
  const long long mine = order[j];
  if (mode == FATHOM_DEPTH_WATERFILL) {
    uint32_t before12 = 0u, before34 = 0u;                    // candidates that rank before planes 1 and 2, 3 and 4 of channel j
#pragma unroll
    for (int u = 0; u < FATHOM_D / 32; ++u) {
      const int i = lane + 32 * u;
      const long long d = order[i] - mine - (i < j ? 0 : 1);
      int e = (int)(d >> 53);                                 // (i = j: the planes above m)
      if (mine >= FIRST_NONFINITE && i != j) e = d >= 0 ? FATHOM_NPLANES : -FATHOM_NPLANES;       // (uniform over the warp)
      auto planes = [&](int m) { return (uint32_t)min(max(m + e, 0), FATHOM_NPLANES); };
      before12 += planes(1) | planes(2) << 16;
      before34 += planes(3) | planes(4) << 16;
    }
    before12 = __reduce_add_sync(0xffffffffu, before12);      // (at most 512 each)
    before34 = __reduce_add_sync(0xffffffffu, before34);
    if (lane == 0) {
      const uint32_t b = (uint32_t)budget;
      out[j] = (uint8_t)(((before12 & 0xffffu) < b) + ((before12 >> 16) < b) + ((before34 & 0xffffu) < b) + ((before34 >> 16) < b));
    }
  } else {
    uint32_t before = 0u;
#pragma unroll
    for (int u = 0; u < FATHOM_D / 32; ++u) {
      const int i = lane + 32 * u;
      before += order[i] > mine || (order[i] == mine && i < j);
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) out[j] = before < (uint32_t)budget ? FATHOM_NPLANES : 0;  // all four planes of a chosen channel
  }
}

}  // namespace

extern "C" int fathom_alloc_depth(fathom_ctx* ctx, const fathom_layout* L, const float* q, const float* var,
                                  int mode, int budget, int heads_per_plan, uint8_t* depth, void* stream) {
  if (!ctx || !q || !depth) return FATHOM_ERR_INVALID_ARG;
  int rc = fathom_check_layout(L);
  if (rc != FATHOM_OK) return rc;
  if (mode != FATHOM_DEPTH_WATERFILL && mode != FATHOM_DEPTH_FIXED_TOP_R && mode != FATHOM_DEPTH_UNIFORM)
    return FATHOM_ERR_UNSUPPORTED;
  if (mode == FATHOM_DEPTH_WATERFILL && !var) return FATHOM_ERR_INVALID_ARG;
  if (budget < 0) return FATHOM_ERR_INVALID_ARG;
  if (mode == FATHOM_DEPTH_UNIFORM && budget > FATHOM_NPLANES) return FATHOM_ERR_INVALID_ARG;
  const int G = L->n_q_heads / L->n_kv_heads;
  if (heads_per_plan < 1 || G % heads_per_plan != 0) return FATHOM_ERR_INVALID_ARG;
  const int plans = L->n_q_heads / heads_per_plan;
  FATHOM_CUDA_TRY(ctx, fathom_launch_dependent(alloc_depth_kernel, dim3(plans * CTAS_PER_PLAN), dim3(AD_THREADS), 0,
                                               static_cast<cudaStream_t>(stream), q, var, mode, budget, heads_per_plan, G, depth));
  return FATHOM_OK;
}
