// Top-k of rows of up to 131,072 scores in ONE kernel: a cluster of up to eight CTAs per head holds the row's keys in
// registers, so whatever the selection has to look at twice is not read twice, and nothing goes through global memory
// between its steps.  What bounded such rows was the chain of launches (histogram, filter, select and emission with a memset
// before them: 30 us for 32 heads of 33,001 scores; sample, collection and selection: 21 us at 131,072) and not the data.
//
// The order of a head's tokens is that of the 64-bit composite (key << 32 | ~token): larger score first, ties to the lower
// token.  The steps, with a cluster barrier after 1, 2 and 3:
//   1. coarse histogram (4096 bins, a thirty-second of an octave where scores usually lie) of the threads' MAXIMA: the bin that holds the want-th largest maximum is a
//      bound - at least `want` tokens reach its lower edge - and a close one: for want = q groups of EPT tokens a share
//      1 - (1 - q)^(1 / EPT) of the tokens reaches the want-th maximum.  Where `want` is most of the number of groups the
//      histogram is of all tokens instead.  Every CTA adds its non-empty bins (a few dozen) to the histograms of all others
//      through distributed shared memory and finds the bound for itself;
//   2. the tokens that reach the bound are listed in token order in every CTA's shared memory;
//   3. the cluster's first CTA pulls the lists, which makes one list in token order of little more than `want` members:
//      fine histogram (2048 bins of 2^13 keys from the bound on), the members of the bin that the threshold splits (a few
//      dozen) ranked against one another, and the chosen tokens written in ascending order by a prefix count.
// (A first form merged whole histograms in every CTA, 64 KB of distributed shared memory each, and exchanged the split bin
// and the counts as well: 8000 of 30,000 cycles went into the first merge alone, 21.5 us at 33,001 scores.)
// A list that would not fit (heavy ties) is not pulled: radix rounds of 11 bits over the composites, the digits' counts pushed
// like in step 1, decide the threshold, and every CTA writes its own tokens.
// The set is unique and the counts are integers: the result does not depend on any order of atomics.
#include "topk_shared.cuh"

#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace {

constexpr int RT_THREADS = 512;
constexpr int RT_WARPS = RT_THREADS / 32;
constexpr int MAX_CLUSTER = 8;
constexpr int COARSE = 4096;
constexpr int FINE = 2048, FINE_SHIFT = 13;
constexpr int SPLIT = 512;                                    // members of a split bin ranked by comparison

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

struct ResidentSmem {
  alignas(16) uint32_t mine[COARSE];                          // this CTA's counts; the selecting CTA's fine histogram; members of its split bin
  alignas(16) uint32_t merged[COARSE];                        // the cluster's
  uint32_t warp_sum[RT_WARPS];
  uint32_t cta_count[MAX_CLUSTER];                            // listed (later: chosen) tokens per CTA, pushed by each of them
  uint32_t found_bin, found_above, found_count, split_count;
  unsigned long long threshold;
  unsigned long long list[1];                                 // [capacity] composites
};
static_assert(SPLIT * 8 <= (COARSE - FINE) * 4, "the members of the split bin lie behind the fine histogram");

// Finds the largest of BINS bins whose suffix count reaches `rank` (> 0) and leaves bin, the count above it and its own count in M
// (all threads may read them afterwards).  If there are fewer than `rank`: bin 0 with everything.
template <int BINS>
__device__ __forceinline__ void find_bin(ResidentSmem& M, const uint32_t* hist, uint32_t rank) {
  constexpr int PER = BINS / RT_THREADS;                      // thread t owns bins BINS - 1 - PER t .. descending
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t c[PER], local = 0u;
#pragma unroll
  for (int v = 0; v < PER / 4; ++v) {
    const uint4 x = *reinterpret_cast<const uint4*>(hist + BINS - PER * tid - 4 * v - 4);
    c[4 * v] = x.w; c[4 * v + 1] = x.z; c[4 * v + 2] = x.y; c[4 * v + 3] = x.x;
    local += x.x + x.y + x.z + x.w;
  }
  uint32_t incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) M.warp_sum[warp] = incl;
  __syncthreads();
  uint32_t above = incl - local;
#pragma unroll
  for (int w = 0; w < RT_WARPS; ++w) above += w < warp ? M.warp_sum[w] : 0u;
  if (above < rank && above + local >= rank) {
    uint32_t run = above;
#pragma unroll
    for (int b = 0; b < PER; ++b) {
      if (run < rank && run + c[b] >= rank) {
        M.found_bin = (uint32_t)(BINS - 1 - (PER * tid + b));
        M.found_above = run;
        M.found_count = c[b];
      }
      run += c[b];
    }
  }
  if (tid == RT_THREADS - 1 && above + local < rank) { M.found_bin = 0u; M.found_above = 0u; M.found_count = above + local; }
  __syncthreads();
}

template <int EPT>
__global__ void __launch_bounds__(RT_THREADS, 2)
topk_resident_kernel(const float* scores, int n, long long score_stride, int elig_lo, int elig_hi, int k, uint32_t want,
                     int by_maxima, uint32_t capacity, int32_t* __restrict__ idx_out, uint32_t* __restrict__ dev_status) {
  extern __shared__ __align__(16) unsigned char resident_smem[];
  ResidentSmem& M = *reinterpret_cast<ResidentSmem*>(resident_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), head = blockIdx.x / ctas;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int b = tid; b < 2 * COARSE / 4; b += RT_THREADS) reinterpret_cast<uint4*>(M.mine)[b] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  auto cleared = cluster.barrier_arrive();                    // my histograms are clear (others will add to one of them)
  FATHOM_PDL_WAIT();                                          // the scores come from the previous kernel
  FATHOM_PDL_RELEASE();                                       // the attention that follows may become resident now

  // ---- my tokens: token(i) = wbase + 128 (i / 4) + 4 lane + i % 4: the warp's loads are runs of 512 bytes.  They are kept as scores
  //      and compared as scores (a key is only formed for the few that matter); NaN stands for a token that is not eligible
  constexpr int V = EPT / 4;
  const int wbase = (rank * RT_WARPS + warp) * 32 * EPT;      // n <= 131072
  const float* row = scores + (size_t)head * (size_t)score_stride;
  const float NONE = __uint_as_float(0x7fffffffu);
  auto token = [&](int i) { return wbase + 128 * (i >> 2) + 4 * lane + (i & 3); };
  float x[EPT];
  {
    const float* src = row + wbase + 4 * lane;                // (score_stride is a multiple of 4: a float4 stays inside the row)
    if (wbase + 32 * EPT <= n) {                              // (uniform over the warp)
#pragma unroll
      for (int v = 0; v < V; ++v) *reinterpret_cast<float4*>(x + 4 * v) = *reinterpret_cast<const float4*>(src + 128 * v);
    } else {
#pragma unroll
      for (int v = 0; v < V; ++v)
        *reinterpret_cast<float4*>(x + 4 * v) = token(4 * v) < n ? *reinterpret_cast<const float4*>(src + 128 * v) : make_float4(NONE, NONE, NONE, NONE);
    }
    if (wbase < elig_lo || wbase + 32 * EPT > elig_hi) {
#pragma unroll
      for (int i = 0; i < EPT; ++i)
        if (token(i) < elig_lo || token(i) >= elig_hi) x[i] = NONE;
    }
  }
  auto composite = [&](int i) { return ((unsigned long long)ordered_key(x[i]) << 32) | (uint32_t)~(uint32_t)token(i); };

  // the non-empty bins of my histogram are added to every CTA's merged one
  auto push = [&](int bins) {
    for (int b = tid; b < bins; b += RT_THREADS) {
      const uint32_t c = M.mine[b];
      if (c)
        for (int r = 0; r < ctas; ++r) atomicAdd(cluster.map_shared_rank(M.merged, r) + b, c);
    }
  };

  // ---- 1. a bound: its coarse bin
  if (by_maxima) {
    float m = x[0];
#pragma unroll
    for (int i = 1; i < EPT; ++i) m = fmaxf(m, x[i]);          // (a NaN is no maximum)
    if (m == m) atomicAdd(&M.mine[coarse_bin(m)], 1u);
  } else {
#pragma unroll
    for (int i = 0; i < EPT; ++i)
      if (x[i] == x[i]) atomicAdd(&M.mine[coarse_bin(x[i])], 1u);
  }
  __syncthreads();
  cluster.barrier_wait(std::move(cleared));                   // (everyone arrived long ago)
  push(COARSE);
  cluster.sync();
  uint32_t base = 0u;                                         // candidates are the scores from bound on, whose key is base
  float bound = NONE;                                         // (nothing wanted: none)
  if (want) {
    find_bin<COARSE>(M, M.merged, want);
    for (int b = tid; b < FINE; b += RT_THREADS) M.mine[b] = 0u;             // (everyone's counts have been pushed)
    bound = M.found_bin == 0u ? -INFINITY : coarse_edge(M.found_bin);       // (bin 0: everything, see find_bin)
    base = ordered_key(bound);
  }

  // ---- places of a set of my tokens (bit i of `set`) among the CTA's, in token order: the counts of a lane's 4-token runs are
  //      prefix-summed over the warp four runs at a time (a byte each: at most 128), run totals and warp totals added
  auto place = [&](uint32_t set, uint32_t (&at)[V]) -> uint32_t {
    uint32_t total = 0u;
#pragma unroll
    for (int g = 0; g < (V + 3) / 4; ++g) {
      uint32_t c = 0u;
#pragma unroll
      for (int v = 4 * g; v < 4 * g + 4 && v < V; ++v) c |= (uint32_t)__popc((set >> (4 * v)) & 15u) << (8 * (v - 4 * g));
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const uint32_t last = __shfl_sync(0xffffffffu, incl, 31), before = incl - c;
#pragma unroll
      for (int v = 4 * g; v < 4 * g + 4 && v < V; ++v) {
        at[v] = total + ((before >> (8 * (v - 4 * g))) & 255u);
        total += (last >> (8 * (v - 4 * g))) & 255u;
      }
    }
    __syncthreads();                                          // (warp_sum may still be read)
    if (lane == 0) M.warp_sum[warp] = total;
    __syncthreads();
    uint32_t ahead = 0u, all = 0u;
#pragma unroll
    for (int w = 0; w < RT_WARPS; ++w) {
      const uint32_t s = M.warp_sum[w];
      ahead += w < warp ? s : 0u;
      all += s;
    }
#pragma unroll
    for (int v = 0; v < V; ++v) at[v] += ahead;
    return all;
  };

  // ---- 2. the tokens that reach the bound
  uint32_t set = 0u, at[V];
#pragma unroll
  for (int i = 0; i < EPT; ++i) set |= (x[i] >= bound ? 1u : 0u) << i;
  const uint32_t listed = place(set, at);
  if (listed <= capacity) {                                   // (uniform) as (score, token) pairs: keys are formed by the CTA that selects
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if ((set >> (4 * v)) & 15u) {
        uint2* to = reinterpret_cast<uint2*>(M.list) + at[v];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if ((set >> (4 * v + c)) & 1u) *to++ = make_uint2(__float_as_uint(x[4 * v + c]), (uint32_t)token(4 * v + c));
      }
    }
  }
  if (tid < ctas) cluster.map_shared_rank(M.cta_count, tid)[rank] = listed;
  cluster.sync();
  uint32_t total = 0u;
  for (int r = 0; r < ctas; ++r) total += M.cta_count[r];
  int32_t* out = idx_out + (size_t)head * k;
  const uint32_t n_sink = (uint32_t)elig_lo, n_local = (uint32_t)(n - elig_hi);

  if (total <= capacity) {                                    // (the same for the whole cluster)
    auto fine = [&](uint32_t key) { return min((key - base) >> FINE_SHIFT, (uint32_t)(FINE - 1)); };
    // ---- 3. the first CTA selects
    if (rank == 0) {
      uint32_t start[MAX_CLUSTER];                            // where each CTA's list starts in the joint one
      start[0] = 0u;
#pragma unroll
      for (int r = 1; r < MAX_CLUSTER; ++r) start[r] = start[r - 1] + (r - 1 < ctas ? M.cta_count[r - 1] : 0u);
      for (uint32_t e0 = 0u; e0 < total; e0 += RT_THREADS * 8) {
        uint2 c[8];                                           // eight loads in flight
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint32_t e = e0 + u * RT_THREADS + tid;
          if (e < total) {
            int r = 0;
            uint32_t s = 0u;
#pragma unroll
            for (int y = 1; y < MAX_CLUSTER; ++y)
              if (y < ctas && e >= start[y]) { r = y; s = start[y]; }
            c[u] = reinterpret_cast<const uint2*>(cluster.map_shared_rank(M.list, r))[e - s];
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint32_t e = e0 + u * RT_THREADS + tid;
          if (e < total) {
            const uint32_t key = ordered_key(__uint_as_float(c[u].x));
            M.list[e] = ((unsigned long long)key << 32) | (uint32_t)~c[u].y;
            atomicAdd(&M.mine[fine(key)], 1u);
          }
        }
      }
      if (tid == 0) M.split_count = 0u;
    }
    auto pulled = cluster.barrier_arrive();
    if (rank != 0) {
      cluster.barrier_wait(std::move(pulled));
      return;
    }
    __syncthreads();
    unsigned long long T = 0ull;                              // fewer than wanted (non-finite scores), or just as many: all of them
    if (total > want) {
      find_bin<FINE>(M, M.mine, want);
      const uint32_t bin = M.found_bin, members = M.found_count, need = want - M.found_above;
      T = (unsigned long long)(base + (bin << FINE_SHIFT)) << 32;
      if (need != members) {                                  // the bin is split: its members are ranked
        unsigned long long* split = reinterpret_cast<unsigned long long*>(M.mine + FINE);
        if (members <= (uint32_t)SPLIT) {
#pragma unroll 4
          for (uint32_t e = tid; e < total; e += RT_THREADS) {
            const unsigned long long c = M.list[e];
            if (fine((uint32_t)(c >> 32)) == bin) split[atomicAdd(&M.split_count, 1u)] = c;
          }
          __syncthreads();
          for (uint32_t i = warp; i < members; i += RT_WARPS) {             // a warp per member, its lanes over the others
            const unsigned long long mine = split[i];
            uint32_t larger = 0u;
            for (uint32_t j = lane; j < members; j += 32) larger += split[j] > mine;
            larger = __reduce_add_sync(0xffffffffu, larger);
            if (lane == 0 && larger + 1u == need) M.threshold = mine;
          }
          __syncthreads();
          T = M.threshold;
        } else {                                              // ties in numbers: 11-bit digits of the members' composites
          unsigned long long prefix = 0ull;
          uint32_t left = need;
          for (int hi = 64; hi > 0;) {
            const int lo = hi > 11 ? hi - 11 : 0;
            for (int b = tid; b < FINE; b += RT_THREADS) M.mine[b] = 0u;
            __syncthreads();
            for (uint32_t e = tid; e < total; e += RT_THREADS) {
              const unsigned long long c = M.list[e];
              if (fine((uint32_t)(c >> 32)) == bin && (hi == 64 || (c >> hi) == (prefix >> hi))) atomicAdd(&M.mine[(uint32_t)(c >> lo) & ((1u << (hi - lo)) - 1u)], 1u);
            }
            __syncthreads();
            find_bin<FINE>(M, M.mine, left);
            prefix |= (unsigned long long)M.found_bin << lo;
            left -= M.found_above;
            const bool whole = left == M.found_count;
            __syncthreads();
            hi = lo;
            if (whole) break;
          }
          T = prefix;
        }
      }
    }
    // ---- ascending output: a warp takes a slice of the list, 32 entries at a time
    const uint32_t slice = ((total + RT_THREADS - 1) / RT_THREADS) * 32, s0 = warp * slice, s1 = min(total, s0 + slice);
    uint32_t count = 0u;
#pragma unroll 4
    for (uint32_t e = s0; e < s1; e += 32) count += __popc(__ballot_sync(0xffffffffu, e + lane < s1 && M.list[e + lane] >= T));
    if (lane == 0) M.warp_sum[warp] = count;
    __syncthreads();
    uint32_t pos = n_sink, chosen = 0u;
#pragma unroll
    for (int w = 0; w < RT_WARPS; ++w) {
      const uint32_t s = M.warp_sum[w];
      pos += w < warp ? s : 0u;
      chosen += s;
    }
#pragma unroll 4
    for (uint32_t e = s0; e < s1; e += 32) {
      const unsigned long long c = e + lane < s1 ? M.list[e + lane] : 0ull;
      const bool take = e + lane < s1 && c >= T;
      const unsigned b = __ballot_sync(0xffffffffu, take);
      if (take) out[pos + __popc(b & ((1u << lane) - 1u))] = (int32_t)~(uint32_t)c;
      pos += __popc(b);
    }
    for (uint32_t e = tid; e < n_sink; e += RT_THREADS) out[e] = (int32_t)e;
    for (uint32_t e = tid; e < n_local; e += RT_THREADS) out[n_sink + chosen + e] = (int32_t)(elig_hi + e);
    const uint32_t filled = n_sink + chosen + n_local;
    if (filled < (uint32_t)k) {                               // short selection (non-finite scores)
      if (tid == 0) atomicOr(dev_status, FATHOM_DEV_TOPK_SHORT);
      for (uint32_t e = filled + tid; e < (uint32_t)k; e += RT_THREADS) out[e] = n - 1;   // pad with the last token
    }
    cluster.barrier_wait(std::move(pulled));
    return;
  }

  // ---- more candidates than the list holds: 11-bit digits of their composites, over the whole cluster
  unsigned long long T = 0ull;
  uint32_t left = want;
  for (int hi = 64; hi > 0;) {
    const int lo = hi > 11 ? hi - 11 : 0;
    for (int b = tid; b < 2 * COARSE / 4; b += RT_THREADS) reinterpret_cast<uint4*>(M.mine)[b] = make_uint4(0u, 0u, 0u, 0u);
    cluster.sync();
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      const unsigned long long c = composite(i);
      if (x[i] >= bound && (hi == 64 || (c >> hi) == (T >> hi))) atomicAdd(&M.mine[(uint32_t)(c >> lo) & ((1u << (hi - lo)) - 1u)], 1u);
    }
    __syncthreads();
    push(FINE);
    cluster.sync();
    find_bin<FINE>(M, M.merged, left);
    T |= (unsigned long long)M.found_bin << lo;
    left -= M.found_above;
    const bool whole = left == M.found_count;
    __syncthreads();
    hi = lo;
    if (whole) break;
  }
  uint32_t chosen = 0u;                                       // bit i: token(i), forced or reaching T
#pragma unroll
  for (int i = 0; i < EPT; ++i) {
    const int t = token(i);
    const bool forced = t < n && (t < elig_lo || t >= elig_hi);
    chosen |= (forced || (x[i] >= bound && composite(i) >= T) ? 1u : 0u) << i;
  }
  const uint32_t own = place(chosen, at);
  if (tid < ctas) cluster.map_shared_rank(M.cta_count, tid)[rank] = own;
  cluster.sync();                                             // (nobody touches another CTA's shared memory after this)
  uint32_t ahead = 0u;
  for (int r = 0; r < rank; ++r) ahead += M.cta_count[r];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    uint32_t pos = ahead + at[v];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if ((chosen >> (4 * v + c)) & 1u) {
        if (pos < (uint32_t)k) out[pos] = token(4 * v + c);
        ++pos;
      }
  }
}

template <int EPT>
cudaError_t launch(const float* scores, long long n, long long score_stride, int Hq, int k, Forced F, uint32_t want, int32_t* idx,
                   uint32_t* dev_status, int ctas, cudaStream_t st) {
  // room for twice what is wanted (the bound lets through 1.05 to 1.5 times), up to 16,384: 164 KB, one CTA per SM; two fit on an SM
  // up to about 10,000
  const uint32_t room = 2u * want < 2048u ? 2048u : 2u * want;
  const uint32_t capacity = room < 16384u ? room : 16384u;
  const size_t smem = sizeof(ResidentSmem) + (size_t)capacity * 8;
  static bool configured[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    e = cudaFuncSetAttribute(topk_resident_kernel<EPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(ResidentSmem) + 16384 * 8));
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(Hq * ctas));
  cfg.blockDim = dim3(RT_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)ctas;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  // maxima bound the threshold closely while `want` leaves a quarter of the groups below it
  const int by_maxima = 4LL * want <= 3LL * (n / EPT) ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, topk_resident_kernel<EPT>, scores, (int)n, score_stride, (int)F.sink_end, (int)F.local_begin, k, want,
                            by_maxima, capacity, idx, dev_status);
}

}  // namespace

// as few tokens per thread as eight CTAs allow (at least 8: more CTAs cost barrier time), then as few CTAs as hold the row
static int tokens_per_thread(long long n) {
  const long long per_cta8 = RT_THREADS * 8;
  return n <= MAX_CLUSTER * per_cta8 ? 8 : (n <= 2 * MAX_CLUSTER * per_cta8 ? 16 : 32);
}
int fathom_topk_resident_ctas(long long n) {
  int ctas = 1;
  while ((long long)ctas * RT_THREADS * tokens_per_thread(n) < n) ctas *= 2;
  return ctas;
}

int fathom_launch_topk_resident(fathom_ctx* ctx, const float* scores, long long n, long long score_stride, int Hq, int k, Forced F,
                                uint32_t want, int32_t* idx, cudaStream_t st) {
  const int ept = tokens_per_thread(n), ctas = fathom_topk_resident_ctas(n);
  cudaError_t e;
  if (ept == 8) e = launch<8>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, ctas, st);
  else if (ept == 16) e = launch<16>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, ctas, st);
  else e = launch<32>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, ctas, st);
  FATHOM_CUDA_TRY(ctx, e);
  return FATHOM_OK;
}
