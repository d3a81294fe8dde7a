// Top-k of rows of up to 131,072 scores in ONE kernel: a cluster of up to eight CTAs per head holds the row's scores in
// registers, so whatever the selection has to look at twice is not read twice, and nothing goes through global memory
// between its steps.  What bounds such rows is not the data but the instructions that every warp executes once, at some nine
// cycles each: 512 threads share out a few hundred candidates.  So a step takes as few instructions per warp as possible (a search
// by one warp over two levels of counts, lists of tokens instead of places computed for every score, one candidate per thread from
// then on).
//
// The order of a head's tokens is that of the 64-bit composite (key << 32 | ~token): larger score first, ties to the lower
// token.  The row is dealt to the CTAs in chunks of 128 tokens, one after the other, so that every CTA holds a sample of the
// whole row.  There is ONE exchange:
//   1. coarse histogram (4096 bins, a thirty-second of an octave where scores usually lie) of the maxima of the threads' groups of
//      tokens, in the CTA's own shared memory: its own bound is the bin that holds the quota-th largest maximum, the quota being its
//      share of `want` and four standard deviations more;
//   2. the tokens that reach the CTA's bound are listed, and list, length and bound are written to every CTA of the cluster.  (Where
//      the large scores lie side by side too many tokens reach what bounds their groups; the bound is then taken from the tokens);
//   3. after the cluster barrier every CTA finds the want-th largest of all lists: fine histogram (2048 bins of 2^13 keys from the
//      lowest bound on), the members of the bin that the threshold splits (a few) ranked against one another.  A threshold
//      that reaches every CTA's bound is exact: all lists are complete down to it.  One that does not is still a bound of the whole
//      row (`want` tokens reach it), and the lists are made once more with it;
//   4. every CTA marks the chosen tokens of all lists in a bitmap of the row, whose prefix counts give its own list's tokens their
//      places in the ascending output.
// (A first form merged whole histograms in every CTA; a second one merged those of the maxima and let the first CTA pull the lists,
// select and write alone: three cluster barriers, and seven of eight CTAs idle for 40 % of the time.  32 heads, back to back, second
// form / this one: 131,072 scores, k = 2048 16.7 / 12.4 us; 65,536, k = 1024 13.4 / 8.6; 33,001, k = 512 12.3 / 7.7; one head of 4096, k = 64 5.8 / 4.3.)
// A list that would not fit (heavy ties) is not copied: radix rounds of 11 bits over the composites, the digits' counts
// pushed to all CTAs, decide the threshold.
// The set is unique and the counts are integers: the result does not depend on any order of atomics.
#include "topk_shared.cuh"

#include <cooperative_groups.h>

#include <cstddef>

namespace cg = cooperative_groups;

namespace {

constexpr int RT_THREADS = 512;
constexpr int RT_WARPS = RT_THREADS / 32;
constexpr int MAX_CLUSTER = 8;
constexpr int FINE = 2048, FINE_SHIFT = 13;
constexpr int SPLIT = 512;                                    // members of a split bin ranked by comparison
constexpr int CHUNK = 128, MAX_CHUNKS = (int)(FATHOM_TOPK_RESIDENT_MAX / CHUNK);
constexpr int MOST_LISTED = 16384;                            // over all lists of a cluster of several CTAs

struct ResidentSmem {
  alignas(16) uint32_t coarse[COARSE];                        // counts of this CTA's maxima; then members of the split bin and places of the chunks,
                                                              // or the digits' counts, this CTA's and the cluster's
  uint32_t coarse_super[COARSE / SUPER];
  uint32_t fine[FINE];                                        // counts of the lists
  uint32_t fine_super[FINE / SUPER];
  alignas(16) uint32_t warp_sum[RT_WARPS];
  uint2 seg[MAX_CLUSTER];                                     // length and bound of every CTA's list, written by each of them
  uint32_t listed, found_bin, found_above, found_count, split_count;
  unsigned long long threshold;
  alignas(16) unsigned long long list[1];                     // [ctas][capacity] composites, [capacity] tokens of this CTA's list, [chunks] uint4 of
                                                              // chosen tokens of the whole row
};
constexpr int COUNTS = COARSE + COARSE / SUPER + FINE + FINE / SUPER;
static_assert(offsetof(ResidentSmem, warp_sum) == COUNTS * 4 && COUNTS % 4 == 0, "the counts lie side by side");
static_assert(SPLIT * 8 + MAX_CHUNKS * 4 <= COARSE * 4, "the split bin and the places fit over the coarse counts");

// All threads of the CTA, after a barrier that completes the counts: what search_bins finds, in M (with a barrier behind it).
template <int BINS>
__device__ __forceinline__ void find_bin(ResidentSmem& M, const uint32_t* bins, const uint32_t* super, uint32_t rank) {
  if (threadIdx.x < 32) {
    uint32_t bin, above, count;
    search_bins<BINS>(bins, super, rank, bin, above, count);
    if (threadIdx.x == 0) { M.found_bin = bin; M.found_above = above; M.found_count = count; }
  }
  __syncthreads();
}

// groups: 1 = one group of tokens per thread, 2 = two, 4 = one per four tokens, 0 = every token a group
template <int EPT>
__global__ void __launch_bounds__(RT_THREADS, 2)
topk_resident_kernel(const float* scores, int n, long long score_stride, int elig_lo, int elig_hi, int k, uint32_t want, uint32_t quota,
                     int groups, uint32_t capacity, int32_t* __restrict__ idx_out, uint32_t* __restrict__ dev_status) {
  extern __shared__ __align__(16) unsigned char resident_smem[];
  ResidentSmem& M = *reinterpret_cast<ResidentSmem*>(resident_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int ctas = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), head = blockIdx.x / ctas;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto started = cluster.barrier_arrive();                    // (nothing is written to a CTA's shared memory before it runs)
  const int chunks = (n + CHUNK - 1) / CHUNK;
  uint32_t* own = reinterpret_cast<uint32_t*>(M.list + (size_t)ctas * capacity);             // (capacity is a multiple of 4)
  uint4* bits = reinterpret_cast<uint4*>(own + capacity);
  unsigned long long* split = reinterpret_cast<unsigned long long*>(M.coarse);
  uint32_t* places = M.coarse + 2 * SPLIT;
  for (int b = tid; b < COUNTS / 4; b += RT_THREADS) reinterpret_cast<uint4*>(M.coarse)[b] = make_uint4(0u, 0u, 0u, 0u);
  for (int b = tid; b < chunks; b += RT_THREADS) bits[b] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) M.listed = M.split_count = 0u;
  __syncthreads();
  FATHOM_PDL_WAIT();                                          // the scores come from the previous kernel
  FATHOM_PDL_RELEASE();                                       // the attention that follows may become resident now

  // ---- my tokens: chunks warp ctas + rank, RT_WARPS ctas further on, .. of the row, 4 consecutive ones per lane.  They are kept as
  //      scores and compared as scores (a key is only formed for the few that matter); NaN stands for a token that is not eligible
  constexpr int V = EPT / 4;
  const int chunk0 = warp * ctas + rank, chunk_step = RT_WARPS * ctas;        // n <= 131072
  const float* row = scores + (size_t)head * (size_t)score_stride;
  const float NONE = __uint_as_float(0x7fffffffu);
  auto token = [&](int i) { return (chunk0 + (i >> 2) * chunk_step) * CHUNK + 4 * lane + (i & 3); };
  float x[EPT];
#pragma unroll
  for (int v = 0; v < V; ++v)                                 // (score_stride is a multiple of 4: a float4 stays inside the row)
    *reinterpret_cast<float4*>(x + 4 * v) = token(4 * v) < n ? *reinterpret_cast<const float4*>(row + token(4 * v)) : make_float4(NONE, NONE, NONE, NONE);
#pragma unroll
  for (int v = 0; v < V; ++v) {
    const int first = (chunk0 + v * chunk_step) * CHUNK;
    if (first < elig_lo || first + CHUNK > elig_hi) {         // (uniform over the warp)
#pragma unroll
      for (int i = 4 * v; i < 4 * v + 4; ++i)
        if (token(i) < elig_lo || token(i) >= elig_hi) x[i] = NONE;
    }
  }

  // ---- 1. my bound
  auto count = [&](float m) {
    if (m == m) {
      const uint32_t b = coarse_bin(m);
      atomicAdd(&M.coarse[b], 1u);
      atomicAdd(&M.coarse_super[b / SUPER], 1u);
    }
  };
  float bound = NONE;                                         // (nothing wanted: none)
  bool exact = false;                                         // the bound is as close as it gets
  bool fits = quota <= capacity;                              // (a quota that no list holds: straight to the radix rounds)
  if (want && fits) {
    auto largest = [&](int i0, int i1) {
      float m = x[i0];
#pragma unroll
      for (int i = i0 + 1; i < i1; ++i) m = fmaxf(m, x[i]);   // (a NaN is no maximum)
      return m;
    };
    if (groups == 1) {
      count(largest(0, EPT));
    } else if (groups == 2) {
      count(largest(0, EPT / 2));
      count(largest(EPT / 2, EPT));
    } else if (groups == 4) {
#pragma unroll
      for (int v = 0; v < V; ++v) count(largest(4 * v, 4 * v + 4));
    } else {
#pragma unroll
      for (int i = 0; i < EPT; ++i) count(x[i]);
    }
    __syncthreads();
    find_bin<COARSE>(M, M.coarse, M.coarse_super, quota);
    bound = M.found_bin == 0u ? -INFINITY : coarse_edge(M.found_bin);         // (bin 0: everything, see search_bins)
  }
  cluster.barrier_wait(std::move(started));                   // (everyone arrived long ago)

  // ---- every warp of a CTA works on one of the lists
  const int per_list = RT_WARPS / ctas, my_list = warp / per_list;            // (ctas is a power of two, at most 8)
  const uint32_t e_first = (uint32_t)(warp % per_list) * 32 + lane, e_step = (uint32_t)per_list * 32;
  const unsigned long long* mine = M.list + (size_t)my_list * capacity;

  unsigned long long T = 0ull;                                // the smallest composite that is selected
  float least = -INFINITY;                                    // no smaller score is selected
  while (fits) {
    // ---- 2. the tokens that reach the bound, in any order
    uint32_t listed;
    for (;;) {
      uint32_t set = 0u;
#pragma unroll
      for (int i = 0; i < EPT; ++i)
        if (x[i] >= bound) set |= 1u << i;
      if (set) {
        uint32_t at = atomicAdd(&M.listed, (uint32_t)__popc(set));
        do {
          const int i = __ffs(set) - 1;
          set &= set - 1u;
          if (at < capacity) own[at] = (uint32_t)token(i);
          ++at;
        } while (set);
      }
      __syncthreads();
      listed = M.listed;
      if (listed <= capacity || exact) break;                 // (the same for the whole CTA)
      // the large scores lie side by side, or in one bin: a bound that the quota of tokens, not of groups, reaches, to 2^10 keys
      exact = true;
      for (int b = tid; b < COARSE + COARSE / SUPER; b += RT_THREADS) M.coarse[b] = 0u;
      __syncthreads();
#pragma unroll
      for (int i = 0; i < EPT; ++i)
        if (x[i] >= bound) count(x[i]);
      __syncthreads();
      find_bin<COARSE>(M, M.coarse, M.coarse_super, quota);
      const uint32_t bin = M.found_bin, rest = quota - M.found_above;
      if (bin != 0u) {
        const uint32_t edge = ordered_key(coarse_edge(bin));
#pragma unroll
        for (int i = 0; i < EPT; ++i)
          if (x[i] >= bound && coarse_bin(x[i]) == bin) {
            const uint32_t b = min((ordered_key(x[i]) - edge) >> 10, (uint32_t)(FINE - 1));
            atomicAdd(&M.fine[b], 1u);
            atomicAdd(&M.fine_super[b / SUPER], 1u);
          }
        __syncthreads();                                      // (found_bin and found_above have been read, too)
        find_bin<FINE>(M, M.fine, M.fine_super, rest);
        bound = fmaxf(bound, key_to_float(edge + (M.found_bin << 10)));
      }
      for (int b = tid; b < FINE + FINE / SUPER; b += RT_THREADS) M.fine[b] = 0u;
      if (tid == 0) M.listed = 0u;
      __syncthreads();
    }
    if (listed <= capacity) {
      for (uint32_t e = tid; e < listed; e += RT_THREADS) {
        const uint32_t t = own[e];
        const unsigned long long c = ((unsigned long long)ordered_key(row[t]) << 32) | (uint32_t)~t;         // (the row's line is in the L1)
        unsigned long long* to = M.list + (size_t)rank * capacity + e;
#pragma unroll 1
        for (int r = 0; r < ctas; ++r) *cluster.map_shared_rank(to, r) = c;
      }
    }
    if (tid < ctas) *cluster.map_shared_rank(&M.seg[rank], tid) = make_uint2(listed, __float_as_uint(bound));
    if (ctas > 1) cluster.sync();
    else __syncthreads();

    // ---- 3. the want-th largest of all lists
    const uint2 theirs = lane < ctas ? M.seg[lane] : make_uint2(0u, __float_as_uint(bound));
    const uint32_t their_key = ordered_key(__uint_as_float(theirs.y));
    const uint32_t total = __reduce_add_sync(0xffffffffu, theirs.x);
    const uint32_t base = __reduce_min_sync(0xffffffffu, their_key), top = __reduce_max_sync(0xffffffffu, their_key);   // keys of the lowest and the highest bound
    const uint32_t count = __shfl_sync(0xffffffffu, theirs.x, my_list);
    fits = !__any_sync(0xffffffffu, theirs.x > capacity);
    if (total >= want) least = key_to_float(base);
    if (!fits || !want) break;                                // (the same for the whole cluster, like every other way out)
    T = 0ull;                                                 // fewer than wanted, or just as many: all of them
    if (total > want) {
      auto fine = [&](uint32_t key) { return min((key - base) >> FINE_SHIFT, (uint32_t)(FINE - 1)); };
      for (uint32_t e = e_first; e < count; e += e_step) {
        const uint32_t b = fine((uint32_t)(mine[e] >> 32));
        atomicAdd(&M.fine[b], 1u);
        atomicAdd(&M.fine_super[b / SUPER], 1u);
      }
      __syncthreads();
      find_bin<FINE>(M, M.fine, M.fine_super, want);
      const uint32_t bin = M.found_bin, members = M.found_count, need = want - M.found_above;
      T = (unsigned long long)(base + (bin << FINE_SHIFT)) << 32;
      if (need != members) {                                  // the bin is split: its members are ranked
        if (members <= (uint32_t)SPLIT) {
          for (uint32_t e = e_first; e < count; e += e_step) {
            const unsigned long long c = mine[e];
            if (fine((uint32_t)(c >> 32)) == bin) split[atomicAdd(&M.split_count, 1u)] = c;
          }
          __syncthreads();
          for (uint32_t i = warp; i < members; i += RT_WARPS) {               // a warp per member, its lanes over the others
            const unsigned long long c = split[i];
            uint32_t larger = 0u;
            for (uint32_t j = lane; j < members; j += 32) larger += split[j] > c;
            larger = __reduce_add_sync(0xffffffffu, larger);
            if (lane == 0 && larger + 1u == need) M.threshold = c;
          }
          __syncthreads();
          T = M.threshold;
        } else {                                              // ties in numbers: 11-bit digits of the members' composites
          unsigned long long prefix = 0ull;
          uint32_t left = need;
          for (int hi = 64; hi > 0;) {
            const int lo = hi > 11 ? hi - 11 : 0;
            for (int b = tid; b < FINE + FINE / SUPER; b += RT_THREADS) M.fine[b] = 0u;
            __syncthreads();
            for (uint32_t e = e_first; e < count; e += e_step) {
              const unsigned long long c = mine[e];
              if (fine((uint32_t)(c >> 32)) == bin && (hi == 64 || (c >> hi) == (prefix >> hi))) {
                const uint32_t digit = (uint32_t)(c >> lo) & ((1u << (hi - lo)) - 1u);
                atomicAdd(&M.fine[digit], 1u);
                atomicAdd(&M.fine_super[digit / SUPER], 1u);
              }
            }
            __syncthreads();
            find_bin<FINE>(M, M.fine, M.fine_super, left);
            prefix |= (unsigned long long)M.found_bin << lo;
            left -= M.found_above;
            hi = lo;
            if (left == M.found_count) break;
            __syncthreads();                                  // (M.found_count has been read)
          }
          T = prefix;
        }
      }
    }
    // complete: the threshold reaches every bound, or every CTA has listed all that it has
    const uint32_t lowest = ordered_key(-INFINITY);
    const uint32_t t_key = total > want ? (uint32_t)(T >> 32) : (total == want ? base : 0u);
    if (t_key >= top || top == lowest) {
      // ---- 4. the chosen tokens of the row
      for (uint32_t e = e_first; e < count; e += e_step) {
        const unsigned long long c = mine[e];
        const uint32_t t = ~(uint32_t)c;
        if (c >= T) atomicOr(reinterpret_cast<uint32_t*>(bits) + t / 32, 1u << (t & 31));
      }
      __syncthreads();
      break;
    }
    // another round: `want` tokens reach the threshold (where fewer than `want` were listed nothing less than everything will do)
    bound = total >= want ? key_to_float(max(t_key, lowest)) : -INFINITY;
    exact = true;
    if (ctas > 1) cluster.sync();                             // (nobody reads the old lists any more)
    else __syncthreads();
    for (int b = tid; b < FINE + FINE / SUPER; b += RT_THREADS) M.fine[b] = 0u;
    if (tid == 0) M.listed = M.split_count = 0u;
    __syncthreads();
  }

  uint32_t chosen = 0u;                                       // without lists, bit i: token(i) is selected by its score
  if (!fits) {
    // ---- more candidates than a list holds: 11-bit digits of the composites, over the whole cluster
    auto composite = [&](int i) { return ((unsigned long long)ordered_key(x[i]) << 32) | (uint32_t)~(uint32_t)token(i); };
    uint32_t *counts = M.coarse, *all = M.coarse + FINE;      // this CTA's and the cluster's
    uint32_t* all_super = M.coarse_super;
    static_assert(2 * FINE <= COARSE, "both fit");
    uint32_t left = want;
    T = 0ull;
    for (int hi = 64; hi > 0;) {
      const int lo = hi > 11 ? hi - 11 : 0;
      for (int b = tid; b < COARSE; b += RT_THREADS) M.coarse[b] = 0u;
      cluster.sync();
#pragma unroll
      for (int i = 0; i < EPT; ++i) {
        const unsigned long long c = composite(i);
        if (x[i] >= least && (hi == 64 || (c >> hi) == (T >> hi))) atomicAdd(&counts[(uint32_t)(c >> lo) & ((1u << (hi - lo)) - 1u)], 1u);
      }
      __syncthreads();
      for (int b = tid; b < FINE; b += RT_THREADS) {          // the non-empty bins are added to every CTA's counts of the cluster
        const uint32_t c = counts[b];
        if (c)
          for (int r = 0; r < ctas; ++r) atomicAdd(cluster.map_shared_rank(all, r) + b, c);
      }
      cluster.sync();
      {                                                       // four bins per thread, eight threads a super bin
        static_assert(FINE == 4 * RT_THREADS && SUPER == 32, "every bin once");
        const uint4 c = *reinterpret_cast<const uint4*>(all + 4 * tid);
        uint32_t sum = c.x + c.y + c.z + c.w;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((tid & 7) == 0) all_super[tid / 8] = sum;
      }
      __syncthreads();
      find_bin<FINE>(M, all, all_super, left);
      T |= (unsigned long long)M.found_bin << lo;
      left -= M.found_above;
      hi = lo;
      if (left == M.found_count) break;
      __syncthreads();                                        // (M.found_count has been read)
    }
#pragma unroll
    for (int i = 0; i < EPT; ++i)
      if (x[i] >= least && composite(i) >= T) chosen |= 1u << i;
#pragma unroll
    for (int v = 0; v < V; ++v) {                             // every warp tells all CTAs its chunks' tokens, eight lanes a word
      uint32_t w = ((chosen >> (4 * v)) & 15u) << (4 * (lane & 7));
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, o);
      const int at = chunk0 + v * chunk_step;
      if ((lane & 7) < ctas && at < chunks) *(cluster.map_shared_rank(reinterpret_cast<uint32_t*>(bits), lane & 7) + 4 * at + (lane >> 3)) = w;
    }
    cluster.sync();                                           // (nobody touches another CTA's shared memory after this)
  }

  // ---- places: the exclusive prefix of the chunks' counts
  uint32_t picked;                                            // tokens selected by score, of the whole row
  {
    static_assert(MAX_CHUNKS == 2 * RT_THREADS, "one or two chunks per thread");
    auto ones = [](const uint4& w) { return (uint32_t)(__popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w)); };
    const bool two = chunks > RT_THREADS;
    const int c0 = two ? 2 * tid : tid;
    uint32_t first = 0u, incl = 0u;
    if (c0 < chunks) {
      first = ones(bits[c0]);
      incl = first + (two && c0 + 1 < chunks ? ones(bits[c0 + 1]) : 0u);
    }
    const uint32_t local = incl;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) M.warp_sum[warp] = incl;
    __syncthreads();
    const uint32_t s = lane < RT_WARPS ? M.warp_sum[lane] : 0u;
    picked = __reduce_add_sync(0xffffffffu, s);
    const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? s : 0u) + incl - local;
    if (c0 < chunks) {
      places[c0] = before;
      if (two) places[c0 + 1] = before + first;
    }
    __syncthreads();
  }
  int32_t* out = idx_out + (size_t)head * k;
  const uint32_t n_sink = (uint32_t)elig_lo, n_local = (uint32_t)(n - elig_hi);
  auto write = [&](uint32_t t) {
    const uint4 w = bits[t / CHUNK];
    const uint32_t part = t % CHUNK / 32, word = part == 0 ? w.x : (part == 1 ? w.y : (part == 2 ? w.z : w.w));
    uint32_t pos = n_sink + places[t / CHUNK] + __popc(word & ((1u << (t & 31)) - 1u));
    pos += part > 0 ? __popc(w.x) : 0;
    pos += part > 1 ? __popc(w.y) : 0;
    pos += part > 2 ? __popc(w.z) : 0;
    if (pos < (uint32_t)k) out[pos] = (int32_t)t;
  };
  if (fits) {
    const uint32_t count = M.seg[rank].x;
    const unsigned long long* list = M.list + (size_t)rank * capacity;
    for (uint32_t e = tid; e < count; e += RT_THREADS) {
      const unsigned long long c = list[e];
      if (c >= T) write(~(uint32_t)c);
    }
  } else {
    for (uint32_t left = chosen; left; left &= left - 1u) write((uint32_t)token(__ffs(left) - 1));
  }
  if (rank == 0) {                                            // the forced tokens
    for (uint32_t e = tid; e < n_sink; e += RT_THREADS) out[e] = (int32_t)e;
    for (uint32_t e = tid; e < n_local; e += RT_THREADS) out[n_sink + picked + e] = (int32_t)(elig_hi + e);
    const uint32_t filled = n_sink + picked + n_local;
    if (filled < (uint32_t)k) {                               // short selection (non-finite scores)
      if (tid == 0) atomicOr(dev_status, FATHOM_DEV_TOPK_SHORT);
      for (uint32_t e = filled + tid; e < (uint32_t)k; e += RT_THREADS) out[e] = n - 1;   // pad with the last token
    }
  }
}

constexpr uint32_t most_listed(int ctas, int per_thread) { return ctas == 1 ? (uint32_t)(RT_THREADS * per_thread) : (uint32_t)(MOST_LISTED / ctas); }
constexpr size_t resident_smem_bytes(int ctas, uint32_t capacity, long long n) {
  return sizeof(ResidentSmem) + (size_t)capacity * ((size_t)ctas * 8 + 4) + (size_t)((n + CHUNK - 1) / CHUNK) * 16;
}
// the most that a launch with that many scores per thread may ask for: full lists, and the longest row that its CTAs hold (one CTA of 32 scores per
// thread, which may list them all, takes more than two that share the lists)
constexpr size_t resident_smem_most(int per_thread) {
  size_t most = 0;
  for (int ctas = 1; ctas <= MAX_CLUSTER; ctas *= 2) {
    const long long held = (long long)ctas * RT_THREADS * per_thread;
    const size_t bytes = resident_smem_bytes(ctas, most_listed(ctas, per_thread), held < FATHOM_TOPK_RESIDENT_MAX ? held : FATHOM_TOPK_RESIDENT_MAX);
    most = bytes > most ? bytes : most;
  }
  return most;
}
static_assert(resident_smem_most(8) <= 227 * 1024 && resident_smem_most(16) <= 227 * 1024 && resident_smem_most(32) <= 227 * 1024, "fits on an SM");

template <int EPT>
cudaError_t launch(const float* scores, long long n, long long score_stride, int Hq, int k, Forced F, uint32_t want, int32_t* idx,
                   uint32_t* dev_status, int ctas, cudaStream_t st) {
  // a CTA's share of what is wanted, with four standard deviations of a sample's count: one head in thousands needs a second round
  const double share = (double)want / ctas;
  const uint32_t quota = ctas == 1 ? want : (uint32_t)(share + 4.0 * sqrt(share) + 8.0);
  // room for 1.75 times the quota (the bound lets through 1.05 to 1.4 times), for 2048 at least and for 16,384 over all lists; two CTAs
  // fit on an SM while k is at most some 4000
  const uint32_t least = (uint32_t)(2048 / ctas), most = most_listed(ctas, EPT);
  uint32_t capacity = (7u * quota / 4u + 3u) & ~3u;
  capacity = capacity < least ? least : (capacity > most ? most : capacity);
  const size_t smem = resident_smem_bytes(ctas, capacity, n);
  static bool configured[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    e = cudaFuncSetAttribute(topk_resident_kernel<EPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)resident_smem_most(EPT));
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
  // the largest groups of which the quota is at most a half: they bound the threshold closely and take the fewest atomics
  const long long lanes = (n + 128LL * ctas - 1) / (128LL * ctas) * 32;       // four tokens each, of a CTA
  const long long threads = lanes < RT_THREADS ? lanes : RT_THREADS, beyond = lanes - EPT / 8 * RT_THREADS;
  const long long halves = threads + (beyond < 0 ? 0 : (beyond < RT_THREADS ? beyond : RT_THREADS));
  const int groups = 2LL * quota <= threads ? 1 : (EPT > 8 && 2LL * quota <= halves ? 2 : (2LL * quota <= lanes ? 4 : 0));
  return cudaLaunchKernelEx(&cfg, topk_resident_kernel<EPT>, scores, (int)n, score_stride, (int)F.sink_end, (int)F.local_begin, k, want,
                            quota, groups, capacity, idx, dev_status);
}

// The fewest tokens per thread (8, 16 or 32) with which all heads' clusters run at a CTA per SM, else with which they have the fewest CTAs:
// more tokens cost a thread less than a second CTA's threads cost the SM.  Clusters of eight leave SMs of a GPC over, so they have to be
// content with two thirds of the chip.  us with 8 / 16 / 32 tokens per thread:
//   8 heads   20,000 scores, k = 1024 6.1 / 6.6 / 8.0; 65,536 scores - / 6.6 / 7.3        16 heads  20,000 scores 7.3 / 6.7 / 8.0
//   32 heads  8000 scores, k = 1024 7.0 / 8.2 / 9.3; 20,000 scores 8.1 / 7.1 / 8.1; 65,536 scores - / 8.6 / 8.4
//   64 heads  20,000 scores, k = 1024 15.5 / 8.4 / 8.2; 33,001 scores - / 16.2 / 9.8
// Lists of eight CTAs for most of a short row are long: 1 head, 20,000 scores, k = 8192 17.6 / 13.7 / 17.4; 32 heads 47.6 / 15.4 / 19.2.
int ctas_for(long long n, int per_thread) {
  int ctas = 1;
  while ((long long)ctas * RT_THREADS * per_thread < n) ctas *= 2;
  return ctas;
}
int tokens_per_thread(long long n, int Hq, uint32_t want) {
  int best = 0;
  for (int per = want > 4096 ? 16 : 8; per <= 32; per *= 2) {
    const int ctas = ctas_for(n, per);
    if (ctas > MAX_CLUSTER) continue;
    if ((ctas == MAX_CLUSTER ? 3LL : 2LL) * ctas * Hq <= 2LL * fathom_sm_count()) return per;
    if (!best || ctas < ctas_for(n, best)) best = per;
  }
  return best;
}

}  // namespace

int fathom_topk_resident_ctas(long long n, int Hq, uint32_t want) { return ctas_for(n, tokens_per_thread(n, Hq, want)); }

int fathom_launch_topk_resident(fathom_ctx* ctx, const float* scores, long long n, long long score_stride, int Hq, int k, Forced F,
                                uint32_t want, int32_t* idx, cudaStream_t st) {
  const int ept = tokens_per_thread(n, Hq, want), ctas = ctas_for(n, ept);
  cudaError_t e;
  if (ept == 8) e = launch<8>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, ctas, st);
  else if (ept == 16) e = launch<16>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, ctas, st);
  else e = launch<32>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, ctas, st);
  FATHOM_CUDA_TRY(ctx, e);
  return FATHOM_OK;
}
