// Top-k of rows of up to 131,072 scores in ONE kernel: a cluster of up to eight CTAs per head holds the row's scores in
// registers, so whatever the selection has to look at twice is not read twice, and nothing goes through global memory
// between its steps.  What bounds such rows is not the data but the instructions that every warp executes once, at some nine
// cycles each: 512 threads share out a few hundred candidates.  So a step takes as few instructions per warp as possible (a search
// by one warp over two levels of counts, lists of tokens instead of places computed for every score, one candidate per thread from
// then on).
//
// The order of a head's tokens is that of the 64-bit composite (key << 32 | ~token): larger score first, ties to the lower
// token.  The row is dealt out in runs of 32 tokens, a line each, and neighbouring ones to different CTAs: neighbours' scores are alike where keys
// are, and every CTA is to hold a sample of the whole row.  (In runs of 128, one after the other, rows of which every eighth run lies above
// the others took 54 us instead of 31.)  A thread's tokens are no neighbours either.  There is ONE exchange:
//   1. coarse histogram (4096 bins, a thirty-second of an octave where scores usually lie) of the maxima of the threads' groups of
//      tokens, in the CTA's own shared memory: its own bound is the bin that holds the quota-th largest maximum, the quota being its
//      share of `want` and four standard deviations more;
//   2. the tokens that reach the CTA's bound are listed, and list, length and bound are written to every CTA of the cluster.  (Where
//      the large scores lie in one bin, or in a few threads, too many tokens reach it; the bound is then taken from the tokens);
//   3. after the cluster barrier every CTA finds the want-th largest of all lists: fine histogram (2048 bins of 2^13 keys from the
//      lowest bound on), the members of the bin that the threshold splits (a few) ranked against one another.  A threshold
//      that reaches every CTA's bound is exact: all lists are complete down to it.  One that does not is still a bound of the whole
//      row (`want` tokens reach it), and the CTAs with a higher one list what lies between;
//   4. every CTA marks the chosen tokens of all lists in a bitmap of the row, whose prefix counts give its own list's tokens their
//      places in the ascending output.
// (A first form merged whole histograms in every CTA; a second one merged those of the maxima and let the first CTA pull the lists,
// select and write alone: three cluster barriers, and seven of eight CTAs idle for 40 % of the time.  32 heads, back to back, second
// form / this one: 131,072 scores, k = 2048 17.0 / 11.7 us; 65,536, k = 1024 13.9 / 8.6; 33,001, k = 512 12.7 / 7.0; one head of 4096, k = 64 6.2 / 4.8.
// Scores alike over runs of 16 to 4096 tokens, 131,072, k = 512: 15 to 34 / 9 to 11.)
// Lists of a large part of a row, or that would not fit (heavy ties), are not made: the counts of all tokens are merged over the cluster and
// the bin that the threshold splits is divided further until few enough members are left to rank them (step 1').
// The set is unique and the counts are integers: the result does not depend on any order of atomics.
#include "topk_shared.cuh"

#include <cooperative_groups.h>

#include <cmath>
#include <cstddef>
#include <type_traits>

namespace cg = cooperative_groups;

namespace {

constexpr int RT_THREADS = 512;
constexpr int RT_WARPS = RT_THREADS / 32;
constexpr int MAX_CLUSTER = 8;
constexpr int FINE = 2048, FINE_SHIFT = 13;
// Members of a split bin that are ranked by comparison: a round of counts takes as long as ranking a hundred, one over the cluster 130.  (With 512,
// 20,000 scores around 1000, k = 512, took 24 us.)
constexpr int SPLIT = 96;
constexpr int CHUNK = 128, MAX_CHUNKS = (int)(FATHOM_TOPK_RESIDENT_MAX / CHUNK);
constexpr uint32_t FEW = 128;                                 // ... where there are no lists
constexpr int TOKEN_BITS = 17;
constexpr uint32_t MOST_WANTED = 9000;                        // by lists
constexpr uint32_t MOST_LISTED = 16384;                       // over all lists of a cluster

struct ResidentSmem {
  alignas(16) uint32_t coarse[COARSE];                        // counts of this CTA's maxima, or tokens; then members of the split bin and places of the chunks
  uint32_t coarse_super[COARSE / SUPER];
  uint32_t fine[FINE];                                        // counts of the lists; or of the cluster, like the first bytes of the lists
  uint32_t fine_super[FINE / SUPER];
  alignas(16) uint32_t warp_sum[RT_WARPS];
  uint2 seg[2][MAX_CLUSTER];                                  // length and bound of every CTA's list in each round, written by each of them
  uint32_t listed, found_bin, found_above, found_count, split_count;
  unsigned long long threshold;
  alignas(16) unsigned long long list[1];                     // [ctas][capacity] composites, [capacity] tokens of this CTA's list, [chunks] uint4 of
                                                              // chosen tokens of the whole row
};
constexpr int COUNTS = COARSE + COARSE / SUPER + FINE + FINE / SUPER;
static_assert(offsetof(ResidentSmem, warp_sum) == COUNTS * 4 && COUNTS % 4 == 0, "the counts lie side by side");
static_assert(SPLIT * 8 + MAX_CHUNKS * 4 <= COARSE * 4, "the split bin and the places fit over the coarse counts");
static_assert(MAX_CLUSTER * FEW * 8 <= COARSE * 4 && FEW * 8 <= FINE * 4 && FATHOM_TOPK_RESIDENT_MAX <= 1LL << TOKEN_BITS, "the few members, too");

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

// All threads, after a barrier that completes the `members` entries of `split`: the need-th largest of them (a warp per entry, its lanes
// over the others).
__device__ __forceinline__ unsigned long long ranked(ResidentSmem& M, const unsigned long long* split, uint32_t members, uint32_t need) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t i = warp; i < members; i += RT_WARPS) {
    const unsigned long long c = split[i];
    uint32_t larger = 0u;
    for (uint32_t j = lane; j < members; j += 32) larger += split[j] > c;
    larger = __reduce_add_sync(0xffffffffu, larger);
    if (lane == 0 && larger + 1u == need) M.threshold = c;
  }
  __syncthreads();
  return M.threshold;
}

// groups: of each thread, that its tokens are dealt to (1, 2, 4, 8 or 16); 0: no lists of candidates (step 1')
template <int EPT, int C>
__global__ void __launch_bounds__(RT_THREADS, 2)
topk_resident_kernel(const float* scores, int n, long long score_stride, int elig_lo, int elig_hi, int k, uint32_t want, uint32_t quota,
                     int groups, uint32_t capacity, int32_t* __restrict__ idx_out, uint32_t* __restrict__ dev_status) {
  extern __shared__ __align__(16) unsigned char resident_smem[];
  ResidentSmem& M = *reinterpret_cast<ResidentSmem*>(resident_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = C > 1 ? (int)cluster.block_rank() : 0, head = blockIdx.x / C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunks = (n + CHUNK - 1) / CHUNK;
  uint32_t* own = reinterpret_cast<uint32_t*>(M.list + (size_t)C * capacity);                // (capacity is a multiple of 4)
  uint4* bits = reinterpret_cast<uint4*>(own + capacity);
  uint32_t* further = reinterpret_cast<uint32_t*>(M.list);    // counts of the cluster, where there are no lists
  unsigned long long* split = reinterpret_cast<unsigned long long*>(M.coarse);
  uint32_t* places = M.coarse + 2 * SPLIT;
  auto clear = [&](uint32_t* p, int words) {
    for (int b = tid; b < words / 4; b += RT_THREADS) reinterpret_cast<uint4*>(p)[b] = make_uint4(0u, 0u, 0u, 0u);
  };
  auto sync = [&] {                                           // all threads of the cluster
    if constexpr (C > 1) cluster.sync();
    else __syncthreads();
  };
  clear(M.coarse, COUNTS);
  if (groups == 0) clear(further, COARSE);
  for (int b = tid; b < chunks; b += RT_THREADS) bits[b] = make_uint4(0u, 0u, 0u, 0u);
  if (tid == 0) M.listed = M.split_count = 0u;
  __syncthreads();
  auto started = cluster.barrier_arrive();                    // (my counts are clear; nothing is written to a CTA's shared memory before it runs)
  FATHOM_PDL_WAIT();                                          // the scores come from the previous kernel
  FATHOM_PDL_RELEASE();                                       // the attention that follows may become resident now

  // ---- my tokens: of every C runs of 32 one is mine, not always the same.  They are kept as scores and compared as scores (a key is only
  //      formed for the few that matter); NaN stands for a token that is not eligible
  constexpr int STEP = RT_WARPS * C * 32;                     // n <= 131072
  const int first = (warp * C + ((rank ^ warp ^ (warp >> 3)) & (C - 1))) * 32 + lane;
  auto token = [&](int i) { return first + i * STEP; };
  const float* row = scores + (size_t)head * (size_t)score_stride;
  const float NONE = __uint_as_float(0x7fffffffu);
  float x[EPT];
  if (first - lane >= elig_lo && first - lane + 32 + (EPT - 1) * STEP <= elig_hi) {          // (uniform over the warp)
#pragma unroll
    for (int i = 0; i < EPT; ++i) x[i] = row[first + i * STEP];
  } else {
    auto before = [&](int end) { return max(end - first + STEP - 1, 0) / STEP; };            // how many of my tokens lie before `end`
    const int i0 = before(elig_lo), i1 = before(elig_hi);
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      x[i] = NONE;
      if (i >= i0 && i < i1) x[i] = row[first + i * STEP];
    }
  }
  auto count = [&](float m) {
    if (m == m) {
      const uint32_t b = coarse_bin(m);
      atomicAdd(&M.coarse[b], 1u);
      atomicAdd(&M.coarse_super[b / SUPER], 1u);
    }
  };

  // ---- 1. my bound
  const bool listing = groups != 0 && want != 0u;
  float bound = NONE;
  if (listing) {
    auto count_groups = [&](auto gc) {
      constexpr int G = decltype(gc)::value;
#pragma unroll
      for (int j = 0; j < G; ++j) {
        float m = x[j];
#pragma unroll
        for (int i = j + G; i < EPT; i += G) m = fmaxf(m, x[i]);              // (a NaN is no maximum)
        count(m);
      }
    };
    if (groups == 1) count_groups(std::integral_constant<int, 1>{});
    else if (groups == 2) count_groups(std::integral_constant<int, 2>{});
    else if (groups == 4) count_groups(std::integral_constant<int, 4>{});
    else if (groups == 8) count_groups(std::integral_constant<int, 8>{});
    else count_groups(std::integral_constant<int, EPT < 16 ? EPT : 16>{});
    __syncthreads();
    find_bin<COARSE>(M, M.coarse, M.coarse_super, quota);
    bound = M.found_bin == 0u ? -INFINITY : coarse_edge(M.found_bin);         // (bin 0: everything, see search_bins)
  }
  cluster.barrier_wait(std::move(started));                   // (everyone arrived long ago)

  // ---- every warp of a CTA works on one of the lists
  constexpr int PER_LIST = RT_WARPS / C;
  const int my_list = warp / PER_LIST;
  const uint32_t e_first = (uint32_t)(warp % PER_LIST) * 32 + lane;
  constexpr uint32_t E_STEP = (uint32_t)PER_LIST * 32;
  const unsigned long long* mine = M.list + (size_t)my_list * capacity;

  unsigned long long T = 0ull;                                // the smallest composite that is selected
  bool by_list = listing;
  float least = -INFINITY;                                    // no smaller score is selected
  if (listing) {
    const uint32_t lowest = ordered_key(-INFINITY);
    float lower = bound, upper = NONE;                        // listed in this round: from `lower` on, what is not listed yet
    uint32_t from = 0u;
#pragma unroll 1
    for (int round = 0;; ++round) {                           // (at most two: the second one's threshold reaches its bound)
      // ---- 2. the tokens that reach the bound, in any order
      uint32_t listed;
      for (bool again = round == 0;; again = false) {
        uint32_t set = 0u;
#pragma unroll
        for (int i = 0; i < EPT; ++i)
          if (x[i] >= lower && !(x[i] >= upper)) set |= 1u << i;
        if (set) {
          uint32_t at = atomicAdd(&M.listed, (uint32_t)__popc(set));
          for (; set && at < capacity; set &= set - 1u) own[at++] = (uint32_t)token(__ffs(set) - 1);
        }
        __syncthreads();
        listed = M.listed;
        if (listed <= capacity || !again) break;              // (the same for the whole CTA)
        // the large scores lie in one bin, or in the groups of a few threads: a bound that the quota of tokens, not of groups, reaches, to a
        // 2048th of what lies between the first bound and the largest
        float m = x[0];
#pragma unroll
        for (int i = 1; i < EPT; ++i) m = fmaxf(m, x[i]);
        const uint32_t largest = __reduce_max_sync(0xffffffffu, m == m ? ordered_key(m) : 0u);
        if (lane == 0) M.warp_sum[warp] = largest;
        __syncthreads();
        const uint32_t edge = ordered_key(lower), range = __reduce_max_sync(0xffffffffu, M.warp_sum[lane % RT_WARPS]) - edge;
        const int shift = max(21 - __clz(range), 0);
#pragma unroll
        for (int i = 0; i < EPT; ++i)
          if (x[i] >= lower) {
            const uint32_t b = (ordered_key(x[i]) - edge) >> shift;
            atomicAdd(&M.fine[b], 1u);
            atomicAdd(&M.fine_super[b / SUPER], 1u);
          }
        __syncthreads();
        find_bin<FINE>(M, M.fine, M.fine_super, quota);
        lower = key_to_float(edge + (M.found_bin << shift));
        clear(M.fine, FINE + FINE / SUPER);
        if (tid == 0) M.listed = 0u;
        __syncthreads();
      }
      if (listed <= capacity) {
        for (uint32_t e = from + tid; e < listed; e += RT_THREADS) {
          const uint32_t t = own[e];
          const unsigned long long c = ((unsigned long long)ordered_key(row[t]) << 32) | (uint32_t)~t;         // (the row's line is in the L1)
          unsigned long long* to = M.list + (size_t)rank * capacity + e;
#pragma unroll
          for (int r = 0; r < C; ++r) *(C > 1 ? cluster.map_shared_rank(to, r) : to) = c;
        }
      }
      from = listed;
      if (tid < C) *(C > 1 ? cluster.map_shared_rank(&M.seg[round][rank], tid) : &M.seg[round][rank]) = make_uint2(listed, __float_as_uint(lower));
      sync();

      // ---- 3. the want-th largest of all lists
      const uint2 theirs = lane < C ? M.seg[round][lane] : make_uint2(0u, __float_as_uint(lower));
      const uint32_t their_key = ordered_key(__uint_as_float(theirs.y));
      const uint32_t total = __reduce_add_sync(0xffffffffu, theirs.x);
      const uint32_t base = __reduce_min_sync(0xffffffffu, their_key), top = __reduce_max_sync(0xffffffffu, their_key);   // keys of the lowest and the highest bound
      const uint32_t length = __shfl_sync(0xffffffffu, theirs.x, my_list);
      by_list = !__any_sync(0xffffffffu, theirs.x > capacity);
      if (!by_list) {                                         // (the same for the whole cluster, like every other way out)
        if (total >= want) least = key_to_float(base);
        break;
      }
      T = 0ull;                                               // fewer than wanted, or just as many: all of them
      if (total > want) {
        auto fine = [&](uint32_t key) { return min((key - base) >> FINE_SHIFT, (uint32_t)(FINE - 1)); };
        for (uint32_t e = e_first; e < length; e += E_STEP) {
          const uint32_t key = (uint32_t)(mine[e] >> 32);
          if (key >= base) {                                  // (in the second round the lists hold less than the new bound, too)
            const uint32_t b = fine(key);
            atomicAdd(&M.fine[b], 1u);
            atomicAdd(&M.fine_super[b / SUPER], 1u);
          }
        }
        __syncthreads();
        find_bin<FINE>(M, M.fine, M.fine_super, want);
        const uint32_t bin = M.found_bin;
        uint32_t members = M.found_count, need = want - M.found_above;
        T = (unsigned long long)(base + (bin << FINE_SHIFT)) << 32;
        // the bin is split: its members are ranked; where there are many (ties, or large scores close together) in ever finer bins
        unsigned long long span = bin == (uint32_t)(FINE - 1) ? ~0ull : 1ull << (32 + FINE_SHIFT);             // (the last one is open above)
        int width = bin == (uint32_t)(FINE - 1) ? 64 : 32 + FINE_SHIFT;
        while (need != members) {
          const unsigned long long low = T;
          if (members <= (uint32_t)SPLIT) {
            for (uint32_t e = e_first; e < length; e += E_STEP) {
              const unsigned long long c = mine[e];
              if (c >= low && c - low < span) split[atomicAdd(&M.split_count, 1u)] = c;
            }
            __syncthreads();
            T = ranked(M, split, members, need);
            break;
          }
          const int shift = width > 11 ? width - 11 : 0;
          __syncthreads();                                    // (the counts and what was found in them have been read)
          clear(M.fine, FINE + FINE / SUPER);
          __syncthreads();
          for (uint32_t e = e_first; e < length; e += E_STEP) {
            const unsigned long long c = mine[e];
            if (c >= low && c - low < span) {
              const uint32_t b = (uint32_t)((c - low) >> shift);
              atomicAdd(&M.fine[b], 1u);
              atomicAdd(&M.fine_super[b / SUPER], 1u);
            }
          }
          __syncthreads();
          find_bin<FINE>(M, M.fine, M.fine_super, need);
          T += (unsigned long long)M.found_bin << shift;
          need -= M.found_above;
          members = M.found_count;
          width = shift;
          span = 1ull << shift;
        }
      }
      // complete: the threshold reaches every bound, or every CTA has listed all that it has
      const uint32_t t_key = total > want ? (uint32_t)(T >> 32) : (total == want ? base : 0u);
      if (t_key >= top || top == lowest) {
        // ---- 4. the chosen tokens of the row
        for (uint32_t e = e_first; e < length; e += E_STEP) {
          const unsigned long long c = mine[e];
          const uint32_t t = ~(uint32_t)c;
          if (c >= T) atomicOr(reinterpret_cast<uint32_t*>(bits) + t / 32, 1u << (t & 31));
        }
        __syncthreads();
        break;
      }
      // another round: `want` tokens reach the threshold (where fewer than `want` were listed nothing less than everything will do)
      upper = lower;
      lower = total >= want ? key_to_float(max(t_key, lowest)) : -INFINITY;
      __syncthreads();                                        // (the counts have been read)
      clear(M.fine, FINE + FINE / SUPER);
      if (tid == 0) M.split_count = 0u;
    }
  }

  if (!by_list && want != 0u) {
    // ---- 1'. no lists: the counts of all tokens, over the whole cluster, then of the tokens of the bin that the threshold splits,
    //      in ever finer bins, until few enough are left to rank them
    auto place = [&](int i) { return ((unsigned long long)ordered_key(x[i]) << TOKEN_BITS) | (unsigned long long)((1u << TOKEN_BITS) - 1u - (uint32_t)token(i)); };
    auto merge = [&](uint32_t* all, int bins) {               // (counts complete) my non-empty bins are added to every CTA's
      if constexpr (C > 1) {
        for (int b = tid; b < bins; b += RT_THREADS) {
          const uint32_t c = M.coarse[b];
          if (c) {
#pragma unroll
            for (int r = 0; r < C; ++r) atomicAdd(cluster.map_shared_rank(all, r) + b, c);
          }
        }
        cluster.sync();
      }
    };
    auto supers = [&](const uint32_t* all, auto binsc) {      // BINS / 512 bins per thread
      constexpr int BINS = decltype(binsc)::value, PER = BINS / RT_THREADS, LANES = SUPER / PER;
      uint32_t sum = 0u;
#pragma unroll
      for (int b = 0; b < PER / 4; ++b) {
        const uint4 c = *reinterpret_cast<const uint4*>(all + PER * tid + 4 * b);
        sum += c.x + c.y + c.z + c.w;
      }
#pragma unroll
      for (int o = 1; o < LANES; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (tid % LANES == 0) M.coarse_super[tid / LANES] = sum;
      __syncthreads();
    };
    if (groups != 0) {                                        // the lists did not hold what they should
      __syncthreads();
      clear(M.coarse, COUNTS);
      clear(further, COARSE);
      sync();
    }
#pragma unroll
    for (int i = 0; i < EPT; ++i)
      if (x[i] >= least) atomicAdd(&M.coarse[coarse_bin(x[i])], 1u);
    __syncthreads();
    uint32_t* all = C > 1 ? further : M.coarse;
    merge(all, COARSE);
    supers(all, std::integral_constant<int, COARSE>{});
    find_bin<COARSE>(M, all, M.coarse_super, want);
    unsigned long long low = 0ull, span = 0ull;               // the places from low to low + span are to be divided, 2^(width - 11) at a time
    uint32_t need = want - M.found_above, members = M.found_count;
    if (M.found_bin != 0u) {
      low = (unsigned long long)ordered_key(coarse_edge(M.found_bin)) << TOKEN_BITS;
      span = ((unsigned long long)ordered_key(coarse_edge(M.found_bin + 1u)) << TOKEN_BITS) - low;
    } else {
      need = members;                                         // fewer than wanted: all of them
    }
    int width = TOKEN_BITS + (span >> TOKEN_BITS <= 1u << 18 ? 18 : 21);      // (the two sizes of bins)
#pragma unroll 1
    for (int level = 1; need != members; ++level) {
      __syncthreads();                                        // (all, found_count .. have been read)
      const float from = key_to_float((uint32_t)(low >> TOKEN_BITS)), to = key_to_float(min((uint32_t)((low + span - 1ull) >> TOKEN_BITS), ordered_key(INFINITY)));
      auto inside = [&](int i) { return x[i] >= from && x[i] <= to && place(i) - low < span; };
      if (members <= FEW) {
        unsigned long long *lists = split, *few = reinterpret_cast<unsigned long long*>(M.fine);         // (nobody reads the coarse counts any more)
        if (tid == 0) M.listed = 0u;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < EPT; ++i)
          if (inside(i)) {
            unsigned long long* to_list = lists + rank * FEW + atomicAdd(&M.listed, 1u);
#pragma unroll
            for (int r = 0; r < C; ++r) *(C > 1 ? cluster.map_shared_rank(to_list, r) : to_list) = place(i);
          }
        __syncthreads();
        if (tid < C) *(C > 1 ? cluster.map_shared_rank(&M.seg[0][rank], tid) : &M.seg[0][rank]) = make_uint2(M.listed, 0u);
        sync();
        for (uint32_t e = tid; e < members; e += RT_THREADS) {
          uint32_t r = 0u, at = e;
          while (at >= M.seg[0][r].x) at -= M.seg[0][r++].x;
          few[e] = lists[r * FEW + at];
        }
        __syncthreads();
        low = ranked(M, few, members, need);
        break;
      }
      // counted in my coarse bins, merged in `fine` and `further` in turn: the next level's counts are cleared a barrier ahead
      uint32_t* next = level & 1 ? further : M.fine;
      all = C == 1 ? M.coarse : (level & 1 ? M.fine : further);
      clear(M.coarse, FINE);
      if (C > 1) clear(next, FINE);
      __syncthreads();
      const int shift = width > 11 ? width - 11 : 0;
#pragma unroll
      for (int i = 0; i < EPT; ++i)
        if (inside(i)) atomicAdd(&M.coarse[(uint32_t)((place(i) - low) >> shift)], 1u);
      __syncthreads();
      merge(all, FINE);
      supers(all, std::integral_constant<int, FINE>{});
      find_bin<FINE>(M, all, M.coarse_super, need);
      low += (unsigned long long)M.found_bin << shift;
      need -= M.found_above;
      members = M.found_count;
      width = shift;
      span = 1ull << shift;
    }
    // every warp tells all CTAs which tokens of its words are chosen
    const float limit = low ? key_to_float((uint32_t)(low >> TOKEN_BITS)) : -INFINITY;
    const int last = (1 << TOKEN_BITS) - 1 - (int)(low & ((1u << TOKEN_BITS) - 1u));         // of that score
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      const uint32_t w = __ballot_sync(0xffffffffu, x[i] > limit || (x[i] == limit && token(i) <= last));
      uint32_t* to = reinterpret_cast<uint32_t*>(bits) + (token(i) - lane) / 32;
      if (lane < C && token(i) - lane < n) *(C > 1 ? cluster.map_shared_rank(to, lane) : to) = w;
    }
    sync();                                                   // (nobody touches another CTA's shared memory after this)
  }

  // ---- places: the exclusive prefix of the chunks' counts
  uint32_t picked;                                            // tokens selected by score, of the whole row
  {
    static_assert(MAX_CHUNKS == 2 * RT_THREADS, "one or two chunks per thread");
    auto ones = [](const uint4& w) { return (uint32_t)(__popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w)); };
    const bool two = chunks > RT_THREADS;
    const int c0 = two ? 2 * tid : tid;
    uint32_t first_of = 0u, incl = 0u;
    if (c0 < chunks) {
      first_of = ones(bits[c0]);
      incl = first_of + (two && c0 + 1 < chunks ? ones(bits[c0 + 1]) : 0u);
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
      if (two) places[c0 + 1] = before + first_of;
    }
    __syncthreads();
  }
  int32_t* out = idx_out + (size_t)head * k;
  const uint32_t n_sink = (uint32_t)elig_lo, n_local = (uint32_t)(n - elig_hi);
  // place of token t, if it is chosen; `word`: the 32 tokens it is one of
  auto place_of = [&](uint32_t t, uint32_t& word) {
    const uint4 w = bits[t / CHUNK];
    const uint32_t part = t % CHUNK / 32;
    word = part == 0 ? w.x : (part == 1 ? w.y : (part == 2 ? w.z : w.w));
    uint32_t pos = n_sink + places[t / CHUNK] + __popc(word & ((1u << (t & 31)) - 1u));
    pos += part > 0 ? __popc(w.x) : 0;
    pos += part > 1 ? __popc(w.y) : 0;
    pos += part > 2 ? __popc(w.z) : 0;
    return pos;
  };
  if (by_list) {
    const uint32_t length = M.listed;
    const unsigned long long* list = M.list + (size_t)rank * capacity;
    for (uint32_t e = tid; e < length; e += RT_THREADS) {
      const unsigned long long c = list[e];
      if (c >= T) {
        const uint32_t t = ~(uint32_t)c;
        uint32_t word;
        const uint32_t pos = place_of(t, word);
        if (pos < (uint32_t)k) out[pos] = (int32_t)t;
      }
    }
  } else {                                                    // the words of my tokens
#pragma unroll 4
    for (int i = 0; i < EPT; ++i) {
      const uint32_t t = (uint32_t)token(i);
      if (t - lane >= (uint32_t)n) break;                     // (uniform over the warp)
      uint32_t word;
      const uint32_t pos = place_of(t, word);
      if ((word >> lane & 1u) && pos < (uint32_t)k) out[pos] = (int32_t)t;
    }
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

constexpr size_t resident_smem_bytes(int ctas, uint32_t capacity, long long n) {
  return sizeof(ResidentSmem) + (size_t)capacity * ((size_t)ctas * 8 + 4) + (size_t)((n + CHUNK - 1) / CHUNK) * 16;
}
// the most of all launches: lists of MOST_LISTED entries, and the longest row, of each number of CTAs
constexpr size_t resident_smem_most() {
  size_t most = 0;
  for (int ctas = 1; ctas <= MAX_CLUSTER; ctas *= 2) {
    const size_t bytes = resident_smem_bytes(ctas, MOST_LISTED / ctas, (long long)ctas * RT_THREADS * 32);
    most = bytes > most ? bytes : most;
  }
  return most;
}
constexpr int SM_SMEM = 227 * 1024;
static_assert(resident_smem_most() <= SM_SMEM && MOST_LISTED % (4 * MAX_CLUSTER) == 0, "fits on an SM");

template <int EPT, int C>
cudaError_t launch(const float* scores, long long n, long long score_stride, int Hq, int k, Forced F, uint32_t want, int32_t* idx,
                   uint32_t* dev_status, cudaStream_t st) {
  // a CTA's share of what is wanted, with four standard deviations of a sample's count
  const double share = (double)want / C;
  const uint32_t quota = C == 1 ? want : (uint32_t)(share + 4.0 * sqrt(share) + 8.0);
  // the largest groups of which the quota is at most a half: they bound the threshold closely and take the fewest atomics
  const long long tokens = (n + 32 * C - 1) / (32 * C) * 32;                  // of a CTA, at most
  int groups = 1;
  while (groups < 16 && 2LL * quota > (tokens < RT_THREADS * groups ? tokens : RT_THREADS * groups)) groups *= 2;
  // room for 1.75 times the quota (the bound lets through 1.05 to 1.4 times), for 2048 in all, where the cluster's counts lie, too
  uint32_t capacity = (7u * quota / 4u + 3u) & ~3u;
  if (capacity < 2048u / C) capacity = 2048u / C;
  if (capacity > MOST_LISTED / C) capacity = MOST_LISTED / C;
  // No lists of more than two sevenths of the tokens, nor of more than MOST_WANTED (in us, lists / none: 4096 scores, one CTA, k = 1024 6.8 / 6.5, 2048
  // 7.6 / 6.1; 16,384, 4 CTAs, k = 4096 10.2 / 9.5, 6000 12.5 / 9.2; 65,536, 8 CTAs, k = 8192 15.1 / 13.2, but 131,072 17 / 23).  Where the CTAs want to
  // share the SMs and their lists leave no room for two, earlier (32 heads: 100,000, k = 6000 39 / 33, 131,072, k = 8192 46 / 39; 40 heads: 33,001, k = 6000 27 / 24,
  // but 131,072 42 / 51)
  const long long ctas = (long long)Hq * C, sms = fathom_sm_count();
  const bool crowded = ctas > sms && 2 * resident_smem_bytes(C, capacity, n) > SM_SMEM;
  if (7LL * quota > 2 * tokens || want > MOST_WANTED || (crowded && quota > 800 && (ctas <= 2 * sms ? 15LL : 10LL) * quota > tokens)) {
    groups = 0;
    capacity = 2048u / C;
  }
  const size_t smem = resident_smem_bytes(C, capacity, n);
  static bool configured[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    e = cudaFuncSetAttribute(topk_resident_kernel<EPT, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)resident_smem_most());
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(Hq * C));
  cfg.blockDim = dim3(RT_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)C;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, topk_resident_kernel<EPT, C>, scores, (int)n, score_stride, (int)F.sink_end, (int)F.local_begin, k, want,
                            quota, groups, capacity, idx, dev_status);
}

// The fewest tokens per thread (8, 16 or 32) with which all heads' clusters run at a CTA per SM, else with which they have the fewest CTAs:
// more tokens cost a thread less than a second CTA's threads cost the SM.  Clusters of eight leave SMs of a GPC over, so they have to be
// content with two thirds of the chip.  us with 8 / 16 / 32 tokens per thread:
//   8 heads   20,000 scores, k = 1024 6.1 / 6.6 / 8.0; 65,536 scores - / 6.6 / 7.3        16 heads  20,000 scores 7.3 / 6.7 / 8.0
//   32 heads  8000 scores, k = 1024 7.0 / 8.2 / 9.3; 20,000 scores 8.1 / 7.1 / 8.1; 65,536 scores - / 8.6 / 8.4
//   64 heads  20,000 scores, k = 1024 15.5 / 8.4 / 8.2; 33,001 scores - / 16.2 / 9.8
int ctas_for(long long n, int per_thread) {
  int ctas = 1;
  while ((long long)ctas * RT_THREADS * per_thread < n) ctas *= 2;
  return ctas;
}
int tokens_per_thread(long long n, int Hq) {
  int best = 0;
  for (int per = 8; per <= 32; per *= 2) {
    const int ctas = ctas_for(n, per);
    if (ctas > MAX_CLUSTER) continue;
    if ((ctas == MAX_CLUSTER ? 3LL : 2LL) * ctas * Hq <= 2LL * fathom_sm_count()) return per;
    if (!best || ctas < ctas_for(n, best)) best = per;
  }
  return best;
}

}  // namespace

int fathom_topk_resident_ctas(long long n, int Hq) { return ctas_for(n, tokens_per_thread(n, Hq)); }

int fathom_launch_topk_resident(fathom_ctx* ctx, const float* scores, long long n, long long score_stride, int Hq, int k, Forced F,
                                uint32_t want, int32_t* idx, cudaStream_t st) {
  const int per = tokens_per_thread(n, Hq), ctas = ctas_for(n, per);
  auto with = [&](auto perc) {
    constexpr int PER = decltype(perc)::value;
    if (ctas == 1) return launch<PER, 1>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, st);
    if (ctas == 2) return launch<PER, 2>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, st);
    if (ctas == 4) return launch<PER, 4>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, st);
    return launch<PER, 8>(scores, n, score_stride, Hq, k, F, want, idx, ctx->dev_status, st);
  };
  const cudaError_t e = per == 8 ? with(std::integral_constant<int, 8>{}) : (per == 16 ? with(std::integral_constant<int, 16>{}) : with(std::integral_constant<int, 32>{}));
  FATHOM_CUDA_TRY(ctx, e);
  return FATHOM_OK;
}
