// fathom_scan: variable-depth bit-plane key scan (Sec. 3.2 prefix dequantiser, Sec. 3.3), accumulate on the tensor cores.
//
// A t-plane read of channel j dequantises to  a * sum_{p<t} (2 b_p - 1) 2^-(p+1)  with a = 8 s the block range, so with
// the active (channel, plane) pairs of a plan as "rows" r = (j, p) a score is
//     score[i][h] = sum_r  sigma[i][r] * s[beta(i)][j(r)]  *  q_h,j(r) 2^(2 - p(r)),        sigma = +1 if the bit is set, else -1:
// a [tokens x rows] . [rows x heads] product whose left operand is the stored fp16 scale with the plane bit as its sign
// - exact in fp16 - and whose right operand depends on neither token nor block.  One add per (token, row, head) on the
// CUDA cores is what bounds the scan (Sec. 7 "Arithmetic per byte": 1.6 G adds at n = 1M, B = 48, 43 us of fp32 pipe
// against 9 us of HBM time for the planes); here the adds go to the tensor cores and the CUDA cores only expand the
// plane bits into the left operand, two integer instructions per pair of elements:
//   * left operand (registers): a lane holds, for 8 consecutive tokens of a block (one byte of each plane word) and 4 of
//     every 16 rows, the half2 (s_r, s_r') of a row pair; the element of token i is that pair with the sign bits flipped
//     where the tokens' bits are clear:  pair ^ (~(bytes << shift_i) & 0x80008000);
//   * right operand: q_hj 2^(2-p) / E_h (E_h a power of two near max_j |q_hj|) split into an fp16 head and an fp16 tail
//     scaled by 2^11 (together 22 significant bits + rounding = the precision of an fp32 weight), columns
//     (head, part) = 4 x 2 = the 8 columns of mma.sync.m16n8k16; built once per session and plan in shared memory;
//   * fp16 x fp16 products are exact in the fp32 accumulators; score = E_h (acc_head + 2^-11 acc_tail).  The order of
//     the accumulation is fixed by the row list alone, so scores do not depend on the launch geometry.
// The tcgen05 path was not taken for this contraction: its left operand must sit in shared or tensor memory, i.e. every
// expanded element would be written and read once more (2 bytes per (token, row) against 1/8 byte of plane bits), and
// the expansion, not the multiply-add, is what costs here (12 mma per 64 tokens x 48 rows against ~100 integer ops).
//
// A tile is 16 blocks (1024 tokens) of one plan (NH query heads that share the planes read).  With the planes in device
// memory the CTAs are persistent: gridDim.x CTAs per plan walk the tiles round-robin, build the plan's row list and right
// operand once, and fetch the next stage's plane words and scales with asynchronous copies (cp.async; a row's words are
// one contiguous run, Sec. 3.6) into the other half of a double buffer.  A stage is a tile and up to 96 rows, or half a tile and up to
// 160; deeper plans take half tiles in passes of up to 96 rows and carry the accumulators over the passes.  The right operand of all rows stays in shared memory.
// With the planes in pinned host memory the grid is one CTA per tile, which keeps the requests on the host link sequential.
// Only planes p < t_j and the scales of active channels are ever read.
#include "scan_shared.cuh"

#include <cstdlib>
#include <cstring>
#include <type_traits>

namespace {

constexpr int THREADS = 128, WARPS = 4;
constexpr int TILE_BLOCKS = FATHOM_SCAN_TILE_BLOCKS;
constexpr int MAX_ROWS = FATHOM_D * FATHOM_NPLANES;          // 512 (channel, plane) pairs
constexpr int MAX_KSTEPS = MAX_ROWS / 16;                    // 16 rows per mma
constexpr int STAGE_ROWS = 96;                               // rows per stage
#ifndef FATHOM_SCAN_CTAS_PER_SM
#define FATHOM_SCAN_CTAS_PER_SM 4                               // 16 warps per SM with ~115 registers each beat 24 warps with 80
#endif
constexpr int CTAS_PER_SM = FATHOM_SCAN_CTAS_PER_SM;

// Sub-tiles of TB blocks.  The row pitches are padded so that the four lanes of a quad, which read rows two apart, hit different
// banks (plane bytes: pitch / 4 = 4 mod 32 for TB = 16, ...).
template <int TB>
struct Geo {
  static constexpr int ROW_BYTES = 8 * TB + 16;               // pitch of a staged plane-word row
  static constexpr int SCALE_ELEMS = TB == 16 ? 24 : 8;       // pitch of a staged scale row, fp16 elements
};
constexpr int STAGE_WORDS = STAGE_ROWS * Geo<16>::ROW_BYTES;           // one buffer of staged plane words
constexpr int STAGE_SCALES = STAGE_ROWS * Geo<16>::SCALE_ELEMS * 2;    // one buffer of staged scales
constexpr int STAGE_KSTEPS = STAGE_ROWS / 16;
// deep plans stage half tiles, which leaves room for the right operand of their further rows behind the staged words
constexpr int DEEP_WORDS = STAGE_ROWS * Geo<8>::ROW_BYTES;
static_assert(2 * DEEP_WORDS + (MAX_KSTEPS - STAGE_KSTEPS) * 32 * 8 <= 2 * STAGE_WORDS, "room for the right operand of deep plans");
// half tiles of up to 160 rows fit in one stage
constexpr int HALF_KSTEPS = 10;
constexpr int HALF_WORDS = 16 * HALF_KSTEPS * Geo<8>::ROW_BYTES;
static_assert(2 * HALF_WORDS + (HALF_KSTEPS - STAGE_KSTEPS) * 32 * 8 <= 2 * STAGE_WORDS, "room for the right operand of their further rows");
static_assert(16 * HALF_KSTEPS * Geo<8>::SCALE_ELEMS * 2 <= STAGE_SCALES, "room for their scales");

// MODE 2.  A lane whose eight scores hold a candidate parks all eight in its warp's ring (three stores, no atomic, no
// loop); when the ring may not take another round of 32, the warp sifts it with all lanes, one parked group per lane,
// into the CTA's four candidate lists (one shared-memory atomic per head); the lists go to the heads' global lists once,
// when the CTA has scanned its last tile (one global atomic per head and CTA).
constexpr int PARK_RING = 64;                                // parked groups per warp
constexpr int CAND_LIST = 512;                               // candidates the CTA keeps, shared out evenly to its heads; beyond that: straight to the global list,
                                                             // with one atomic per warp, head and round (one per candidate: 500,003 tokens, 4096 of 32 heads
                                                             // with a plan each, budget 48: 155 us instead of 102; 8192 of 32 heads, budget 16: 96 instead of 76)

template <int MODE>
struct alignas(16) Smem {
  uint16_t row_id[MAX_ROWS];                                  // active row r: channel * 4 + plane
  int nrows;
  int warp_tot[WARPS];
  float wmax[WARPS][4];                                       // per warp: max_j |q_hj| of its channels
  float hscale[4], hinv[4];                                   // E_h and 1 / E_h
  float q[4][FATHOM_D];                                       // the heads' queries
  float thr[4];                                               // MODE 2: score a token must reach, per head
  uint32_t ccount[4], cbase[4];                               // MODE 2: candidates in the CTA's lists; where they go in the global lists
  uint32_t elig[2];                                           // MODE 2: eligible tokens lo <= t < hi of the session
  alignas(16) float4 park_lo[MODE == 2 ? WARPS * PARK_RING : 1];     // MODE 2: scores 0..3 of a parked group
  alignas(16) float4 park_hi[MODE == 2 ? WARPS * PARK_RING : 1];     //         scores 4..7
  uint32_t park_tok[MODE == 2 ? WARPS * PARK_RING : 1];       //         its first token (30 bits) and the head within the CTA (2 bits)
  uint2 clist[MODE == 2 ? CAND_LIST : 1];                     // MODE 2: (score bits, token) per head
  alignas(16) uint2 bfr[STAGE_KSTEPS][32];                    // right operand of the first 96 rows: per 16 rows, the two B registers of every lane
  alignas(16) unsigned char words[2 * STAGE_WORDS];           // staged plane words, double buffered; deep plans: + the other rows' right operand
  alignas(16) unsigned char scale[2 * STAGE_SCALES];          // staged fp16 scales, double buffered
};

// D += A B, A 16 x 16 (row), B 16 x 8 (col), fp16 operands, fp32 accumulators
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// D = A B
__device__ __forceinline__ void mma_16816_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.0f));
}

// byte k of two rows' plane words at the top of the two halves of a register: bits 8..15 and 24..31 (the others are masked later)
__device__ __forceinline__ uint32_t row_bytes(uint32_t w0, uint32_t w1, int k) { return __byte_perm(w0, w1, 0x4000 + 0x1010 * k); }
// the scale pair with each half's sign flipped where bit J of the half's byte is clear (J = 7 sits on the sign: no shift)
template <int J>
__device__ __forceinline__ uint32_t signed_pair(uint32_t pair, uint32_t bytes) {
  return pair ^ (~(bytes << (7 - J)) & 0x80008000u);
}

// eight consecutive scores: one 32-byte store where the address allows it (a whole sector per lane), else two of 16 bytes
__device__ __forceinline__ void store_scores8(float* row, const float (&v)[8]) {
  if ((reinterpret_cast<uintptr_t>(row) & 31u) == 0) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(row), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]),
                 "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
  } else {
    *reinterpret_cast<float4*>(row) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4*>(row + 4) = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// Eight tokens of a lane (one byte of every row's plane word; x0, x1: row_bytes of the lane's two row pairs of 16 rows) times 16 rows.  Slice j of the accumulators: mma row gq = token 2 j, row gq + 8 = token 2 j + 1.
template <bool FIRST>
__device__ __forceinline__ void mma_tokens8(float (&acc)[4][4], uint32_t x0, uint32_t x1, uint32_t S0, uint32_t S1, uint2 bf) {
  auto mma = [&](float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3) {
    if (FIRST) mma_16816_first(c, a0, a1, a2, a3, bf.x, bf.y);
    else mma_16816(c, a0, a1, a2, a3, bf.x, bf.y);
  };
  mma(acc[0], signed_pair<0>(S0, x0), signed_pair<1>(S0, x0), signed_pair<0>(S1, x1), signed_pair<1>(S1, x1));
  mma(acc[1], signed_pair<2>(S0, x0), signed_pair<3>(S0, x0), signed_pair<2>(S1, x1), signed_pair<3>(S1, x1));
  mma(acc[2], signed_pair<4>(S0, x0), signed_pair<5>(S0, x0), signed_pair<4>(S1, x1), signed_pair<5>(S1, x1));
  mma(acc[3], signed_pair<6>(S0, x0), signed_pair<7>(S0, x0), signed_pair<6>(S1, x1), signed_pair<7>(S1, x1));
}

// MODE 0: scores of every token are written (fathom_scan, fathom_scan_batch).
// MODE 1: only every tile_step-th tile is scanned and its scores are written compactly (tile i of the launch at
//         token positions 1024 i ..) - the sample from which fathom_scan_topk derives a safe threshold.
// MODE 2: every tile is scanned, nothing is written but the tokens whose score reaches the head's threshold:
//         (score, token) pairs appended to the head's candidate list.
// grid = (CTAs per plan, groups of NH query heads); MODE 1 and 2 are launched with one item.
// IN_HBM: every store of the launch lies in device memory (its rows are staged past the L1).
// UNIT: blocks that a CTA takes at a time, 16 (a tile) or 8.
template <int NH, int MODE, bool IN_HBM, int CAP, int UNIT>
__global__ void __launch_bounds__(THREADS, CTAS_PER_SM)
scan_kernel(const __grid_constant__ ScanBatchOf<CAP> B, int G, int heads_per_plan, fathom_scan_fuse fz) {
  extern __shared__ __align__(16) unsigned char scan_smem[];   // sizeof(Smem<MODE>): more than the static limit in MODE 2
  Smem<MODE>& M = *reinterpret_cast<Smem<MODE>*>(scan_smem);

  FATHOM_PDL_WAIT();                                          // depths (and thresholds) come from the previous kernels
  const int total = (int)B.tile_end[B.items - 1];              // tiles of this launch (tile and block indices fit 32 bits)
  if ((int)blockIdx.x >= total) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr bool in_hbm = IN_HBM;
  constexpr int HEAD_LIST = CAND_LIST / NH;
  const int gq = lane >> 2, t4 = lane & 3;                     // mma fragment coordinates: lane = (row group, column pair)
  const int h0 = blockIdx.y * NH;                              // first of the NH query heads of this CTA
  // second attempt of the fused selection: may have nothing to do
  if (MODE == 2 && fz.gate.mode == 2 && !__syncthreads_or(fathom_gate_wants(fz.gate, h0 + tid % NH))) return;
  const int plan = h0 / heads_per_plan;                        // NH divides heads_per_plan: one plan per CTA
  const int kv = h0 / G;
  const int myh = t4 < NH ? t4 : 0;                            // the head whose scores this lane receives (lanes t4 >= NH: none)
  if (MODE == 2 && tid < 4) M.ccount[tid] = 0u;
  if (MODE == 2 && tid == 0) {                                 // (MODE 2 is launched with one session)
    const long long n0 = B.n[0];
    const long long hi = fz.local_begin < n0 ? fz.local_begin : n0, lo = fz.sink_end < hi ? fz.sink_end : hi;
    M.elig[0] = (uint32_t)lo;
    M.elig[1] = (uint32_t)hi;
  }
  if (MODE == 2 && tid < NH)                                   // read after the barriers of the first item's row list
    M.thr[tid] = !fathom_gate_wants(fz.gate, h0 + tid) ? __uint_as_float(0x7fc00000u)              // (nothing reaches a NaN)
               : fz.state_is_score ? __uint_as_float(fz.state[(h0 + tid) * 8]) : fathom_bin_lower_edge(fz.state[(h0 + tid) * 8]);

  int item = -1, nrows = 0, nb_item = 0;
  uint32_t half_stride = 0, eighth_stride = 0;                 // rows of plane words and of scales in 16-byte units, and my KV head's first
  const uint4 *planes_kv = nullptr, *scales_kv = nullptr;
  float hs = 1.0f, hs_tail = 0.0f;                             // E of my head and E 2^-11

  auto bfr_of = [&](int ks) {                                  // the right operand of 16 rows, [32 lanes]
    return ks < STAGE_KSTEPS ? M.bfr[ks]
                             : reinterpret_cast<uint2*>(M.words + (nrows <= 16 * HALF_KSTEPS ? 2 * HALF_WORDS : 2 * DEEP_WORDS)) + (ks - STAGE_KSTEPS) * 32;
  };
  // ---- right operand of all rows (made visible by the barrier that precedes the first stage's arithmetic): entry
  //      (kstep, lane, i) holds rows 16 kstep + 2 (lane & 3) + 8 i and the next one, column lane >> 2 = (head, part)
  auto fill_bfr = [&]() {
    const int entries = max(1, (nrows + 15) >> 4) * 64;        // (a plan without rows: 16 of weight and scale 0)
    for (int e = tid; e < entries; e += THREADS) {
      const int ks = e >> 6, ln = (e >> 1) & 31, i = e & 1;
      const int col = ln >> 2, head = col >> 1, part = col & 1;
      const int r0 = ks * 16 + 2 * (ln & 3) + 8 * i;
      uint32_t packed = 0u;
      if (head < NH) {
        const float inv = M.hinv[head];
#pragma unroll
        for (int z = 0; z < 2; ++z) {
          const int r = r0 + z;
          float v = 0.0f;
          if (r < nrows) {
            const int id = M.row_id[r];
            v = M.q[head][id >> 2] * inv * __int_as_float((129 - (id & 3)) << 23);
          }
          const __half hi = __float2half_rn(v);
          const __half out = part ? __float2half_rn((v - __half2float(hi)) * 2048.0f) : hi;
          packed |= (uint32_t)__half_as_ushort(out) << (16 * z);
        }
      }
      reinterpret_cast<uint32_t*>(bfr_of(ks) + ln)[i] = packed;
    }
  };

  // ---- a new session: the active row list of this plan, ordered by channel then plane (thread = channel), the
  //      heads' power-of-two scales (the right operand of every 16 rows follows once the first stage has been requested)
  auto enter_item = [&](int tile) {
    int it = item < 0 ? 0 : item;
    while (tile >= B.tile_end[it]) ++it;                       // uniform over the CTA; items only move forward
    if (it == item) return;
    item = it;
    nb_item = (int)((B.n[it] + FATHOM_BLOCK - 1) / FATHOM_BLOCK);
    const int t = min((int)B.depth[it][(size_t)plan * FATHOM_D + tid], FATHOM_NPLANES);   // a depth above 4 (an unwritten buffer) must not index past the row list
    int incl = t;                                              // inclusive prefix of depths over channels
    float qa[NH];
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      const float x = *(const volatile float*)(B.q[it] + (size_t)(h0 + h) * FATHOM_D + tid);   // (a predecessor may have written it)
      M.q[h][tid] = x;
      qa[h] = fabsf(x);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
#pragma unroll
      for (int h = 0; h < NH; ++h) qa[h] = fmaxf(qa[h], __shfl_xor_sync(0xffffffffu, qa[h], o));
    }
    if (lane == 31) M.warp_tot[warp] = incl;
#pragma unroll
    for (int h = 0; h < NH; ++h)
      if (lane == h) M.wmax[warp][h] = qa[h];
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += M.warp_tot[w];
    const int start = before + incl - t;
    for (int p = 0; p < t; ++p) M.row_id[start + p] = (uint16_t)(tid * FATHOM_NPLANES + p);
    if (tid == FATHOM_D - 1) M.nrows = before + incl;
    if (tid < NH) {                                            // E = 2^floor(log2 max|q|), kept inside the normal range
      float m = 0.0f;
#pragma unroll
      for (int w = 0; w < WARPS; ++w) m = fmaxf(m, M.wmax[w][tid]);
      int eb = (int)(__float_as_uint(m) >> 23);
      eb = eb < 1 ? 1 : (eb > 253 ? 253 : eb);
      M.hscale[tid] = __int_as_float(eb << 23);
      M.hinv[tid] = __int_as_float((254 - eb) << 23);
    }
    __syncthreads();
    nrows = M.nrows;
    half_stride = (uint32_t)(B.plane_stride[it] >> 1);          // (511 * half_stride < 2^32: fathom_check_layout)
    eighth_stride = (uint32_t)(B.scale_stride[it] >> 3);
    planes_kv = reinterpret_cast<const uint4*>(B.planes[it]) + (uint64_t)(kv * FATHOM_D * FATHOM_NPLANES) * (uint64_t)half_stride;
    scales_kv = reinterpret_cast<const uint4*>(B.scales[it]) + (uint64_t)(kv * FATHOM_D) * (uint64_t)eighth_stride;
    hs = M.hscale[myh];
    hs_tail = hs * 4.8828125e-4f;                              // 2^-11
  };

  // first block of launch tile `tile` within its session
  auto first_block = [&](int tile) -> int {
    const int tl = tile - (item ? (int)B.tile_end[item - 1] : 0);
    return tl * (MODE == 1 ? fz.tile_step : 1) * UNIT;
  };

  // a buffer's scale rows from `first` up to the next multiple of 16 (at least 16) hold 0, so that whatever the stale plane bytes of
  // those rows say they contribute +-0
  auto clear_pad = [&](auto tbc, int first, int buf) {
    const int pad = max(16, (first + 15) & ~15) - first;
    constexpr int WPR = Geo<decltype(tbc)::value>::SCALE_ELEMS / 2;           // 32-bit words per scale row
    for (int e = tid; e < pad * WPR; e += THREADS) reinterpret_cast<uint32_t*>(M.scale + buf * STAGE_SCALES)[first * WPR + e] = 0u;
  };

  uint32_t parked = 0u, stages = 0u;                           // MODE 2: groups in my warp's ring (the same in every lane); stages done
  float my_thr = 0.0f;

  // ---- MODE 2, whole warp: the parked groups, one per lane and round, into the CTA's candidate lists.  A lane marks the
  //      candidates among its group's eight scores (score reaches the head's threshold, token eligible).  Nearly always
  //      there is one: the lanes that have any are ranked per head with a ballot, lanes 0..3 reserve the heads' places
  //      with one shared-memory atomic each, and every such lane writes its first candidate; further candidates of a
  //      group take a place of their own.  All warps of a CTA sift at the same stages (every fourth): a warp that did
  //      it alone would keep the others waiting at the stage barrier.
  auto sift = [&]() {
    if (MODE != 2) return;
    __syncwarp();                                              // the parked groups are visible to the whole warp
    const uint32_t elo = M.elig[0], ehi = M.elig[1];
    auto append = [&](uint32_t h, uint32_t pos, float val, uint32_t token, uint32_t beyond) {
      if (pos < (uint32_t)HEAD_LIST) {
        M.clist[h * HEAD_LIST + pos] = make_uint2(__float_as_uint(val), token);
      } else {                                                 // list full: straight to the global list, where a place has been reserved, or at one's own
        const uint32_t at = beyond != 0xffffffffu ? beyond : atomicAdd(&fz.cand_count[h0 + h], 1u);
        if ((long long)at < fz.capacity) {
          fz.cand_score[(size_t)(h0 + h) * fz.capacity + at] = val;
          fz.cand_idx[(size_t)(h0 + h) * fz.capacity + at] = (int32_t)token;
        }
      }
    };
    for (uint32_t e0 = 0; e0 < parked; e0 += 32) {
      const uint32_t e = warp * PARK_RING + e0 + lane;
      const bool mine = e0 + lane < parked;
      const uint32_t tk = mine ? M.park_tok[e] : 0u;
      const uint32_t h = tk >> 30, tok = tk & 0x3fffffffu;
      const float th = M.thr[h];
      uint32_t mask = 0u;
      if (mine) {
        const float4 a = M.park_lo[e], b = M.park_hi[e];
        const float w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int x = 0; x < 8; ++x) mask |= (w[x] >= th && tok + x - elo < ehi - elo ? 1u : 0u) << x;
      }
      auto score_at = [&](uint32_t x) { return reinterpret_cast<const float*>(x < 4u ? &M.park_lo[e] : &M.park_hi[e])[x & 3u]; };
      uint32_t rank = 0u, tot = 0u, base = 0u;
#pragma unroll
      for (int hh = 0; hh < 4; ++hh) {
        const unsigned with = __ballot_sync(0xffffffffu, mask != 0u && h == (uint32_t)hh);
        if (h == (uint32_t)hh) rank = __popc(with & ((1u << lane) - 1u));
        if (lane == hh) tot = __popc(with);
      }
      uint32_t over = 0u;                                      // where those of my head that do not fit start in the global list
      if (lane < 4 && tot) {
        base = atomicAdd(&M.ccount[lane], tot);
        const uint32_t fits = base < (uint32_t)HEAD_LIST ? min(tot, (uint32_t)HEAD_LIST - base) : 0u;
        if (fits < tot) over = atomicAdd(&fz.cand_count[h0 + lane], tot - fits) - fits;
      }
      base = __shfl_sync(0xffffffffu, base, (int)h);
      over = __shfl_sync(0xffffffffu, over, (int)h);
      if (mask) {
        const uint32_t x = (uint32_t)__ffs((int)mask) - 1u;
        mask &= mask - 1u;
        append(h, base + rank, score_at(x), tok + x, over + rank);
      }
      while (mask) {                                           // a second candidate in one group of eight: rare
        const uint32_t x = (uint32_t)__ffs((int)mask) - 1u;
        mask &= mask - 1u;
        append(h, atomicAdd(&M.ccount[h], 1u), score_at(x), tok + x, 0xffffffffu);
      }
    }
    parked = 0u;
    __syncwarp();                                              // the ring may be written again
  };

  // ---- eight consecutive scores of head t4 (lanes with t4 < NH, tokens of an existing block): tokens tok .. tok + 7 of
  //      the session, written at position dst of the head's row (MODE 0, 1) or tested against the head's threshold (MODE 2)
  auto emit = [&](const float (&v)[8], uint32_t tok, uint32_t dst, uint32_t n, bool live) {
    if (MODE != 2) {
      if (!live) return;
      float* row = B.scores[item] + (size_t)(h0 + t4) * (size_t)B.score_stride[item] + dst;
      if (tok + 8 <= n) {
        store_scores8(row, v);
      } else {
#pragma unroll
        for (int x = 0; x < 8; ++x)
          if (tok + x < n) row[x] = v[x];
      }
    } else {
      // a lane with a candidate among its eight scores parks them (called by all lanes of the warp; `live`: the lane
      // has scores at all).  Eligibility of the tokens is checked when the ring is sifted.
      const float vmax = fmaxf(fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])), fmaxf(fmaxf(v[4], v[5]), fmaxf(v[6], v[7])));
      const bool has = live && vmax >= my_thr;
      const unsigned bal = __ballot_sync(0xffffffffu, has);
      if (bal) {                                             // (the same for every lane)
        if (has) {
          const uint32_t e = warp * PARK_RING + parked + __popc(bal & ((1u << lane) - 1u));
          M.park_lo[e] = make_float4(v[0], v[1], v[2], v[3]);
          M.park_hi[e] = make_float4(v[4], v[5], v[6], v[7]);
          M.park_tok[e] = tok | ((uint32_t)t4 << 30);
        }
        parked += __popc(bal);
        if (parked > (uint32_t)(PARK_RING - 32)) sift();
      }
    }
  };

  // ---- eight tokens' accumulators -> scores of head t4: columns 2 t4 (head part) and 2 t4 + 1 (tail part)
  auto finish = [&](const float (&acc)[4][4], uint32_t tok, uint32_t dst, uint32_t n) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[2 * j] = fmaf(acc[j][1], hs_tail, acc[j][0] * hs);
      v[2 * j + 1] = fmaf(acc[j][3], hs_tail, acc[j][2] * hs);
    }
    emit(v, tok, dst, n, t4 < NH);
  };
  // A warp's TB / 4 blocks of a stage are 16 TB tokens, and a lane takes 2 TB consecutive ones (TB = 16: half a block, TB = 8: a
  // quarter): ONE load of TB / 4 bytes per row gives all their bits, and one scale pair per row pair serves them all.  They
  // are worked eight at a time (byte k of the loaded words).  Tokens past the end of the sequence are computed from zeros or from
  // what pads the rows and never leave.
  struct Place { const unsigned char* wp; const uint16_t* sp; uint32_t tok0, dst0; };
  auto place = [&](auto tbc, int g, int u, int blk0, int buf, int buf_words) {     // blk0: the stage's first block
    constexpr int TB = decltype(tbc)::value, BYTES = TB / 4;   // plane bytes per row and lane
    const int mine = warp * (TB / 4) + (gq * BYTES) / 8;       // my block of the stage
    const int off = (gq * BYTES) % 8;                          // where my bytes start in its words
    Place p;
    p.wp = M.words + buf * buf_words + (2 * t4) * Geo<TB>::ROW_BYTES + mine * 8 + off;
    p.sp = reinterpret_cast<const uint16_t*>(M.scale + buf * STAGE_SCALES) + (2 * t4) * Geo<TB>::SCALE_ELEMS + mine;
    p.tok0 = (uint32_t)(blk0 + mine) * FATHOM_BLOCK + off * 8;                               // my first token
    p.dst0 = MODE == 1 ? (uint32_t)g * (TILE_BLOCKS * FATHOM_BLOCK) + (uint32_t)(u * TB + mine) * FATHOM_BLOCK + off * 8 : p.tok0;
    return p;
  };
  auto load_rows = [&](auto tbc, const unsigned char* wk, const uint16_t* sk, uint32_t (&w)[4], uint32_t (&S)[2]) {
    constexpr int TB = decltype(tbc)::value, RB = Geo<TB>::ROW_BYTES, SE = Geo<TB>::SCALE_ELEMS;
    auto plane_bytes = [](const unsigned char* p) -> uint32_t {
      return TB == 16 ? *reinterpret_cast<const uint32_t*>(p) : (uint32_t)*reinterpret_cast<const uint16_t*>(p);
    };
    w[0] = plane_bytes(wk);
    w[1] = plane_bytes(wk + RB);
    w[2] = plane_bytes(wk + 8 * RB);
    w[3] = plane_bytes(wk + 9 * RB);
    S[0] = __byte_perm(sk[0], sk[SE], 0x5410);
    S[1] = __byte_perm(sk[8 * SE], sk[9 * SE], 0x5410);
  };
  // A stage holds all rows, NKS x 16 of them (the last 16 may be padded), of TB blocks: a tile of up to 96 rows, or half a tile of up to
  // 160.  A thread copies the same 16-byte column of the same rows in every stage, so where they start is kept in registers.  Up to 96
  // rows the words and scales a lane reads are in registers before the first MMA, and so is the right operand of up to four steps (of
  // more it would spill); of more rows the accumulators of all the lane's tokens are kept and the rows walked once.  (In two passes of up to 96
  // rows, with a barrier and copy offsets made anew for each, 136 rows took 127 us at 1,048,576 tokens, 8 plans, against 104, and 7.9 at 4096
  // tokens against 4.7.)
  auto run_single = [&](auto tbc, auto nksc, int g, int end) {
    constexpr int TB = decltype(tbc)::value, NKS = decltype(nksc)::value, RB = Geo<TB>::ROW_BYTES, SE = Geo<TB>::SCALE_ELEMS;
    constexpr int BYTES = TB / 4;                              // plane bytes per row and lane
    constexpr bool KEEP = NKS <= 4, WALK = NKS > STAGE_KSTEPS;
    constexpr int WC = TB / 2, WR = THREADS / WC, WS = (16 * NKS + WR - 1) / WR;          // columns of a row of words, rows and sweeps of the CTA over them
    constexpr int SC = TB / 8, SR = THREADS / SC, SS = (16 * NKS + SR - 1) / SR;          // ... of the scales
    constexpr int BUF = TB == 16 ? STAGE_WORDS : HALF_WORDS;
    // half tiles of one device-resident session's whole-tile launch are dealt out one by one all the same: the shares are even to a half tile
    // (decode step, 136 rows, 500,003 tokens 98.7 -> 96.6 us; a plan per head, 262,144 tokens 145.6 -> 141.0).  Over the host link a CTA takes its
    // tile's halves one after the other: they are the two ends of the same lines (136 rows, 8192 tokens, 8 plans 46.8 -> 39.5 us)
    constexpr bool SINGLY = TB < UNIT && MODE == 0 && CAP == 1 && IN_HBM;
    const int last = SINGLY ? (nb_item + TB - 1) / TB : end;
    auto block_of = [&](int g, int u) { return SINGLY ? g * TB : first_block(g) + u * TB; };
    const int wc = tid % WC, wr = tid / WC, sc = tid % SC, sr = tid / SC;
    uint32_t wo[WS], so[SS];
#pragma unroll
    for (int i = 0; i < WS; ++i) wo[i] = (uint32_t)M.row_id[min(wr + WR * i, MAX_ROWS - 1)] * half_stride;
#pragma unroll
    for (int i = 0; i < SS; ++i) so[i] = (uint32_t)(M.row_id[min(sr + SR * i, MAX_ROWS - 1)] >> 2) * eighth_stride;
    auto prefetch = [&](int blk0, int buf) {
      const int nblk = nb_item - blk0;                         // >= 1
      const bool vw = 2 * wc < nblk, vs = 8 * sc < nblk;
      const uint4* words_src = planes_kv + (vw ? (blk0 >> 1) + wc : 0);       // (nothing is read where there is no block)
      const uint4* scales_src = scales_kv + (vs ? (blk0 >> 3) + sc : 0);
      unsigned char* wd = M.words + buf * BUF + wr * RB + wc * 16;
      unsigned char* sd = M.scale + buf * STAGE_SCALES + sr * (SE * 2) + sc * 16;
#pragma unroll
      for (int i = 0; i < WS; ++i)
        if ((!WALK && WR * (i + 1) <= 16 * (NKS - 1)) || wr + WR * i < nrows) fathom_copy_async<16>(wd + i * (WR * RB), words_src + wo[i], vw, in_hbm);
#pragma unroll
      for (int i = 0; i < SS; ++i)
        if (sr + SR * i < nrows) fathom_copy_async<16>(sd + i * (SR * SE * 2), scales_src + so[i], vs, in_hbm);
      fathom_copies_commit();
    };
    prefetch(block_of(g, 0), 0);                               // the first stage's rows are on their way ...
    clear_pad(tbc, nrows, 0);
    clear_pad(tbc, nrows, 1);
    fill_bfr();                                                // ... while the right operand is made
    const uint32_t n = (uint32_t)B.n[item];                    // n < 2^31
    uint2 bf[KEEP ? NKS : 1];
    for (int u = 0, buf = 0;; buf ^= 1) {
      int g_next = g, u_next = u + 1;                          // (of half tiles: the tile's second, where it has blocks)
      if (SINGLY || TB == UNIT || u_next == UNIT / TB || first_block(g) + u_next * TB >= nb_item) {
        u_next = 0;
        g_next = g + gridDim.x;
      }
      const bool more = g_next < last;
      fathom_copies_wait<0>();
      __syncthreads();                                         // this stage's words and scales are in place, and every warp has
                                                               // left the previous stage: its buffer may be refilled
      if (more) prefetch(block_of(g_next, u_next), buf ^ 1);   // lands while this stage is scanned
      const Place at = place(tbc, g, u, block_of(g, u), buf, BUF);
      if constexpr (WALK) {
        float acc[BYTES][4][4];
        auto step = [&](auto first, int ks, uint2 b) {
          uint32_t w[4], S[2];
          load_rows(tbc, at.wp + ks * (16 * RB), at.sp + ks * (16 * SE), w, S);
#pragma unroll
          for (int k = 0; k < BYTES; ++k)
            mma_tokens8<decltype(first)::value>(acc[k], row_bytes(w[0], w[1], k), row_bytes(w[2], w[3], k), S[0], S[1], b);
        };
        step(std::true_type{}, 0, M.bfr[0][lane]);
#pragma unroll
        for (int ks = 1; ks < STAGE_KSTEPS; ++ks) step(std::false_type{}, ks, M.bfr[ks][lane]);
        const uint2* further = bfr_of(STAGE_KSTEPS) + lane;
#pragma unroll 1
        for (int ks = STAGE_KSTEPS; 16 * ks < nrows; ++ks, further += 32) step(std::false_type{}, ks, *further);
#pragma unroll
        for (int k = 0; k < BYTES; ++k) finish(acc[k], at.tok0 + 8 * k, at.dst0 + 8 * k, n);
      } else {
        uint32_t w[NKS][4], S[NKS][2];
#pragma unroll
        for (int ks = 0; ks < NKS; ++ks) {
          if (KEEP) bf[ks] = M.bfr[ks][lane];
          load_rows(tbc, at.wp + ks * (16 * RB), at.sp + ks * (16 * SE), w[ks], S[ks]);
        }
#pragma unroll
        for (int k = 0; k < BYTES; ++k) {
          float acc[4][4];
#pragma unroll
          for (int ks = 0; ks < NKS; ++ks) {
            const uint32_t x0 = row_bytes(w[ks][0], w[ks][1], k), x1 = row_bytes(w[ks][2], w[ks][3], k);
            const uint2 b = KEEP ? bf[KEEP ? ks : 0] : M.bfr[ks][lane];
            if (ks == 0) mma_tokens8<true>(acc, x0, x1, S[ks][0], S[ks][1], b);
            else mma_tokens8<false>(acc, x0, x1, S[ks][0], S[ks][1], b);
          }
          finish(acc, at.tok0 + 8 * k, at.dst0 + 8 * k, n);
        }
      }
      if (MODE == 2 && (++stages & 3u) == 0u) sift();          // (every warp of the CTA at the same stages)
      if (!more) return;
      g = g_next;
      u = u_next;
    }
  };
  // plans of more than 160 rows: the accumulators of the lane's tokens are carried over the passes of a half tile (those of a whole
  // tile, 64 registers, would spill)
  auto run_passes = [&](int g, int end) {
    constexpr std::integral_constant<int, 8> tbc{};
    constexpr int TB = 8, BYTES = TB / 4;
    const int npass = (nrows + STAGE_ROWS - 1) / STAGE_ROWS;
    const int rows_stage = ((nrows + npass - 1) / npass + 15) & ~15;          // equal passes of whole ksteps, at most 96 rows
    // plane words and scales of one stage: half tile u of tile g, rows of `pass`
    auto prefetch = [&](int g, int u, int pass, int buf) {
      const int blk0 = first_block(g) + u * TB;
      const int nblk = nb_item - blk0;                         // >= 1: stages past the last block are never entered
      const int s0 = pass * rows_stage, sc = min(rows_stage, nrows - s0);
      const int c = tid & 3;                                   // my 16-byte column of every row I copy
      const bool valid = 2 * c < nblk;
      const uint4* words_src = planes_kv + (valid ? (blk0 >> 1) + c : 0);
      unsigned char* wd = M.words + buf * DEEP_WORDS + c * 16;
      for (int r = tid >> 2; r < sc; r += THREADS >> 2)
        fathom_copy_async<16>(wd + r * Geo<TB>::ROW_BYTES, words_src + (uint32_t)M.row_id[s0 + r] * half_stride, valid, in_hbm);
      unsigned char* sd = M.scale + buf * STAGE_SCALES;
      for (int r = tid; r < sc; r += THREADS)
        fathom_copy_async<16>(sd + r * (Geo<TB>::SCALE_ELEMS * 2), scales_kv + (blk0 >> 3) + (uint32_t)(M.row_id[s0 + r] >> 2) * eighth_stride, true, in_hbm);
      clear_pad(tbc, sc, buf);
      fathom_copies_commit();
    };
    prefetch(g, 0, 0, 0);
    fill_bfr();
    float acc[BYTES][4][4];
    for (int u = 0, pass = 0, buf = 0;; buf ^= 1) {
      int g_next = g, u_next = u, pass_next = pass + 1;
      if (pass_next == npass) {
        pass_next = 0;
        u_next = u + 1;
        if (u_next * TB >= UNIT || first_block(g) + u_next * TB >= nb_item) { u_next = 0; g_next = g + gridDim.x; }
      }
      const bool more = g_next < end;
      fathom_copies_wait<0>();
      __syncthreads();
      if (more) prefetch(g_next, u_next, pass_next, buf ^ 1);
      if (pass == 0) {
#pragma unroll
        for (int k = 0; k < BYTES; ++k)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[k][j][0] = acc[k][j][1] = acc[k][j][2] = acc[k][j][3] = 0.0f;
      }
      const Place at = place(tbc, g, u, first_block(g) + u * TB, buf, DEEP_WORDS);
      const int ks0 = pass * (rows_stage >> 4), nks = (min(rows_stage, nrows - pass * rows_stage) + 15) >> 4;
#pragma unroll 2
      for (int ks = 0; ks < nks; ++ks) {
        uint32_t w[4], S[2];
        const uint2 bf = bfr_of(ks0 + ks)[lane];
        load_rows(tbc, at.wp + ks * (16 * Geo<TB>::ROW_BYTES), at.sp + ks * (16 * Geo<TB>::SCALE_ELEMS), w, S);
#pragma unroll
        for (int k = 0; k < BYTES; ++k)
          mma_tokens8<false>(acc[k], row_bytes(w[0], w[1], k), row_bytes(w[2], w[3], k), S[0], S[1], bf);
      }
      if (pass == npass - 1) {
        const uint32_t n = (uint32_t)B.n[item];
#pragma unroll
        for (int k = 0; k < BYTES; ++k) finish(acc[k], at.tok0 + 8 * k, at.dst0 + 8 * k, n);
        if (MODE == 2 && (++stages & 3u) == 0u) sift();
      }
      if (!more) return;
      g = g_next;
      u = u_next;
      pass = pass_next;
    }
  };

  for (int g = blockIdx.x; g < total;) {                       // session by session
    if (item >= 0) __syncthreads();                            // every warp is done with the previous session's row list
    enter_item(g);
    if (MODE == 2) my_thr = M.thr[myh];
    const int end = min(total, (int)B.tile_end[item]);
    const int nks = (nrows + 15) >> 4;
    auto shallow = [&](auto nksc) { run_single(std::integral_constant<int, UNIT>{}, nksc, g, end); };
    if (nks <= 1) shallow(std::integral_constant<int, 1>{});
    else if (nks == 2) shallow(std::integral_constant<int, 2>{});
    else if (nks == 3) shallow(std::integral_constant<int, 3>{});
    else if (nks == 4) shallow(std::integral_constant<int, 4>{});
    else if (nks == 5) shallow(std::integral_constant<int, 5>{});
    else if (nks == 6) shallow(std::integral_constant<int, 6>{});
    else if (nks <= HALF_KSTEPS) run_single(std::integral_constant<int, 8>{}, std::integral_constant<int, HALF_KSTEPS>{}, g, end);
    else run_passes(g, end);
    g += (end - g + (int)gridDim.x - 1) / (int)gridDim.x * (int)gridDim.x;      // my first tile of a later session
  }
  if (MODE == 2) {
    // ---- the CTA has scanned its last tile: what is still parked is sifted, then the four lists go to the heads' global
    //      lists, one atomic per head
    sift();
    __syncthreads();
    if (tid < NH) {
      const uint32_t c = min(M.ccount[tid], (uint32_t)HEAD_LIST);
      M.ccount[tid] = c;
      M.cbase[tid] = c ? atomicAdd(&fz.cand_count[h0 + tid], c) : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < NH && h < 4; ++h) {
      const uint32_t c = M.ccount[h], at = M.cbase[h];
      for (uint32_t e = tid; e < c; e += THREADS)
        if ((long long)(at + e) < fz.capacity) {
          const uint2 it = M.clist[h * HEAD_LIST + e];
          fz.cand_score[(size_t)(h0 + h) * fz.capacity + at + e] = __uint_as_float(it.x);
          fz.cand_idx[(size_t)(h0 + h) * fz.capacity + at + e] = (int32_t)it.y;
        }
    }
  }
}

template <int NH, int MODE, int CAP, int UNIT>
int launch_units(const ScanBatchOf<CAP>& B, int Hkv, int Hq, int heads_per_plan, const fathom_scan_fuse& fz, bool host, bool dependent,
                 cudaStream_t st) {
  const int plans = Hq / NH;
  dim3 grid((unsigned)fathom_scan_grid_ctas(B.tile_end[B.items - 1], plans, host, CTAS_PER_SM), (unsigned)plans);
  constexpr size_t smem = sizeof(Smem<MODE>);                 // dynamic: MODE 2 needs more than the static limit
  auto kernel = scan_kernel<NH, MODE, true, CAP, UNIT>;
  if (UNIT == TILE_BLOCKS && host) kernel = scan_kernel<NH, MODE, false, CAP, TILE_BLOCKS>;
  if (smem > 48 * 1024) {
    static bool configured[64][2] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FATHOM_ERR_CUDA;
    if (dev >= 0 && dev < 64 && !configured[dev][host ? 0 : 1]) {
      if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return FATHOM_ERR_CUDA;
      configured[dev][host ? 0 : 1] = true;
    }
  }
  if (dependent) {                                            // may become resident while the previous kernel of the stream runs
    if (fathom_launch_dependent(kernel, grid, dim3(THREADS), smem, st, B, Hq / Hkv, heads_per_plan, fz) != cudaSuccess)
      return FATHOM_ERR_CUDA;
    return FATHOM_OK;
  }
  kernel<<<grid, THREADS, smem, st>>>(B, Hq / Hkv, heads_per_plan, fz);
  return FATHOM_OK;
}

template <int NH, int MODE, int CAP>
int launch_scan(const ScanBatchOf<CAP>& B, int Hkv, int Hq, int heads_per_plan, const fathom_scan_fuse& fz, bool dependent, cudaStream_t st) {
  const long long tiles = B.tile_end[B.items - 1];
  if (tiles <= 0) return FATHOM_OK;
  bool host = false;                                          // any store of the launch in pinned host memory
  for (int i = 0; i < B.items; ++i) host = host || fathom_planes_in_host_memory(B.planes[i]);
  // Half tiles as the CTAs' units where all of them are resident at once, and where, over several waves of whole tiles, the busiest
  // CTA then has a tenth fewer blocks.  (Decode steps on stores that no cache holds, whole / half, 8 KV and 32 query heads, budget 48: 8192 tokens 15.7 /
  // 15.3 us, 16,384 16.5 / 16.1, 33,001 20.8 / 20.3, 100,000 36.5 / 35.9, but 200,000 45.8 / 46.1, 500,003 60.5 / 63.2; two heads per plan, 16,384
  // tokens 17.7 / 16.6; one head 33,001 16.0 / 15.4; a plan per head 8192 17.5 / 16.5, 33,001 24.1 / 24.5.)
  if constexpr (MODE == 0 && CAP == 1) {
    const int plans = Hq / NH;
    if (!host && fathom_scan_ctas_override() == 0) {
      ScanBatchOf<CAP> U = B;
      const long long halves = (fathom_nblocks(B.n[0]) + TILE_BLOCKS / 2 - 1) / (TILE_BLOCKS / 2);
      const long long x16 = fathom_scan_grid_ctas(tiles, plans, false, CTAS_PER_SM), x8 = fathom_scan_grid_ctas(halves, plans, false, CTAS_PER_SM);
      const bool resident = halves == x8, waves = tiles > x16;
      if (resident || (waves && (halves + x8 - 1) / x8 * 10 <= (tiles + x16 - 1) / x16 * 2 * 9)) {
        U.tile_end[0] = halves;
        return launch_units<NH, MODE, CAP, TILE_BLOCKS / 2>(U, Hkv, Hq, heads_per_plan, fz, false, dependent, st);
      }
    }
  }
  return launch_units<NH, MODE, CAP, TILE_BLOCKS>(B, Hkv, Hq, heads_per_plan, fz, host, dependent, st);
}

// FATHOM_SCAN_PATH=simt (read once) selects the CUDA-core kernel of scan_simt.cu for every scan of the process
bool simt_path() {
  static const bool v = [] { const char* e = getenv("FATHOM_SCAN_PATH"); return e && strcmp(e, "simt") == 0; }();
  return v;
}

template <int MODE, int CAP>
int dispatch_scan(const ScanBatchOf<CAP>& B, int Hkv, int Hq, int heads_per_plan, const fathom_scan_fuse& fz, bool dependent,
                  cudaStream_t st) {
  if (simt_path()) {
    ScanBatch W = {};
    W.items = B.items;
    for (int i = 0; i < B.items; ++i) {
      W.planes[i] = B.planes[i]; W.scales[i] = B.scales[i]; W.q[i] = B.q[i]; W.depth[i] = B.depth[i]; W.scores[i] = B.scores[i];
      W.n[i] = B.n[i]; W.plane_stride[i] = B.plane_stride[i]; W.scale_stride[i] = B.scale_stride[i]; W.score_stride[i] = B.score_stride[i];
      W.tile_end[i] = B.tile_end[i];
    }
    return fathom_scan_simt_dispatch(MODE, W, Hkv, Hq, heads_per_plan, fz, dependent, st);
  }
  switch (heads_per_plan) {
    case 1: return launch_scan<1, MODE>(B, Hkv, Hq, 1, fz, dependent, st);
    case 2: return launch_scan<2, MODE>(B, Hkv, Hq, 2, fz, dependent, st);
    case 4: return launch_scan<4, MODE>(B, Hkv, Hq, 4, fz, dependent, st);
    case 8: return launch_scan<4, MODE>(B, Hkv, Hq, 8, fz, dependent, st);   // two CTAs of four heads share a plan
    default: return FATHOM_ERR_UNSUPPORTED;
  }
}

// one session as a batch of one; `tile_step` > 1 lists only the sampled tiles
ScanBatchOf<1> single_item(const fathom_layout* L, const uint64_t* planes, const uint16_t* scales, const float* q, const uint8_t* depth,
                           float* scores, long long score_stride, int tile_step) {
  ScanBatchOf<1> B = {};
  B.items = 1;
  B.planes[0] = planes; B.scales[0] = scales; B.q[0] = q; B.depth[0] = depth; B.scores[0] = scores;
  B.n[0] = L->n; B.plane_stride[0] = L->plane_stride_words; B.scale_stride[0] = L->scale_stride; B.score_stride[0] = score_stride;
  const long long tiles = (fathom_nblocks(L->n) + TILE_BLOCKS - 1) / TILE_BLOCKS;
  B.tile_end[0] = (tiles + tile_step - 1) / tile_step;
  return B;
}

int g_ctas_override = 0;                                       // fathom_scan_set_ctas_per_plan

}  // namespace

// Whether the planes are read over the host link (pinned host memory mapped into the device's address space)
bool fathom_planes_in_host_memory(const void* planes) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, planes) != cudaSuccess) { cudaGetLastError(); return false; }
  return a.type == cudaMemoryTypeHost;
}

int fathom_scan_ctas_override() { return g_ctas_override; }

int fathom_scan_grid_ctas(long long tiles, int plans, bool host_planes, int ctas_per_sm) {
  if (g_ctas_override >= 1) return (int)(g_ctas_override < tiles ? g_ctas_override : tiles);
  if (host_planes) return (int)tiles;
  static int sms[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!sms[dev]) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 148;
    sms[dev] = v;
  }
  long long x = (long long)sms[dev] * ctas_per_sm / plans;
  if (x < 1) x = 1;
  return (int)(x < tiles ? x : tiles);
}

int fathom_scan_tile_tokens() { return TILE_BLOCKS * FATHOM_BLOCK; }

int fathom_launch_scan_sample(const fathom_layout* L, const uint64_t* planes, const uint16_t* scales, const float* q,
                              const uint8_t* depth, int heads_per_plan, float* sample, long long sample_stride,
                              int tile_step, cudaStream_t st) {
  fathom_scan_fuse fz = {};
  fz.tile_step = tile_step;
  return dispatch_scan<1>(single_item(L, planes, scales, q, depth, sample, sample_stride, tile_step), L->n_kv_heads, L->n_q_heads,
                          heads_per_plan, fz, true, st);
}

int fathom_launch_scan_filter(const fathom_layout* L, const uint64_t* planes, const uint16_t* scales, const float* q,
                              const uint8_t* depth, int heads_per_plan, const fathom_scan_fuse& fz, cudaStream_t st) {
  // (a programmatic dependent: the second, gated attempt then costs no launch latency when it has nothing to do)
  if (L->n > (1ll << 30)) return FATHOM_ERR_UNSUPPORTED;      // a parked group keeps its first token in 30 bits
  return dispatch_scan<2>(single_item(L, planes, scales, q, depth, nullptr, 0, 1), L->n_kv_heads, L->n_q_heads, heads_per_plan, fz,
                          true, st);
}

extern "C" int fathom_scan_set_ctas_per_plan(int ctas) {
  g_ctas_override = ctas > 0 ? ctas : 0;
  return FATHOM_OK;
}

extern "C" int fathom_scan(fathom_ctx* ctx, const fathom_layout* L, const uint64_t* planes, const uint16_t* scales,
                           const float* q, const uint8_t* depth, int heads_per_plan, float* scores, void* stream) {
  if (!ctx || !planes || !scales || !q || !depth || !scores) return FATHOM_ERR_INVALID_ARG;
  int rc = fathom_check_layout(L);
  if (rc != FATHOM_OK) return rc;
  const int G = L->n_q_heads / L->n_kv_heads;
  if (heads_per_plan < 1 || G % heads_per_plan != 0) return FATHOM_ERR_INVALID_ARG;
  if (!fathom_aligned16(planes) || !fathom_aligned16(scales) || !fathom_aligned16(scores)) return FATHOM_ERR_ALIGNMENT;
  fathom_scan_fuse fz = {};
  fz.tile_step = 1;
  rc = dispatch_scan<0>(single_item(L, planes, scales, q, depth, scores, L->score_stride, 1), L->n_kv_heads, L->n_q_heads, heads_per_plan,
                        fz, true, static_cast<cudaStream_t>(stream));
  if (rc != FATHOM_OK) return rc;
  FATHOM_CUDA_TRY(ctx, cudaGetLastError());
  return FATHOM_OK;
}

extern "C" int fathom_scan_batch(fathom_ctx* ctx, const fathom_scan_item* items, int n_items, int heads_per_plan, void* stream) {
  if (!ctx || !items || n_items < 1) return FATHOM_ERR_INVALID_ARG;
  const int Hkv = items[0].layout.n_kv_heads, Hq = items[0].layout.n_q_heads;
  for (int i = 0; i < n_items; ++i) {
    const fathom_scan_item& it = items[i];
    int rc = fathom_check_layout(&it.layout);
    if (rc != FATHOM_OK) return rc;
    if (it.layout.n_kv_heads != Hkv || it.layout.n_q_heads != Hq) return FATHOM_ERR_INVALID_ARG;   // one model, many sessions
    if (!it.planes || !it.scales || !it.q || !it.depth || !it.scores) return FATHOM_ERR_INVALID_ARG;
    if (!fathom_aligned16(it.planes) || !fathom_aligned16(it.scales) || !fathom_aligned16(it.scores)) return FATHOM_ERR_ALIGNMENT;
  }
  const int G = Hq / Hkv;
  if (heads_per_plan < 1 || G % heads_per_plan != 0) return FATHOM_ERR_INVALID_ARG;
  if (heads_per_plan != 1 && heads_per_plan != 2 && heads_per_plan != 4 && heads_per_plan != 8) return FATHOM_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  fathom_scan_fuse fz = {};
  fz.tile_step = 1;
  for (int first = 0; first < n_items; first += ScanBatch::MAX_ITEMS) {       // at most 32 sessions per launch
    ScanBatch B = {};
    B.items = n_items - first < ScanBatch::MAX_ITEMS ? n_items - first : ScanBatch::MAX_ITEMS;
    long long tiles = 0;
    for (int i = 0; i < B.items; ++i) {
      const fathom_scan_item& it = items[first + i];
      B.planes[i] = it.planes; B.scales[i] = it.scales; B.q[i] = it.q; B.depth[i] = it.depth; B.scores[i] = it.scores;
      B.n[i] = it.layout.n; B.plane_stride[i] = it.layout.plane_stride_words; B.scale_stride[i] = it.layout.scale_stride;
      B.score_stride[i] = it.layout.score_stride;
      tiles += (fathom_nblocks(it.layout.n) + TILE_BLOCKS - 1) / TILE_BLOCKS;
      B.tile_end[i] = tiles;
    }
    const int rc = dispatch_scan<0>(B, Hkv, Hq, heads_per_plan, fz, false, st);
    if (rc != FATHOM_OK) return rc;
  }
  FATHOM_CUDA_TRY(ctx, cudaGetLastError());
  return FATHOM_OK;
}
