// fathom_rotate_keys and fathom_build_planes_rotated on the 5th-generation tensor cores: K' = (K - mu) V  (Sec. 3.5 "Basis
// rule"), and the covariance of fathom_calibrate.
//
// The rotation is the one dense contraction next to the decode path (n x 128 by 128 x 128 per KV head), so it runs
// as tcgen05.mma with the accumulator in tensor memory.  The rotated keys feed a quantiser, so 11 significant bits are not
// enough; both operands are split into an fp16 head and an fp16 tail, x = xh + xl, v = vh + vl, and three products are
// accumulated in fp32:  xh vh + xh vl + xl vh  (the dropped xl vl term is below 2^-22 of |x||v|).  fp16 has the significant bits
// of tf32 at half the bytes and twice the rate; its range is made up for by powers of two: every token and every rotated channel
// is scaled so that its largest element lies in [2^14, 2^15), and the accumulator is scaled back (exactly) where it is read.  A
// tail has no bits below 2^-24: elements above 2^-18 of the largest keep 22 bits, smaller ones an absolute error of 2^-39 of it.
// Against fp64, keys of 0.1 to 4 with four channels at 16: 7.0e-7 of the norm (both parts in tf32, cut off: 1.7e-6); with one channel at
// 1e5 times the others and a basis that leaves it alone, the others are off by 7e-7 of theirs.
//
// The BASIS is the left operand (M = 128 rotated channels) and the tokens are the right one (N = 128):
//   * the split basis stays in tensor memory (128 columns) for all of a head's tiles, so an MMA reads only the tokens from
//     shared memory (with both operands there the MMAs alone took the whole shared-memory data path);
//   * the accumulator has a rotated channel per lane and a token per column, which is what both epilogues want: a thread
//     holds 64 tokens = one block of ONE channel.  A warp writes 128 contiguous bytes of a rotated key per store straight from
//     registers, and the quantiser's block maximum and plane words need no exchange between threads (with a token per
//     lane they took a redux, four ballots and a shuffle per element: 9.5 us a tile).
//
// One persistent CTA per SM walks a contiguous range of 128-token tiles in three roles:
//   16 producer warps  own eight rows of every tile each: one bulk copy brings them into the stage two tiles ahead, and where
//                      they lie the warp subtracts the mean, scales (a row's scale is one reduction over its lanes), splits and
//                      writes head and tail back (64 channels are one row of the 128-byte swizzle): fp32 keys take exactly
//                      the bytes of their head and tail, so a stage is one buffer for both, and three stages fit.  With the keys
//                      of the next tile in registers, two stages fitted: 403 us for 262,144 fp32 tokens x 8 heads, against 386 us;
//   1 MMA thread       issues a tile's 8 x 3 MMAs (M = N = 128, K = 16), commits them to the stage's barrier and to the
//                      accumulator's (two accumulators alternate);
//   8 epilogue warps   read the accumulator with tcgen05.ld (warp w: lanes 32 (w mod 4).., block w div 4 of the tile), hand it
//                      back, scale, and store or quantise.
// Measured: 262,144 fp32 tokens x 8 heads to planes 1057 us (both operands in shared memory, tf32) -> 375 us = 2.9 TB/s; 200,001 bf16
// tokens to rotated keys 233 us = 5.3 TB/s.  Stamps inside the kernel (fp32 to planes, ~5000 cycles a tile): a tile's MMAs take 2300
// cycles, its conversion 2100 while the epilogue rests and up to 4000 beside it, its epilogue 4900 (2500 of them the
// quantiser): the roles share the ALU's issue slots, and eight epilogue warps set the pace.  Tried: 8 producer and 16 epilogue warps, a block on
// two threads, the accumulator handed back before the quantiser runs: the producers set the pace instead (411 us).
//
// Every wait on an mbarrier is bounded; a wait that runs out sets FATHOM_DEV_WAIT_EXPIRED in the context status and
// the thread stops waiting; every role still finishes its loops, and the CTA frees its tensor memory and returns.
#include "quantise.cuh"

namespace {

constexpr int TC_THREADS = 256;                              // covariance kernel
constexpr int TILE_M = 128;                                  // tokens per tile
constexpr int KC = 32;                                       // channels per chunk = 128 bytes of tf32
constexpr int NCHUNK = FATHOM_D / KC;                        // 4
constexpr int SLAB = TILE_M * KC * 4;                        // 16 KB: 128 rows of 128 bytes
constexpr int UMMA_K = 8;                                    // tf32 elements per MMA along K (32 bytes)
constexpr uint32_t WAIT_TRIES = 1u << 22;

// rotation kernel: roles, ring of stages, shared-memory map (bytes from a 1024-byte aligned base)
constexpr int PRODUCERS = 512, EPILOGUE = 256;
constexpr int RT_THREADS = PRODUCERS + EPILOGUE + 32;        // the last warp issues the MMAs
constexpr int RK = 16;                                       // fp16 elements per MMA along K (32 bytes)
constexpr int HALF_CH = 64;                                  // channels per 128-byte row of fp16
constexpr int STAGES = 3;                                    // one arrives, one is converted, one is multiplied
constexpr int STAGE_BYTES = 4 * SLAB;                        // a tile: per group of eight rows, heads of channels 0..63, 64..127, tails of the same
constexpr int GROUP = 8, GROUPS = TILE_M / GROUP;            // rows that a producer warp owns; 1 KB per group and quarter
constexpr int GROUP_BYTES = 4 * 1024;
static_assert(GROUPS == PRODUCERS / 32 && GROUPS * GROUP_BYTES == STAGE_BYTES, "a producer warp per group");
constexpr int FACTORS = 8;                                   // ring of the tiles' token scales (producers are at most four tiles ahead)
constexpr int UNIT_BLOCKS = 4;                               // quantiser: blocks whose plane words are written together (32 bytes a row)
constexpr int OUT_PITCH = FATHOM_NPLANES * UNIT_BLOCKS * 2 + 1;             // words per channel of staged plane words, odd: no bank conflicts
constexpr int OUT_BYTES = FATHOM_D * OUT_PITCH * 4;
template <bool BUILD>
struct Map {
  static constexpr int OUT = STAGES * STAGE_BYTES;            // BUILD: 128 x OUT_PITCH words
  static constexpr int SCALE = OUT + (BUILD ? OUT_BYTES : 0); // BUILD: 128 x 4 fp16
  static constexpr int MU = SCALE + (BUILD ? FATHOM_D * UNIT_BLOCKS * 2 : 0);   // 128 floats
  static constexpr int VSCALE = MU + FATHOM_D * 4;            // 128 floats: what a rotated channel is scaled back by
  static constexpr int FACTOR = VSCALE + FATHOM_D * 4;        // FACTORS x 128 floats: what a token is scaled back by
  static constexpr int BAR = FACTOR + FACTORS * TILE_M * 4;   // full and empty barriers of the stages, full and empty of the accumulators,
  static constexpr int BARS = 2 * STAGES + 4 + STAGES * GROUPS;   // arrival of every group's keys
  static constexpr int BYTES = BAR + BARS * 8 + 16 + 1024;    // + tensor-memory base, slack for the manual 1024-byte alignment
  static_assert(BYTES <= 227 * 1024, "shared memory");
};
constexpr uint32_t COL_VH = 0, COL_VL = COL_VH + FATHOM_D / 2, COL_ACC = 128;   // tensor memory: basis head and tail (two fp16 a column), two accumulators
constexpr uint32_t RT_TMEM_COLS = 512;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float tf32_head(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// byte offset inside a group's quarter of the 16-byte piece `c4` (0..7) of row `row`: rows are 128 bytes and piece c4 of row r sits
// at position c4 ^ r (the 128-byte swizzle)
__device__ __forceinline__ int swizzled(int row, int c4) { return row * 128 + ((c4 ^ row) << 4); }

// K-major, 128-byte swizzle: start address, leading offset 1 (unused), GROUP_BYTES between 8-row groups, version 1
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3ffffu) >> 4) | (1ull << 16) | ((uint64_t)(GROUP_BYTES >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// fp32 accumulator, tf32 A and B, both K-major, N = 128, M = 128
constexpr uint32_t UMMA_IDESC = (1u << 4) | (2u << 7) | (2u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

// fp16 operands: left in tensor memory (lane = row, elements 2 c and 2 c + 1 in column c), right in shared memory
constexpr uint32_t UMMA_IDESC_F16 = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
__device__ __forceinline__ void umma_f16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, {%5, %5, %5, %5}, p;\n\t}\n"
      :: "r"(tmem_d), "r"(tmem_a), "l"(b), "r"(UMMA_IDESC_F16), "r"(accumulate), "r"(0u) : "memory");
}
// The power of two that brings `largest` (not negative) into [2^14, 2^15), and its inverse
__device__ __forceinline__ float scale_up(float largest, float& back) {
  const uint32_t e = min(max(__float_as_uint(largest) >> 23, 15u), 254u);
  back = __uint_as_float((e - 14u) << 23);
  return __uint_as_float((268u - e) << 23);
}
// fp16 head and tail of two scaled values
__device__ __forceinline__ void split2(float2 v, uint32_t& head, uint32_t& tail) {
  const __half2 h = __float22half2_rn(v);
  const __half2 l = __float22half2_rn(fathom_fma2(__half22float2(h), make_float2(-1.0f, -1.0f), v));
  head = *reinterpret_cast<const uint32_t*>(&h);
  tail = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(reinterpret_cast<unsigned long long&>(d))
      : "l"(reinterpret_cast<const unsigned long long&>(a)), "l"(reinterpret_cast<const unsigned long long&>(b)));
  return d;
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
               : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done != 0;
}
// Bounded wait for the phase with the given parity; false when the limit ran out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t tries = WAIT_TRIES) {
  for (uint32_t i = 0; i < tries; ++i) {
    if (mbar_test(bar, parity)) return true;
    if (i > 64) __nanosleep(32);
  }
  return false;
}

// The same for a whole warp whose lanes all poll (each of them reads what has arrived): false in every lane if the limit ran out for
// any.  A warp that disagreed would split at the next branch on the answer, and lanes that give up would leave the others in a
// full-mask shuffle.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, uint32_t tries = WAIT_TRIES) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, tries)) != 0;
}

// The give-up path of the bounded waits, exercised on its own (no copy, no MMA, nothing asynchronous is outstanding): one warp
// waits `tries` times on a barrier that nothing will ever arrive on, and on one whose phase is complete with a limit that has run
// out for its odd lanes.  If all lanes say that both waits gave up, FATHOM_DEV_WAIT_EXPIRED is reported.
__global__ void wait_expiry_selftest_kernel(uint32_t* dev_status, uint32_t tries) {
  __shared__ __align__(8) uint64_t bars[2];
  const uint32_t never = (uint32_t)__cvta_generic_to_shared(&bars[0]), complete = never + 8;
  if (threadIdx.x == 0) {
    mbar_init(never, 1);
    mbar_init(complete, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" :: "r"(complete) : "memory");
  }
  __syncwarp();
  const bool gave_up = !mbar_wait_warp(never, 0, tries), split = !mbar_wait_warp(complete, 0, threadIdx.x & 1 ? 0u : tries);
  const bool all = __all_sync(0xffffffffu, gave_up && split) != 0;
  if (threadIdx.x == 0 && all) atomicOr(dev_status, FATHOM_DEV_WAIT_EXPIRED);
}

__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" :: "r"(bar) : "memory");
}
// 32 columns of the warp's 32 lanes
__device__ __forceinline__ void tmem_load32(uint32_t taddr, float (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
        "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15]), "=f"(r[16]),
        "=f"(r[17]), "=f"(r[18]), "=f"(r[19]), "=f"(r[20]), "=f"(r[21]), "=f"(r[22]), "=f"(r[23]), "=f"(r[24]),
        "=f"(r[25]), "=f"(r[26]), "=f"(r[27]), "=f"(r[28]), "=f"(r[29]), "=f"(r[30]), "=f"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_store32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n"
      :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
         "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
         "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
         "r"(r[30]), "r"(r[31]) : "memory");
}
// the two epilogue warps that share 32 channels
__device__ __forceinline__ void pair_barrier(int pair) { asm volatile("bar.sync %0, 64;" :: "r"(1 + pair) : "memory"); }
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {   // one arrival; bytes may be 0
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
  if (bytes)
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// 16 bytes of a key row: four fp32 or eight bf16 channels
__device__ __forceinline__ void unpack16(const uint4& u, float (&x)[4]) {
  x[0] = __uint_as_float(u.x); x[1] = __uint_as_float(u.y); x[2] = __uint_as_float(u.z); x[3] = __uint_as_float(u.w);
}
__device__ __forceinline__ void unpack16(const uint4& u, float (&x)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int c = 0; c < 4; ++c) { x[2 * c] = __uint_as_float(w[c] << 16); x[2 * c + 1] = __uint_as_float(w[c] & 0xffff0000u); }
}
// four channels of a key, as loaded; converted where they are used (a conversion behind the load waited for it there, before the MMAs of
// the stage were issued: calibration of 131,072 bf16 tokens x 8 heads 274 -> 146 us)
template <typename T> struct Row4;
template <> struct Row4<float> { using type = float4; };
template <> struct Row4<__nv_bfloat16> { using type = uint2; };
__device__ __forceinline__ float4 row4(const float4& r) { return r; }
__device__ __forceinline__ float4 row4(const uint2& u) {
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}

// One kernel for both entry points (so that every accumulator is bit for bit the same in both).  BUILD: planes and scales of the
// rotated keys, tiles in pairs (a unit of 256 tokens = four blocks = 32 bytes of every plane row, written together:
// partial-sector writes cost a fill read each); otherwise the rotated keys themselves.
template <typename T, bool BUILD>
__global__ void __launch_bounds__(RT_THREADS, 1)
rotate_tc_kernel(const T* __restrict__ K, const float* __restrict__ mean, const float* __restrict__ basis, float* __restrict__ K_rot,
                 uint64_t* __restrict__ planes, uint16_t* __restrict__ scales, long long n, long long plane_stride, long long scale_stride,
                 long long tiles_per_head, long long total_tiles, uint32_t* __restrict__ dev_status) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // 1024-byte aligned in the shared window
  const uint32_t sm_base = smem_u32(sm);
  using MP = Map<BUILD>;
  float* s_mu = reinterpret_cast<float*>(sm + MP::MU);
  float* s_vscale = reinterpret_cast<float*>(sm + MP::VSCALE);
  float* s_factor = reinterpret_cast<float*>(sm + MP::FACTOR);
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(sm + MP::BAR + MP::BARS * 8);
  const uint32_t bar_full = sm_base + MP::BAR, bar_empty = bar_full + STAGES * 8, bar_acc_full = bar_empty + STAGES * 8,
                 bar_acc_empty = bar_acc_full + 16, bar_raw = bar_acc_empty + 16;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (uniform)
  constexpr int MMA_WARP = (PRODUCERS + EPILOGUE) / 32;

  // contiguous range of tiles of this CTA over the (KV head, tile) space
  constexpr long long UNIT = BUILD ? UNIT_BLOCKS * FATHOM_BLOCK / TILE_M : 1;
  const long long units = total_tiles / UNIT;
  const long long g0 = units * blockIdx.x / gridDim.x * UNIT, g1 = units * (blockIdx.x + 1) / gridDim.x * UNIT;

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(bar_full + 8 * s, PRODUCERS / 32);
      mbar_init(bar_empty + 8 * s, 1);
      for (int w = 0; w < GROUPS; ++w) mbar_init(bar_raw + 8 * (s * GROUPS + w), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bar_acc_full + 8 * a, 2);                     // the commit, and an arrival that passes the producers' scales on
      mbar_init(bar_acc_empty + 8 * a, EPILOGUE / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {                                     // one warp owns the tensor-memory allocation
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(s_tmem)), "r"(RT_TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *s_tmem;

  bool alive = true;                                          // false once a bounded wait ran out; the same in all lanes of a warp
  // one lane polls for its warp
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (alive) {
      bool ok = true;
      if (lane == 0) ok = mbar_wait(bar, parity);
      alive = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    }
  };
  uint32_t tcount = 0;                                        // tiles so far: accumulator and its parity
  uint32_t requested = 0;                                     // producers: tiles whose keys are on their way or here (each is waited for)

  for (long long g = g0; g < g1;) {                           // head by head
    const long long kv = g / tiles_per_head, tile0 = g - kv * tiles_per_head;
    const long long count = min(g1, (kv + 1) * tiles_per_head) - g;
    g += count;
    // keys of this warp's rows of the head's tile t into their stage (bytes past the end of the sequence are left as they are: they become
    // columns of the accumulator that are never used); c: its number among all tiles of this CTA
    constexpr int ROW = FATHOM_D * sizeof(T);
    auto request = [&](long long t, uint32_t c) {
      if (t >= count) return;
      const uint32_t stage = c % STAGES;
      wait(bar_empty + 8 * stage, ((c / STAGES) & 1u) ^ 1u);  // (a fresh barrier lets the first round through)
      if (!alive) return;
      requested = c + 1;
      if (lane != 0) return;
      const long long r0 = (tile0 + t) * TILE_M + warp * GROUP;
      const int rows = (int)max(0ll, min((long long)GROUP, n - r0));
      bulk_load(sm_base + stage * STAGE_BYTES + warp * GROUP_BYTES, reinterpret_cast<const unsigned char*>(K) + ((size_t)kv * (size_t)n + (size_t)r0) * ROW,
                (uint32_t)(rows * ROW), bar_raw + 8 * (stage * GROUPS + warp));
    };
    if (warp < GROUPS) {
      request(0, tcount);
      request(1, tcount + 1);
    }
    // ---- the head's split basis into tensor memory (lane = rotated channel j, column = channel c), its mean into shared memory
    if (warp < 4) {
      const float* V = basis + (size_t)kv * FATHOM_D * FATHOM_D + tid;
      float largest = 0.0f, back;
#pragma unroll 32
      for (int c = 0; c < FATHOM_D; ++c) largest = fmaxf(largest, fabsf(__ldg(V + c * FATHOM_D)));
      const float up = scale_up(largest, back);
      s_vscale[tid] = back;
#pragma unroll 1
      for (int c0 = 0; c0 < 2 * FATHOM_D; c0 += 64) {         // heads, then tails (32 registers at a time)
        uint32_t part[32];
#pragma unroll
        for (int c = 0; c < 64; c += 2) {
          const float* v = V + ((c0 & (FATHOM_D - 1)) + c) * FATHOM_D;
          uint32_t head, tail;
          split2(make_float2(__ldg(v) * up, __ldg(v + FATHOM_D) * up), head, tail);
          part[c / 2] = c0 < FATHOM_D ? head : tail;
        }
        tmem_store32(tmem + ((uint32_t)(warp * 32) << 16) + COL_VH + c0 / 2, part);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    } else if (warp < 8) {
      s_mu[tid - 128] = mean[(size_t)kv * FATHOM_D + tid - 128];
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    if (tid < PRODUCERS) {
      // ---- producers: 16 bytes of a row per lane
      constexpr int CH = 16 / sizeof(T);                      // channels per load
      constexpr int LANES = FATHOM_D / CH, STEP = 32 / LANES, LOADS = GROUP / STEP;   // lanes per row, rows per load
      const int row0 = lane / LANES, c0 = (lane % LANES) * CH, byte = (c0 % HALF_CH) * 2;
      float2 mu[CH / 2];                                      // negated
#pragma unroll
      for (int c = 0; c < CH / 2; ++c) mu[c] = make_float2(-s_mu[c0 + 2 * c], -s_mu[c0 + 2 * c + 1]);
      const float2 one = make_float2(1.0f, 1.0f);
      for (long long t = 0; t < count; ++t, ++tcount) {
        const uint32_t stage = tcount % STAGES;
        unsigned char* group = sm + stage * STAGE_BYTES + warp * GROUP_BYTES;
        unsigned char* to = group + (c0 / HALF_CH) * 1024;
        float* factor = s_factor + (tcount % FACTORS) * TILE_M + warp * GROUP;
        if (tcount < requested && !mbar_wait_warp(bar_raw + 8 * (stage * GROUPS + warp), (tcount / STAGES) & 1u)) alive = false;
        uint4 xr[LOADS];
#pragma unroll
        for (int i = 0; i < LOADS; ++i) xr[i] = reinterpret_cast<const uint4*>(group)[i * 32 + lane];
        __syncwarp();                                         // (what is read here is written below)
#pragma unroll
        for (int i = 0; i < LOADS; ++i) {
          float x[CH];
          float2 d[CH / 2];
          unpack16(xr[i], x);
          float largest = 0.0f;                               // the row's largest magnitude (non-negative floats order like integers)
#pragma unroll
          for (int c = 0; c < CH / 2; ++c) {
            d[c] = fathom_fma2(make_float2(x[2 * c], x[2 * c + 1]), one, mu[c]);
            largest = fmaxf(largest, fmaxf(fabsf(d[c].x), fabsf(d[c].y)));
          }
          uint32_t m = __float_as_uint(largest);
          if (LANES == 32) {
            m = __reduce_max_sync(0xffffffffu, m);
          } else {
#pragma unroll
            for (int o = LANES / 2; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
          }
          float back;
          const float up = scale_up(__uint_as_float(m), back);
          const int row = row0 + STEP * i;
          if (c0 == 0) factor[row] = back;
          uint32_t h[CH / 2], l[CH / 2];
#pragma unroll
          for (int c = 0; c < CH / 2; ++c) split2(mul2(d[c], make_float2(up, up)), h[c], l[c]);
          unsigned char* p = to + swizzled(row, byte >> 4) + (byte & 15);
          if constexpr (CH == 8) {
            *reinterpret_cast<uint4*>(p) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(p + 2048) = make_uint4(l[0], l[1], l[2], l[3]);
          } else {
            *reinterpret_cast<uint2*>(p) = make_uint2(h[0], h[1]);
            *reinterpret_cast<uint2*>(p + 2048) = make_uint2(l[0], l[1]);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy stores -> visible to the MMA
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_full + 8 * stage);
        request(t + 2, tcount + 2);
      }
    } else if (warp == MMA_WARP) {
      // (the whole warp runs the loop, one elected lane issues: addresses and descriptors then stay in uniform registers; issued
      // from a divergent branch an MMA took 66 to 80 cycles to issue, as long as it takes to run)
      const uint32_t base = __shfl_sync(0xffffffffu, sm_base, 0), tm = __shfl_sync(0xffffffffu, tmem, 0);
      bool ready = false;                                     // what the full barrier said when it was asked ahead of time: an answer takes
                                                              // ~300 cycles while the other warps store, several MMAs' worth
      for (long long t = 0; t < count; ++t, ++tcount) {
        const uint32_t buf = tcount & 1u, acc = tm + COL_ACC + buf * 128u;
        const uint32_t stage = tcount % STAGES, phase = (tcount / STAGES) & 1u;
        if (alive && !mbar_wait_warp(bar_acc_empty + 8 * buf, ((tcount >> 1) & 1u) ^ 1u)) alive = false;
        if (alive && !ready && !mbar_wait_warp(bar_full + 8 * stage, phase)) alive = false;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t slab = base + stage * STAGE_BYTES;
        if (elect_one()) {
#pragma unroll
          for (int hc = 0; hc < FATHOM_D / HALF_CH; ++hc) {
            const uint64_t xh = umma_desc(slab + hc * 1024), xl = umma_desc(slab + (2 + hc) * 1024);
#pragma unroll
            for (int ks = 0; ks < HALF_CH / RK; ++ks) {
              const uint32_t vh = tm + COL_VH + (hc * HALF_CH + ks * RK) / 2, vl = tm + COL_VL + (hc * HALF_CH + ks * RK) / 2;
              const uint64_t ko = ks * RK * 2 >> 4;           // 16-byte units along K inside the swizzled row
              umma_f16_ts(acc, vh, xl + ko, (hc | ks) ? 1u : 0u);
              umma_f16_ts(acc, vl, xh + ko, 1u);
              umma_f16_ts(acc, vh, xh + ko, 1u);
            }
          }
          umma_commit(bar_empty + 8 * stage);
          umma_commit(bar_acc_full + 8 * buf);
          mbar_arrive(bar_acc_full + 8 * buf);
        }
        ready = __all_sync(0xffffffffu, mbar_test(bar_full + 8 * ((tcount + 1) % STAGES), ((tcount + 1) / STAGES) & 1u)) != 0;
        __syncwarp();
      }
    } else {
      // ---- epilogue: my channel, my block of every tile
      const int lq = warp & 3, blk = (warp - PRODUCERS / 32) >> 2, ch = lq * 32 + lane;
      const float vscale = s_vscale[ch];
      for (long long t = 0; t < count; ++t, ++tcount) {
        const long long tile = tile0 + t;
        const uint32_t buf = tcount & 1u;
        float r[32];
        const float4* factor = reinterpret_cast<const float4*>(s_factor + (tcount % FACTORS) * TILE_M + blk * FATHOM_BLOCK);
        wait(bar_acc_full + 8 * buf, (tcount >> 1) & 1u);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t taddr = tmem + ((uint32_t)(lq * 32) << 16) + COL_ACC + buf * 128u + (uint32_t)(blk * FATHOM_BLOCK);
        auto load_half = [&](int half) {                      // 32 tokens at a time: 64 would spill
          tmem_load32(taddr + 32 * half, r);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int i = 0; i < 32; i += 4) {                   // the token's scale taken back (powers of two: exact); the channel's is left
            const float4 f = factor[8 * half + i / 4];
            const float2 a = mul2(make_float2(r[i], r[i + 1]), make_float2(f.x, f.y));
            const float2 b = mul2(make_float2(r[i + 2], r[i + 3]), make_float2(f.z, f.w));
            r[i] = a.x; r[i + 1] = a.y; r[i + 2] = b.x; r[i + 3] = b.y;
          }
        };
        auto hand_back = [&]() {                              // a later MMA overwrites the accumulator
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_acc_empty + 8 * buf);
        };
        const long long tok0 = tile * TILE_M + blk * FATHOM_BLOCK;
        const int valid = (int)min((long long)FATHOM_BLOCK, n - tok0);       // tokens of this block (may be <= 0)
        if (!BUILD) {
          float* out = K_rot + ((size_t)kv * (size_t)n + (size_t)tok0) * FATHOM_D + ch;
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            load_half(half);
            if (half == 1) hand_back();
            if (valid == FATHOM_BLOCK) {
#pragma unroll
              for (int i = 0; i < 32; ++i) out[(32 * half + i) * FATHOM_D] = r[i] * vscale;
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (32 * half + i < valid) out[(32 * half + i) * FATHOM_D] = r[i] * vscale;
            }
          }
        } else {
          // the plane builder's quantiser (build_planes.cu) on one thread's block; absent tail tokens count as 0
          float a = 0.0f;
          auto largest = [&](int half) {
            if (valid < 32 * half + 32) {
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (32 * half + i >= valid) r[i] = 0.0f;
            }
#pragma unroll
            for (int i = 0; i < 32; i += 2) a = fmaxf(a, fmaxf(fabsf(r[i]), fabsf(r[i + 1])));
          };
          load_half(1);
          largest(1);
          load_half(0);
          largest(0);
          const __half sh = __float2half_rn(a * vscale * 0.125f);   // (exact but for the one rounding to fp16)
          // the quantiser compares multiples of the stored scale with the values, so it may have both without the channel's scale
          const float sc = __half2float(sh) / vscale, inv = 1.0f / sc;
          const int bu = (int)(tile % UNIT) * (TILE_M / FATHOM_BLOCK) + blk;
          uint32_t* o = reinterpret_cast<uint32_t*>(sm + MP::OUT) + ch * OUT_PITCH + bu * 2;
          if (tile % UNIT == 0) pair_barrier(lq);             // the last unit's flush has read them
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            if (half == 1) {
              load_half(1);
              hand_back();
            }
            const int left = valid - 32 * half;
            const uint32_t keep = left >= 32 ? ~0u : (left <= 0 ? 0u : (~0u >> (32 - left)));   // absent tail tokens carry 0 bits
            uint32_t w[FATHOM_NPLANES];
            fathom_quantise32(r, sc, inv, w);
            if (!(sc > 0.0f)) { w[0] = ~0u; w[1] = w[2] = w[3] = 0u; }      // zero scale: every code is 8 = 0b1000
#pragma unroll
            for (int p = 0; p < FATHOM_NPLANES; ++p) o[p * UNIT_BLOCKS * 2 + half] = w[p] & keep;
          }
          reinterpret_cast<uint16_t*>(sm + MP::SCALE)[ch * UNIT_BLOCKS + bu] = __half_as_ushort(sh);
          if ((tile + 1) % UNIT == 0) {
            // ---- flush: the unit's four blocks of every (channel, plane) row are 32 contiguous bytes
            pair_barrier(lq);
            const int et = blk * 32 + lane;                   // of the 64 threads that have these 32 channels
            const long long nb = (n + FATHOM_BLOCK - 1) / FATHOM_BLOCK, b0 = tile / UNIT * UNIT_BLOCKS;
            const int nblk = (int)min((long long)UNIT_BLOCKS, nb - b0);
            const uint32_t* staged = reinterpret_cast<const uint32_t*>(sm + MP::OUT);
            for (int e = lq * 32 * FATHOM_NPLANES + et; e < (lq + 1) * 32 * FATHOM_NPLANES; e += 64) {
              const uint32_t* src = staged + (e >> 2) * OUT_PITCH + (e & 3) * UNIT_BLOCKS * 2;
              uint64_t* dst = planes + ((size_t)kv * FATHOM_D * FATHOM_NPLANES + e) * (size_t)plane_stride + b0;
              if (nblk == UNIT_BLOCKS && (reinterpret_cast<uintptr_t>(dst) & 31u) == 0) {   // a whole sector
                asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst), "r"(src[0]), "r"(src[1]), "r"(src[2]), "r"(src[3]),
                             "r"(src[4]), "r"(src[5]), "r"(src[6]), "r"(src[7]) : "memory");
                continue;
              }
#pragma unroll
              for (int pair = 0; pair < UNIT_BLOCKS / 2; ++pair) {
                if (2 * pair + 1 < nblk) {
                  *reinterpret_cast<uint4*>(dst + 2 * pair) = make_uint4(src[4 * pair], src[4 * pair + 1], src[4 * pair + 2], src[4 * pair + 3]);
                } else if (2 * pair < nblk) {
                  dst[2 * pair] = ((uint64_t)src[4 * pair + 1] << 32) | src[4 * pair];
                }
              }
            }
            if (blk == 0) {
              const uint16_t* src = reinterpret_cast<const uint16_t*>(sm + MP::SCALE) + ch * UNIT_BLOCKS;
              uint16_t* dst = scales + ((size_t)kv * FATHOM_D + ch) * (size_t)scale_stride + b0;
              if (nblk == UNIT_BLOCKS) {
                *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(src);
              } else {
                for (int x = 0; x < nblk; ++x) dst[x] = src[x];
              }
            }
          }
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();                                          // the epilogue has waited for every MMA of the head: basis and mean may change
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }

  if (!alive && dev_status) atomicOr(dev_status, FATHOM_DEV_WAIT_EXPIRED);
  __syncthreads();
  if (warp == MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(RT_TMEM_COLS) : "memory");
}

// ---- covariance partials on the tensor cores: C = sum_t (x_t - mu)(x_t - mu)^T ----------------------------------------
// D[i][j] += sum_t A[i][t] B[j][t] with A = B = (X - mu)^T, i.e. M = N = 128 channels and K = tokens.  X is stored token
// by token with the channels contiguous, which is the MN-major operand form: a slab holds 64 tokens x 32 channels in
// rows of 128 bytes (row = token; swizzled in 32-byte pieces over groups of four rows, the only form MN-major tf32
// operands take), four slabs side by side cover the 128 channels (leading offset = slab size), eight token rows
// (1024 bytes) are one K step.  Head and tail of the split keys serve as both operands:
// xh xh^T + xh xl^T + xl xh^T.  A CTA accumulates a contiguous token range of one KV head in tensor memory and writes
// one 128 x 128 partial at the end; the partials are summed in fp64 by the caller's reduction kernel.
constexpr int CV_TOK = 64;                                   // tokens per stage
constexpr int CV_SLAB = CV_TOK * 128;                        // 8 KB: 64 token rows of 128 bytes (32 channels)
constexpr int CV_PART = NCHUNK * CV_SLAB;                    // 32 KB: head (or tail) of one stage, 128 channels
constexpr int CV_OFF_STAGE = 4 * CV_PART;                    // two stages x (head, tail), then the epilogue staging
constexpr int CV_OFF_MU = CV_OFF_STAGE + 8 * 32 * 32 * 4;
constexpr int CV_OFF_BAR = CV_OFF_MU + FATHOM_D * 4;
constexpr int CV_SMEM = CV_OFF_BAR + 64 + 1024;
// MN-major operands of 32-bit elements take the 128-byte swizzle with a 32-byte base: rows of 128 bytes (32 channels) in
// groups of FOUR, and inside a group the 32-byte piece p of row r sits at position p ^ (r & 3).
__device__ __forceinline__ int slab_offset_mn(int row, int c4) { return row * 128 + (((((c4 >> 1) ^ (row & 3)) << 1) | (c4 & 1)) << 4); }
// descriptor: leading offset = bytes between 32-channel slabs, stride offset = bytes between 4-token groups, layout type 1
__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3ffffu) >> 4) | ((uint64_t)(CV_SLAB >> 4) << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (1ull << 61);
}
constexpr uint32_t UMMA_IDESC_MN = UMMA_IDESC | (1u << 15) | (1u << 16);   // A and B MN-major
__device__ __forceinline__ void umma_tf32_mn(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, {%5, %5, %5, %5}, p;\n\t}\n"
      :: "r"(tmem_d), "l"(a), "l"(b), "r"(UMMA_IDESC_MN), "r"(accumulate), "r"(0u) : "memory");
}

// shift[kv][c] = mean of channel c over 64 keys spread evenly over the head's sequence (any value near the data would
// do; it only has to keep S S^T / n small against the sum of squares - keys from one place, e.g. the first tokens of a
// prompt, may sit far from the rest)
// (sixteen keys per thread, requested together: eight at a time per channel took 11 us)
constexpr int SHIFT_KEYS = 64, SHIFT_GROUPS = 4;
template <typename T>
__global__ void __launch_bounds__(FATHOM_D * SHIFT_GROUPS)
cov_shift_kernel(const T* K, long long n, float* __restrict__ shift) {
  constexpr int EACH = SHIFT_KEYS / SHIFT_GROUPS;
  __shared__ float s_sum[SHIFT_GROUPS][FATHOM_D];
  FATHOM_PDL_WAIT();
  FATHOM_PDL_RELEASE();
  const int kv = blockIdx.x, c = threadIdx.x % FATHOM_D, g = threadIdx.x / FATHOM_D;
  const T* Kh = K + (size_t)kv * (size_t)n * FATHOM_D;
  const int rows = (int)min((long long)SHIFT_KEYS, n);
  const long long step = n / rows;                            // >= 1
  float v[EACH], sum = 0.0f;
#pragma unroll
  for (int u = 0; u < EACH; ++u) v[u] = g * EACH + u < rows ? (float)Kh[(size_t)((g * EACH + u) * step) * FATHOM_D + c] : 0.0f;
#pragma unroll
  for (int u = 0; u < EACH; ++u) sum += v[u];
  s_sum[g][c] = sum;
  __syncthreads();
  if (g == 0) shift[(size_t)kv * FATHOM_D + c] = ((s_sum[0][c] + s_sum[1][c]) + (s_sum[2][c] + s_sum[3][c])) / (float)rows;
}

template <typename T>
__global__ void __launch_bounds__(TC_THREADS, 1)
cov_partial_tc_kernel(const T* K, const float* shift, float* __restrict__ partial,
                      float* __restrict__ partial_sum, long long n, uint32_t* __restrict__ dev_status) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sm_base = smem_u32(sm);
  float* s_mu = reinterpret_cast<float*>(sm + CV_OFF_MU);
  float* s_stage = reinterpret_cast<float*>(sm + CV_OFF_STAGE);
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(sm + CV_OFF_BAR + 32);
  const uint32_t bar_empty0 = sm_base + CV_OFF_BAR, bar_empty1 = sm_base + CV_OFF_BAR + 8, bar_acc = sm_base + CV_OFF_BAR + 16;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, kv = blockIdx.y;
  // this CTA's tokens: stages of 64 tokens, split evenly over the CTAs of the head
  const long long stages_total = (n + CV_TOK - 1) / CV_TOK;
  const long long s0 = stages_total * blockIdx.x / gridDim.x, s1 = stages_total * (blockIdx.x + 1) / gridDim.x;
  const T* Kh = K + (size_t)kv * (size_t)n * FATHOM_D;

  if (tid == 0) {
    mbar_init(bar_empty0, 1);
    mbar_init(bar_empty1, 1);
    mbar_init(bar_acc, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(s_tmem)), "r"(256u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  FATHOM_PDL_WAIT();                                          // the shift comes from the previous kernel
  if (tid < FATHOM_D) s_mu[tid] = shift[(size_t)kv * FATHOM_D + tid];
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = *s_tmem;

  // the thread's share of a stage: eight 16-byte pieces; piece f = tid + 256 i is token f / 32, channels 4 (f % 32)..
  const int q4 = tid & 31, kc = q4 >> 3, c4 = q4 & 7, tok0 = tid >> 5;      // token tok0 + 8 i
  const int x_off = kc * CV_SLAB + slab_offset_mn(tok0, c4);                 // + 1024 i (tokens 8 apart: eight rows further)
  const float4 mu = *reinterpret_cast<const float4*>(s_mu + 4 * q4);
  using Raw = typename Row4<T>::type;
  Raw xr[8];
  auto load_stage = [&](long long st) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const long long t = st * CV_TOK + tok0 + 8 * i;
      if constexpr (sizeof(T) == 4) xr[i] = mu;               // tokens past the end count as the shift: they add nothing
      else xr[i] = Raw{};
      if (st < s1 && t < n) xr[i] = *reinterpret_cast<const Raw*>(Kh + (size_t)t * FATHOM_D + 4 * q4);
    }
  };
  load_stage(s0);
  bool alive = true;
  uint32_t q = 0;
  float4 sum4 = make_float4(0.f, 0.f, 0.f, 0.f);              // sum of (x - shift) over this thread's tokens, 4 channels
  for (long long st = s0; st < s1; ++st, ++q) {
    const int buf = q & 1;
    const uint32_t bar_empty = buf ? bar_empty1 : bar_empty0;
    if (q >= 2 && alive && !mbar_wait(bar_empty, ((q >> 1) - 1) & 1)) alive = false;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4 x = sizeof(T) == 4 || st * CV_TOK + tok0 + 8 * i < n ? row4(xr[i]) : mu;
      const float a0 = x.x - mu.x, a1 = x.y - mu.y, a2 = x.z - mu.z, a3 = x.w - mu.w;
      sum4.x += a0; sum4.y += a1; sum4.z += a2; sum4.w += a3;
      const float h0 = tf32_head(a0), h1 = tf32_head(a1), h2 = tf32_head(a2), h3 = tf32_head(a3);
      const int off = buf * 2 * CV_PART + x_off + i * 1024;
      *reinterpret_cast<float4*>(sm + off) = make_float4(h0, h1, h2, h3);
      *reinterpret_cast<float4*>(sm + off + CV_PART) = make_float4(tf32_head(a0 - h0), tf32_head(a1 - h1), tf32_head(a2 - h2), tf32_head(a3 - h3));
    }
    load_stage(st + 1);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t xh = sm_base + buf * 2 * CV_PART, xl = xh + CV_PART;
#pragma unroll
      for (int ks = 0; ks < CV_TOK / UMMA_K; ++ks) {          // eight tokens per MMA = one 1024-byte group of rows
        const uint64_t dh = umma_desc_mn(xh + ks * 1024), dl = umma_desc_mn(xl + ks * 1024);
        const uint32_t accumulate = (q | (uint32_t)ks) ? 1u : 0u;
        umma_tf32_mn(tmem_d, dh, dh, accumulate);             // first accumulator:  sum xh xh^T
        umma_tf32_mn(tmem_d + 128u, dh, dl, accumulate);      // second accumulator: sum xh xl^T (its transpose is xl xh^T)
      }
      umma_commit(bar_empty);
      if (st == s1 - 1) umma_commit(bar_acc);
    }
  }
  // (not before: CTAs of the merge that wait beside this one for the whole pass take issue slots from it - 131,072 bf16 tokens x 4 heads
  // 150 -> 144 us; beside fp32 keys they do not fit)
  FATHOM_PDL_RELEASE();
  // ---- per-channel sums of (x - shift): the eight threads of a channel quad (one per warp) are added in warp order
  {
    float4* red = reinterpret_cast<float4*>(s_stage);         // [8 warps][32 quads]
    red[warp * 32 + q4] = sum4;
    __syncthreads();
    if (warp == 0) {
      float4 t = red[q4];
#pragma unroll
      for (int w = 1; w < 8; ++w) { const float4 u = red[w * 32 + q4]; t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w; }
      *reinterpret_cast<float4*>(partial_sum + ((size_t)kv * gridDim.x + blockIdx.x) * FATHOM_D + 4 * q4) = t;
    }
    __syncthreads();                                          // the staging area is reused by the epilogue below
  }
  // ---- the partial: accumulator -> registers -> staging -> global memory (zeros if the CTA had no tokens)
  float* out_base = partial + ((size_t)kv * gridDim.x + blockIdx.x) * 2 * FATHOM_D * FATHOM_D;   // two matrices per CTA
  if (s0 < s1) {
    if (alive && !mbar_wait(bar_acc, 0)) alive = false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
#pragma unroll 1
  for (int which = 0; which < 2; ++which) {
    const int lq = warp & 3, cb = (warp >> 2) * 64;
    float4* st4 = reinterpret_cast<float4*>(s_stage + warp * 1024);
    float* out = out_base + (size_t)which * FATHOM_D * FATHOM_D + (size_t)(lq * 32) * FATHOM_D + cb;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      uint32_t r[32];
      if (s0 < s1) {
        const uint32_t taddr = tmem_d + ((uint32_t)(lq * 32) << 16) + (uint32_t)(which * 128 + cb + p * 32);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
            "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
              "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
              "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
            : "r"(taddr) : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      } else {
#pragma unroll
        for (int c = 0; c < 32; ++c) r[c] = 0u;
      }
      __syncwarp();
#pragma unroll
      for (int f = 0; f < 8; ++f)
        st4[lane * 8 + (f ^ (lane & 7))] = make_float4(__uint_as_float(r[4 * f]), __uint_as_float(r[4 * f + 1]),
                                                        __uint_as_float(r[4 * f + 2]), __uint_as_float(r[4 * f + 3]));
      __syncwarp();
#pragma unroll
      for (int it = 0; it < 8; ++it) {
        const int rr = it * 4 + (lane >> 3), f = lane & 7;
        *reinterpret_cast<float4*>(out + (size_t)rr * FATHOM_D + p * 32 + f * 4) = st4[rr * 8 + (f ^ (rr & 7))];
      }
    }
  }
  if (!alive && dev_status) atomicOr(dev_status, FATHOM_DEV_WAIT_EXPIRED);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem_d), "r"(256u) : "memory");
  }
}

}  // namespace

namespace {
template <typename T, bool BUILD>
int launch_rotate(fathom_ctx* ctx, const fathom_layout* L, const void* K, const float* mean, const float* basis, float* K_rot,
                  uint64_t* planes, uint16_t* scales, cudaStream_t st) {
  static bool configured[64] = {};
  static int sms[64] = {};
  int dev = 0;
  FATHOM_CUDA_TRY(ctx, cudaGetDevice(&dev));
  const int slot = dev >= 0 && dev < 64 ? dev : 0;
  if (!configured[slot] || slot != dev) {
    FATHOM_CUDA_TRY(ctx, cudaDeviceGetAttribute(&sms[slot], cudaDevAttrMultiProcessorCount, dev));
    FATHOM_CUDA_TRY(ctx, cudaFuncSetAttribute(rotate_tc_kernel<T, BUILD>, cudaFuncAttributeMaxDynamicSharedMemorySize, Map<BUILD>::BYTES));
    configured[slot] = true;
  }
  constexpr int UNIT = BUILD ? UNIT_BLOCKS * FATHOM_BLOCK / TILE_M : 1;
  const long long per_head = (L->n + TILE_M * UNIT - 1) / (TILE_M * UNIT) * UNIT, total = per_head * L->n_kv_heads;
  const unsigned grid = (unsigned)(total / UNIT < sms[slot] ? total / UNIT : sms[slot]);
  rotate_tc_kernel<T, BUILD><<<grid, RT_THREADS, Map<BUILD>::BYTES, st>>>(static_cast<const T*>(K), mean, basis, K_rot, planes, scales, L->n,
                                                                L->plane_stride_words, L->scale_stride, per_head, total, ctx->dev_status);
  FATHOM_CUDA_TRY(ctx, cudaGetLastError());
  return FATHOM_OK;
}
}  // namespace

int fathom_launch_rotate_tc(fathom_ctx* ctx, const fathom_layout* L, const void* K, int k_dtype, const float* mean,
                            const float* basis, float* K_rot, cudaStream_t st) {
  return k_dtype == FATHOM_F32 ? launch_rotate<float, false>(ctx, L, K, mean, basis, K_rot, nullptr, nullptr, st)
                               : launch_rotate<__nv_bfloat16, false>(ctx, L, K, mean, basis, K_rot, nullptr, nullptr, st);
}

int fathom_launch_rotate_build_tc(fathom_ctx* ctx, const fathom_layout* L, const void* K, int k_dtype, const float* mean,
                                  const float* basis, uint64_t* planes, uint16_t* scales, cudaStream_t st) {
  return k_dtype == FATHOM_F32 ? launch_rotate<float, true>(ctx, L, K, mean, basis, nullptr, planes, scales, st)
                               : launch_rotate<__nv_bfloat16, true>(ctx, L, K, mean, basis, nullptr, planes, scales, st);
}

// CTAs per KV head of the tensor-core covariance pass (one 128 x 128 partial each)
int fathom_cov_tc_ctas_per_head(int Hkv) {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int c = sms / (Hkv > 0 ? Hkv : 1);
  return c < 1 ? 1 : c;
}

namespace {
template <typename T>
int launch_cov(fathom_ctx* ctx, const fathom_layout* L, const void* K, float* shift, float* partial, float* partial_sum, dim3 grid, cudaStream_t st) {
  FATHOM_CUDA_TRY(ctx, cudaFuncSetAttribute(cov_partial_tc_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, CV_SMEM));
  FATHOM_CUDA_TRY(ctx, fathom_launch_dependent(cov_shift_kernel<T>, dim3(L->n_kv_heads), dim3(FATHOM_D * SHIFT_GROUPS), 0, st, static_cast<const T*>(K),
                                               (long long)L->n, shift));
  FATHOM_CUDA_TRY(ctx, fathom_launch_dependent(cov_partial_tc_kernel<T>, grid, dim3(TC_THREADS), CV_SMEM, st, static_cast<const T*>(K), shift, partial,
                                               partial_sum, (long long)L->n, ctx->dev_status));
  return FATHOM_OK;
}
}  // namespace

// Enqueues the shift, the covariance partials [Hkv][ctas][2][128][128] (sum xh xh^T and sum xh xl^T of the shifted
// keys, per CTA) and the per-channel sums [Hkv][ctas][128].
int fathom_launch_cov_tc(fathom_ctx* ctx, const fathom_layout* L, const void* K, int k_dtype, float* shift, float* partial,
                         float* partial_sum, int ctas_per_head, cudaStream_t st) {
  dim3 grid((unsigned)ctas_per_head, (unsigned)L->n_kv_heads);
  return k_dtype == FATHOM_F32 ? launch_cov<float>(ctx, L, K, shift, partial, partial_sum, grid, st)
                               : launch_cov<__nv_bfloat16>(ctx, L, K, shift, partial, partial_sum, grid, st);
}

extern "C" int fathom_selftest_wait_expiry(fathom_ctx* ctx, int tries, void* stream) {
  if (!ctx || tries < 1 || tries > 4096) return FATHOM_ERR_INVALID_ARG;
  wait_expiry_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(ctx->dev_status, (uint32_t)tries);
  FATHOM_CUDA_TRY(ctx, cudaGetLastError());
  return FATHOM_OK;
}
