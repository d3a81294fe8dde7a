// fathom_build_planes: K -> channel-major bit planes + fp16 block scales (Sec. 3.2, Eq. 2).
//
// Two threads own one channel of a 64-token block (32 tokens each): the 128 threads of a token half read
// every token row as 512 contiguous bytes, keep their 32 values in registers, exchange the two half maxima
// through shared memory, round a/8 to fp16 and take the codes and their plane words from fathom_quantise32
// (quantise.cuh).  A CTA walks BLOCKS_PER_CTA consecutive blocks and
// collects their plane words and scales in shared memory, then writes every (channel, plane) row segment
// as whole 32-byte sectors (partial-sector writes cost a fill read each).
// A short sequence - appended tokens - takes one block per CTA instead: there the serial walk is what costs.
#include "quantise.cuh"

namespace {

constexpr int BP_THREADS = 2 * FATHOM_D;
constexpr int HALF = FATHOM_BLOCK / 2;                         // tokens per thread

__device__ __forceinline__ float load_k(const float* p) { return *p; }
__device__ __forceinline__ float load_k(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// BLOCKS_PER_CTA: 8, or 1 for short sequences
template <typename T, int BLOCKS_PER_CTA>
__global__ void __launch_bounds__(BP_THREADS, 4)
build_planes_kernel(const T* K, uint32_t* __restrict__ planes32, uint16_t* __restrict__ scales,
                    long long n, long long nb, long long plane_stride, long long scale_stride) {
  constexpr int OUT_PITCH = FATHOM_NPLANES * BLOCKS_PER_CTA * 2 + 1;
  __shared__ float s_amax[2][2][FATHOM_D];                     // [parity of block][token half][channel]
  __shared__ uint32_t s_out[FATHOM_D][OUT_PITCH];              // [channel][plane][block][half], padded against bank conflicts
  __shared__ uint16_t s_scale[FATHOM_D][BLOCKS_PER_CTA];
  const int j = threadIdx.x & (FATHOM_D - 1);                  // channel
  const int half = threadIdx.x >> 7;                           // 0: tokens 0..31 of the block, 1: tokens 32..63
  const int h = blockIdx.y;                                    // KV head
  const long long b0 = (long long)blockIdx.x * BLOCKS_PER_CTA;
  const T* Kh = K + (size_t)h * (size_t)n * FATHOM_D;
  FATHOM_PDL_WAIT();                                           // the keys may come from the previous kernel
  FATHOM_PDL_RELEASE();

  for (int bb = 0; bb < BLOCKS_PER_CTA; ++bb) {
    const long long b = b0 + bb;
    if (b >= nb) break;                                        // uniform over the CTA
    const long long i0 = b * FATHOM_BLOCK + half * HALF;
    const int valid = (int)min((long long)HALF, n - i0);       // of this thread's 32 tokens (may be <= 0)

    float v[HALF];
    if (valid >= HALF) {
#pragma unroll
      for (int i = 0; i < HALF; ++i) v[i] = load_k(Kh + (size_t)(i0 + i) * FATHOM_D + j);
    } else {
#pragma unroll
      for (int i = 0; i < HALF; ++i) v[i] = (i < valid) ? load_k(Kh + (size_t)(i0 + i) * FATHOM_D + j) : 0.0f;
    }
    float a = 0.0f;
#pragma unroll
    for (int i = 0; i < HALF; ++i) a = fmaxf(a, fabsf(v[i]));
    s_amax[bb & 1][half][j] = a;
    __syncthreads();
    a = fmaxf(a, s_amax[bb & 1][half ^ 1][j]);

    const __half sh = __float2half_rn(a * 0.125f);             // a/8 is exact; one rounding to fp16
    const float sc = __half2float(sh);

    const uint32_t keep = (valid >= HALF) ? ~0u : (valid <= 0 ? 0u : (~0u >> (32 - valid)));   // absent tail tokens carry 0 bits
    uint32_t w[FATHOM_NPLANES];
    fathom_quantise32(v, sc, 1.0f / sc, w);
    if (!(sc > 0.0f)) { w[0] = ~0u; w[1] = w[2] = w[3] = 0u; }  // zero scale: every code is 8 = 0b1000
#pragma unroll
    for (int p = 0; p < FATHOM_NPLANES; ++p) w[p] &= keep;
    // little-endian halves of the 64-bit plane word: tokens 0..31 in the low 32 bits
#pragma unroll
    for (int p = 0; p < FATHOM_NPLANES; ++p) s_out[j][(p * BLOCKS_PER_CTA + bb) * 2 + half] = w[p];
    if (half == 0) s_scale[j][bb] = __half_as_ushort(sh);
  }
  __syncthreads();

  // ---- flush: each (channel, plane) row segment is BLOCKS_PER_CTA words (64 contiguous bytes)
  const int nblk = (int)min((long long)BLOCKS_PER_CTA, nb - b0);
  uint64_t* planes64 = reinterpret_cast<uint64_t*>(planes32);
  if (BLOCKS_PER_CTA == 1) {
    for (int e = threadIdx.x; e < FATHOM_D * FATHOM_NPLANES; e += BP_THREADS) {
      const uint32_t* src = &s_out[e / FATHOM_NPLANES][e % FATHOM_NPLANES * 2];
      planes64[((size_t)h * FATHOM_D * FATHOM_NPLANES + e) * (size_t)plane_stride + b0] = ((uint64_t)src[1] << 32) | src[0];
    }
    if (threadIdx.x < FATHOM_D) scales[((size_t)h * FATHOM_D + threadIdx.x) * (size_t)scale_stride + b0] = s_scale[threadIdx.x][0];
    return;
  }
  constexpr int PAIRS = BLOCKS_PER_CTA / 2 > 0 ? BLOCKS_PER_CTA / 2 : 1;
  for (int e = threadIdx.x; e < FATHOM_D * FATHOM_NPLANES * PAIRS; e += BP_THREADS) {
    const int pair = e % PAIRS;                                // two words = one 16-byte store
    const int p = (e / PAIRS) % FATHOM_NPLANES;
    const int c = e / (PAIRS * FATHOM_NPLANES);
    const uint32_t* src = &s_out[c][(p * BLOCKS_PER_CTA + 2 * pair) * 2];
    uint64_t* dst = planes64 + (((size_t)h * FATHOM_D + c) * FATHOM_NPLANES + p) * (size_t)plane_stride + b0 + 2 * pair;
    if (2 * pair + 1 < nblk) {
      *reinterpret_cast<uint4*>(dst) = make_uint4(src[0], src[1], src[2], src[3]);
    } else if (2 * pair < nblk) {
      dst[0] = ((uint64_t)src[1] << 32) | src[0];
    }
  }
  for (int e = threadIdx.x; e < FATHOM_D; e += BP_THREADS) {
    uint16_t* dst = scales + ((size_t)h * FATHOM_D + e) * (size_t)scale_stride + b0;
    if (nblk == BLOCKS_PER_CTA) {
      uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int x = 0; x < BLOCKS_PER_CTA; ++x) w[x / 2] |= (uint32_t)s_scale[e][x] << (16 * (x & 1));
      *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
      for (int x = 0; x < nblk; ++x) dst[x] = s_scale[e][x];
    }
  }
}

template <typename T, int BLOCKS_PER_CTA>
int launch_blocks(fathom_ctx* ctx, const fathom_layout* L, const T* K, uint64_t* planes, uint16_t* scales, cudaStream_t st) {
  const long long nb = fathom_nblocks(L->n);
  dim3 grid((unsigned)((nb + BLOCKS_PER_CTA - 1) / BLOCKS_PER_CTA), (unsigned)L->n_kv_heads);
  FATHOM_CUDA_TRY(ctx, fathom_launch_dependent(build_planes_kernel<T, BLOCKS_PER_CTA>, grid, dim3(BP_THREADS), 0, st, K,
                                               reinterpret_cast<uint32_t*>(planes), scales, (long long)L->n, nb,
                                               (long long)L->plane_stride_words, (long long)L->scale_stride));
  return FATHOM_OK;
}

// A CTA per block while that is less than one wave of CTAs (four of 64 registers x 256 threads are resident per SM): the partial
// sectors it writes are few then, and the walk over eight blocks is a chain of eight load latencies (one head, 424 tokens of
// fp32: 5.9 -> 2.9 us).
template <typename T>
int launch_build(fathom_ctx* ctx, const fathom_layout* L, const T* K, uint64_t* planes, uint16_t* scales, cudaStream_t st) {
  if (fathom_nblocks(L->n) * L->n_kv_heads <= 4LL * fathom_sm_count()) return launch_blocks<T, 1>(ctx, L, K, planes, scales, st);
  return launch_blocks<T, 8>(ctx, L, K, planes, scales, st);
}

}  // namespace

extern "C" int fathom_build_planes(fathom_ctx* ctx, const fathom_layout* L, const void* K, int k_dtype,
                                   uint64_t* planes, uint16_t* scales, void* stream) {
  if (!ctx || !K || !planes || !scales) return FATHOM_ERR_INVALID_ARG;
  int rc = fathom_check_layout(L);
  if (rc != FATHOM_OK) return rc;
  if (k_dtype != FATHOM_F32 && k_dtype != FATHOM_BF16) return FATHOM_ERR_UNSUPPORTED;
  if (!fathom_aligned16(K) || !fathom_aligned16(planes) || !fathom_aligned16(scales)) return FATHOM_ERR_ALIGNMENT;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (k_dtype == FATHOM_F32) return launch_build<float>(ctx, L, static_cast<const float*>(K), planes, scales, st);
  return launch_build<__nv_bfloat16>(ctx, L, static_cast<const __nv_bfloat16*>(K), planes, scales, st);
}
