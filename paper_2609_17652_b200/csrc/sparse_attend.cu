// fathom_sparse_attend: gather of the selected K/V rows + exact softmax attention (Sec. 2 "Top-k decoding").
//
// Split-k: CTA (split, head) handles FATHOM_ATTN_CHUNK selected rows.  Logits and the weighted V sum both give half a warp to a row (a row is
// 256 B in bf16: 16 lanes x 16 bytes, one fully coalesced row per half-warp and load instruction), 16 rows per
// half-warp with eight in flight; the partial sums are combined in a fixed order.  Every CTA
// publishes its (max, denominator, weighted sum) triple and takes a ticket; the CTA that draws the last
// ticket of a head merges all triples in split order, so the output is bit-reproducible whichever CTA
// that is, and no second launch is needed.
//
// Few rows (k <= 1024) are a chain of latencies, not bytes, and take a kernel of their own: a cluster of up to eight CTAs per head,
// each lane requests its share of 4 or 8 K rows AND of their V rows as soon as the indices are here, and the CTAs' triples meet
// in the first one's shared memory instead of in global memory behind a fence, a ticket and a second fence.
// Decode steps with it: 4096 tokens, k = 64, one head 19.3 -> 15.9 us; 33,001 tokens, k = 512, 32 heads 32.3 -> 28.5 us.
#include "fathom_common.cuh"

#include <cooperative_groups.h>
#include <mutex>

namespace cg = cooperative_groups;

namespace {

constexpr int AT_THREADS = FATHOM_ATTN_CHUNK;   // 128 threads: one per row, then one per channel
constexpr int AT_WARPS = AT_THREADS / 32;

// eight consecutive channels of a row, as loaded (converted to fp32 only when used, to keep many rows in flight)
struct Raw8h { uint4 x; };
struct Raw8f { float4 a, b; };
__device__ __forceinline__ Raw8h load_raw(const __nv_bfloat16* p) { Raw8h r; r.x = *reinterpret_cast<const uint4*>(p); return r; }
__device__ __forceinline__ Raw8f load_raw(const float* p) {
  Raw8f r; r.a = reinterpret_cast<const float4*>(p)[0]; r.b = reinterpret_cast<const float4*>(p)[1]; return r;
}
__device__ __forceinline__ void unpack(const Raw8h& r, float v[8]) {
  const uint32_t w[4] = {r.x.x, r.x.y, r.x.z, r.x.w};
#pragma unroll
  for (int c = 0; c < 4; ++c) { v[2 * c] = __uint_as_float(w[c] << 16); v[2 * c + 1] = __uint_as_float(w[c] & 0xffff0000u); }
}
__device__ __forceinline__ void unpack(const Raw8f& r, float v[8]) {
  v[0] = r.a.x; v[1] = r.a.y; v[2] = r.a.z; v[3] = r.a.w; v[4] = r.b.x; v[5] = r.b.y; v[6] = r.b.z; v[7] = r.b.w;
}
template <typename T> struct RawOf;
template <> struct RawOf<__nv_bfloat16> { using type = Raw8h; };
template <> struct RawOf<float> { using type = Raw8f; };
template <typename T>
__global__ void __launch_bounds__(AT_THREADS, 8)
attend_partial_kernel(const float* q, const T* Krows, const T* Vrows, const int32_t* idx, int k, long long n, int G, float softmax_scale,
                      float* __restrict__ partial, int splits, unsigned int* __restrict__ tickets,
                      float* __restrict__ result) {
  __shared__ float s_q[FATHOM_D];
  __shared__ float s_p[AT_THREADS];
  __shared__ int32_t s_idx[AT_THREADS];
  __shared__ float s_red[AT_WARPS];
  __shared__ float s_acc[AT_THREADS / 16][FATHOM_D];          // one partial sum per half-warp
  const int split = blockIdx.x, head = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int kv = head / G;
  FATHOM_PDL_WAIT();                                          // the indices come from the previous kernel
  FATHOM_PDL_RELEASE();                                       // (the next step's first kernel may become resident)
  const T* Kh = Krows + (size_t)kv * (size_t)n * FATHOM_D;
  const T* Vh = Vrows + (size_t)kv * (size_t)n * FATHOM_D;
  s_q[tid] = q[(size_t)head * FATHOM_D + tid];
  const int pos = split * AT_THREADS + tid;
  const bool valid = pos < k;
  int32_t row = 0;
  if (valid) {
    row = idx[(size_t)head * k + pos];
    row = (row < 0) ? 0 : ((long long)row >= n ? (int32_t)(n - 1) : row);   // out-of-range indices are clamped, never dereferenced
  }
  s_idx[tid] = row;
  __syncthreads();

  // Half a warp per row (16 lanes x 8 channels = one fully coalesced row per load instruction), 16 rows per half-warp: the K rows, then
  // the V rows, FLY of them in flight all the time, so that V rows arrive while the chunk maximum and the exponentials are
  // computed.  (All sixteen in flight take 96 and 168 registers, so that fewer CTAs are resident: 32 heads of 4096 bf16 rows
  // 14.5 us instead of 13.6, 64 heads of 2048 fp32 rows 25.4 instead of 23.1.)
  using Raw = typename RawOf<T>::type;
  constexpr int FLY = sizeof(T) == 2 ? 8 : 4;
  const int hw = tid >> 4, l16 = tid & 15;
  Raw raw[FLY];
  auto request = [&](int u) {                                 // u < 16: K row u, else V row u - 16
    raw[u % FLY] = load_raw((u < 16 ? Kh : Vh) + (size_t)s_idx[hw * 16 + u % 16] * FATHOM_D + l16 * 8);
  };
#pragma unroll
  for (int u = 0; u < FLY; ++u) request(u);
  {
    float qv[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) qv[c] = s_q[l16 * 8 + c];
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      float x[8];
      unpack(raw[u % FLY], x);
      float part = 0.0f;
#pragma unroll
      for (int c = 0; c < 8; ++c) part = fmaf(x[c], qv[c], part);
      request(u + FLY);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);   // fixed butterfly order
      if (l16 == 0) s_p[hw * 16 + u] = part;
    }
  }
  __syncthreads();
  const float e = valid ? s_p[tid] * softmax_scale : -INFINITY;
  __syncthreads();                                           // s_p is reused for the probabilities below
  float m = e;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) s_red[warp] = m;
  __syncthreads();
  m = fmaxf(fmaxf(s_red[0], s_red[1]), fmaxf(s_red[2], s_red[3]));
  const float p = valid ? expf(e - m) : 0.0f;
  s_p[tid] = p;
  float l = p;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  __syncthreads();                                           // s_red reads done, s_p visible
  if (lane == 0) s_red[warp] = l;

  // weighted V sum (lane = 8 channels); the eight half-warps are summed in a fixed order
  {
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      float x[8];
      unpack(raw[u % FLY], x);
      const float pr = s_p[hw * 16 + u];                       // rows past k carry probability 0
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[c] = fmaf(pr, x[c], acc[c]);
      if (u + FLY < 16) request(16 + u + FLY);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) s_acc[hw][l16 * 8 + c] = acc[c];
  }
  __syncthreads();
  float* out = partial + ((size_t)head * splits + split) * (FATHOM_D + 2);
  out[2 + tid] = (((s_acc[0][tid] + s_acc[1][tid]) + (s_acc[2][tid] + s_acc[3][tid])) +
                  ((s_acc[4][tid] + s_acc[5][tid]) + (s_acc[6][tid] + s_acc[7][tid])));
  if (tid == 0) { out[0] = m; out[1] = ((s_red[0] + s_red[1]) + s_red[2]) + s_red[3]; }

  // ---- publish; the CTA that draws the head's last ticket merges all chunks (and re-arms the ticket counter)
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    const unsigned int t = atomicAdd(&tickets[head], 1u);
    s_last = (t == (unsigned int)splits - 1u);
    if (s_last) tickets[head] = 0u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const float* P = partial + (size_t)head * splits * (FATHOM_D + 2);
  float M = -INFINITY;
#pragma unroll 8
  for (int s = 0; s < splits; ++s) M = fmaxf(M, __ldcg(P + (size_t)s * (FATHOM_D + 2)));
  float num = 0.0f, den = 0.0f;
#pragma unroll 8
  for (int s = 0; s < splits; ++s) {
    const float* ps = P + (size_t)s * (FATHOM_D + 2);
    const float w = expf(__ldcg(ps) - M);
    den = fmaf(w, __ldcg(ps + 1), den);
    num = fmaf(w, __ldcg(ps + 2 + tid), num);
  }
  result[(size_t)head * FATHOM_D + tid] = num / den;
}

// ---- few rows: one cluster per head, gridDim.x CTAs of 16 half-warps x ROWS rows
constexpr int FEW_THREADS = 256, FEW_HW = FEW_THREADS / 16, FEW_CLUSTER = 8;
template <typename T, int ROWS>
__global__ void __launch_bounds__(FEW_THREADS)
attend_few_kernel(const float* q, const T* Krows, const T* Vrows, const int32_t* idx, int k, long long n, int G, float softmax_scale, float* __restrict__ result) {
  __shared__ float s_max[FEW_HW], s_sum[FEW_HW];
  __shared__ __align__(16) float s_acc[FEW_HW][FATHOM_D];     // one partial sum per half-warp
  __shared__ float s_num[FEW_CLUSTER][FATHOM_D], s_m[FEW_CLUSTER], s_den[FEW_CLUSTER];   // first CTA: the cluster's triples
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = blockIdx.x, ctas = gridDim.x, head = blockIdx.y, tid = threadIdx.x, hw = tid >> 4, l16 = tid & 15;
  auto started = cluster.barrier_arrive();                    // (its shared memory may be written once everyone has started)
  FATHOM_PDL_WAIT();                                          // the indices come from the previous kernel
  FATHOM_PDL_RELEASE();
  const size_t rows0 = (size_t)(head / G) * (size_t)n;
  const int pos = (rank * FEW_HW + hw) * ROWS;                // first of the half-warp's positions
  int32_t mine = 0;
  if (l16 < ROWS && pos + l16 < k) {
    mine = idx[(size_t)head * k + pos + l16];
    mine = (mine < 0) ? 0 : ((long long)mine >= n ? (int32_t)(n - 1) : mine);   // out-of-range indices are clamped, never dereferenced
  }
  const float4* qp = reinterpret_cast<const float4*>(q + (size_t)head * FATHOM_D + l16 * 8);
  float qv[8];
  if ((reinterpret_cast<uintptr_t>(q) & 15u) == 0) {
    const float4 a = qp[0], b = qp[1];
    qv[0] = a.x; qv[1] = a.y; qv[2] = a.z; qv[3] = a.w; qv[4] = b.x; qv[5] = b.y; qv[6] = b.z; qv[7] = b.w;
  } else {
#pragma unroll
    for (int c = 0; c < 8; ++c) qv[c] = q[(size_t)head * FATHOM_D + l16 * 8 + c];
  }
  using Raw = typename RawOf<T>::type;
  Raw kr[ROWS], vr[ROWS];
  size_t at[ROWS];
#pragma unroll
  for (int u = 0; u < ROWS; ++u) at[u] = (rows0 + (size_t)__shfl_sync(0xffffffffu, mine, u, 16)) * FATHOM_D + l16 * 8;
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {                            // (positions past k: nothing is loaded)
    kr[u] = Raw{};
    if (pos + u < k) kr[u] = load_raw(Krows + at[u]);
  }
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    vr[u] = Raw{};
    if (pos + u < k) vr[u] = load_raw(Vrows + at[u]);
  }
  float e[ROWS], m = -INFINITY;
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    float x[8], part = 0.0f;
    unpack(kr[u], x);
#pragma unroll
    for (int c = 0; c < 8; ++c) part = fmaf(x[c], qv[c], part);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);   // every lane has the sum
    e[u] = pos + u < k ? part * softmax_scale : -INFINITY;
    m = fmaxf(m, e[u]);
  }
  if (l16 == 0) s_max[hw] = m;
  __syncthreads();
  m = -INFINITY;
#pragma unroll
  for (int h = 0; h < FEW_HW; ++h) m = fmaxf(m, s_max[h]);    // of the CTA (it has at least one row)
  float l = 0.0f, acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    const float p = pos + u < k ? expf(e[u] - m) : 0.0f;
    float x[8];
    unpack(vr[u], x);
    l += p;
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = fmaf(p, x[c], acc[c]);
  }
  float4* to = reinterpret_cast<float4*>(&s_acc[hw][l16 * 8]);
  to[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
  to[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
  if (l16 == 0) s_sum[hw] = l;
  __syncthreads();
  float num = 0.0f, den = 0.0f;
  if (tid < FATHOM_D) {
#pragma unroll
    for (int h = 0; h < FEW_HW; ++h) { num += s_acc[h][tid]; den += s_sum[h]; }
  }
  cluster.barrier_wait(std::move(started));
  if (ctas == 1) {
    if (tid < FATHOM_D) result[(size_t)head * FATHOM_D + tid] = num / den;
    return;
  }
  if (tid < FATHOM_D) {
    cluster.map_shared_rank(&s_num[0][0], 0)[rank * FATHOM_D + tid] = num;
    if (tid == 0) {
      cluster.map_shared_rank(s_m, 0)[rank] = m;
      cluster.map_shared_rank(s_den, 0)[rank] = den;
    }
  }
  cluster.sync();
  if (rank != 0 || tid >= FATHOM_D) return;
  m = s_m[0];
  for (int c = 1; c < ctas; ++c) m = fmaxf(m, s_m[c]);
  num = den = 0.0f;
  for (int c = 0; c < ctas; ++c) {                            // in rank order
    const float w = expf(s_m[c] - m);
    den = fmaf(w, s_den[c], den);
    num = fmaf(w, s_num[c][tid], num);
  }
  result[(size_t)head * FATHOM_D + tid] = num / den;
}

template <typename T, int ROWS>
cudaError_t launch_few(const float* q, const void* K, const void* V, const int32_t* idx, int k, long long n, int Hq, int G, float scale, float* out,
                       cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  const unsigned ctas = (unsigned)((k + FEW_HW * ROWS - 1) / (FEW_HW * ROWS));
  cfg.gridDim = dim3(ctas, (unsigned)Hq);
  cfg.blockDim = dim3(FEW_THREADS);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ctas;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, attend_few_kernel<T, ROWS>, q, static_cast<const T*>(K), static_cast<const T*>(V), idx, k, n, G, scale, out);
}

// The kernel for k rows, the same for both entry points.  Beyond 1024 rows the gather is bound by memory, which the CTAs of 128 rows
// fill better than clusters do.  Clusters that are not all resident at once lose more: the next one waits until a whole cluster has
// left.  That costs more than they gain where the other kernel is at its best, with eight chunks (their triples are merged in one
// round of loads, fewer of them one after the other), and with more than 128 heads.  Us with clusters / with CTAs of 128 rows: 1024 bf16 rows,
// 48 heads 6.1 / 6.8, 64 heads 9.5 / 7.3, 128 heads 15.1 / 10.6; 1024 fp32 rows, 32 heads 6.1 / 7.6, 40 heads 10.2 / 8.5; 896 bf16
// rows, 64 heads 8.6 / 10.4, 128 heads 14.0 / 13.9; 512 bf16 rows, 128 heads 9.3 / 8.8, 256 heads 15.5 / 12.2.
constexpr int FEW_ROWS = FEW_CLUSTER * FEW_HW * 8;
template <typename T>
bool takes_clusters(int k, int Hq) {
  if (k > FEW_ROWS) return false;
  if (k <= FEW_ROWS - FATHOM_ATTN_CHUNK && Hq <= 128) return true;
  const bool short_rows = k <= FEW_ROWS / 2;                  // (four rows per half-warp)
  const int rows = short_rows ? 4 : 8, per_sm = sizeof(T) == 2 ? (short_rows ? 5 : 3) : (short_rows ? 4 : 2);   // by their registers: 48, 80; 62, 102
  return (long long)Hq * ((k + FEW_HW * rows - 1) / (FEW_HW * rows)) <= (long long)per_sm * fathom_sm_count();
}
template <typename T>
cudaError_t launch_attend(const float* q, const void* K, const void* V, const int32_t* idx, int k, long long n, int Hq, int G, float scale,
                          float* partial, int splits, unsigned int* tickets, float* out, cudaStream_t st) {
  if (takes_clusters<T>(k, Hq))
    return (k <= FEW_ROWS / 2 ? launch_few<T, 4> : launch_few<T, 8>)(q, K, V, idx, k, n, Hq, G, scale, out, st);
  // (launched so that its CTAs may become resident while the selection kernel still runs)
  return fathom_launch_dependent(attend_partial_kernel<T>, dim3((unsigned)splits, (unsigned)Hq), dim3(AT_THREADS), 0, st, q, static_cast<const T*>(K),
                                 static_cast<const T*>(V), idx, k, n, G, scale, partial, splits, tickets, out);
}

}  // namespace

extern "C" int fathom_sparse_attend(fathom_ctx* ctx, const fathom_layout* L, const float* q, const void* Krows,
                                    const void* Vrows, int row_dtype, const int32_t* idx, int k, float softmax_scale,
                                    float* out, void* stream) {
  if (!ctx || !q || !Krows || !Vrows || !idx || !out) return FATHOM_ERR_INVALID_ARG;
  int rc = fathom_check_layout(L);
  if (rc != FATHOM_OK) return rc;
  if (k < 1 || k > L->n) return FATHOM_ERR_INVALID_ARG;
  if (row_dtype != FATHOM_BF16 && row_dtype != FATHOM_F32) return FATHOM_ERR_UNSUPPORTED;
  if (!fathom_aligned16(Krows) || !fathom_aligned16(Vrows)) return FATHOM_ERR_ALIGNMENT;
  const int Hq = L->n_q_heads, G = Hq / L->n_kv_heads;
  if (Hq > FATHOM_CTL_MAX_HEADS) return FATHOM_ERR_UNSUPPORTED;
  fathom_attn_scratch S = fathom_carve_attn(ctx->scratch, Hq, k);
  if (S.bytes > ctx->scratch_bytes) return FATHOM_ERR_SCRATCH_TOO_SMALL;
  unsigned int* tickets = ctx->dev_status + FATHOM_CTL_TICKETS;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  FATHOM_CUDA_TRY(ctx, (row_dtype == FATHOM_BF16 ? launch_attend<__nv_bfloat16> : launch_attend<float>)(
      q, Krows, Vrows, idx, k, (long long)L->n, Hq, G, softmax_scale, S.partial, S.splits, tickets, out, st));
  return FATHOM_OK;
}

// ---- allocation-free variant --------------------------------------------------------------------------
// Scratch for callers that cannot allocate: the per-chunk (max, denominator, weighted sum) triples live in
// this array instead of a context's arena.  In host code the name below is only a handle for the runtime,
// not a device address, so the address is fetched once per device with cudaGetSymbolAddress and that
// pointer is what the kernels receive.
static __device__ __align__(256) float g_attend_static_partials[FATHOM_ATTEND_STATIC_MAX_CHUNKS * (FATHOM_D + 2)];
// Ticket counters of the merge step, one per query head; zero when the library is loaded and re-armed by
// the merging CTA of every call, so they never need clearing either.
static __device__ __align__(256) unsigned int g_attend_static_tickets[FATHOM_ATTEND_STATIC_MAX_CHUNKS];

namespace {
constexpr int STATIC_MAX_DEVICES = 64;
float* g_static_partials_ptr[STATIC_MAX_DEVICES];            // device address per device ordinal, null until first use
unsigned int* g_static_tickets_ptr[STATIC_MAX_DEVICES];
std::mutex g_static_mutex;
}  // namespace

extern "C" int fathom_sparse_attend_static(const fathom_layout* L, const float* q, const void* Krows, const void* Vrows,
                                           int row_dtype, const int32_t* idx, int k, float softmax_scale, float* out,
                                           void* stream) {
  if (!q || !Krows || !Vrows || !idx || !out) return FATHOM_ERR_INVALID_ARG;
  int rc = fathom_check_layout(L);
  if (rc != FATHOM_OK) return rc;
  if (k < 1 || k > L->n) return FATHOM_ERR_INVALID_ARG;
  if (row_dtype != FATHOM_BF16 && row_dtype != FATHOM_F32) return FATHOM_ERR_UNSUPPORTED;
  if (!fathom_aligned16(Krows) || !fathom_aligned16(Vrows)) return FATHOM_ERR_ALIGNMENT;
  const int Hq = L->n_q_heads, G = Hq / L->n_kv_heads;
  const int splits = (k + FATHOM_ATTN_CHUNK - 1) / FATHOM_ATTN_CHUNK;
  if ((long long)Hq * splits > FATHOM_ATTEND_STATIC_MAX_CHUNKS) return FATHOM_ERR_STATIC_LIMIT;

  // set-up, once per device, with that device current
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return FATHOM_ERR_CUDA;
  if (dev < 0 || dev >= STATIC_MAX_DEVICES) return FATHOM_ERR_UNSUPPORTED;
  float* partial = nullptr;
  unsigned int* tickets = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_partials_ptr[dev]) {
      void *p = nullptr, *t = nullptr;
      if (cudaGetSymbolAddress(&p, g_attend_static_partials) != cudaSuccess || !p) return FATHOM_ERR_CUDA;
      if (cudaGetSymbolAddress(&t, g_attend_static_tickets) != cudaSuccess || !t) return FATHOM_ERR_CUDA;
      g_static_tickets_ptr[dev] = static_cast<unsigned int*>(t);
      g_static_partials_ptr[dev] = static_cast<float*>(p);
    }
    partial = g_static_partials_ptr[dev];
    tickets = g_static_tickets_ptr[dev];
  }

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if ((row_dtype == FATHOM_BF16 ? launch_attend<__nv_bfloat16> : launch_attend<float>)(
          q, Krows, Vrows, idx, k, (long long)L->n, Hq, G, softmax_scale, partial, splits, tickets, out, st) != cudaSuccess)
    return FATHOM_ERR_CUDA;
  return FATHOM_OK;
}
