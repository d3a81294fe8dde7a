// fathom_klt_basis: eigenbasis and eigenvalues of the 128 x 128 key covariance of every KV head (Sec. 3.5 "Basis rule";
// Appendix B5: mean, eigenbasis and eigenvalues of a layer's keys from the session's own prefill cache), so that a rotated
// store can be built with library calls alone: fathom_calibrate -> fathom_klt_basis -> fathom_rotate_keys / _query.
//
// Two-sided cyclic Jacobi, a cluster of eight CTAs per KV head.  A sweep is 127 steps of 64 disjoint pairs (p_k, q_k) in
// round-robin order (player 127 stays, the others move round a ring), so every pair meets once per sweep and the 64
// rotations of a step commute.  Two passes over the full fp64 matrix per step (columns, then rows) and the accumulation of
// the rotations beside them took 5.5 us a step on one SM's shared-memory data path: 2.8 ms for 8 covariances of 4 sweeps.  So:
//   * CTA 0 keeps one triangle of the symmetric matrix (fp64, the diagonal apart) and touches each element ONCE per step: the
//     2 x 2 block of pairs k and l is rotated from both sides in registers.  The matrix is stored by SLOT (the p and the q side
//     of pair 0 .. 63), not by player: a step reads one buffer and writes every element where the next step's slots want it in
//     the other one, so that all addresses of a thread are the same in every step (indexing by player in place was bound by
//     the index arithmetic: 1.8 us a step) and a warp's accesses are runs of consecutive doubles;
//   * the rotations of the next step are computed in the same phase by the 64 threads that update the elements (p', q') they
//     need: one barrier per step, and the chain of a rotation (two reciprocal square roots) runs beside the other warps' updates;
//   * CTA 0 logs a sweep's rotations (fp32 c, s); the seven other CTAs fetch the log through distributed shared memory and apply
//     it to their rows of the accumulated basis (fp32) while CTA 0 runs the next sweep.  A row is owned by one warp, so
//     nothing but __syncwarp separates the steps.
// Sweeps stop when the off-diagonal mass has fallen below 1e-24 of the diagonal's (at most 16 sweeps; a covariance of
// keys takes 4 to 10).  The order of operations is fixed, so the result is bit-reproducible.  Eigenvalues come out
// in descending order (ties: lower original index first) and every direction is signed so that its largest component is
// positive; the rotated store does not depend on either choice.  Eigenvalues are clamped at zero.
#include "fathom_common.cuh"

#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace {

constexpr int N = FATHOM_D;                                   // 128
constexpr int PAIRS = N / 2, STEPS = N - 1;
constexpr int MAX_SWEEPS = 16;
constexpr int EIG_CLUSTER = 8;                                // CTA 0: the matrix; CTAs 1..7: rows of the basis
constexpr int V_ROWS = (N + EIG_CLUSTER - 2) / (EIG_CLUSTER - 1);   // 19 rows per basis CTA (the last one 14)

constexpr int DIST = PAIRS / 2;                                // block (i, i + d mod 64), d = 1 .. 32 (d = 32: i < 32 only)
constexpr int TYPE = DIST * PAIRS;                            // blocks; element type (side of i) * 2 + side of i + d at TYPE * type
constexpr int BUF = 4 * TYPE;                                 // 8192 doubles: one triangle by slots
constexpr int TRIANGLES = 10;
constexpr int EIG_THREADS = PAIRS * (TRIANGLES + 1) + 32;     // 736: the pivots' blocks, the triangles, d = 32
static_assert(EIG_THREADS / 32 >= V_ROWS && EIG_THREADS / 32 <= 32, "a warp per basis row; one warp sums the warps' partial sums");
// Distances 1, 3 .. 31 in triples a, b, c with c = a + b or a + b + c = 64: the pairs k, k + a, k + a + b are the corners of three
// blocks, so a thread reads three rotations for three blocks (two blocks of one pair took three as well: 128 of 1600 wavefronts)
__constant__ const unsigned char TRIPLE[TRIANGLES][3] = {{1, 30, 31}, {3, 26, 29}, {4, 24, 28}, {10, 17, 27}, {11, 14, 25},
                                                         {19, 22, 23}, {6, 15, 21}, {8, 12, 20}, {5, 13, 18}, {7, 9, 16}};

struct EigSmem {
  double A[2][BUF + PAIRS];                                   // CTA 0: the matrix before this step and before the next; the last 64
                                                              // of a buffer take the stores of elements that became a pivot
  float2 log[STEPS][PAIRS];                                   // (c, s) of a sweep: written by CTA 0, copied by the others
  double2 cs[2][PAIRS];                                       // rotations of this step and of the next
  double diag[2][N];                                          // diagonal by slot (side * 64 + pair) after this step and after the next
  double pivot[PAIRS];                                        // a_pq of the step that follows the sweep (for the off-diagonal mass)
  double red[EIG_THREADS / 32][2];
  int rank[N];
  float big[N];                                               // basis CTAs: the largest component of every column over my rows
  int done;
};
static_assert(sizeof(float) * V_ROWS * N <= sizeof(double) * 2 * (BUF + PAIRS), "the basis rows lie where CTA 0 keeps the matrix");

// the pair k of a step: p = step + k, q = step - k (mod 127), q = 127 for k = 0
__device__ __forceinline__ int player_p(int step, int k) { const int x = step + k; return x >= STEPS ? x - STEPS : x; }
__device__ __forceinline__ int player_q(int step, int k) { const int x = step - k; return k == 0 ? N - 1 : (x < 0 ? x + STEPS : x); }

struct Slot { int pair, side; };                              // side 0: p, 1: q
__device__ __forceinline__ Slot slot_of_player(int x, int step) {
  if (x == N - 1) return Slot{0, 1};
  const int e = x >= step ? x - step : x - step + STEPS;      // 0 .. 126 round the ring from the step's p_0
  return e < PAIRS ? Slot{e, 0} : Slot{STEPS - e, 1};
}
// where a slot's player sits in the next step: one place back round the ring
__device__ __forceinline__ Slot next_slot(Slot s) {
  if (s.side == 0) return s.pair == 0 ? Slot{1, 1} : Slot{s.pair - 1, 0};
  if (s.pair == 0) return s;
  return s.pair == PAIRS - 1 ? Slot{PAIRS - 1, 0} : Slot{s.pair + 1, 1};
}
// index of the element of two slots of different pairs
__device__ __forceinline__ int element(Slot a, Slot b) {
  int d = (b.pair - a.pair) & (PAIRS - 1);
  if (d > DIST || (d == DIST && a.pair >= DIST)) { const Slot t = a; a = b; b = t; d = PAIRS - d; }
  return (a.side * 2 + b.side) * TYPE + (d - 1) * PAIRS + a.pair;
}

// rotation that zeroes apq: with r = 1 / sqrt(d^2 + 4 apq^2), d = aqq - app:  c^2 = (1 + |d| r) / 2,  s = sgn(d) apq r / c
__device__ __forceinline__ double2 rotation(double app, double aqq, double apq, double& app_new, double& aqq_new) {
  const double d = aqq - app, h2 = fma(d, d, 4.0 * apq * apq);
  double c = 1.0, s = 0.0, t = 0.0;
  if (fabs(apq) > 1e-150) {
    const double r = rsqrt(h2);
    const double c2 = fma(0.5 * fabs(d), r, 0.5), inv = rsqrt(c2);
    c = c2 * inv;
    s = copysign(1.0, d) * (apq * r) * inv;
    t = s * inv;
  }
  app_new = fma(-t, apq, app);
  aqq_new = fma(t, apq, aqq);
  return make_double2(c, s);
}

// what a thread keeps of a block for the whole kernel: where it is read, the pairs, where its elements go
struct Unit { int load, i, j, to[4]; };
__device__ __forceinline__ Unit unit_of(int i, int d, int trash) {
  Unit u;
  u.i = i;
  u.j = (i + d) & (PAIRS - 1);
  u.load = (d - 1) * PAIRS + i;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const Slot a = next_slot(Slot{u.i, e >> 1}), b = next_slot(Slot{u.j, e & 1});
    u.to[e] = a.pair == b.pair ? trash : element(a, b);       // the two players meet in the next step: a pivot
  }
  return u;
}
// the 2 x 2 block, rotated from both sides: rows (pair i) by ri, columns (pair j) by rj
__device__ __forceinline__ void rotate_block(const double* __restrict__ from, double* __restrict__ to, const Unit& u, double2 ri, double2 rj,
                                             double (&z)[4]) {
  const double x0 = from[u.load], x1 = from[u.load + TYPE], x2 = from[u.load + 2 * TYPE], x3 = from[u.load + 3 * TYPE];
  const double y0 = ri.x * x0 - ri.y * x2, y1 = ri.x * x1 - ri.y * x3;
  const double y2 = ri.y * x0 + ri.x * x2, y3 = ri.y * x1 + ri.x * x3;
  z[0] = rj.x * y0 - rj.y * y1;
  z[1] = rj.y * y0 + rj.x * y1;
  z[2] = rj.x * y2 - rj.y * y3;
  z[3] = rj.y * y2 + rj.x * y3;
#pragma unroll
  for (int e = 0; e < 4; ++e) to[u.to[e]] = z[e];
}

__global__ void __cluster_dims__(EIG_CLUSTER, 1, 1) __launch_bounds__(EIG_THREADS, 1)
klt_eig_kernel(const float* __restrict__ cov, float* __restrict__ basis, float* __restrict__ eigenvalues) {
  extern __shared__ __align__(16) unsigned char raw[];
  EigSmem& M = *reinterpret_cast<EigSmem*>(raw);
  cg::cluster_group cluster = cg::this_cluster();
  const int part = (int)cluster.block_rank(), kv = blockIdx.x / EIG_CLUSTER;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  EigSmem& M0 = *cluster.map_shared_rank(&M, 0);

  if (part == 0) {
    const float* C = cov + (size_t)kv * N * N;
    for (int e = tid; e < 2 * (BUF + PAIRS); e += EIG_THREADS) M.A[0][e] = 0.0;   // (the unused half of d = 32 stays zero)
    if (tid < N) {                                            // "after step -1", in the slots of step -1 = 126 (mod 127)
      const Slot s = slot_of_player(tid, STEPS - 1);
      M.diag[1][s.side * PAIRS + s.pair] = (double)C[tid * N + tid];
    }
    __syncthreads();
    for (int e = tid; e < N * N; e += EIG_THREADS) {
      const int i = e >> 7, j = e & (N - 1);
      if (i < j) {
        const double a = 0.5 * ((double)C[i * N + j] + (double)C[j * N + i]);   // the symmetric part, exactly
        const Slot si = slot_of_player(i, 0), sj = slot_of_player(j, 0);
        if (si.pair == sj.pair) M.pivot[si.pair] = a;
        else M.A[0][element(si, sj)] = a;
      }
    }
    __syncthreads();
    // ---- thread's blocks.  Threads 0..63 take the block whose element becomes the pivot of the next step's pair k = tid: its
    //      p' is now pair k + 1's p (k = 63: its own q), its q' pair k - 1's q (k = 1: pair 0's p; k = 0: pair 0's q), so that
    //      is the block (k - 1, k + 1) of distance 2, (0, 1) for k = 0 and (62, 63) for k = 63.  Ten groups of 64 threads take
    //      a triangle of three blocks each; where (0, 1) and (62, 63) are taken already, (62, 0) and (63, 1) of d = 2 stand in.
    //      The last warp takes d = 32
    const int k = tid & (PAIRS - 1), group = (tid >> 6) - 1, trash = BUF + k;
    const bool ahead = group < 0, opposite = group == TRIANGLES;
    Unit u0, u1, u2;
    int pivot_element = 0, own = 0, src_p = 0, src_q = 0;
    if (ahead) {
      u0 = k == 0 ? unit_of(0, 1, trash) : k == PAIRS - 1 ? unit_of(PAIRS - 2, 1, trash) : unit_of(k - 1, 2, trash);
      pivot_element = k == PAIRS - 1 ? 3 : (k == 1 ? 0 : 2);
      own = element(next_slot(Slot{k, 0}), next_slot(Slot{k, 1}));             // where this step's pivot (now zero) goes
      src_p = k == PAIRS - 1 ? PAIRS + k : k + 1;
      src_q = k == 0 ? PAIRS : (k == 1 ? 0 : PAIRS + k - 1);
      u1 = u2 = u0;
      const int p = player_p(0, k), q = player_q(0, k);
      M.cs[0][k] = rotation((double)C[p * N + p], (double)C[q * N + q], M.pivot[k], M.diag[0][k], M.diag[0][PAIRS + k]);
    } else if (opposite) {
      u0 = u1 = u2 = unit_of(k & (DIST - 1), DIST, trash);
    } else {
      const int da = TRIPLE[group][0], db = TRIPLE[group][1], dc = TRIPLE[group][2];
      u0 = unit_of(k, da, trash);
      u1 = unit_of((k + da) & (PAIRS - 1), db, trash);
      u2 = unit_of(dc == da + db ? k : (k + da + db) & (PAIRS - 1), dc, trash);
      if (da == 1 && k == 0) u0 = unit_of(PAIRS - 2, 2, trash);
      if (da == 1 && k == PAIRS - 2) u0 = unit_of(PAIRS - 1, 2, trash);
    }
    const bool closed = u2.i == k;                            // third block (k, k + a + b), else (k + a + b, k)
    const int corner = closed ? u2.j : u2.i;
    int g = 0;                                                // steps so far (parity of the double buffers)
    for (int sweep = 0;; ++sweep) {
      // ---- how far from diagonal?  (fixed-order reduction: per thread, per warp, then over the warps)
      double off = 0.0, dg = 0.0;
      for (int e = tid; e < BUF; e += EIG_THREADS) {
        const double a = M.A[g & 1][e];
        off = fma(a, 2.0 * a, off);
      }
      if (ahead) off = fma(M.pivot[k], 2.0 * M.pivot[k], off);
      if (tid < N) dg = M.diag[(g & 1) ^ 1][tid] * M.diag[(g & 1) ^ 1][tid];
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        off += __shfl_xor_sync(0xffffffffu, off, o);
        dg += __shfl_xor_sync(0xffffffffu, dg, o);
      }
      if (lane == 0) { M.red[warp][0] = off; M.red[warp][1] = dg; }
      __syncthreads();
      off = lane < EIG_THREADS / 32 ? M.red[lane][0] : 0.0;
      dg = lane < EIG_THREADS / 32 ? M.red[lane][1] : 0.0;
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        off += __shfl_xor_sync(0xffffffffu, off, o);
        dg += __shfl_xor_sync(0xffffffffu, dg, o);
      }
      const bool done = sweep == MAX_SWEEPS || off <= 1e-24 * dg;   // the same for every thread
      if (sweep > 0) cluster.sync();                          // the others have copied the previous sweep's log
      if (tid == 0) M.done = done;
      if (!done) {
        for (int step = 0; step < STEPS; ++step, ++g) {
          const int par = g & 1;
          const double* from = M.A[par];
          double* to = M.A[par ^ 1];
          const double2* cs = M.cs[par];
          double z[4];
          if (ahead) {
            const double2 mine = cs[k];
            const double app = M.diag[par][src_p], aqq = M.diag[par][src_q];
            rotate_block(from, to, u0, cs[u0.i], cs[u0.j], z);
            const double apq = pivot_element == 0 ? z[0] : (pivot_element == 2 ? z[2] : z[3]);
            double* after = M.diag[par ^ 1];
            M.cs[par ^ 1][k] = rotation(app, aqq, apq, after[k], after[PAIRS + k]);
            to[own] = 0.0;
            M.log[step][k] = make_float2((float)mine.x, (float)mine.y);
            if (step == STEPS - 1) M.pivot[k] = apq;
          } else {
            const double2 ri = cs[u0.i], rj = cs[u0.j];
            rotate_block(from, to, u0, ri, rj, z);
            if (!opposite) {
              const double2 r0 = group == 0 ? cs[k] : ri, r1 = group == 0 ? cs[u1.i] : rj, r2 = cs[corner];
              rotate_block(from, to, u1, r1, r2, z);
              rotate_block(from, to, u2, closed ? r0 : r2, closed ? r2 : r0, z);
            }
          }
          __syncthreads();
        }
      }
      cluster.sync();                                         // log and flag are complete
      if (done) break;
    }
    // ---- eigenvalues in descending order (ties: lower index first)
    if (tid < N) {
      const double* D = M.diag[(g & 1) ^ 1];
      auto of = [&](int x) { const Slot s = slot_of_player(x, STEPS - 1); return D[s.side * PAIRS + s.pair]; };
      const double mine = of(tid);
      int r = 0;
      for (int i = 0; i < N; ++i) { const double x = of(i); r += (x > mine || (x == mine && i < tid)) ? 1 : 0; }
      M.rank[tid] = r;
      eigenvalues[(size_t)kv * N + r] = (float)fmax(mine, 0.0);   // a variance: rounding may leave -1e-20 on a rank-deficient input
    }
  } else {
    // ---- rows of the basis: a warp keeps one
    float* V = reinterpret_cast<float*>(M.A);                 // [V_ROWS][N]
    const int first_row = (part - 1) * V_ROWS, rows = min(V_ROWS, N - first_row);
    for (int e = tid; e < rows * N; e += EIG_THREADS) V[e] = (e >> 7) + first_row == (e & (N - 1)) ? 1.0f : 0.0f;
    while (true) {
      cluster.sync();                                         // a sweep's log is complete
      if (M0.done) break;                                     // (the same for every thread)
      for (int e = tid; e < STEPS * PAIRS / 2; e += EIG_THREADS)
        reinterpret_cast<float4*>(M.log)[e] = reinterpret_cast<const float4*>(M0.log)[e];
      cluster.sync();                                         // CTA 0 may write the next sweep's (also: my copy is complete)
      if (warp < rows) {
        float* row = V + warp * N;
        for (int step = 0; step < STEPS; ++step) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int k = lane + 32 * h, p = player_p(step, k), q = player_q(step, k);
            const float2 r = M.log[step][k];
            const float vp = row[p], vq = row[q];
            row[p] = __fsub_rn(__fmul_rn(r.x, vp), __fmul_rn(r.y, vq));
            row[q] = __fadd_rn(__fmul_rn(r.y, vp), __fmul_rn(r.x, vq));
          }
          __syncwarp();
        }
      }
      __syncthreads();                                        // the log may be overwritten
    }
    __syncthreads();
    if (tid < N) {
      float big = 0.0f;
      for (int i = 0; i < rows; ++i) {
        const float v = V[i * N + tid];
        if (fabsf(v) > fabsf(big)) big = v;
      }
      M.big[tid] = big;
    }
  }
  cluster.sync();                                             // ranks and largest components are published
  if (part != 0) {
    // ---- direction j goes to column rank[j], signed so that its largest component is positive
    const float* V = reinterpret_cast<const float*>(M.A);
    const int first_row = (part - 1) * V_ROWS, rows = min(V_ROWS, N - first_row);
    for (int e = tid; e < N; e += EIG_THREADS) M.rank[e] = M0.rank[e];         // (my own copy)
    float* sign = reinterpret_cast<float*>(M.log);
    for (int j = tid; j < N; j += EIG_THREADS) {
      float big = 0.0f;
      for (int c = 1; c < EIG_CLUSTER; ++c) {
        const float v = cluster.map_shared_rank(&M, c)->big[j];
        if (fabsf(v) > fabsf(big)) big = v;
      }
      sign[j] = big < 0.0f ? -1.0f : 1.0f;
    }
    __syncthreads();
    for (int e = tid; e < rows * N; e += EIG_THREADS) {
      const int i = e >> 7, j = e & (N - 1);
      basis[((size_t)kv * N + first_row + i) * N + M.rank[j]] = V[e] * sign[j];
    }
  }
  cluster.sync();                                             // nobody leaves while its shared memory may be read
}

}  // namespace

extern "C" int fathom_klt_basis(fathom_ctx* ctx, const fathom_layout* L, const float* cov, float* basis, float* eigenvalues,
                                void* stream) {
  if (!ctx || !cov || !basis || !eigenvalues) return FATHOM_ERR_INVALID_ARG;
  const int rc = fathom_check_layout(L);
  if (rc != FATHOM_OK) return rc;
  if (!fathom_aligned16(cov) || !fathom_aligned16(basis)) return FATHOM_ERR_ALIGNMENT;
  static bool configured[64] = {};
  int dev = 0;
  FATHOM_CUDA_TRY(ctx, cudaGetDevice(&dev));
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    FATHOM_CUDA_TRY(ctx, cudaFuncSetAttribute(klt_eig_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(EigSmem)));
    configured[dev] = true;
  }
  klt_eig_kernel<<<L->n_kv_heads * EIG_CLUSTER, EIG_THREADS, sizeof(EigSmem), static_cast<cudaStream_t>(stream)>>>(cov, basis, eigenvalues);
  FATHOM_CUDA_TRY(ctx, cudaGetLastError());
  return FATHOM_OK;
}
