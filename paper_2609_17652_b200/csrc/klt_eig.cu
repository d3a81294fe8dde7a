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
//   * CTA 0 logs the rotations (fp32 c, s); the seven other CTAs fetch the log through distributed shared memory, 32 steps at a
//     time, and apply them to their rows of the accumulated basis (fp32) while CTA 0 goes on.  A row is owned by one warp, so
//     nothing but __syncwarp separates the steps.  (A sweep at a time, CTA 0 stood still for 20 K cycles while its log was copied,
//     and 38 K at the end while the last sweep was applied: a step takes 1.2 K.)
// A step in fp64 is bound by the shared-memory data path all the same (128 KB read and written), so the sweeps that only have to
// come close run in fp32 (half the bytes, a shorter chain), and fp64 finishes, the columns dealt out over the eight CTAs: the
// accumulated basis is made orthonormal by one Newton-Schulz step W = V (3 I - V^T V) / 2, B = W^T C W is formed from the
// covariance itself, and what is left off its diagonal is removed by rotating all pairs at once, W + W K with
// K_ij = -K_ji = the tangent of the pair's Jacobi angle, columns normalised.  That is exact for a pair by itself, and otherwise off by
// products of two angles that share a column: it is the last step if no such product exceeds 5e-7 (fp32 rotations leave more than
// that in the basis), and if none exceeds 1e-2 the finish starts again from the basis it gave, which squares them.  Otherwise
// (several close eigenvalues) fp64 sweeps go on from B as described above.  8 covariances of
// 131,072 keys: fp64 sweeps alone 632 us; three fp32 sweeps and two rounds of the finish about 345 us.
// The fp64 sweeps stop when the off-diagonal mass has fallen below 1e-24 of the diagonal's (at most 16 sweeps).  The order of
// operations is fixed, so the result is bit-reproducible.  Eigenvalues come out in descending order (ties: lower original index
// first) and every direction is signed so that its largest component is positive; the rotated store does not depend on either
// choice.  Eigenvalues are clamped at zero.
#include "fathom_common.cuh"

#include <climits>
#include <cooperative_groups.h>
#include <utility>

namespace cg = cooperative_groups;

namespace {

constexpr int N = FATHOM_D;                                   // 128
constexpr int PAIRS = N / 2, STEPS = N - 1;
constexpr int MAX_SWEEPS = 16, MAX_SWEEPS_FP32 = 10;
constexpr double TOL = 1e-24, TOL_FP32 = 1e-11;               // off-diagonal over diagonal mass at which the sweeps stop
constexpr double MAX_TANGENT = 0.25, MAX_PRODUCT = 5e-7, AGAIN_PRODUCT = 1e-2;   // of the rotations that finish: each, any two in a column
constexpr int MAX_FINISHES = 4;
constexpr int EIG_CLUSTER = 8;                                // CTA 0: the matrix; CTAs 1..7: rows of the basis
constexpr int V_ROWS = (N + EIG_CLUSTER - 2) / (EIG_CLUSTER - 1);   // 19 rows per basis CTA (the last one 14)

constexpr int DIST = PAIRS / 2;                                // block (i, i + d mod 64), d = 1 .. 32 (d = 32: i < 32 only)
constexpr int TYPE = DIST * PAIRS;                            // blocks; element type (side of i) * 2 + side of i + d at TYPE * type
constexpr int BUF = 4 * TYPE;                                 // 8192 doubles: one triangle by slots
constexpr int TRIANGLES = 10;
constexpr int EIG_THREADS = PAIRS * (TRIANGLES + 1) + 32;     // 736: the pivots' blocks, the triangles, d = 32
constexpr int SEG = 32, SEGS = (STEPS + SEG - 1) / SEG;        // steps that are handed over together; a sweep's (the log is a ring of these)
constexpr int COLS = N / EIG_CLUSTER;                         // columns of the finish per CTA: 16
constexpr int LDC = COLS + 1;                                 // their pitch: lanes walk rows and columns
constexpr int KPARTS = 4;                                     // a product's sum is split over this many groups of 128 threads
static_assert(KPARTS * 128 <= EIG_THREADS, "threads of a product");
static_assert(EIG_THREADS / 32 >= V_ROWS && EIG_THREADS / 32 <= 32, "a warp per basis row; one warp sums the warps' partial sums");
// Distances 1, 3 .. 31 in triples a, b, c with c = a + b or a + b + c = 64: the pairs k, k + a, k + a + b are the corners of three
// blocks, so a thread reads three rotations for three blocks (two blocks of one pair took three as well: 128 of 1600 wavefronts)
__constant__ const unsigned char TRIPLE[TRIANGLES][3] = {{1, 30, 31}, {3, 26, 29}, {4, 24, 28}, {10, 17, 27}, {11, 14, 25},
                                                         {19, 22, 23}, {6, 15, 21}, {8, 12, 20}, {5, 13, 18}, {7, 9, 16}};

struct EigSmem {
  double A[2 * (BUF + PAIRS)];                                // CTA 0: the matrix (fp32 or fp64) before this step and before the next; the last
                                                              // 64 of a buffer take the stores of elements that became a pivot.
                                                              // Other CTAs: rows of the basis.  Finish: a full matrix in fp64
  union {
    float2 log[STEPS][PAIRS];                                 // (c, s) of the last SEGS segments: written by CTA 0, copied by the others
    struct {                                                  // finish: [row][my columns]
      double G[N][LDC];                                       // V^T V, later B
      double W[N][LDC], T[N][LDC];                            // W; C W, later the angles
      double P[KPARTS - 2][N][LDC];                           // partial sums of a product
    };
  };
  double2 cs[2][PAIRS];                                       // rotations of this step and of the next
  double diag[2][N];                                          // diagonal by slot (side * 64 + pair) after this step and after the next
  double pivot[PAIRS];                                        // a_pq of the step that follows the sweep (for the off-diagonal mass)
  double red[EIG_THREADS / 32][2];
  double lambda[N];
  double cta_red[EIG_CLUSTER];
  int rank[N];
  float big[N];                                               // basis CTAs: the largest component of every column over my rows
  int segments;                                               // CTA 0: how many there are in all, once that is known
};

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

template <typename Real> struct Pair2;
template <> struct Pair2<double> { using type = double2; };
template <> struct Pair2<float> { using type = float2; };
template <typename Real> __device__ __forceinline__ typename Pair2<Real>::type make2(Real x, Real y) { typename Pair2<Real>::type r; r.x = x; r.y = y; return r; }
__device__ __forceinline__ double inverse_sqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ float inverse_sqrt(float x) { return rsqrtf(x); }

// rotation that zeroes apq: with r = 1 / sqrt(d^2 + 4 apq^2), d = aqq - app:  c^2 = (1 + |d| r) / 2,  s = sgn(d) apq r / c
template <typename Real>
__device__ __forceinline__ typename Pair2<Real>::type rotation(Real app, Real aqq, Real apq, Real& app_new, Real& aqq_new) {
  const Real d = aqq - app, h2 = fma(d, d, Real(4) * apq * apq);
  Real c = Real(1), s = Real(0), t = Real(0);
  if (fabs(apq) > (sizeof(Real) == 8 ? Real(1e-150) : Real(1e-18))) {        // (fp32: the matrix is scaled to a diagonal of at most one)
    const Real r = inverse_sqrt(h2);
    const Real c2 = fma(Real(0.5) * fabs(d), r, Real(0.5)), inv = inverse_sqrt(c2);
    c = c2 * inv;
    s = copysign(Real(1), d) * (apq * r) * inv;
    t = s * inv;
  }
  app_new = fma(-t, apq, app);
  aqq_new = fma(t, apq, aqq);
  return make2<Real>(c, s);
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
// A thread reads all its blocks before it writes the first (the compiler cannot: the two buffers might be one, for all it knows)
template <typename Real>
__device__ __forceinline__ void load_block(const Real* from, const Unit& u, Real (&x)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) x[e] = from[u.load + e * TYPE];
}
// the 2 x 2 block, rotated from both sides: rows (pair i) by ri, columns (pair j) by rj
template <typename Real, typename R2>
__device__ __forceinline__ void rotate_block(Real* to, const Unit& u, R2 ri, R2 rj, const Real (&x)[4], Real (&z)[4]) {
  const Real y0 = ri.x * x[0] - ri.y * x[2], y1 = ri.x * x[1] - ri.y * x[3];
  const Real y2 = ri.y * x[0] + ri.x * x[2], y3 = ri.y * x[1] + ri.x * x[3];
  z[0] = rj.x * y0 - rj.y * y1;
  z[1] = rj.y * y0 + rj.x * y1;
  z[2] = rj.x * y2 - rj.y * y3;
  z[3] = rj.y * y2 + rj.x * y3;
#pragma unroll
  for (int e = 0; e < 4; ++e) to[u.to[e]] = z[e];
}

// CTA 0: sweeps over the symmetric matrix whose elements (i <= j) `get` returns, until off-diagonal mass <= tol * diagonal mass or
// max_sweeps have been done.  Returns the number of steps; the diagonal is left in M.diag by slot of step 126.
template <typename Real, typename Cluster, typename Get>
__device__ __forceinline__ int sweeps(EigSmem& M, Cluster& cluster, int max_sweeps, double tol, Get get) {
  using R2 = typename Pair2<Real>::type;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  Real* const A = reinterpret_cast<Real*>(M.A);
  Real* const diag = reinterpret_cast<Real*>(M.diag);         // [2][N]
  Real* const pivot = reinterpret_cast<Real*>(M.pivot);
  R2* const rot = reinterpret_cast<R2*>(M.cs);                // [2][PAIRS]
  constexpr int LDB = BUF + PAIRS;
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
    own = element(next_slot(Slot{k, 0}), next_slot(Slot{k, 1}));               // where this step's pivot (now zero) goes
    src_p = k == PAIRS - 1 ? PAIRS + k : k + 1;
    src_q = k == 0 ? PAIRS : (k == 1 ? 0 : PAIRS + k - 1);
    u1 = u2 = u0;
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
  const bool closed = u2.i == k;                              // third block (k, k + a + b), else (k + a + b, k)
  const int corner = closed ? u2.j : u2.i;

  for (int e = tid; e < 2 * LDB; e += EIG_THREADS) A[e] = Real(0);             // (the unused half of d = 32 stays zero)
  __syncthreads();
  if (tid == 0) M.segments = INT_MAX;
  constexpr int BATCH = 8;                                    // elements a thread fetches together
  for (int e0 = tid; e0 < N * N; e0 += BATCH * EIG_THREADS) {
    Real fetched[BATCH];
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int e = e0 + u * EIG_THREADS, i = e >> 7, j = e & (N - 1);
      fetched[u] = e < N * N && i <= j ? get(i, j) : Real(0);
    }
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int e = e0 + u * EIG_THREADS, i = e >> 7, j = e & (N - 1);
      if (e >= N * N || i > j) continue;
      const Real a = fetched[u];
      const Slot si = slot_of_player(i, 0), sj = slot_of_player(j, 0);
      if (i == j) {                                           // "after step -1", in the slots of step -1 = 126 (mod 127)
        const Slot s = slot_of_player(i, STEPS - 1);
        diag[N + s.side * PAIRS + s.pair] = a;
        diag[si.side * PAIRS + si.pair] = a;                  // (and where the first rotations read it)
      } else if (si.pair == sj.pair) pivot[si.pair] = a;
      else A[element(si, sj)] = a;
    }
  }
  __syncthreads();
  if (ahead) {
    const Real app = diag[k], aqq = diag[PAIRS + k];
    rot[k] = rotation<Real>(app, aqq, pivot[k], diag[k], diag[PAIRS + k]);
  }
  int g = 0;                                                  // steps so far (parity of the double buffers)
  int handed = 0;                                             // segments so far: one phase of the cluster barrier each, arrived at when the segment is
                                                              // complete and waited for one segment later.  The others arrive at a phase when they
                                                              // have copied the segments before it, so a ring of SEGS is never overrun
  typename Cluster::arrival_token phase;
  auto hand_over = [&]() {
    if (handed++ > 0) cluster.barrier_wait(std::move(phase));
    phase = cluster.barrier_arrive();
  };
  for (int sweep = 0;; ++sweep) {
    // ---- how far from diagonal?  (fixed-order reduction: per thread, per warp, then over the warps)
    double off = 0.0, dg = 0.0;
    for (int e = tid; e < BUF; e += EIG_THREADS) {
      const double a = (double)A[(g & 1) * LDB + e];
      off = fma(a, 2.0 * a, off);
    }
    if (ahead) off = fma((double)pivot[k], 2.0 * (double)pivot[k], off);
    if (tid < N) dg = (double)diag[((g & 1) ^ 1) * N + tid] * (double)diag[((g & 1) ^ 1) * N + tid];
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
    const bool done = sweep == max_sweeps || off <= tol * dg;  // the same for every thread
    if (!done) {
      for (int step = 0; step < STEPS; ++step, ++g) {
        const int par = g & 1;
        const Real* from = A + par * LDB;
        Real* to = A + (par ^ 1) * LDB;
        const R2* cs = rot + par * PAIRS;
        Real x0[4], x1[4], x2[4], z[4];
        load_block(from, u0, x0);
        if (ahead) {
          const R2 mine = cs[k];
          const Real app = diag[par * N + src_p], aqq = diag[par * N + src_q];
          rotate_block<Real, R2>(to, u0, cs[u0.i], cs[u0.j], x0, z);
          const Real apq = pivot_element == 0 ? z[0] : (pivot_element == 2 ? z[2] : z[3]);
          Real* after = diag + (par ^ 1) * N;
          rot[(par ^ 1) * PAIRS + k] = rotation<Real>(app, aqq, apq, after[k], after[PAIRS + k]);
          to[own] = Real(0);
          M.log[step][k] = make_float2((float)mine.x, (float)mine.y);
          if (step == STEPS - 1) pivot[k] = apq;
        } else {
          const R2 ri = cs[u0.i], rj = cs[u0.j];
          if (opposite) {
            rotate_block<Real, R2>(to, u0, ri, rj, x0, z);
          } else {
            const R2 r0 = group == 0 ? cs[k] : ri, r1 = group == 0 ? cs[u1.i] : rj, r2 = cs[corner];
            load_block(from, u1, x1);
            load_block(from, u2, x2);
            rotate_block<Real, R2>(to, u0, ri, rj, x0, z);
            rotate_block<Real, R2>(to, u1, r1, r2, x1, z);
            rotate_block<Real, R2>(to, u2, closed ? r0 : r2, closed ? r2 : r0, x2, z);
          }
        }
        __syncthreads();
        if (step % SEG == SEG - 1 || step == STEPS - 1) hand_over();
      }
    } else {
      if (tid == 0) M.segments = handed;
      hand_over();                                            // the last phase, without a segment
      cluster.barrier_wait(std::move(phase));                 // everything is applied
      return g;
    }
  }
}

// The other CTAs: the logged rotations applied to `rows` rows of the basis, a warp per row
template <typename Cluster>
__device__ __forceinline__ void apply_sweeps(EigSmem& M, EigSmem& M0, Cluster& cluster, float* V, int rows) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int segment = 0;; ++segment) {
    cluster.sync();                                           // the segment's log is complete
    if (segment >= M0.segments) return;                       // (the same for every thread)
    const int first = segment % SEGS * SEG, last = min(first + SEG, STEPS);
    for (int e = first * PAIRS / 2 + tid; e < last * PAIRS / 2; e += EIG_THREADS)
      reinterpret_cast<float4*>(M.log)[e] = reinterpret_cast<const float4*>(M0.log)[e];
    __syncthreads();                                          // (a warp that is still in the segment before has that in another part of the ring)
    if (warp < rows) {
      float* row = V + warp * N;
      for (int step = first; step < last; ++step) {
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
  }
}

__global__ void __cluster_dims__(EIG_CLUSTER, 1, 1) __launch_bounds__(EIG_THREADS, 1)
klt_eig_kernel(const float* cov, float* basis_out, float* __restrict__ eigenvalues) {
  extern __shared__ __align__(16) unsigned char raw[];
  EigSmem& M = *reinterpret_cast<EigSmem*>(raw);
  cg::cluster_group cluster = cg::this_cluster();
  const int part = (int)cluster.block_rank(), kv = blockIdx.x / EIG_CLUSTER;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  EigSmem& M0 = *cluster.map_shared_rank(&M, 0);
  const float* C = cov + (size_t)kv * N * N;
  float* basis = basis_out + (size_t)kv * N * N;
  float* V = reinterpret_cast<float*>(M.A);                   // CTAs 1..7: [V_ROWS][N]
  const int first_row = (part - 1) * V_ROWS, rows = min(V_ROWS, N - first_row);

  FATHOM_PDL_WAIT();                                          // the covariance comes from the previous kernel
  FATHOM_PDL_RELEASE();
  // ---- 1. fp32 sweeps.  (The output is written when the covariance has been read for the last time: it may be the same buffer)
  if (part == 0) {
    float m = 0.0f;                                           // scaled by a power of two so that the largest diagonal element is near one
    for (int i = lane; i < N; i += 32) m = fmaxf(m, fabsf(C[i * N + i]));
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const double scale = m > 0.0f ? ldexp(1.0, -ilogbf(m)) : 1.0;
    sweeps<float>(M, cluster, MAX_SWEEPS_FP32, TOL_FP32, [&](int i, int j) { return (float)(0.5 * ((double)C[i * N + j] + (double)C[j * N + i]) * scale); });
  } else {
    for (int e = tid; e < rows * N; e += EIG_THREADS) V[e] = (e >> 7) + first_row == (e & (N - 1)) ? 1.0f : 0.0f;
    __syncthreads();
    apply_sweeps(M, M0, cluster, V, rows);
  }
  cluster.sync();

  // ---- 2. the finish in fp64, columns J0 .. J0 + 15 in this CTA.  X: a full matrix, row pitch N + 1 (rows and columns are walked)
  double* const X = M.A;
  constexpr int LDX = N + 1;
  static_assert(N * LDX <= 2 * (BUF + PAIRS), "a full fp64 matrix lies where the sweeps keep theirs");
  const int J0 = part * COLS;
  // Products of 128 x 128 by 128 x 16: a thread has four rows (row, + 32, ..) by four columns and a quarter of the sum, so that ten 128-byte
  // reads of shared memory serve 512 multiply-adds (a row by four columns took three times as many); 512 threads (half as many, and
  // results at a pitch of 16, where 32 rows share a bank: 13.5 K cycles a product)
  const int row = tid & 31, pj = ((tid >> 5) & 3) * 4, kpart = tid >> 7;
  // out[i][j] = finish(i, j, sum over k of (by_column ? X[k][i] : X[i][k]) * R[k][j]); R and out are different arrays
  auto product = [&](bool by_column, const double* right, int ld_right, double (*out)[LDC], auto finish) {
    double s[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) s[r][0] = s[r][1] = s[r][2] = s[r][3] = 0.0;
    if (kpart < KPARTS) {
      const double* x = by_column ? X + row : X + row * LDX;
      const int step = by_column ? LDX : 1, rows32 = by_column ? 32 : 32 * LDX;
#pragma unroll 2
      for (int k = kpart * (N / KPARTS); k < (kpart + 1) * (N / KPARTS); ++k) {
        double a[4], b[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) a[r] = x[k * step + r * rows32];
#pragma unroll
        for (int c = 0; c < 4; ++c) b[c] = right[k * ld_right + pj + c];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) s[r][c] = fma(a[r], b[c], s[r][c]);
      }
    }
    if (kpart > 0 && kpart < KPARTS) {
      double (*part)[LDC] = kpart == 1 ? out : M.P[kpart - 2];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) part[row + 32 * r][pj + c] = s[r][c];
    }
    __syncthreads();
    if (kpart == 0) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int i = row + 32 * r, j = pj + c;
          double sum = s[r][c] + out[i][j];
#pragma unroll
          for (int h = 0; h < KPARTS - 2; ++h) sum += M.P[h][i][j];
          out[i][j] = finish(i, j, sum);
        }
    }
    __syncthreads();
  };
  auto as_is = [](int, int, double v) { return v; };
  constexpr int FULL = (N * N / 4 + EIG_THREADS - 1) / EIG_THREADS;
  auto store_full = [&](const float4 (&v)[FULL]) {
#pragma unroll
    for (int u = 0; u < FULL; ++u) {
      const int e = 4 * (tid + u * EIG_THREADS);
      if (e < N * N) {
        double* to = X + (e >> 7) * LDX + (e & (N - 1));
        to[0] = v[u].x; to[1] = v[u].y; to[2] = v[u].z; to[3] = v[u].w;
      }
    }
    __syncthreads();
  };
  auto load_covariance = [&]() {                              // all loads in flight together
    float4 v[FULL];
#pragma unroll
    for (int u = 0; u < FULL; ++u)
      if (tid + u * EIG_THREADS < N * N / 4) v[u] = __ldcg(reinterpret_cast<const float4*>(C) + tid + u * EIG_THREADS);
    store_full(v);
  };
  auto load_basis = [&]() {                                   // the rows that the sweeps left in the other CTAs
    float4 v[FULL];
#pragma unroll
    for (int u = 0; u < FULL; ++u) {
      const int e = tid + u * EIG_THREADS, i = e / (N / 4);
      if (e < N * N / 4) v[u] = reinterpret_cast<const float4*>(cluster.map_shared_rank(M.A, 1 + i / V_ROWS))[i % V_ROWS * (N / 4) + e % (N / 4)];
    }
    cluster.sync();                                           // (X lies where the rows do)
    store_full(v);
  };
  auto gather = [&]() {                                       // X = the columns M.W of all CTAs, four CTAs' in flight together
    constexpr int PER = (N * COLS + EIG_THREADS - 1) / EIG_THREADS;
#pragma unroll
    for (int c0 = 0; c0 < EIG_CLUSTER; c0 += 4) {
      double v[4][PER];
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int u = 0; u < PER; ++u)
          if (tid + u * EIG_THREADS < N * COLS) v[c][u] = cluster.map_shared_rank(&M, c0 + c)->W[(tid + u * EIG_THREADS) / COLS][(tid + u * EIG_THREADS) % COLS];
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          const int e = tid + u * EIG_THREADS;
          if (e < N * COLS) X[(e / COLS) * LDX + (c0 + c) * COLS + e % COLS] = v[c][u];
        }
    }
    __syncthreads();
  };
  load_basis();
  double worst = 0.0;                                         // the largest product of two tangents in a column
  for (int round = 0; round < MAX_FINISHES; ++round) {
    // one step squares the distance from orthonormal, 1e-6 after the fp32 sweeps; after a round it is the worst product
    for (bool last = round == 0 || worst <= 1e-4;; last = true) {
      product(true, X + J0, LDX, M.G, as_is);                                                                // V^T V
      product(false, &M.G[0][0], LDC, M.W, [&](int i, int j, double v) { return 1.5 * X[i * LDX + J0 + j] - 0.5 * v; });   // V (3 I - V^T V) / 2
      if (last) break;
      cluster.sync();
      gather();
      cluster.sync();                                         // (read by everyone before they are rewritten)
    }
    load_covariance();
    for (int e = tid; e < N * N; e += EIG_THREADS) {          // the symmetric part, exactly
      const int i = e >> 7, j = e & (N - 1);
      if (i < j) X[i * LDX + j] = X[j * LDX + i] = 0.5 * (X[i * LDX + j] + X[j * LDX + i]);
    }
    __syncthreads();
    product(true, &M.W[0][0], LDC, M.T, as_is);                                                             // C W
    cluster.sync();                                           // every CTA's columns of W
    gather();
    product(true, &M.T[0][0], LDC, M.G, as_is);                                                             // B = W^T C W
    if (tid < COLS * EIG_CLUSTER) cluster.map_shared_rank(&M, tid / COLS)->lambda[J0 + tid % COLS] = M.G[J0 + tid % COLS][tid % COLS];
    cluster.sync();                                           // B, and its diagonal everywhere

    // ---- 3. the rotations that finish, if they do not disturb one another (b_ij that the sweeps would have left are left)
    double diag2 = 0.0;
    for (int i = lane; i < N; i += 32) diag2 = fma(M.lambda[i], M.lambda[i], diag2);
#pragma unroll
    for (int o = 16; o; o >>= 1) diag2 += __shfl_xor_sync(0xffffffffu, diag2, o);
    for (int e = tid; e < N * COLS; e += EIG_THREADS) {
      const int i = e / COLS, c = e % COLS;
      const double b = M.G[i][c], d = M.lambda[J0 + c] - M.lambda[i];
      M.T[i][c] = i != J0 + c && b * b > TOL / (N * N) * diag2 ? 2.0 * b / (d + copysign(sqrt(fma(d, d, 4.0 * b * b)), d)) : 0.0;
    }
    __syncthreads();
    worst = 0.0;                                                // of my columns; 1 if a tangent is too large
    if (warp < COLS) {
      double first = 0.0, second = 0.0;
      for (int i = lane; i < N; i += 32) {
        const double x = fabs(M.T[i][warp]);
        second = fmax(second, fmin(first, x));
        first = fmax(first, x);
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const double f = __shfl_xor_sync(0xffffffffu, first, o), g = __shfl_xor_sync(0xffffffffu, second, o);
        second = fmax(fmax(second, g), fmin(first, f));
        first = fmax(first, f);
      }
      worst = first <= MAX_TANGENT ? first * second : 1.0;
    }
    if (lane == 0) M.red[warp][0] = worst;
    __syncthreads();
    worst = lane < EIG_THREADS / 32 ? M.red[lane][0] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    if (tid < EIG_CLUSTER) cluster.map_shared_rank(&M, tid)->cta_red[part] = worst;
    cluster.sync();
    for (int r = 0; r < EIG_CLUSTER; ++r) worst = fmax(worst, M.cta_red[r]);
    if (worst > (round == MAX_FINISHES - 1 ? MAX_PRODUCT : AGAIN_PRODUCT)) break;   // (the same for the whole cluster)
    product(false, &M.T[0][0], LDC, M.W, [&](int i, int j, double v) { return X[i * LDX + J0 + j] + v; });  // W + W K
    if (warp < COLS) {                                        // a warp per column: its length
      double len = 0.0;
      for (int i = lane; i < N; i += 32) len = fma(M.W[i][warp], M.W[i][warp], len);
#pragma unroll
      for (int o = 16; o; o >>= 1) len += __shfl_xor_sync(0xffffffffu, len, o);
      const double scale = rsqrt(len);
      for (int i = lane; i < N; i += 32) M.W[i][warp] *= scale;
    }
    __syncthreads();
    if (worst <= MAX_PRODUCT) break;
    cluster.sync();                                           // every CTA's new columns
    gather();
    cluster.sync();                                           // (read by everyone before they are rewritten)
  }

  if (worst <= MAX_PRODUCT) {
    double* lambda = M.diag[0];                               // the corrected eigenvalues of all columns
    if (warp < COLS) {                                        // a warp per column: largest component (ties: the positive one), eigenvalue
      double big = 0.0, add = 0.0;
      for (int i = lane; i < N; i += 32) {
        const double v = M.W[i][warp];
        if (fabs(v) > fabs(big)) big = v;
        add = fma(M.G[i][warp], M.T[i][warp], add);
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        add += __shfl_xor_sync(0xffffffffu, add, o);
        const double other = __shfl_xor_sync(0xffffffffu, big, o);
        if (fabs(other) > fabs(big) || (fabs(other) == fabs(big) && other > big)) big = other;
      }
      if (lane == 0) {
        M.pivot[warp] = big < 0.0 ? -1.0 : 1.0;
        for (int r = 0; r < EIG_CLUSTER; ++r) cluster.map_shared_rank(&M, r)->diag[0][J0 + warp] = M.lambda[J0 + warp] + add;
      }
    }
    cluster.sync();
    if (tid < COLS) {
      const double mine = lambda[J0 + tid];
      int r = 0;
      for (int i = 0; i < N; ++i) r += (lambda[i] > mine || (lambda[i] == mine && i < J0 + tid)) ? 1 : 0;
      M.rank[tid] = r;
      eigenvalues[(size_t)kv * N + r] = (float)fmax(mine, 0.0);   // a variance: rounding may leave -1e-20 on a rank-deficient input
    }
    __syncthreads();
    for (int e = tid; e < N * COLS; e += EIG_THREADS) basis[(e / COLS) * N + M.rank[e % COLS]] = (float)(M.W[e / COLS][e % COLS] * M.pivot[e % COLS]);
    return;                                                   // (nobody reads another CTA's shared memory any more)
  }

  // ---- 4. close eigenvalues: fp64 sweeps from B
  if (part == 0) {
    const int g = sweeps<double>(M, cluster, MAX_SWEEPS, TOL, [&](int i, int j) { return cluster.map_shared_rank(&M, j / COLS)->G[i][j % COLS]; });
    if (tid < N) {                                            // eigenvalues in descending order (ties: lower index first)
      const double* D = M.diag[(g & 1) ^ 1];
      auto of = [&](int x) { const Slot sl = slot_of_player(x, STEPS - 1); return D[sl.side * PAIRS + sl.pair]; };
      const double mine = of(tid);
      int r = 0;
      for (int i = 0; i < N; ++i) { const double x = of(i); r += (x > mine || (x == mine && i < tid)) ? 1 : 0; }
      M.rank[tid] = r;
      eigenvalues[(size_t)kv * N + r] = (float)fmax(mine, 0.0);
    }
  } else {
    constexpr int PER = (V_ROWS * N + EIG_THREADS - 1) / EIG_THREADS;
    float keep[PER];                                          // my rows of W, to where the sweeps want them (the same memory)
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int e = tid + u * EIG_THREADS;
      keep[u] = e < rows * N ? (float)X[(first_row + (e >> 7)) * LDX + (e & (N - 1))] : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PER; ++u)
      if (tid + u * EIG_THREADS < rows * N) V[tid + u * EIG_THREADS] = keep[u];
    __syncthreads();
    apply_sweeps(M, M0, cluster, V, rows);
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
      basis[(first_row + i) * N + M.rank[j]] = V[e] * sign[j];
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
  FATHOM_CUDA_TRY(ctx, fathom_launch_dependent(klt_eig_kernel, dim3(L->n_kv_heads * EIG_CLUSTER), dim3(EIG_THREADS), sizeof(EigSmem),
                                               static_cast<cudaStream_t>(stream), cov, basis, eigenvalues));
  return FATHOM_OK;
}
