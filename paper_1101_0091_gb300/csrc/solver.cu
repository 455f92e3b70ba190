// Iterative consumers of the product: conjugate gradients (Hestenes-Stiefel)
// and the Lanczos three-term recurrence, each on k independent columns, so that
// every iteration's product is one k-column SpMM through the plan (Sec. 1.3.1
// names Lanczos and Jacobi-Davidson as the methods whose run time the product
// dominates).
//
// Vectors are row-major n x k blocks (ld = k, 16-byte aligned: the vector
// kernels move 16 bytes per access).  The vector work of an iteration is three
// fused grid-stride kernels on a grid of at most one wave; each writes
// its per-column inner products as one partial per CTA, and every CTA of the kernel
// that uses them adds the partials again in a fixed order.  Reductions are
// therefore deterministic for a given solver.  Columns freeze on the device the
// iteration they converge (or break down), so the host only polls a counter
// every `check_every` iterations; those iterations are replayed from a CUDA
// graph captured once per (B, X, check_every).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "device.cuh"
#include "internal.h"

namespace spmv {

constexpr int kVecCtasPerSm = 2;  // CTAs of the vector kernels per SM (their launch bounds hold them resident)
constexpr int kMaxCols = 16;

// Per-column scalars.  Every CTA of a kernel reads them and CTA 0 writes, so no kernel writes a field
// that it reads: k_cg_direction writes rr, active, iters and n_active, k_cg_update the others, with
// copies (rr_old) or working sets (running) of what k_cg_direction needs; k_lz_alpha writes uu, scale
// and live, k_lz_beta their copies.
struct CgScalars {
  double rr[kMaxCols], rr_old[kMaxCols], tol2[kMaxCols], alpha[kMaxCols];
  int active[kMaxCols], running[kMaxCols], iters[kMaxCols], breakdown[kMaxCols];
  int n_active;
};

struct LzScalars {
  double uu[kMaxCols], uu_old[kMaxCols], scale[kMaxCols], scale_old[kMaxCols];
  int live[kMaxCols], live_old[kMaxCols];
};

// ---------------------------------------------------------------- block walking
// How the threads of a kernel walk a row-major n x k block, one unit per thread and grid stride:
//  PAIRS (k = 1): two consecutive entries, one 16-byte access;
//  VROWS (k = K = 2, 4): one row of K values, K/2 16-byte accesses;
//  VGROUPS (k = K = 8, 16): a group of 4 columns of one row (K/4 units per row), two 16-byte accesses;
//  FLAT (other k): one entry; the largest multiple of k threads of a CTA take part, so that a thread
//    stays on its column and a warp reads consecutive entries.
// In every mode the stride keeps a thread on the same columns.  PAIRS, VROWS and VGROUPS need 16-byte
// aligned blocks (checked on the host).
enum { FLAT = 0, VROWS = 1, PAIRS = 2, VGROUPS = 3 };

constexpr int kVecThreads = 512;  // threads per CTA of the vector kernels

template <int K, int MODE>
struct Seg {
  static constexpr int NG = MODE == VGROUPS ? K / 4 : 1;                                        // units per row
  static constexpr int W = MODE == FLAT ? 1 : MODE == PAIRS ? 2 : (MODE == VGROUPS ? 4 : K);  // values per unit
  static constexpr int KC = MODE == PAIRS ? 1 : W;                // accumulators (columns) per thread
  static constexpr int KP = MODE == FLAT ? kMaxCols : (MODE == PAIRS ? 1 : K);  // columns at most
  static constexpr int U = MODE == FLAT ? 4 : (W == 2 ? 2 : 1);   // units in flight per thread and vector
  static_assert(kVecThreads % NG == 0, "a thread's units must share one column group");
  // units of an n x k block, threads of a CTA that take part, first column of thread t
  __host__ __device__ static int64_t units(int64_t n, int k) {
    return MODE == FLAT ? n * k : MODE == PAIRS ? (n + 1) / 2 : n * NG;
  }
  __host__ __device__ static int threads(int k) { return MODE == FLAT ? kVecThreads / k * k : kVecThreads; }
  __device__ static int column(int t, int k) { return MODE == FLAT ? t % k : MODE == VGROUPS ? (t % NG) * 4 : 0; }
  __device__ static int acc(int w) { return MODE == PAIRS ? 0 : w; }  // accumulator of value w
  __device__ static void load(const double* p, int64_t u, int64_t n, double (&v)[W]) {
    if constexpr (MODE == FLAT) {
      v[0] = p[u];
    } else if constexpr (MODE == PAIRS) {
      if (2 * u + 1 < n) {
        const double2 t = reinterpret_cast<const double2*>(p)[u];
        v[0] = t.x;
        v[1] = t.y;
      } else {
        v[0] = p[2 * u];
        v[1] = 0.0;
      }
    } else {
      // VGROUPS: u * 4 is the offset of group u % NG of row u / NG
#pragma unroll
      for (int h = 0; h < W / 2; ++h) {
        const double2 t = reinterpret_cast<const double2*>(p + u * W)[h];
        v[2 * h] = t.x;
        v[2 * h + 1] = t.y;
      }
    }
  }
  __device__ static void store(double* p, int64_t u, int64_t n, const double (&v)[W]) {
    if constexpr (MODE == FLAT) {
      p[u] = v[0];
    } else if constexpr (MODE == PAIRS) {
      if (2 * u + 1 < n)
        reinterpret_cast<double2*>(p)[u] = make_double2(v[0], v[1]);
      else
        p[2 * u] = v[0];
    } else {
#pragma unroll
      for (int h = 0; h < W / 2; ++h) reinterpret_cast<double2*>(p + u * W)[h] = make_double2(v[2 * h], v[2 * h + 1]);
    }
  }
};

// The walk of one thread: U units per step, all loads of a step before its arithmetic and stores.
template <typename G>
struct Walk {
  int64_t u, stride, units, n;
  __device__ Walk(int64_t n_, int k) : n(n_) {
    const int t = G::threads(k);
    units = (int)threadIdx.x < t ? G::units(n, k) : 0;
    stride = (int64_t)gridDim.x * t;
    u = (int64_t)blockIdx.x * t + threadIdx.x;
  }
  __device__ bool more() const { return u < units; }
  __device__ bool has(int j) const { return j == 0 || u + j * stride < units; }  // of a step that more() allows
  __device__ void next() { u += stride * G::U; }
  __device__ void load(const double* p, double (&v)[G::U][G::W]) const {
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (u + j * stride < units) {
        G::load(p, u + j * stride, n, v[j]);
      } else {
#pragma unroll
        for (int w = 0; w < G::W; ++w) v[j][w] = 0.0;
      }
    }
  }
  __device__ void store(double* p, const double (&v)[G::U][G::W]) const {
#pragma unroll
    for (int j = 0; j < G::U; ++j)
      if (has(j)) G::store(p, u + j * stride, n, v[j]);
  }
};

// ---------------------------------------------------------------- reductions
// Per-column sums over a CTA and then over the CTAs, in a fixed order (so a solver's results do not
// depend on timing).  No CTA waits to be the last: each writes its column sums (a partial), and every
// CTA of the kernel that needs the totals adds all partials again in the same order.  A warp's FP64 add
// occupies the SM for 16 cycles whatever it adds, so the sums go through shared memory in passes that
// keep 32 lanes busy; an xor-shuffle tree per warp and column spent as many cycles on the sums as on the
// vectors' arithmetic (320 against 66 warp adds for 512 threads and four columns).
struct VecShared {
  double sums[kVecThreads * 4], part[128];
};

// Thread c < period gets the sum of the values of column c among the N values in sh.sums, value i
// belonging to column i % period.  (period = KP, a power of two, or in FLAT mode k; N <= 2048.)
template <typename G>
__device__ __forceinline__ double column_sum(VecShared& sh, int N, int k) {
  const int t = threadIdx.x;
  __syncthreads();
  double x = 0.0;
  if constexpr (G::KP == kMaxCols && G::KC == 1 && G::W == 1) {  // FLAT
    const int r1 = 128 / k * k, r2 = 32 / k * k;
    if (t < r1) {
      for (int i = t; i < N; i += r1) x += sh.sums[i];
      sh.part[t] = x;
    }
    __syncthreads();
    if (t < 32) {
      x = 0.0;
      if (t < r2)
        for (int i = t; i < r1; i += r2) x += sh.part[i];
      __syncwarp();
      sh.part[t] = x;
      __syncwarp();
      x = 0.0;
      if (t < k)
        for (int i = t; i < r2; i += k) x += sh.part[i];
    }
  } else {
    if (t < 128) {
      x = sh.sums[t];
      for (int i = t + 128; i < N; i += 128) x += sh.sums[i];
      sh.part[t] = x;
    }
    __syncthreads();
    if (t < 32) {
      x = (sh.part[t] + sh.part[t + 32]) + (sh.part[t + 64] + sh.part[t + 96]);
#pragma unroll
      for (int off = 16; off >= G::KP; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    }
  }
  return x;
}

// This CTA's column sums of the threads' accumulators, to partial[blockIdx.x * period + c].
template <typename G>
__device__ __forceinline__ void write_partial(const double (&acc)[G::KC], int k, double* partial, VecShared& sh) {
  __syncthreads();
#pragma unroll
  for (int w = 0; w < G::KC; ++w) sh.sums[threadIdx.x * G::KC + w] = acc[w];
  const int period = G::NG * G::KC == G::KP ? G::KP : k;
  const double x = column_sum<G>(sh, G::threads(k) * G::KC, k);
  if ((int)threadIdx.x < period) partial[(size_t)blockIdx.x * period + threadIdx.x] = x;
}

// Thread c < period gets the total of column c over n_partials partials.
template <typename G>
__device__ __forceinline__ double read_partials(const double* partial, unsigned n_partials, int k, VecShared& sh) {
  const int period = G::NG * G::KC == G::KP ? G::KP : k;
  const unsigned step = G::threads(k), count = n_partials * period;
  double x = 0.0;
  if (threadIdx.x < step) {
    unsigned i = threadIdx.x;
    for (; i + 3 * step < count; i += 4 * step) {
      double v[4];
#pragma unroll
      for (unsigned j = 0; j < 4; ++j) v[j] = __ldcg(partial + i + j * step);
      x += (v[0] + v[1]) + (v[2] + v[3]);
    }
    for (; i < count; i += step) x += __ldcg(partial + i);
  }
  sh.sums[threadIdx.x] = x;
  return column_sum<G>(sh, step, k);
}

// ---------------------------------------------------------------- CG kernels
// R = B - AX (AX in Q), P = R; column sums of R.R and B.B.
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads) k_cg_init(int64_t n, int k, const double* B,
                                                         const double* Q, double* R,
                                                         double* P, double* rr_partial,
                                                         double* bb_partial) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  double rr[G::KC], bb[G::KC];
#pragma unroll
  for (int q = 0; q < G::KC; ++q) rr[q] = bb[q] = 0.0;
  for (Walk<G> w(n, k); w.more(); w.next()) {
    double b[G::U][G::W], r[G::U][G::W];
    w.load(B, b);
    w.load(Q, r);
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (!w.has(j)) break;
#pragma unroll
      for (int i = 0; i < G::W; ++i) {
        r[j][i] = b[j][i] - r[j][i];
        rr[G::acc(i)] = fma(r[j][i], r[j][i], rr[G::acc(i)]);
        bb[G::acc(i)] = fma(b[j][i], b[j][i], bb[G::acc(i)]);
      }
    }
    w.store(R, r);
    w.store(P, r);
  }
  write_partial<G>(rr, k, rr_partial, sh);
  write_partial<G>(bb, k, bb_partial, sh);
}

// One CTA: the scalars of the start, tol2 = rtol^2 B.B, active = rr > tol2.
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads) k_cg_begin(int k, const double* rr_partial, const double* bb_partial,
                                                          unsigned n_partials, CgScalars* S, double rtol2) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  __shared__ int n_active;
  const int c = threadIdx.x;
  if (c == 0) n_active = 0;
  const double rr = read_partials<G>(rr_partial, n_partials, k, sh);
  __syncthreads();
  const double bb = read_partials<G>(bb_partial, n_partials, k, sh);
  if (c < k) {
    S->rr[c] = rr;
    S->tol2[c] = rtol2 * bb;
    S->active[c] = rr > rtol2 * bb;
    S->iters[c] = 0;
    S->breakdown[c] = 0;
    if (rr > rtol2 * bb) atomicAdd(&n_active, 1);
  }
  __syncthreads();
  if (c == 0) S->n_active = n_active;
}

// Column sums of P.Q.
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads, 2) k_cg_dot(int64_t n, int k, const double* P,
                                                           const double* Q, double* partial) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  double acc[G::KC];
#pragma unroll
  for (int q = 0; q < G::KC; ++q) acc[q] = 0.0;
  for (Walk<G> w(n, k); w.more(); w.next()) {
    double p[G::U][G::W], q2[G::U][G::W];
    w.load(P, p);
    w.load(Q, q2);
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (!w.has(j)) break;
#pragma unroll
      for (int i = 0; i < G::W; ++i) acc[G::acc(i)] = fma(p[j][i], q2[j][i], acc[G::acc(i)]);
    }
  }
  write_partial<G>(acc, k, partial, sh);
}

// alpha = R.R / P.Q (breakdown when P.Q <= 0); running columns: R -= alpha Q; column sums of R.R.  (The
// first step's loads are issued before the scalars are known; so in the kernels below.)
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads, 2)
    k_cg_update(int64_t n, int k, double* R, const double* Q, const double* pq_partial,
                double* rr_partial, CgScalars* S) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  __shared__ double s_alpha[kMaxCols];
  __shared__ int s_run[kMaxCols];
  Walk<G> w(n, k);
  double r[G::U][G::W], q2[G::U][G::W];
  w.load(R, r);
  w.load(Q, q2);
  const double pq = read_partials<G>(pq_partial, gridDim.x, k, sh);
  const int c = threadIdx.x;
  if (c < k) {
    const int active = S->active[c], run = active && pq > 0.0;
    const double rr = S->rr[c];
    s_run[c] = run;
    s_alpha[c] = run ? rr / pq : 0.0;
    if (blockIdx.x == 0) {
      if (active && !run) S->breakdown[c] = 1;
      S->running[c] = run;
      S->alpha[c] = s_alpha[c];
      S->rr_old[c] = rr;
    }
  }
  __syncthreads();
  double alpha[G::KC], acc[G::KC];
  bool run[G::KC];
  const int c0 = G::column(threadIdx.x, k);
#pragma unroll
  for (int q = 0; q < G::KC; ++q) {
    alpha[q] = s_alpha[c0 + q];
    run[q] = s_run[c0 + q];
    acc[q] = 0.0;
  }
  while (w.more()) {
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (!w.has(j)) break;
#pragma unroll
      for (int i = 0; i < G::W; ++i) {
        const int q = G::acc(i);
        const double x = fma(-alpha[q], q2[j][i], r[j][i]);  // (a select: a branch issued both sides' multiply-adds)
        r[j][i] = run[q] ? x : r[j][i];
        acc[q] = fma(r[j][i], r[j][i], acc[q]);
      }
    }
    w.store(R, r);
    w.next();
    w.load(R, r);
    w.load(Q, q2);
  }
  write_partial<G>(acc, k, rr_partial, sh);
}

// beta = R.R(new) / R.R(old); running columns: X += alpha P, P = R + beta P; then the columns that met
// the tolerance stop.  (X is updated here, where P is read anyway.)
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads, 2)
    k_cg_direction(int64_t n, int k, double* X, const double* R, double* P,
                   const double* rr_partial, CgScalars* S) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  __shared__ double s_alpha[kMaxCols], s_beta[kMaxCols];
  __shared__ int s_run[kMaxCols], s_next[kMaxCols];
  Walk<G> w(n, k);
  double x[G::U][G::W], r[G::U][G::W], p[G::U][G::W];
  w.load(X, x);
  w.load(R, r);
  w.load(P, p);
  const double rr = read_partials<G>(rr_partial, gridDim.x, k, sh);
  const int c = threadIdx.x;
  if (c < k) {
    const int run = S->running[c];
    s_run[c] = run;
    s_alpha[c] = S->alpha[c];
    s_beta[c] = run ? rr / S->rr_old[c] : 0.0;
    s_next[c] = run && rr > S->tol2[c];
    if (blockIdx.x == 0) {
      if (run) {
        S->rr[c] = rr;
        S->iters[c] += 1;
      }
      S->active[c] = s_next[c];
    }
  }
  __syncthreads();
  if (blockIdx.x == 0 && c == 0) {
    int na = 0;
    for (int q = 0; q < k; ++q) na += s_next[q];
    S->n_active = na;
  }
  double alpha[G::KC], beta[G::KC];
  bool run[G::KC];
  const int c0 = G::column(threadIdx.x, k);
#pragma unroll
  for (int q = 0; q < G::KC; ++q) {
    alpha[q] = s_alpha[c0 + q];
    beta[q] = s_beta[c0 + q];
    run[q] = s_run[c0 + q];
  }
  while (w.more()) {
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (!w.has(j)) break;
#pragma unroll
      for (int i = 0; i < G::W; ++i) {
        const int q = G::acc(i);
        const double xn = fma(alpha[q], p[j][i], x[j][i]), pn = fma(beta[q], p[j][i], r[j][i]);
        x[j][i] = run[q] ? xn : x[j][i];
        p[j][i] = run[q] ? pn : p[j][i];
      }
    }
    w.store(X, x);
    w.store(P, p);
    w.next();
    w.load(X, x);
    w.load(R, r);
    w.load(P, p);
  }
}

// ---------------------------------------------------------------- Lanczos kernels
// Column sums of V0.V0.
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads, 2) k_lz_norm(int64_t n, int k, const double* V0,
                                                            double* partial) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  double acc[G::KC];
#pragma unroll
  for (int q = 0; q < G::KC; ++q) acc[q] = 0.0;
  for (Walk<G> w(n, k); w.more(); w.next()) {
    double v[G::U][G::W];
    w.load(V0, v);
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (!w.has(j)) break;
#pragma unroll
      for (int i = 0; i < G::W; ++i) acc[G::acc(i)] = fma(v[j][i], v[j][i], acc[G::acc(i)]);
    }
  }
  write_partial<G>(acc, k, partial, sh);
}

// A power of two near 1 / sqrt(uu): a vector of squared norm uu > 0 is scaled by it without rounding, to a
// squared norm of 1 .. 4.
__device__ __forceinline__ double unit_scale(double uu) { return ldexp(1.0, -(ilogb(uu) >> 1)); }

// u_1 = V0 scaled by unit_scale (0 in a column of norm 0), so that no product or sum depends on |V0|; column
// sums of u_1.u_1.  One pass over V0 a call: 500,009 rows, k = 4, 20 steps 1794 -> 1808 us; 1,000,000 rows, k = 1,
// 12 steps 902 -> 908.
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads, 2)
    k_lz_start(int64_t n, int k, const double* V0, double* u1, const double* norm_partial, double* uu_partial) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  __shared__ double s_scale[kMaxCols];
  Walk<G> w(n, k);
  double v[G::U][G::W];
  w.load(V0, v);
  const double norm2 = read_partials<G>(norm_partial, gridDim.x, k, sh);
  const int c = threadIdx.x;
  if (c < k) s_scale[c] = norm2 > 0.0 ? unit_scale(norm2) : 0.0;
  __syncthreads();
  double scale[G::KC], acc[G::KC];
  const int c0 = G::column(threadIdx.x, k);
#pragma unroll
  for (int q = 0; q < G::KC; ++q) {
    scale[q] = s_scale[c0 + q];
    acc[q] = 0.0;
  }
  while (w.more()) {
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (!w.has(j)) break;
#pragma unroll
      for (int i = 0; i < G::W; ++i) {
        const int q = G::acc(i);
        v[j][i] = scale[q] > 0.0 ? v[j][i] * scale[q] : 0.0;
        acc[q] = fma(v[j][i], v[j][i], acc[q]);
      }
    }
    w.store(u1, v);
    w.next();
    w.load(V0, v);
  }
  write_partial<G>(acc, k, uu_partial, sh);
}

// The beta of the step before, from uu = u_j.u_j.  uu_old is multiplied by the square of its own scale, a power
// of two, so the quotient is beta^2 whatever size u_{j-1} had.
__device__ __forceinline__ double last_beta(const LzScalars* S, int c, double uu) {
  return S->live_old[c] ? sqrt(uu / (S->scale_old[c] * S->uu_old[c] * S->scale_old[c])) : 0.0;
}

// The Lanczos vectors are not normalised: u_j = |u_j| v_j, and the pass that divided by the norm is gone
// (seven vector passes instead of nine; k = 4, 500,009 rows: 92.2 -> 89.2 us a step).  W (= A u_j) is scaled by
// s_j, a power of two near 1 / |u_j| (0 for a column that has stopped), so that nothing is rounded, and
// becomes s_j |u_j| (A v_j - beta_{j-1} v_{j-1}) = s_j W - (s_j u_j.u_j / s_{j-1} u_{j-1}.u_{j-1}) u_{j-1}; column sums
// of W.u_j.  Each column scalar is one quotient of such sums: its error is alike in every row.  beta_{j-1} is
// |u_j| / (s_{j-1} |u_{j-1}|), stored to beta_out unless that is NULL (j = 1; every column was live before).
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads, 2)
    k_lz_alpha(int64_t n, int k, double* W, const double* u, const double* u_prev, const double* uu_partial,
               double* wu_partial, LzScalars* S, double* beta_out) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  __shared__ double s_inv[kMaxCols], s_prev[kMaxCols];
  Walk<G> w(n, k);
  double x[G::U][G::W], uj[G::U][G::W], up[G::U][G::W];
  w.load(W, x);
  w.load(u, uj);
  const double uu = read_partials<G>(uu_partial, gridDim.x, k, sh);
  const int c = threadIdx.x;
  if (c < k) {
    const bool first = beta_out == nullptr;
    const bool live = (first || S->live_old[c]) && uu > 0.0;
    const double scale = live ? unit_scale(uu) : 0.0;
    s_inv[c] = scale;
    s_prev[c] = !first && live ? scale * uu / (S->scale_old[c] * S->uu_old[c]) : 0.0;
    if (blockIdx.x == 0) {
      if (!first) beta_out[c] = last_beta(S, c, uu);
      S->live[c] = live;
      S->scale[c] = scale;
      S->uu[c] = uu;
    }
  }
  __syncthreads();
  double inv[G::KC], prev[G::KC], acc[G::KC];
  const int c0 = G::column(threadIdx.x, k);
#pragma unroll
  for (int q = 0; q < G::KC; ++q) {
    inv[q] = s_inv[c0 + q];
    prev[q] = s_prev[c0 + q];
    acc[q] = 0.0;
  }
  while (w.more()) {
    w.load(u_prev, up);
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (!w.has(j)) break;
#pragma unroll
      for (int i = 0; i < G::W; ++i) {
        const int q = G::acc(i);
        x[j][i] = fma(-prev[q], up[j][i], inv[q] * x[j][i]);
        acc[q] = fma(x[j][i], uj[j][i], acc[q]);
      }
    }
    w.store(W, x);
    w.next();
    w.load(W, x);
    w.load(u, uj);
  }
  write_partial<G>(acc, k, wu_partial, sh);
}

// alpha_j = W.u_j / (s_j u_j.u_j) (live columns), stored to alpha_out; W = W - (W.u_j / u_j.u_j) u_j = u_{j+1}; column
// sums of W.W.
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads, 2)
    k_lz_beta(int64_t n, int k, double* W, const double* u, const double* wu_partial, double* uu_partial,
              LzScalars* S, double* alpha_out) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  __shared__ double s_a[kMaxCols];
  Walk<G> w(n, k);
  double x[G::U][G::W], uj[G::U][G::W];
  w.load(W, x);
  w.load(u, uj);
  const double wu = read_partials<G>(wu_partial, gridDim.x, k, sh);
  const int c = threadIdx.x;
  if (c < k) {
    const bool live = S->live[c];
    s_a[c] = live ? wu / S->uu[c] : 0.0;
    if (blockIdx.x == 0) {
      alpha_out[c] = live ? wu / (S->scale[c] * S->uu[c]) : 0.0;
      S->uu_old[c] = S->uu[c];
      S->scale_old[c] = S->scale[c];
      S->live_old[c] = S->live[c];
    }
  }
  __syncthreads();
  double a[G::KC], acc[G::KC];
  const int c0 = G::column(threadIdx.x, k);
#pragma unroll
  for (int q = 0; q < G::KC; ++q) {
    a[q] = s_a[c0 + q];
    acc[q] = 0.0;
  }
  while (w.more()) {
#pragma unroll
    for (int j = 0; j < G::U; ++j) {
      if (!w.has(j)) break;
#pragma unroll
      for (int i = 0; i < G::W; ++i) {
        const int q = G::acc(i);
        x[j][i] = fma(-a[q], uj[j][i], x[j][i]);
        acc[q] = fma(x[j][i], x[j][i], acc[q]);
      }
    }
    w.store(W, x);
    w.next();
    w.load(W, x);
    w.load(u, uj);
  }
  write_partial<G>(acc, k, uu_partial, sh);
}

// One CTA: the last beta.
template <int K, int MODE>
__global__ void __launch_bounds__(kVecThreads) k_lz_end(int k, const double* uu_partial, unsigned n_partials,
                                                        const LzScalars* S, double* beta_out) {
  using G = Seg<K, MODE>;
  grid_wait();
  grid_dependents();
  __shared__ VecShared sh;
  const double uu = read_partials<G>(uu_partial, n_partials, k, sh);
  if ((int)threadIdx.x < k) beta_out[threadIdx.x] = last_beta(S, threadIdx.x, uu);
}

// ---------------------------------------------------------------- dispatch
template <template <int, int> class F, typename... Args>
static cudaError_t by_k(int k, Args... args) {
  switch (k) {
    case 1: return F<1, PAIRS>::run(args...);
    case 2: return F<2, VROWS>::run(args...);
    case 4: return F<4, VROWS>::run(args...);
    case 8: return F<8, VGROUPS>::run(args...);
    case 16: return F<16, VGROUPS>::run(args...);
    default: return F<1, FLAT>::run(args...);
  }
}

#define SOLVER_LAUNCHER(NAME, ...)                                   \
  template <int K, int MODE>                                         \
  struct NAME {                                                      \
    template <typename... A>                                         \
    static cudaError_t run(unsigned grid, cudaStream_t s, A... a) { \
      return launch_dependent(__VA_ARGS__, grid, kVecThreads, s, a...); \
    }                                                                \
  };
SOLVER_LAUNCHER(LCgInit, k_cg_init<K, MODE>)
SOLVER_LAUNCHER(LCgBegin, k_cg_begin<K, MODE>)
SOLVER_LAUNCHER(LCgDot, k_cg_dot<K, MODE>)
SOLVER_LAUNCHER(LCgUpdate, k_cg_update<K, MODE>)
SOLVER_LAUNCHER(LCgDirection, k_cg_direction<K, MODE>)
SOLVER_LAUNCHER(LLzNorm, k_lz_norm<K, MODE>)
SOLVER_LAUNCHER(LLzStart, k_lz_start<K, MODE>)
SOLVER_LAUNCHER(LLzAlpha, k_lz_alpha<K, MODE>)
SOLVER_LAUNCHER(LLzBeta, k_lz_beta<K, MODE>)
SOLVER_LAUNCHER(LLzEnd, k_lz_end<K, MODE>)
#undef SOLVER_LAUNCHER

// CTAs of the vector kernels on an n x k block: enough for its units, at most `most`.
template <int K, int MODE>
struct LGrid {
  static cudaError_t run(int64_t n, int k, int64_t most, unsigned* grid) {
    using G = Seg<K, MODE>;
    const int64_t per_cta = G::threads(k);
    *grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((G::units(n, k) + per_cta - 1) / per_cta, most));
    return cudaSuccess;
  }
};

}  // namespace spmv

using namespace spmv;

struct spmv_solver {
  spmv_handle A = nullptr;
  int device = 0, k = 0;
  int64_t n = 0;
  unsigned grid = 1;               // CTAs of the vector kernels (one wave at most)
  double *buf[3] = {nullptr, nullptr, nullptr};  // CG: R, P, Q; Lanczos: u_{j-1}, u_j, W in turn
  double *partial = nullptr, *partial2 = nullptr;  // column sums per CTA (two, one read while the other is written)
  CgScalars* cg = nullptr;
  LzScalars* lz = nullptr;
  double* lz_out = nullptr;        // alpha[m][16], beta[m][16] on the device
  int lz_cap = 0;
  int* host_active = nullptr;      // pinned
  cudaStream_t cap = nullptr;
  cudaEvent_t ev = nullptr;
  cudaGraphExec_t graph = nullptr;
  const double* g_B = nullptr;
  double* g_X = nullptr;
  int g_steps = 0;
  uint64_t g_gen = 0;              // plan generation the graph was captured at
};

static void solver_free(spmv_solver* s) {
  if (s->graph) cudaGraphExecDestroy(s->graph);
  for (double* b : s->buf) if (b) cudaFree(b);
  if (s->partial) cudaFree(s->partial);
  if (s->partial2) cudaFree(s->partial2);
  if (s->cg) cudaFree(s->cg);
  if (s->lz) cudaFree(s->lz);
  if (s->lz_out) cudaFree(s->lz_out);
  if (s->host_active) cudaFreeHost(s->host_active);
  if (s->cap) cudaStreamDestroy(s->cap);
  if (s->ev) cudaEventDestroy(s->ev);
}

namespace {
struct SolverDeviceGuard {
  int prev = -1;
  explicit SolverDeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
  }
  ~SolverDeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

// One CG iteration on stream s: Q = A P, then P.Q, the R update, and X with the new direction.
spmv_status cg_iteration(spmv_solver* S, double* X, cudaStream_t s) {
  double *R = S->buf[0], *P = S->buf[1], *Q = S->buf[2];
  spmv_status st = spmv_apply_block(S->A, P, S->k, S->k, Q, S->k, s);
  if (st != SPMV_OK) return st;
  cudaError_t e = by_k<LCgDot>(S->k, S->grid, s, S->n, S->k, (const double*)P, (const double*)Q, S->partial);
  if (e == cudaSuccess)
    e = by_k<LCgUpdate>(S->k, S->grid, s, S->n, S->k, R, (const double*)Q, (const double*)S->partial, S->partial2,
                        S->cg);
  if (e == cudaSuccess)
    e = by_k<LCgDirection>(S->k, S->grid, s, S->n, S->k, X, (const double*)R, P, (const double*)S->partial2, S->cg);
  return e == cudaSuccess ? SPMV_OK : cuda_fail(e, "CG kernel launch");
}
}  // namespace

extern "C" {

spmv_status spmv_solver_create(spmv_handle A, int32_t k, spmv_solver_handle* out) {
  if (!A || !out) return fail(SPMV_ERR_ARG, "NULL argument");
  *out = nullptr;
  spmv_info info;
  spmv_status st = spmv_get_info(A, &info);
  if (st != SPMV_OK) return st;
  if (info.n_rows != info.n_cols) return fail(SPMV_ERR_ARG, "the solvers need a square matrix");
  if (k < 1 || k > plan_max_k(A)) return fail(SPMV_ERR_ARG, "k out of range 1..max_k of the plan");
  auto* S = new (std::nothrow) spmv_solver;
  if (!S) return fail(SPMV_ERR_OOM, "host allocation failed");
  S->A = A;
  S->device = plan_device(A);
  S->k = k;
  S->n = info.n_rows;
  SolverDeviceGuard g(S->device);
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, S->device);
  if (e == cudaSuccess)
    e = by_k<LGrid>(k, S->n, k, (int64_t)(sms > 0 ? sms : 1) * kVecCtasPerSm, &S->grid);
  const size_t vec = sizeof(double) * (size_t)(S->n > 0 ? S->n : 1) * (size_t)k;
  for (int b = 0; b < 3 && e == cudaSuccess; ++b) e = cudaMalloc(&S->buf[b], vec);
  if (e == cudaSuccess) e = cudaMalloc(&S->partial, sizeof(double) * S->grid * kMaxCols);
  if (e == cudaSuccess) e = cudaMalloc(&S->partial2, sizeof(double) * S->grid * kMaxCols);
  if (e == cudaSuccess) e = cudaMalloc(&S->cg, sizeof(CgScalars));
  if (e == cudaSuccess) e = cudaMemset(S->cg, 0, sizeof(CgScalars));
  if (e == cudaSuccess) e = cudaMalloc(&S->lz, sizeof(LzScalars));
  if (e == cudaSuccess) e = cudaMallocHost(&S->host_active, sizeof(int));
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&S->cap, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&S->ev, cudaEventDisableTiming);
  if (e != cudaSuccess) {
    solver_free(S);
    delete S;
    return e == cudaErrorMemoryAllocation ? fail(SPMV_ERR_OOM, "solver work vectors")
                                          : cuda_fail(e, "solver setup");
  }
  *out = S;
  return SPMV_OK;
}

spmv_status spmv_solver_destroy(spmv_solver_handle S) {
  if (!S) return SPMV_OK;
  {
    SolverDeviceGuard g(S->device);
    cudaDeviceSynchronize();
    solver_free(S);
  }
  delete S;
  return SPMV_OK;
}

spmv_status spmv_cg_solve(spmv_solver_handle S, const double* B_dev, double* X_dev, int32_t max_iter, double rtol,
                          int32_t check_every, void* stream, int32_t* iterations_host, double* rr_host,
                          spmv_cg_summary* summary) {
  if (!S) return fail(SPMV_ERR_ARG, "solver handle is NULL");
  if (max_iter < 0 || check_every < 1 || !(rtol >= 0.0)) return fail(SPMV_ERR_ARG, "bad max_iter, check_every or rtol");
  if (S->n > 0 && (!B_dev || !X_dev)) return fail(SPMV_ERR_ARG, "B or X is NULL");
  if ((((uintptr_t)B_dev) | ((uintptr_t)X_dev)) & 15) return fail(SPMV_ERR_ARG, "B and X must be 16-byte aligned");
  SolverDeviceGuard g(S->device);
  cudaStream_t s = (cudaStream_t)stream;
  CgScalars host{};
  if (S->n > 0) {
    // R = B - A X0, P = R, scalars
    spmv_status st = spmv_apply_block(S->A, X_dev, S->k, S->k, S->buf[2], S->k, s);
    if (st != SPMV_OK) return st;
    cudaError_t e = by_k<LCgInit>(S->k, S->grid, s, S->n, S->k, B_dev, (const double*)S->buf[2], S->buf[0], S->buf[1],
                                  S->partial, S->partial2);
    if (e == cudaSuccess)
      e = by_k<LCgBegin>(S->k, 1u, s, S->k, (const double*)S->partial, (const double*)S->partial2, S->grid, S->cg,
                         rtol * rtol);
    if (e != cudaSuccess) return cuda_fail(e, "CG init launch");
    const int steps = check_every < max_iter ? check_every : (max_iter > 0 ? max_iter : 1);
    const uint64_t gen = plan_generation(S->A);
    if (max_iter > 0 &&
        (!S->graph || S->g_B != B_dev || S->g_X != X_dev || S->g_steps != steps || S->g_gen != gen)) {
      if (S->graph) cudaGraphExecDestroy(S->graph);
      S->graph = nullptr;
      cudaGraph_t gr = nullptr;
      SPMV_CUDA(cudaStreamBeginCapture(S->cap, cudaStreamCaptureModeThreadLocal));
      spmv_status cst = SPMV_OK;
      for (int it = 0; it < steps && cst == SPMV_OK; ++it) cst = cg_iteration(S, X_dev, S->cap);
      cudaError_t ce = cudaStreamEndCapture(S->cap, &gr);
      if (cst != SPMV_OK) {
        if (gr) cudaGraphDestroy(gr);
        return cst;
      }
      if (ce != cudaSuccess) return cuda_fail(ce, "CG graph capture");
      ce = cudaGraphInstantiate(&S->graph, gr, 0);
      cudaGraphDestroy(gr);
      if (ce != cudaSuccess) {
        S->graph = nullptr;
        return cuda_fail(ce, "CG graph instantiate");
      }
      S->g_B = B_dev;
      S->g_X = X_dev;
      S->g_steps = steps;
      S->g_gen = gen;
    }
    int done = 0;
    while (done < max_iter) {
      // whole graphs while they fit; the remainder one iteration at a time
      if (max_iter - done >= S->g_steps) {
        SPMV_CUDA(cudaGraphLaunch(S->graph, s));
        done += S->g_steps;
      } else {
        spmv_status ist = cg_iteration(S, X_dev, s);
        if (ist != SPMV_OK) return ist;
        done += 1;
        if (done < max_iter && (done % S->g_steps) != 0) continue;
      }
      SPMV_CUDA(cudaMemcpyAsync(S->host_active, &S->cg->n_active, sizeof(int), cudaMemcpyDeviceToHost, s));
      SPMV_CUDA(cudaEventRecord(S->ev, s));
      SPMV_CUDA(cudaEventSynchronize(S->ev));
      if (*S->host_active == 0) break;
    }
    SPMV_CUDA(cudaMemcpyAsync(&host, S->cg, sizeof(CgScalars), cudaMemcpyDeviceToHost, s));
    SPMV_CUDA(cudaStreamSynchronize(s));
  }
  int it_max = 0, conv = 0, bd = 0;
  for (int q = 0; q < S->k; ++q) {
    if (iterations_host) iterations_host[q] = host.iters[q];
    if (rr_host) rr_host[q] = host.rr[q];
    it_max = host.iters[q] > it_max ? host.iters[q] : it_max;
    bd += host.breakdown[q];
    conv += !host.breakdown[q] && !(host.rr[q] > host.tol2[q]);
  }
  if (summary) {
    std::memset(summary, 0, sizeof(*summary));
    summary->iterations = it_max;
    summary->converged = S->n > 0 ? conv : S->k;
    summary->breakdown = bd;
  }
  return SPMV_OK;
}

spmv_status spmv_lanczos(spmv_solver_handle S, const double* V0_dev, int32_t m, double* alpha_host,
                         double* beta_host, void* stream) {
  if (!S) return fail(SPMV_ERR_ARG, "solver handle is NULL");
  if (m < 1) return fail(SPMV_ERR_ARG, "m must be >= 1");
  if (S->n > 0 && !V0_dev) return fail(SPMV_ERR_ARG, "V0 is NULL");
  if (((uintptr_t)V0_dev) & 15) return fail(SPMV_ERR_ARG, "V0 must be 16-byte aligned");
  if (!alpha_host || !beta_host) return fail(SPMV_ERR_ARG, "alpha or beta is NULL");
  SolverDeviceGuard g(S->device);
  cudaStream_t s = (cudaStream_t)stream;
  const int k = S->k;
  if (S->n == 0) {
    std::memset(alpha_host, 0, sizeof(double) * (size_t)m * k);
    std::memset(beta_host, 0, sizeof(double) * (size_t)m * k);
    return SPMV_OK;
  }
  if (S->lz_cap < m) {
    if (S->lz_out) cudaFree(S->lz_out);
    S->lz_out = nullptr;
    S->lz_cap = 0;
    SPMV_CUDA(cudaMalloc(&S->lz_out, sizeof(double) * 2 * (size_t)m * kMaxCols));
    S->lz_cap = m;
  }
  double* a_out = S->lz_out;
  double* b_out = S->lz_out + (size_t)m * kMaxCols;
  // u_{j+1} is the W of step j; the three buffers hold u_{j-1}, u_j and W in turn, u_0 = 0 and u_1 (V0
  // scaled) first
  const double *u_prev = S->buf[0], *u = S->buf[1];
  cudaError_t e = by_k<LLzNorm>(k, S->grid, s, S->n, k, V0_dev, S->partial2);
  if (e == cudaSuccess)
    e = by_k<LLzStart>(k, S->grid, s, S->n, k, V0_dev, S->buf[1], (const double*)S->partial2, S->partial);
  // (The memset last: without it between them the first product is launched while k_lz_start runs, and all
  // steps behind it take 2 us longer, 1,000,000 rows, k = 1.)
  if (e == cudaSuccess) e = cudaMemsetAsync(S->buf[0], 0, sizeof(double) * (size_t)S->n * (size_t)k, s);
  if (e != cudaSuccess) return cuda_fail(e, "Lanczos start");
  for (int j = 0; j < m; ++j) {
    double* W = S->buf[(j + 2) % 3];
    spmv_status st = spmv_apply_block(S->A, u, k, k, W, k, s);
    if (st != SPMV_OK) return st;
    e = by_k<LLzAlpha>(k, S->grid, s, S->n, k, W, u, u_prev, (const double*)S->partial, S->partial2, S->lz,
                       j ? b_out + (size_t)(j - 1) * kMaxCols : (double*)nullptr);
    if (e == cudaSuccess)
      e = by_k<LLzBeta>(k, S->grid, s, S->n, k, W, u, (const double*)S->partial2, S->partial, S->lz,
                        a_out + (size_t)j * kMaxCols);
    if (e != cudaSuccess) return cuda_fail(e, "Lanczos kernel launch");
    u_prev = u;
    u = W;
  }
  e = by_k<LLzEnd>(k, 1u, s, k, (const double*)S->partial, S->grid, (const LzScalars*)S->lz,
                   b_out + (size_t)(m - 1) * kMaxCols);
  if (e != cudaSuccess) return cuda_fail(e, "Lanczos kernel launch");
  std::vector<double> tmp((size_t)2 * m * kMaxCols);
  SPMV_CUDA(cudaMemcpyAsync(tmp.data(), S->lz_out, sizeof(double) * tmp.size(), cudaMemcpyDeviceToHost, s));
  SPMV_CUDA(cudaStreamSynchronize(s));
  for (int j = 0; j < m; ++j)
    for (int q = 0; q < k; ++q) {
      alpha_host[(size_t)j * k + q] = tmp[(size_t)j * kMaxCols + q];
      beta_host[(size_t)j * k + q] = tmp[(size_t)(m + j) * kMaxCols + q];
    }
  return SPMV_OK;
}

}  // extern "C"
