// CRS_L{1,2,4,8,16,32}: L lanes per row, loads straight from HBM (Sec. 1.2 loop).
//
// L >= 2 (k_crs_lanes): a group of L consecutive lanes owns one row; lane t of the
// group takes entries rs + t, rs + t + L, ... (for L >= 8 a group's loads of
// val/col_idx coalesce), gathers B with read-only loads and keeps FP64 partial sums,
// which an xor-shuffle tree of log2(L) steps adds at the end.
//
// CRS_L1 is a family of its own (crs_l1): one vector on short rows
// (k_crs_row) or on rows of eight and more entries on average (k_crs_wide), blocks of
// k >= 2 columns with a row's columns split over k / W lanes (k_crs_cols), and, when
// AUTO asks for it, a few long rows on a warp or a CTA each (k_crs_long).  Except for
// those long rows a row's entries go to one lane in order, each column's sum is
// formed in the same order whatever the block's width and alignment are, and the
// bits are the same.
#include <type_traits>

#include "device.cuh"
#include "internal.h"

namespace spmv {

// Bring the val/col slices of rows [f0, f0 + rows) into L2 (one thread).
template <typename VT>
__device__ __forceinline__ void prefetch_rows(int64_t f0, int64_t rows, int64_t n_rows,
                                              const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                              const VT* __restrict__ val) {
  if (f0 >= n_rows) return;
  const int64_t f1 = f0 + rows < n_rows ? f0 + rows : n_rows;
  const int bs = __ldg(row_ptr + f0), be = __ldg(row_ptr + f1);
  constexpr int VA = 16 / (int)sizeof(VT);
  const int v_lo = bs & ~(VA - 1), v_hi = (be + VA - 1) & ~(VA - 1);
  const int c_lo = bs & ~3, c_hi = (be + 3) & ~3;
  if (be > bs) {
    prefetch_l2(val + v_lo, (uint32_t)(v_hi - v_lo) * (uint32_t)sizeof(VT));
    prefetch_l2(col + c_lo, (uint32_t)(c_hi - c_lo) * 4u);
  }
}

// VEC (L > 1, a full block of K >= 2 columns with 16-byte aligned B rows): each
// entry's K values are gathered with K / 2 16-byte loads instead of K 8-byte ones.
template <typename VT, int L, int K, bool VEC>
__global__ void __launch_bounds__(kThreads, (K == 1 ? 8 : 1))
    k_crs_lanes(int64_t n_rows, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
                const VT* __restrict__ val, const double* __restrict__ B, int64_t ldb, double* __restrict__ C,
                int64_t ldc, int k, int prefetch) {
  constexpr int RPC = kThreads / L;  // rows per CTA
  // bring the val/col slices of the CTA `prefetch` positions ahead into L2
  if (threadIdx.x == 0 && prefetch > 0)
    prefetch_rows(((int64_t)blockIdx.x + prefetch) * RPC, RPC, n_rows, row_ptr, col, val);
  const int64_t g = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / L;
  const int t = threadIdx.x % L;
  const bool active = g < n_rows;
  int rs = 0, re = 0;
  if (active) {
    rs = __ldg(row_ptr + g);
    re = __ldg(row_ptr + g + 1);
  }
  double acc[K];
#pragma unroll
  for (int q = 0; q < K; ++q) acc[q] = 0.0;
  // batches of NB entries per lane: all gathers of a batch are issued before its FMAs
  // (K >= 4: one entry per batch; its K gathers already keep the FP64 pipe fed, and two entries
  // measured 9 % slower at K = 4)
  constexpr int NB = K < 4 && L == 2 ? 4 / K : 1;
  for (int j = rs + t; j < re; j += NB * L) {
    double v[NB];
    const double* b[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int jj = (j + u * L < re) ? j + u * L : j;
      v[u] = to_f64(L >= 8 ? ldcs(val + jj) : ldg(val + jj));
      b[u] = B + (int64_t)(L >= 8 ? ldcs(col + jj) : ldg(col + jj)) * ldb;
    }
    double gv[NB][K];
    if constexpr (VEC) {
#pragma unroll
      for (int u = 0; u < NB; ++u)
#pragma unroll
        for (int q = 0; q < K; q += 2) {
          const double2 x = j + u * L < re ? __ldg(reinterpret_cast<const double2*>(b[u] + q)) : make_double2(0.0, 0.0);
          gv[u][q] = x.x;
          gv[u][q + 1] = x.y;
        }
    } else {
#pragma unroll
      for (int u = 0; u < NB; ++u)
#pragma unroll
        for (int q = 0; q < K; ++q) gv[u][q] = (j + u * L < re && q < k) ? __ldg(b[u] + q) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < NB; ++u)
#pragma unroll
      for (int q = 0; q < K; ++q)
        if (j + u * L < re && q < k) acc[q] = fma(v[u], gv[u][q], acc[q]);
  }
#pragma unroll
  for (int q = 0; q < K; ++q) acc[q] = warp_sum_xor(acc[q], L);
  if (!active) return;
  double* out = C + g * ldc;
#pragma unroll
  for (int q = 0; q < K; ++q)
    if (q < k && t == q % L) out[q] = acc[q];
}

// The last 0..3 entries of a row (r of them, gathers x): no multiply-add is issued that no lane of the
// warp needs.  A masked-off warp instruction occupies the FP64 pipe (16 cycles of an SM) like any other.
template <typename VT, int W>
__device__ __forceinline__ void add_tail(int r, const VT* v, const double (*x)[W], double (&acc)[W]) {
  const unsigned lanes = __activemask();
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    if (!__any_sync(lanes, u < r)) break;
    if (u < r)
#pragma unroll
      for (int q = 0; q < W; ++q) acc[q] = fma(to_f64(v[u]), x[u][q], acc[q]);
  }
}

// CRS_L1, one vector: thread per row, four entries at a time (their gathers in flight together), then
// the last 0..3.  Padding each row's last batch of eight (FP32 values: four) with masked multiply-adds
// cost what it padded: 280^3 Poisson (7 entries a row) 326.5 -> 323.2 us (HBM-bound), with FP32 values
// 303.9 -> 272.4 us; 1500^2 Laplacian 39.0 -> 33.2 us; 3,000,000 rows of 5 entries 48.9 -> 41.1 us.  The
// two pipes together bound it: 7 multiply-adds per row are 0.74 of the HBM time at 280^3, with FP32
// values 0.99 of it.  Among uneven rows a warp waits for its longest anyway, and with FP32 values the
// batches are masked (MASKED): 1,500,000 rows of 0 .. 12 / 4 .. 9 / 10 .. 30 entries 42.0 -> 35.1, 42.6 ->
// 35.8, 53.9 -> 42.4 us, power-law rows of up to 16 35.0 -> 30.7.  (Doubles of the first, second and last: 44.3 ->
// 40.9, 39.0 -> 40.8, 32.6 -> 37.0; not masked.)
template <typename VT, bool UNIT, bool MASKED>  // UNIT: ldb = 1 (its multiplication and two registers saved)
__global__ void __launch_bounds__(kThreads, 8)
    k_crs_row(int64_t n_rows, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
              const VT* __restrict__ val, const double* B, int64_t ldb, double* C,
              int64_t ldc, int prefetch) {
  if (threadIdx.x == 0 && prefetch > 0)
    prefetch_rows(((int64_t)blockIdx.x + prefetch) * kThreads, kThreads, n_rows, row_ptr, col, val);
  const int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (g >= n_rows) return;
  int j = __ldg(row_ptr + g);
  const int re = __ldg(row_ptr + g + 1);
  grid_wait();
  if (gridDim.x > 4 * kOneWave) grid_dependents();
  double acc[1] = {0.0};
  if constexpr (MASKED) {
    for (int left = re - j; left > 0; left -= 4, j = (int)((uint32_t)j + 4)) {
      double v[4], x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = u < left ? j + u : j;
        v[u] = to_f64(ldg(val + i));
        const double* b = UNIT ? B + ldg(col + i) : B + (int64_t)ldg(col + i) * ldb;
        x[u] = u < left ? *b : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (u < left) acc[0] = fma(v[u], x[u], acc[0]);
    }
    grid_dependents();
    C[g * ldc] = acc[0];
    return;
  }
  for (; (uint32_t)j + 4 <= (uint32_t)re; j += 4) {
    const VT* vj = val + j;
    const int32_t* cj = col + j;
    double v[4], x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u] = to_f64(ldg(vj + u));
      x[u] = *(UNIT ? B + ldg(cj + u) : B + (int64_t)ldg(cj + u) * ldb);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[0] = fma(v[u], x[u], acc[0]);
  }
  double v[3], x[3][1];
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    v[u] = x[u][0] = 0.0;
    if ((uint32_t)j + u < (uint32_t)re) {
      v[u] = to_f64(ldg(val + j + u));
      x[u][0] = *(UNIT ? B + ldg(col + j + u) : B + (int64_t)ldg(col + j + u) * ldb);
    }
  }
  add_tail(re - j, v, x, acc);
  grid_dependents();
  C[g * ldc] = acc[0];
}

// The halo pass of the local/halo split: C[rows[t]] += (halo row t) * B, as k_crs_row.
template <typename VT>
__global__ void __launch_bounds__(kThreads, 8)
    k_crs_halo(int64_t n_rows, const int32_t* __restrict__ rows, const int32_t* __restrict__ row_ptr,
               const int32_t* __restrict__ col, const VT* __restrict__ val, const double* B, double* C) {
  const int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (g >= n_rows) return;
  const int64_t row = __ldg(rows + g);
  const int rs = __ldg(row_ptr + g), re = __ldg(row_ptr + g + 1);
  grid_wait();
  grid_dependents();
  const double c = C[row];
  double acc = 0.0;
  for (int j = rs; j < re; ++j) acc = fma(to_f64(ldg(val + j)), B[ldg(col + j)], acc);
  C[row] = c + acc;
}

// k columns of a row on G = k / W lanes, W columns each (A16: the blocks' rows start on 16 bytes; even W).
template <typename VT, int W, bool A16>
__global__ void __launch_bounds__(kThreads, (W == 1 ? 8 : 6))
    k_crs_cols(int64_t n_rows, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
               const VT* __restrict__ val, const double* B, int64_t ldb, double* C,
               int64_t ldc, int G, int prefetch) {
  const int rpc = kThreads / G;  // rows per CTA
  if (threadIdx.x == 0 && prefetch > 0)
    prefetch_rows(((int64_t)blockIdx.x + prefetch) * rpc, rpc, n_rows, row_ptr, col, val);
  const int r = (int)threadIdx.x / G;
  const int64_t g = (int64_t)blockIdx.x * rpc + r;
  if (r >= rpc || g >= n_rows) return;
  const int c0 = ((int)threadIdx.x - r * G) * W;  // first column of this lane
  const int rs = __ldg(row_ptr + g), re = __ldg(row_ptr + g + 1);
  grid_wait();
  if (gridDim.x > kOneWave) grid_dependents();
  double acc[W];
#pragma unroll
  for (int q = 0; q < W; ++q) acc[q] = 0.0;
  const double* Bc = B + c0;
  for (int j = rs; j < re; ++j) {
    const double v = to_f64(ldg(val + j));
    double gv[W];
    load_cols<W, A16>(Bc + (int64_t)ldg(col + j) * ldb, gv);
#pragma unroll
    for (int q = 0; q < W; ++q) acc[q] = fma(v, gv[q], acc[q]);
  }
  grid_dependents();
  store_cols<W, A16>(C + g * ldc + c0, acc);
}

template <typename VT, int W, bool A16 = (W % 2 == 0)>
static cudaError_t launch_cols(int64_t n_rows, const int32_t* row_ptr, const int32_t* col, const VT* val,
                               const double* B, int64_t ldb, double* C, int64_t ldc, int k, int pf, cudaStream_t s) {
  const int G = k / W, rpc = kThreads / G;
  const int64_t grid = (n_rows + rpc - 1) / rpc;
  return launch_dependent(k_crs_cols<VT, W, A16>, (unsigned)grid, kThreads, s, n_rows, row_ptr, col, val, B, ldb, C,
                          ldc, G, pf);
}

// out[i] = (a, b)[i + phase], i < 4, phase < 4: four consecutive entries that straddle two aligned groups.
template <typename T>
__device__ __forceinline__ void realign(const T (&a)[4], const T (&b)[4], int phase, T (&out)[4]) {
  const bool one = phase & 1, two = phase & 2;
  T t[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const T x = i < 4 ? a[i % 4] : b[i % 4], y = i < 3 ? a[(i + 1) % 4] : b[(i + 1) % 4];
    t[i] = one ? y : x;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) out[i] = two ? t[i + 2] : t[i];
}

// CRS_L1 on matrices of longer rows, k = W columns on the row's one lane: val and col_idx are read in
// aligned groups of four entries (32 and 16 bytes), realigned in registers to the row's own start, so
// that no multiply-add is issued for an entry of another row and the order of the sum is the scalar
// kernel's.  One entry at a time, the 32 lanes of a load touch 32 lines of which each gives 8 or 4
// bytes, and at 27 entries a row L1 loses most of them before their next use: 569 MB came from DRAM for
// 330 MB of matrix.  Now every sector is used by the load that fetches it.  On a 27-point stencil of
// 999,900 rows 131.0 -> 71.2 us (HBM floor 50, FP64 floor 42): the gathers' latency at 40 warps
// per SM bounds it, and what L1 keeps for them.  So the doubles take no line there (76.5 -> 74.4 us; the
// column groups of half a sector must: 110 us without) and CTAs are of 64 threads, whose slots are
// refilled sooner (128: 72.6, 64: 71.2).  20 million entries in rows of 8 / 16 / 32 / 64, doubles, against 256
// threads and all in L1: 52.8 -> 49.7, 54.0 -> 49.3, 62.8 -> 52.5, 61.8 -> 51.8 us.  Staging a warp's 32 rows in
// shared memory instead (one bulk copy) took 75 us, but 248 against 93 us at 32 entries a row, where the
// lanes meet in one bank, and rows of 60 entries left 8 warps on an SM.  An L2 prefetch of the CTAs
// ahead slows it (152 ahead 79, 456 100 us), and so do a second group or its columns in flight (79 and
// 81 us), columns in groups of eight (72 registers: 74.5 us) and more warps with spilled registers (75 us).
constexpr int kWideThreads = 64;

template <typename VT, int W>
__global__ void __launch_bounds__(kWideThreads, (W == 4 ? 12 : 20))
    k_crs_wide(int64_t n_rows, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
               const VT* __restrict__ val, const double* B, int64_t ldb, double* C,
               int64_t ldc) {
  const int64_t g = (int64_t)blockIdx.x * kWideThreads + threadIdx.x;
  if (g >= n_rows) return;
  const int rs = __ldg(row_ptr + g), re = __ldg(row_ptr + g + 1);
  double acc[W];
#pragma unroll
  for (int q = 0; q < W; ++q) acc[q] = 0.0;
  const int phase = rs & 3;
  // the next four entries straddle the aligned groups a and b (a group is read only if it holds an
  // entry of the row)
  VT va[4] = {}, vb[4] = {};
  int32_t ca[4] = {}, cb[4] = {};
  // (at goes up to four beyond a row that may end at 2^31 - 1; 64 bits where registers are left for them: floats,
  // 300,000 rows of 3 or 40 entries, 26.9 us with 32 and 25.5 with 64)
  using At = typename std::conditional<sizeof(VT) == 8, uint32_t, int64_t>::type;
  const At end = re;
  At at = rs & ~3;
  if (at < end) {
    ldg4(val + at, va);
    ldg4(col + at, ca);
  }
  grid_wait();
  for (int n = re - rs; n > 0; n -= 4) {
    at += 4;
    if (at < end) {
      ldg4(col + at, cb);
      ldg4(val + at, vb);
    }
    VT v[4];
    int32_t c[4];
    realign(ca, cb, phase, c);
    double x[4][W];
    if (n >= 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) load_cols(B + (int64_t)c[u] * ldb, x[u]);
      realign(va, vb, phase, v);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < W; ++q) acc[q] = fma(to_f64(v[u]), x[u][q], acc[q]);
    } else {
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (u < n) load_cols(B + (int64_t)c[u] * ldb, x[u]);
      realign(va, vb, phase, v);
      add_tail(n, v, x, acc);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      va[u] = vb[u];
      ca[u] = cb[u];
    }
  }
  grid_dependents();
  store_cols(C + g * ldc, acc);
}

template <typename VT, int W>
static cudaError_t launch_wide(const CsrDev& A, const VT* val, const double* B, int64_t ldb, double* C, int64_t ldc,
                               cudaStream_t s) {
  const int64_t grid = (A.n_rows + kWideThreads - 1) / kWideThreads;
  return launch_dependent(k_crs_wide<VT, W>, (unsigned)grid, kWideThreads, s, A.n_rows, A.row_ptr, A.col, val, B,
                          ldb, C, ldc);
}

// One row on NT threads (a warp or the CTA; thread t of them): EP entry lanes, a power of two, times
// k column lanes.  Entry lane e adds entries rs + e, rs + e + EP, ...; a tree over sh (NT sums) adds
// the entry lanes in a fixed order.  One column per lane for every k: the tree's FP64 adds are what
// a row of a few dozen entries spends most on, and each step of it adds 32 useful sums this way.
template <typename VT, int NT>
__device__ __forceinline__ void long_row(int row, int t, int k, const int32_t* __restrict__ row_ptr,
                                         const int32_t* __restrict__ col, const VT* __restrict__ val,
                                         const double* B, int64_t ldb, double* C,
                                         int64_t ldc, double* sh) {
  const int rs = __ldg(row_ptr + row), re = __ldg(row_ptr + row + 1);
  const int ep = 1 << (31 - __clz(NT / k));
  const int e = t / k, c = t - e * k;
  double acc = 0.0;
  grid_wait();
  if (e < ep) {
    constexpr int U = 4;  // entries in flight per lane
    // (unsigned: the steps of a CTA's lanes go up to 1024 beyond a row that may end at 2^31 - 1)
    const uint32_t end = re, step = ep;
    for (uint32_t j = (uint32_t)rs + e; j < end; j += U * step) {
      double v[U], g[U];
#pragma unroll
      for (uint32_t u = 0; u < U; ++u) {
        const uint32_t jj = j + u * step < end ? j + u * step : j;
        v[u] = to_f64(ldcs(val + jj));
        g[u] = B[(int64_t)ldcs(col + jj) * ldb + c];
      }
#pragma unroll
      for (uint32_t u = 0; u < U; ++u)
        if (j + u * step < end) acc = fma(v[u], g[u], acc);
    }
  }
  sh[t] = acc;
  for (int h = ep >> 1; h > 0; h >>= 1) {
    if (NT == 32) __syncwarp(); else __syncthreads();
    if (e < h) sh[t] = acc += sh[t + h * k];
  }
  if (e == 0) C[(int64_t)row * ldc + c] = acc;
}

// CRS_L1 as AUTO runs it on matrices with long rows: the listed long rows first (longest first), each on
// a CTA or a warp, then the others with a lane per row and column.  What bounded these products was the
// longest row, walked by one thread with one or eight gathers in flight: a 200,000-row matrix with
// power-law lengths up to 2000 took 212.9 us at k = 1 and takes 10.2 now; what is left is the dependent loads
// of a lane's rounds and, back to back, the host's launch.  One column per lane for every k: a warp that
// covers fewer of these uneven rows waits less for its longest (1,000,000 rows, lengths up to 500, k = 4 / 8,
// four columns per lane 121.9 / 171.5 us, one 69.6 / 112.6).
template <typename VT>
__global__ void __launch_bounds__(kThreads, 8)
    k_crs_long(const int32_t* __restrict__ long_rows, int n_long, int n_cta, int64_t n_rows,
               const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col, const VT* __restrict__ val,
               const double* B, int64_t ldb, double* C, int64_t ldc, int k, int short_row, int prefetch) {
  __shared__ double sh[kThreads];
  constexpr int WARPS = kThreads / 32;
  const int tid = (int)threadIdx.x;
  int64_t blk = blockIdx.x;
  if (blk < n_cta) {
    long_row<VT, kThreads>(__ldg(long_rows + blk), tid, k, row_ptr, col, val, B, ldb, C, ldc, sh);
    return;
  }
  blk -= n_cta;
  const int warp_ctas = (n_long - n_cta + WARPS - 1) / WARPS;
  if (blk < warp_ctas) {
    const int i = n_cta + (int)blk * WARPS + tid / 32;
    if (i < n_long)
      long_row<VT, 32>(__ldg(long_rows + i), tid % 32, k, row_ptr, col, val, B, ldb, C, ldc,
                       sh + (tid & ~31));
    return;
  }
  blk -= warp_ctas;
  const int rpc = kThreads / k;
  if (tid == 0 && prefetch > 0) prefetch_rows((blk + prefetch) * rpc, rpc, n_rows, row_ptr, col, val);
  const int r = tid / k;
  const int64_t g = blk * rpc + r;
  if (r >= rpc || g >= n_rows) return;
  const int rs = __ldg(row_ptr + g), re = __ldg(row_ptr + g + 1);
  grid_wait();
  grid_dependents();
  if (re - rs > short_row) return;
  const double* Bc = B + (tid - r * k);
  double acc = 0.0;
  // four entries in flight, then one by one: large matrices are bound by the FP64 pipe, and a batch
  // padded with masked multiply-adds issues them (3,000,000 rows of 5 entries, k = 3: 127.5 us padded,
  // 94.6 us so)
  int j = rs;
  for (; re - j >= 4; j += 4) {
    double v[4], x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u] = to_f64(ldg(val + j + u));
      x[u] = Bc[(int64_t)ldg(col + j + u) * ldb];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) acc = fma(v[u], x[u], acc);
  }
  for (; j < re; ++j) acc = fma(to_f64(ldg(val + j)), Bc[(int64_t)ldg(col + j) * ldb], acc);
  C[g * ldc + (tid - r * k)] = acc;
}

template <typename VT>
static cudaError_t launch_long(const CsrDev& A, const VT* val, const double* B, int64_t ldb, double* C, int64_t ldc,
                               int k, cudaStream_t s) {
  const LongRows& lr = A.long_rows;
  const int rpc = kThreads / k, warps = kThreads / 32, n_cta = lr.n_cta[k];
  const int64_t grid = n_cta + (lr.n - n_cta + warps - 1) / warps + (A.n_rows + rpc - 1) / rpc;
  return launch_dependent(k_crs_long<VT>, (unsigned)grid, kThreads, s, lr.rows, lr.n, n_cta, A.n_rows, A.row_ptr,
                          A.col, val, B, ldb, C, ldc, k, lr.short_row, A.prefetch);
}

template <typename VT, int L, int K>
static cudaError_t launch_lanes_t(const CsrDev& A, const VT* val, const double* B, int64_t ldb, double* C,
                                  int64_t ldc, int k, cudaStream_t s) {
  const int64_t rows_per_cta = kThreads / L;
  const int64_t grid = (A.n_rows + rows_per_cta - 1) / rows_per_cta;
  // a full block with 16-byte aligned B rows: 16-byte gathers
  if (K >= 2 && k == K && ldb % 2 == 0 && (((uintptr_t)B) & 15) == 0)
    k_crs_lanes<VT, L, K, (K >= 2)><<<(unsigned)grid, kThreads, 0, s>>>(A.n_rows, A.row_ptr, A.col, val, B, ldb, C,
                                                                          ldc, k, A.prefetch);
  else
    k_crs_lanes<VT, L, K, false><<<(unsigned)grid, kThreads, 0, s>>>(A.n_rows, A.row_ptr, A.col, val, B, ldb, C, ldc,
                                                                       k, A.prefetch);
  return cudaGetLastError();
}

template <typename VT, int L>
static cudaError_t lanes_k(const CsrDev& A, const VT* val, const double* B, int64_t ldb, double* C, int64_t ldc, int k,
                           cudaStream_t s) {
  if (A.n_rows == 0) return cudaSuccess;
  if (k <= 1) return launch_lanes_t<VT, L, 1>(A, val, B, ldb, C, ldc, k, s);
  if (k <= 2) return launch_lanes_t<VT, L, 2>(A, val, B, ldb, C, ldc, k, s);
  if (k <= 4) return launch_lanes_t<VT, L, 4>(A, val, B, ldb, C, ldc, k, s);
  if (k <= 8) return launch_lanes_t<VT, L, 8>(A, val, B, ldb, C, ldc, k, s);
  return launch_lanes_t<VT, L, 16>(A, val, B, ldb, C, ldc, k, s);
}

// CRS_L1: the kernel for the plan's rows and the block's width and alignment.
template <typename VT>
static cudaError_t crs_l1(const CsrDev& A, const VT* val, const double* B, int64_t ldb, double* C, int64_t ldc, int k,
                          cudaStream_t s) {
  const int64_t n = A.n_rows;
  if (n == 0) return cudaSuccess;
  const int32_t *rp = A.row_ptr, *col = A.col;
  const int pf = A.prefetch;
  const bool a16 = rows_on_16_bytes(B, ldb, C, ldc);
  if (A.long_rows.n > 0) return launch_long(A, val, B, ldb, C, ldc, k, s);
  const bool even = A.lane_cols == 4;
  if (k == 1) {
    // (not with longer rows: 200,000 rows of 4 or 60 entries 28.8 -> 35.5 us masked, power-law rows of up to 2000
    // 173 -> 211)
    const bool masked = sizeof(VT) == 4 && !even && A.longest <= kShortRowWide;
    if (!masked && A.nnz >= kWideRow * n) return launch_wide<VT, 1>(A, val, B, ldb, C, ldc, s);
    auto* row = masked ? (ldb == 1 ? k_crs_row<VT, true, sizeof(VT) == 4> : k_crs_row<VT, false, sizeof(VT) == 4>)
                       : (ldb == 1 ? k_crs_row<VT, true, false> : k_crs_row<VT, false, false>);
    return launch_dependent(row, (unsigned)((n + kThreads - 1) / kThreads), kThreads, s, n, rp, col, val, B, ldb, C,
                            ldc, pf);
  }
  // (uneven rows: a row's columns on one lane keep its warp waiting for its longest row.  Rows of 10 .. 30 entries,
  // 300,000 of them, k = 2 / 4: 51.8 / 97.2 us on k_crs_wide, 37.6 / 65.3 on k_crs_cols)
  const bool long_average = A.nnz >= kWideRowCols * n;
  if (long_average && even && a16 && k == 2) return launch_wide<VT, 2>(A, val, B, ldb, C, ldc, s);
  if (long_average && even && a16 && k == 4) return launch_wide<VT, 4>(A, val, B, ldb, C, ldc, s);
  // (rows of 16 and more entries: one column per lane rather than 3, 5 or 7; the lanes of a row share its
  // uncoalesced entries.  27-point stencil on 60^3, k = 3 / 5, one / several: 32.5 / 34.8, 51.4 / 54.9 us)
  int w = cols_per_lane(k, a16, n, A.lane_cols, A.lane_cols > 1 && !long_average);
  // Short rows gain by two columns from fewer threads on where they are uneven (100,000 / 300,000 rows of 4 .. 9
  // entries, k = 4 / 2, one -> two columns 13.0 -> 10.6, 18.2 -> 14.1 us; of 0 .. 12 13.0 -> 13.5, 18.2 -> 18.0; 30,000
  // of 0 .. 12, k = 16, 11.2 -> 12.9), and in
  // 8-byte accesses too (1,500,000 rows of 4 .. 9, k = 4, ld = 5 150.4 -> 113.1, of 1 49.0 -> 38.6, 160^3 Poisson
  // 199.5 -> 192.3; 300,000 rows of 8 18.4 -> 20.0).  Not where one long row is walked by its lanes alone (100,000
  // rows of 4 and one of 4000, k = 2: 446 -> 620).
  const bool many = even ? n * (k / 2) >= kMinColThreads : n >= 100000 && A.longest <= kWalkedRow;
  if (w == 1 && k % 2 == 0 && A.lane_cols > 1 && A.nnz < kWideRow * n && many) w = 2;
  switch (w) {
    case 7: return launch_cols<VT, 7>(n, rp, col, val, B, ldb, C, ldc, k, pf, s);
    case 5: return launch_cols<VT, 5>(n, rp, col, val, B, ldb, C, ldc, k, pf, s);
    case 4: return launch_cols<VT, 4>(n, rp, col, val, B, ldb, C, ldc, k, pf, s);
    case 3: return launch_cols<VT, 3>(n, rp, col, val, B, ldb, C, ldc, k, pf, s);
    case 2:
      return a16 ? launch_cols<VT, 2>(n, rp, col, val, B, ldb, C, ldc, k, pf, s)
                 : launch_cols<VT, 2, false>(n, rp, col, val, B, ldb, C, ldc, k, pf, s);
    default: return launch_cols<VT, 1>(n, rp, col, val, B, ldb, C, ldc, k, pf, s);
  }
}

template <typename VT>
static cudaError_t crs_dispatch(const CsrDev& A, int lanes, const VT* val, const double* B, int64_t ldb, double* C,
                                int64_t ldc, int k, cudaStream_t s) {
  switch (lanes) {
    case 1: return crs_l1(A, val, B, ldb, C, ldc, k, s);
    case 2: return lanes_k<VT, 2>(A, val, B, ldb, C, ldc, k, s);
    case 4: return lanes_k<VT, 4>(A, val, B, ldb, C, ldc, k, s);
    case 8: return lanes_k<VT, 8>(A, val, B, ldb, C, ldc, k, s);
    case 16: return lanes_k<VT, 16>(A, val, B, ldb, C, ldc, k, s);
    case 32: return lanes_k<VT, 32>(A, val, B, ldb, C, ldc, k, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_crs_lanes(const CsrDev& A, bool fp32, int lanes, const double* B, int64_t ldb, double* C,
                             int64_t ldc, int k, cudaStream_t s) {
  if (fp32 && A.val32_special) return crs_dispatch<float>(A, lanes, A.val32, B, ldb, C, ldc, k, s);
  if (fp32) return crs_dispatch<f32n>(A, lanes, reinterpret_cast<const f32n*>(A.val32), B, ldb, C, ldc, k, s);
  return crs_dispatch<double>(A, lanes, A.val, B, ldb, C, ldc, k, s);
}

template <typename VT>
static cudaError_t launch_halo_v(const HaloDev& H, const VT* val, const double* B, double* C, cudaStream_t s) {
  if (H.n_rows == 0) return cudaSuccess;
  return launch_dependent(k_crs_halo<VT>, (unsigned)((H.n_rows + kThreads - 1) / kThreads), kThreads, s, H.n_rows,
                          H.rows, H.row_ptr, H.col, val, B, C);
}

cudaError_t launch_halo(const HaloDev& H, bool fp32, const double* B, double* C, cudaStream_t s) {
  if (fp32 && H.val32_special) return launch_halo_v<float>(H, H.val32, B, C, s);
  if (fp32) return launch_halo_v<f32n>(H, reinterpret_cast<const f32n*>(H.val32), B, C, s);
  return launch_halo_v<double>(H, H.val, B, C, s);
}

}  // namespace spmv
