// SELL-C-sigma product, C = 32 (Kreutzer et al. 2014 format; the paper's CRS
// loop of Sec. 1.2 applied to the sliced, sorted, column-major form).
//
// One warp per chunk, one lane per sorted row: slot j of lane t lives at
// chunk_ptr[c] + 32*j + t, so each load instruction of a warp reads 32
// consecutive entries (256 B of FP64 values, 128 B of indices).  Every lane
// runs chunk_len[c] steps; padding slots hold +0.0 and a valid column, so they
// add exactly +0.0 and need no test.  The row sum goes to C[perm[r]].  Sorting
// rows by length inside sigma-windows keeps the padding (idle FP64 issue
// slots) small.
//
// A block of k >= 2 columns runs k_sell_cols: each sorted row is shared by
// G = k / W lanes with W columns each (sell_cols), and the G lanes of a row
// read one contiguous piece of its B row; a row's slots are still summed in
// order, so every W gives the same bits.  Here a lane stops at its row's own
// length (from the CRS row_ptr): a warp's rows are fewer than a chunk's, and the
// padding that they leave out is FP64 work, which bounds these products (600,011-row
// eigenproblem matrix, k = 6: 106.3 -> 96.7 us, now 93.9, FP64 floor 79).  One vector is bound by
// the SMs' requests to L2 on scattered matrices (2,000,003 rows: 92.3 us, request
// floor 73); there the two dependent loads in front of each row cost more than
// its padding (99.9 us).
#include "device.cuh"
#include "internal.h"

namespace spmv {

// Bring the slots of chunks [c0, c0 + chunks) into L2 (one thread; chunk
// offsets are multiples of 32 slots, so the ranges are 16-byte aligned).
template <typename VT>
__device__ __forceinline__ void prefetch_chunks(int64_t c0, int64_t chunks, int64_t n_chunks,
                                                const int64_t* __restrict__ chunk_ptr,
                                                const int32_t* __restrict__ col, const VT* __restrict__ val) {
  if (c0 >= n_chunks) return;
  const int64_t c1 = c0 + chunks < n_chunks ? c0 + chunks : n_chunks;
  const int64_t s0 = __ldg(chunk_ptr + c0), s1 = __ldg(chunk_ptr + c1);
  if (s1 > s0) {
    prefetch_l2(val + s0, (uint32_t)((s1 - s0) * (int64_t)sizeof(VT)));
    prefetch_l2(col + s0, (uint32_t)((s1 - s0) * 4));
  }
}

template <typename VT>
__global__ void __launch_bounds__(kThreads)
    k_sell(int64_t n_rows, int64_t n_chunks, const int32_t* __restrict__ perm,
           const int64_t* __restrict__ chunk_ptr, const int32_t* __restrict__ chunk_len,
           const int32_t* __restrict__ col, const VT* __restrict__ val, const double* B,
           int64_t ldb, double* C, int64_t ldc, int prefetch) {
  constexpr int CPC = kThreads / kSellC;  // chunks per CTA
  // bring the slots of the CTA `prefetch` positions ahead into L2
  if (threadIdx.x == 0 && prefetch > 0)
    prefetch_chunks(((int64_t)blockIdx.x + prefetch) * CPC, CPC, n_chunks, chunk_ptr, col, val);
  const int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  const int64_t c = r >> 5;
  if (c >= n_chunks) return;
  const int t = threadIdx.x & 31;
  const int len = __ldg(chunk_len + c);
  const int64_t base = __ldg(chunk_ptr + c) + t;
  grid_wait();
  double acc = 0.0;
  // batches of NB slots, software-pipelined: all gathers of a batch are issued before its FMAs, and behind
  // them the next batch's values and columns (len is the warp's, so the last slots take a branch, not
  // masked multiply-adds).  Without and with the pipeline: eigenproblem matrices of 400,009 / 2,000,003 rows
  // 23.9 -> 22.8, 93.3 -> 92.3 us; 130^3 Poisson 40.4 -> 36.3 (FP32 values 35.0 -> 29.7; HBM floor 33 and 24).
  constexpr int NB = 2;
  VT v[NB];
  int32_t cc[NB];
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    v[u] = VT();
    cc[u] = 0;
    if (u < len) {
      v[u] = ldcs(val + base + u * kSellC);
      cc[u] = ldcs(col + base + u * kSellC);
    }
  }
  int j = 0;
  for (; j + NB <= len; j += NB) {
    double g[NB];
    VT vn[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) g[u] = B[(int64_t)cc[u] * ldb];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int64_t nxt = base + (int64_t)(j + NB + u < len ? j + NB + u : j) * kSellC;
      vn[u] = ldcs(val + nxt);
      cc[u] = ldcs(col + nxt);
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) acc = fma(to_f64(v[u]), g[u], acc);
#pragma unroll
    for (int u = 0; u < NB; ++u) v[u] = vn[u];
  }
#pragma unroll
  for (int u = 0; u < NB - 1; ++u)
    if (j + u < len) acc = fma(to_f64(v[u]), B[(int64_t)cc[u] * ldb], acc);
  grid_dependents();
  if (r >= n_rows) return;
  C[(int64_t)__ldg(perm + r) * ldc] = acc;
}

// Slots of a lane's step in k_sell_cols, whose values and columns are loaded behind the gathers of the step
// before (0: no such pipeline).  Means over rows of 1 .. 200 entries, 20,000 .. 2,000,000 of them, in units
// of the fastest of 0 / 1 / 2 slots: doubles one column 1.06 / 1.02 / 1.03, two in 16 bytes 1.03 / 1.03 / 1.02
// (eigenproblem matrices of 600,011 and 2,000,003 rows, k = 6, 94.8 / 93.8 / 95.1 and 300 / 297 / 300 us), two, three
// and four in 8 bytes 1.05 / 1.02 / 1.01, four in 16 bytes 1.02 / 1.01 / 1.04, five and seven 1.04 / 1.01 / 1.04;
// floats one column 1.02 / 1.09 / 1.10, two 1.03 / 1.05 / 1.01, three and four 1.03 / 1.02 / 1.02.
// Two columns where a long row bounds the product (LONG, kWalkedRow): unrolled slots without the pipeline, 200,000
// power-law rows of up to 2000, k = 2 / 4 561 -> 523, 575 -> 525 us (FP32 values, k = 2, 456 -> 400).
template <typename VT, int W, bool A16, bool LONG>
constexpr int kSellStep = LONG ? 0
                          : sizeof(VT) == 4 ? (W == 1 ? 0 : W == 2 ? 2 : 1) : (!A16 && W >= 2 && W <= 4 ? 2 : 1);

// k columns of a sorted row on G = k / W lanes, W columns each (as k_crs_cols).
template <typename VT, int W, bool A16, bool LONG>
__global__ void __launch_bounds__(kThreads, (W == 1 ? 8 : 6))
    k_sell_cols(int64_t n_rows, int64_t n_chunks, const int32_t* __restrict__ perm, const int32_t* __restrict__ row_ptr,
                const int64_t* __restrict__ chunk_ptr, const int32_t* __restrict__ chunk_len,
                const int32_t* __restrict__ col, const VT* __restrict__ val, const double* B,
                int64_t ldb, double* C, int64_t ldc, int G, int prefetch) {
  const int rpc = kThreads / G;  // sorted rows per CTA
  if (threadIdx.x == 0 && prefetch > 0) {
    // the chunks that start in the rows of the CTA `prefetch` positions ahead
    const int64_t f0 = (((int64_t)blockIdx.x + prefetch) * rpc + kSellC - 1) / kSellC;
    const int64_t f1 = (((int64_t)blockIdx.x + prefetch + 1) * rpc + kSellC - 1) / kSellC;
    if (f1 > f0) prefetch_chunks(f0, f1 - f0, n_chunks, chunk_ptr, col, val);
  }
  const int rl = (int)threadIdx.x / G;
  const int64_t r = (int64_t)blockIdx.x * rpc + rl;  // sorted row
  if (rl >= rpc || r >= n_rows) return;
  const int64_t c = r >> 5;
  const int c0 = ((int)threadIdx.x - rl * G) * W;  // first column of this lane
  const int row = __ldg(perm + r);
  const int len = __ldg(row_ptr + row + 1) - __ldg(row_ptr + row);
  const int64_t base = __ldg(chunk_ptr + c) + (r & (kSellC - 1));
  grid_wait();
  double acc[W];
#pragma unroll
  for (int q = 0; q < W; ++q) acc[q] = 0.0;
  const double* Bc = B + c0;
  const VT* vp = val + base;  // (advanced slot by slot: 32 slots of a row of 2^26 entries are out of 32 bits)
  const int32_t* cp = col + base;
  constexpr int NB = kSellStep<VT, W, A16, LONG>;
  if constexpr (NB == 2) {
    VT v[NB];
    int32_t cc[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      v[u] = VT();
      cc[u] = 0;
      if (u < len) {
        v[u] = ldcs(vp + u * kSellC);
        cc[u] = ldcs(cp + u * kSellC);
      }
    }
    int j = 0;
    for (; j + NB <= len; j += NB) {
      double g[NB][W];
      VT vn[NB];
#pragma unroll
      for (int u = 0; u < NB; ++u) load_cols<W, A16>(Bc + (int64_t)cc[u] * ldb, g[u]);
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int64_t nxt = (int64_t)(j + NB + u < len ? j + NB + u : j) * kSellC;
        vn[u] = ldcs(vp + nxt);
        cc[u] = ldcs(cp + nxt);
      }
#pragma unroll
      for (int u = 0; u < NB; ++u)
#pragma unroll
        for (int q = 0; q < W; ++q) acc[q] = fma(to_f64(v[u]), g[u][q], acc[q]);
#pragma unroll
      for (int u = 0; u < NB; ++u) v[u] = vn[u];
    }
#pragma unroll
    for (int u = 0; u < NB - 1; ++u)
      if (j + u < len) {
        double g[W];
        load_cols<W, A16>(Bc + (int64_t)cc[u] * ldb, g);
#pragma unroll
        for (int q = 0; q < W; ++q) acc[q] = fma(to_f64(v[u]), g[q], acc[q]);
      }
  } else if constexpr (NB == 1) {
    double g[W];
    if (len > 0) {
      VT v = ldcs(vp);
      int32_t c = ldcs(cp);
#pragma unroll 4
      for (int j = 1; j < len; ++j) {
        load_cols<W, A16>(Bc + (int64_t)c * ldb, g);
        vp += kSellC;
        cp += kSellC;
        const VT vn = ldcs(vp);
        c = ldcs(cp);
#pragma unroll
        for (int q = 0; q < W; ++q) acc[q] = fma(to_f64(v), g[q], acc[q]);
        v = vn;
      }
      load_cols<W, A16>(Bc + (int64_t)c * ldb, g);
#pragma unroll
      for (int q = 0; q < W; ++q) acc[q] = fma(to_f64(v), g[q], acc[q]);
    }
  } else {
    double g[W];
#pragma unroll 4
    for (int j = 0; j < len; ++j) {
      const double v = to_f64(ldcs(vp));
      load_cols<W, A16>(Bc + (int64_t)ldcs(cp) * ldb, g);
      vp += kSellC;
      cp += kSellC;
#pragma unroll
      for (int q = 0; q < W; ++q) acc[q] = fma(v, g[q], acc[q]);
    }
  }
  grid_dependents();
  store_cols<W, A16>(C + (int64_t)row * ldc + c0, acc);
}

template <typename VT, int W, bool A16 = (W % 2 == 0), bool LONG = false>
static cudaError_t launch_cols(const SellDev& S, const VT* val, const double* B, int64_t ldb, double* C, int64_t ldc,
                               int k, cudaStream_t s) {
  const int G = k / W, rpc = kThreads / G;
  const int64_t grid = (S.n_rows + rpc - 1) / rpc;
  return launch_dependent(k_sell_cols<VT, W, A16, LONG>, (unsigned)grid, kThreads, s, S.n_rows, S.n_chunks, S.perm,
                          S.row_ptr, S.chunk_ptr, S.chunk_len, S.col, val, B, ldb, C, ldc, G, S.prefetch);
}

// Columns per lane of a block product.  Several read a row's slots and its B rows in fewer, longer accesses, as
// long as the threads still fill the GPU.
static int sell_cols(const SellDev& S, int k, bool a16) {
  const int64_t n = S.n_rows;
  // Four for many short rows (in an uneven chunk the padding is idle FP64 time, more of it the more rows a warp
  // holds).  Two -> four columns, k = 16: 1,500,000 rows of 2 / 5 / 8 entries 168 -> 121, 271 -> 205, 341 -> 319 us,
  // 300,000 rows of 3 34.6 -> 27.2, of 13 106.6 -> 106.6; eigenproblem matrix of 600,011 rows (12.8 a row), k = 8,
  // 120.4 -> 126.2; of 60,000 rows, one -> four, 15.3 -> 19.8.
  // (1,000,000 power-law rows of up to 2000, k = 4 679 -> 1079.)
  if (k % 4 == 0 && n * (k / 4) >= 1000000 && S.slots <= 9 * n && S.longest <= kWalkedRow) return 4;
  // Two: k = 2 from 100,000 rows on or in long rows (one -> two columns: 20,000 rows of 48 / 200 entries 21.9 -> 15.4,
  // 57.8 -> 43.6 us, 200,000 rows of 4 or 60 39.9 -> 32.8, eigenproblem matrices of 60,000 / 150,000 rows 9.3 -> 9.4,
  // 16.6 -> 15.0, 300^2 Laplacian 4.0 -> 4.7), other k from as many threads on as k_crs_cols (k = 8, 60,000 / 150,000
  // rows 15.3 -> 17.8, 33.4 -> 34.2).
  const bool wide2 = k == 2 ? n >= 100000 || S.slots >= 24 * n : n * (k / 2) >= kMinColThreads;
  if (a16 && k % 2 == 0 && wide2) return 2;
  // 8-byte accesses.  One -> two columns: 1,500,000 rows, k = 2, of 1 / 2 / 3 / 5 / 8 entries 23.2 -> 19.9, 32.5 ->
  // 30.4, 37.2 -> 36.3, 44.1 -> 50.0, 63.2 -> 70.9 us, k = 4, of 8 entries 118 -> 94; unsorted rows of 4 or 60, k = 16,
  // 180 -> 208.
  if (!(a16 && k % 2 == 0))
    for (int w : {7, 5, 3})
      if (k % w == 0 && n * (k / w) >= kMinColThreads) return w;
  if (!a16 && k % 2 == 0 && n * (k / 2) >= kMinColThreads && (k > 2 || S.slots <= 3 * n) &&
      (double)S.nnz >= kAutoSellFill * (double)S.slots)
    return 2;
  return 1;
}

template <typename VT>
static cudaError_t sell_k(const SellDev& S, const VT* val, const double* B, int64_t ldb, double* C, int64_t ldc,
                          int k, cudaStream_t s) {
  if (S.n_chunks == 0) return cudaSuccess;
  if (k > 1) {
    const bool a16 = rows_on_16_bytes(B, ldb, C, ldc);
    switch (sell_cols(S, k, a16)) {
      case 7: return launch_cols<VT, 7>(S, val, B, ldb, C, ldc, k, s);
      case 5: return launch_cols<VT, 5>(S, val, B, ldb, C, ldc, k, s);
      case 4:
        return a16 ? launch_cols<VT, 4>(S, val, B, ldb, C, ldc, k, s)
                   : launch_cols<VT, 4, false>(S, val, B, ldb, C, ldc, k, s);
      case 3: return launch_cols<VT, 3>(S, val, B, ldb, C, ldc, k, s);
      case 2:
        if (S.longest > kWalkedRow)
          return a16 ? launch_cols<VT, 2, true, true>(S, val, B, ldb, C, ldc, k, s)
                     : launch_cols<VT, 2, false, true>(S, val, B, ldb, C, ldc, k, s);
        return a16 ? launch_cols<VT, 2>(S, val, B, ldb, C, ldc, k, s)
                   : launch_cols<VT, 2, false>(S, val, B, ldb, C, ldc, k, s);
      default: return launch_cols<VT, 1>(S, val, B, ldb, C, ldc, k, s);
    }
  }
  const int64_t grid = (S.n_chunks * kSellC + kThreads - 1) / kThreads;
  return launch_dependent(k_sell<VT>, (unsigned)grid, kThreads, s, S.n_rows, S.n_chunks, S.perm, S.chunk_ptr,
                          S.chunk_len, S.col, val, B, ldb, C, ldc, S.prefetch);
}

cudaError_t launch_sell(const SellDev& S, bool fp32, const double* B, int64_t ldb, double* C, int64_t ldc, int k,
                        cudaStream_t s) {
  if (fp32 && S.val32_special) return sell_k<float>(S, S.val32, B, ldb, C, ldc, k, s);
  if (fp32) return sell_k<f32n>(S, reinterpret_cast<const f32n*>(S.val32), B, ldb, C, ldc, k, s);
  return sell_k<double>(S, S.val, B, ldb, C, ldc, k, s);
}

}  // namespace spmv
