// Device side of the batched product: member table, work items and the
// persistent kernel (shared by the batch API and its allocation-free entry).
#pragma once

#include "device.cuh"

namespace spmv {

struct BatchMat {
  const int32_t* row_ptr;
  const int32_t* col;
  const double* val;
  const double* B;
  double* C;
  int64_t ldb, ldc;
  int64_t n_rows;
};

// Work item.  mode 0: rows [p0, p1) of member `mat`, bounds from row_ptr.
// mode 1: the rows listed at positions [p0, p1) of the (row, first entry)
// list, all of length `len` (the length-binned rows of the adaptive policy).
// mode 2: listed rows of unequal lengths (ends from row_ptr); mode 4 the same, of a member whose
// entries end within a long step of 2^31 - 1 (listed_mode).
// mode 3: chunks [p0, p1) of the length-sorted SELL-32 copy (sorted policy),
// all of length `len`, stored back to back from slot `base`: one lane per row,
// slots column-major inside a chunk.
// L lanes share one row; 32/L rows per warp pass.
struct BatchItem {
  int32_t mat, p0, p1, len;
  int16_t lanes, mode;
  int32_t pad;
  int64_t base;
};

// At k = 2 mode 2 steps by up to 4 entries on each of 32 lanes, counted in 32 bits.
inline int listed_mode(int64_t nnz) { return nnz <= INT32_MAX - 4 * 32 ? 2 : 4; }

// Length-sorted SELL-32 copy of the short rows of the members with the sorted
// policy: chunk c holds 32 rows (row index perm[32c + t], -1 for padding) of
// chunk_len[c] slots each at chunk_ptr[c] + 32 j + t.
struct BatchSell {
  const int64_t* chunk_ptr;
  const int32_t* chunk_len;
  const int32_t* perm;
  const int32_t* col;
  const double* val;
};

// C is written once per product: streaming (evict-first) stores leave L2 to
// the B blocks of the members in flight.
__device__ __forceinline__ void st_c(double* p, double x) { __stcs(p, x); }
__device__ __forceinline__ void st_c(double2* p, double2 x) { __stcs(p, x); }

__device__ __forceinline__ void st_c4(double* p, const double* x) {
  asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(x[0]), "d"(x[1]), "d"(x[2]), "d"(x[3])
               : "memory");
}

// A row of k values in accesses of VEC doubles (1, 2, 4).  VEC > 1: every member's B and C rows start on VEC
// doubles and k is a multiple of VEC.  One lane gathers a whole row, so the accesses are what L1 serves
// one by one (0.73 of its rate at k = 4 in 16 bytes): 512 members, k = 4, 16 -> 32 bytes 491 -> 475 us, 96 members,
// k = 8 235 -> 229 us.  Rows are stored in 32 bytes from K = 16 on (96 members, k = 16: 444 -> 392 us); a row of one
// sector gains nothing (475 -> 479), one of two is mixed (96 members 229 -> 225, 16 members 88 -> 92).
template <int K, int VEC>
__device__ __forceinline__ void gather_row(const double* __restrict__ b, int k, double (&g)[K]) {
#pragma unroll
  for (int q = 0; q < K; q += VEC) {
    if constexpr (VEC == 1) {
      // (a select: behind a branch a column the gathers no longer go out together: 300 members, k = 8, ld = 9 1199
      // us, 1115 so)
      g[q] = q < k ? __ldg(b + q) : 0.0;
    } else if (q >= k) {
#pragma unroll
      for (int u = 0; u < VEC; ++u) g[q + u] = 0.0;
    } else if constexpr (VEC == 4) {
      asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];"
          : "=d"(g[q]), "=d"(g[q + 1]), "=d"(g[q + 2]), "=d"(g[q + 3])
          : "l"(b + q));
    } else {
      const double2 t = __ldg(reinterpret_cast<const double2*>(b + q));
      g[q] = t.x;
      g[q + 1] = t.y;
    }
  }
}

template <int K, int VEC>
__device__ __forceinline__ void store_row(double* out, int k, const double (&acc)[K]) {
  constexpr int SV = VEC == 4 && K < 16 ? 2 : VEC;  // doubles per store
#pragma unroll
  for (int q = 0; q < K; q += SV) {
    if (q >= k) break;
    if constexpr (SV == 4) st_c4(out + q, acc + q);
    if constexpr (SV == 2) st_c(reinterpret_cast<double2*>(out + q), make_double2(acc[q], acc[q + 1]));
    if constexpr (SV == 1) st_c(out + q, acc[q]);
  }
}

// NB entries per lane have their gathers issued before their FMAs.
template <int L, int K, int VEC, int NB = (L == 1 && K <= 2 ? 4 / K : 1)>
__device__ __forceinline__ void batch_rows(const BatchMat* __restrict__ Mp, const int2* __restrict__ rowlist,
                                           const BatchItem& item, int k, int lane) {
  const BatchMat& M = *Mp;  // fields are read where used, not held across the item
  constexpr int RPP = 32 / L;  // rows per warp pass
  const int t = lane % L;
  for (int base = item.p0; base < item.p1; base += RPP) {
    const int i = base + lane / L;
    const bool active = i < item.p1;
    int r = 0, rs = 0, re = 0;
    if (active) {
      if (item.mode) {
        const int2 e = __ldg(rowlist + i);
        r = e.x;
        rs = e.y;
        re = item.mode == 1 ? rs + item.len : __ldg(M.row_ptr + r + 1);
      } else {
        r = i;
        rs = __ldg(M.row_ptr + r);
        re = __ldg(M.row_ptr + r + 1);
      }
    }
    double acc[K];
#pragma unroll
    for (int q = 0; q < K; ++q) acc[q] = 0.0;
    for (int j = rs + t; j < re; j += NB * L) {
      double v[NB];
      const double* b[NB];
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int jj = (j + u * L < re) ? j + u * L : j;
        v[u] = ldcs(M.val + jj);
        b[u] = M.B + (int64_t)ldcs(M.col + jj) * M.ldb;
      }
      double g[NB][K];
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        if (j + u * L < re) {
          gather_row<K, VEC>(b[u], k, g[u]);
        } else {
#pragma unroll
          for (int q = 0; q < K; ++q) g[u][q] = 0.0;
        }
      }
#pragma unroll
      for (int u = 0; u < NB; ++u)
#pragma unroll
        for (int q = 0; q < K; ++q)
          if (j + u * L < re && q < k) acc[q] = fma(v[u], g[u][q], acc[q]);
    }
    if (L > 1) {
#pragma unroll
      for (int q = 0; q < K; ++q) acc[q] = warp_sum_xor(acc[q], L);
    }
    if (active) {
      double* out = M.C + (int64_t)r * M.ldc;
      if constexpr (L == 1) {
        store_row<K, VEC>(out, k, acc);
      } else {
#pragma unroll
        for (int q = 0; q < K; ++q)
          if (q < k && t == q % L) st_c(out + q, acc[q]);
      }
    }
  }
}

// A round is a dependent pair of loads, a round trip to L2 or DRAM.  Long rows of
// the same length class (mode 2, some 32 entries per lane) at K = 2 take four
// entries a round, which costs no occupancy (512 members, k = 2: 355 -> 337 us; 32
// members 46.7 -> 41.6).  Items of unsorted rows keep to one: slots past the end of
// a short row still occupy the FP64 pipe (512 members on 8 lanes per row: 2.77 -> 4.05
// ms).  So does K = 4, where two a round lengthen the launch (499 -> 507 us), and K = 1
// (293 -> 301).
template <int K, int VEC>
__device__ __forceinline__ void batch_row_item(const BatchMat* __restrict__ Mp, const int2* __restrict__ rowlist,
                                               const BatchItem& item, int k, int lane) {
  if constexpr (K == 2) {
    if (item.mode == 2) switch (item.lanes) {
      case 2: batch_rows<2, K, VEC, 4>(Mp, rowlist, item, k, lane); return;
      case 4: batch_rows<4, K, VEC, 4>(Mp, rowlist, item, k, lane); return;
      case 8: batch_rows<8, K, VEC, 4>(Mp, rowlist, item, k, lane); return;
      case 16: batch_rows<16, K, VEC, 4>(Mp, rowlist, item, k, lane); return;
      case 32: batch_rows<32, K, VEC, 4>(Mp, rowlist, item, k, lane); return;
    }
  }
  switch (item.lanes) {
    case 1: batch_rows<1, K, VEC>(Mp, rowlist, item, k, lane); break;
    case 2: batch_rows<2, K, VEC>(Mp, rowlist, item, k, lane); break;
    case 4: batch_rows<4, K, VEC>(Mp, rowlist, item, k, lane); break;
    case 8: batch_rows<8, K, VEC>(Mp, rowlist, item, k, lane); break;
    case 16: batch_rows<16, K, VEC>(Mp, rowlist, item, k, lane); break;
    default: batch_rows<32, K, VEC>(Mp, rowlist, item, k, lane); break;
  }
}

// Chunks whose rows all have exactly LEN entries, CH chunks per step; returns
// the first chunk left for the generic loop.  Same FMA order per row as the
// generic loop.
template <int LEN, int CH, int K, int VEC>
__device__ __forceinline__ int chunks_fixed(const BatchMat* __restrict__ Mp, const double* __restrict__ B,
                                            int64_t ldb, const BatchSell& S, const BatchItem& item, int k,
                                            int lane) {
  int c = item.p0;
  for (; c + CH - 1 < item.p1; c += CH) {
    const int64_t s0 = item.base + (int64_t)(c - item.p0) * 32 * LEN + lane;
    int r[CH];
    double v[CH][LEN];
    const double* b[CH][LEN];
#pragma unroll
    for (int h = 0; h < CH; ++h) {
      r[h] = __ldg(S.perm + (int64_t)(c + h) * 32 + lane);
#pragma unroll
      for (int j = 0; j < LEN; ++j) {
        const int64_t slot = s0 + (int64_t)(h * LEN + j) * 32;
        v[h][j] = ldcs(S.val + slot);
        b[h][j] = B + (int64_t)ldcs(S.col + slot) * ldb;
      }
    }
    double g[CH][LEN][K];
#pragma unroll
    for (int h = 0; h < CH; ++h)
#pragma unroll
      for (int j = 0; j < LEN; ++j) gather_row<K, VEC>(b[h][j], k, g[h][j]);
#pragma unroll
    for (int h = 0; h < CH; ++h) {
      double acc[K];
#pragma unroll
      for (int q = 0; q < K; ++q) acc[q] = 0.0;
#pragma unroll
      for (int j = 0; j < LEN; ++j)
#pragma unroll
        for (int q = 0; q < K; ++q) acc[q] = fma(v[h][j], g[h][j][q], acc[q]);
      if (r[h] < 0) continue;
      double* out = Mp->C + (int64_t)r[h] * Mp->ldc;
      store_row<K, VEC>(out, k, acc);
    }
  }
  return c;
}

template <int K, int VEC>
__device__ __forceinline__ void batch_chunks(const BatchMat* __restrict__ Mp, const BatchSell& S,
                                             const BatchItem& item, int k, int lane) {
  struct {
    const double* B;
    int64_t ldb;
  } M = {Mp->B, Mp->ldb};  // only what the inner loop needs stays in registers
  const int len = item.len;  // every chunk of the item has this length: no per-chunk metadata loads
  int c = item.p0;
  // short rows (most rows of a power-law matrix): a fixed length, several
  // chunks per step, every load and gather of a step in flight together
  if (len == 1) c = chunks_fixed<1, K <= 4 ? 4 : 2, K, VEC>(Mp, M.B, M.ldb, S, item, k, lane);
  else if (len == 2) c = chunks_fixed<2, K <= 4 ? 2 : 1, K, VEC>(Mp, M.B, M.ldb, S, item, k, lane);
  else if (len == 3 && K <= 4) c = chunks_fixed<3, 1, K, VEC>(Mp, M.B, M.ldb, S, item, k, lane);
  else if (len == 4 && K <= 4) c = chunks_fixed<4, 1, K, VEC>(Mp, M.B, M.ldb, S, item, k, lane);
  for (; c < item.p1; ++c) {
    const int64_t base = item.base + (int64_t)(c - item.p0) * 32 * len + lane;
    const int r = __ldg(S.perm + (int64_t)c * 32 + lane);
    double acc[K];
#pragma unroll
    for (int q = 0; q < K; ++q) acc[q] = 0.0;
    // NB slots a step, software-pipelined: the next step's values and columns are in flight while this
    // step's gathers are, so only the gathers stay on the critical path.  512 members, against four / two slots
    // without the pipeline at k = 1 / 2 and one slot with it at k = 4: 287 -> 281, 334 -> 330, 476 -> 468 us.
    constexpr int NB = K == 1 ? 4 : K <= 4 ? 2 : 1;
    double v[NB];
    int32_t cc[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      v[u] = u < len ? ldcs(S.val + base + u * 32) : 0.0;
      cc[u] = u < len ? ldcs(S.col + base + u * 32) : 0;
    }
    int j = 0;
    for (; j + NB <= len; j += NB) {
      double g[NB][K], vn[NB];
      int32_t cn[NB];
#pragma unroll
      for (int u = 0; u < NB; ++u) gather_row<K, VEC>(M.B + (int64_t)cc[u] * M.ldb, k, g[u]);
#pragma unroll
      for (int u = 0; u < NB; ++u) {
        const int64_t nxt = base + (int64_t)(j + NB + u < len ? j + NB + u : j) * 32;
        vn[u] = ldcs(S.val + nxt);
        cn[u] = ldcs(S.col + nxt);
      }
#pragma unroll
      for (int u = 0; u < NB; ++u)
#pragma unroll
        for (int q = 0; q < K; ++q)
          if (q < k) acc[q] = fma(v[u], g[u][q], acc[q]);
#pragma unroll
      for (int u = 0; u < NB; ++u) v[u] = vn[u], cc[u] = cn[u];
    }
#pragma unroll
    for (int u = 0; u < NB - 1; ++u)
      if (j + u < len) {
        double g[K];
        gather_row<K, VEC>(M.B + (int64_t)cc[u] * M.ldb, k, g);
#pragma unroll
        for (int q = 0; q < K; ++q)
          if (q < k) acc[q] = fma(v[u], g[q], acc[q]);
      }
    if (r >= 0) {
      double* out = Mp->C + (int64_t)r * Mp->ldc;
      store_row<K, VEC>(out, k, acc);
    }
  }
}

// Threads per CTA of the persistent kernels, and the CTAs per SM the register
// budget is sized for: for k <= 4 at 72 registers seven 128-thread CTAs (28
// warps) stay resident (256-thread CTAs held to 64 registers spilled, and only
// three of them fitted on an SM, not four: 24 warps); the wider gathers of
// k = 8 / 16 keep about 100 registers (four or five CTAs) rather than spill.
constexpr int kBatchThreads = 128;
constexpr int kBatchCtasPerSm = 7;
template <int K>
struct BatchMinCtas {
  static constexpr int value = K <= 4 ? kBatchCtasPerSm : 4;
};

// Persistent kernel: warps take items round-robin (dynamic = 0) or from the
// atomic counter (dynamic = 1, counter zeroed before the launch).
// Next item index of the calling warp: round-robin or from the atomic counter.
__device__ __forceinline__ int next_item(int it, int nw, int dynamic, int* counter, int lane) {
  if (!dynamic) return it + nw;
  int v = 0;
  if (lane == 0) v = atomicAdd(counter, 1);
  return __shfl_sync(0xffffffffu, v, 0);
}

// Persistent kernel over row items (modes 0-2).
template <int K, int VEC>
__global__ void __launch_bounds__(kBatchThreads, BatchMinCtas<K>::value)
    k_batch_rows(const BatchMat* __restrict__ mats, const BatchItem* __restrict__ items, int n_items,
                 const int2* __restrict__ rowlist, int* __restrict__ counter, int dynamic, int k) {
  const int lane = threadIdx.x & 31;
  const int wid = blockIdx.x * (kBatchThreads / 32) + (threadIdx.x >> 5);
  const int nw = gridDim.x * (kBatchThreads / 32);
  int it = dynamic ? next_item(0, nw, 1, counter, lane) : wid;
  while (it < n_items) {
    const BatchItem item = items[it];
    batch_row_item<K, VEC>(mats + item.mat, rowlist, item, k, lane);
    it = next_item(it, nw, dynamic, counter, lane);
  }
}

// Persistent kernel over all item modes.  Sorted-chunk items and row items of
// one member stay next to each other in the list, so a member's B block is
// gathered while it is resident in L2 (two separate kernels, one per mode,
// would stream every B block twice).
template <int K, int VEC>
__global__ void __launch_bounds__(kBatchThreads, BatchMinCtas<K>::value)
    k_batch(const BatchMat* __restrict__ mats, const BatchItem* __restrict__ items, int n_items,
            const int2* __restrict__ rowlist, BatchSell sell, int* __restrict__ counter, int dynamic, int k) {
  const int lane = threadIdx.x & 31;
  const int wid = blockIdx.x * (kBatchThreads / 32) + (threadIdx.x >> 5);
  const int nw = gridDim.x * (kBatchThreads / 32);
  int it = dynamic ? next_item(0, nw, 1, counter, lane) : wid;
  while (it < n_items) {
    const BatchItem item = items[it];
    if (item.mode == 3)
      batch_chunks<K, VEC>(mats + item.mat, sell, item, k, lane);
    else
      batch_row_item<K, VEC>(mats + item.mat, rowlist, item, k, lane);
    it = next_item(it, nw, dynamic, counter, lane);
  }
}

template <int VEC>
static const void* batch_rows_kernel_t(int k) {
  if constexpr (VEC == 1) {
    if (k == 1) return (const void*)k_batch_rows<1, 1>;
    if (k == 3) return (const void*)k_batch_rows<3, 1>;
  }
  if constexpr (VEC <= 2)
    if (k <= 2) return (const void*)k_batch_rows<2, VEC>;
  if (k <= 4) return (const void*)k_batch_rows<4, VEC>;
  if (k <= 8) return (const void*)k_batch_rows<8, VEC>;
  return (const void*)k_batch_rows<16, VEC>;
}

template <int VEC>
static const void* batch_kernel_t(int k) {
  if constexpr (VEC == 1) {
    if (k == 1) return (const void*)k_batch<1, 1>;
    if (k == 3) return (const void*)k_batch<3, 1>;  // (as four columns, one masked: 603.6 us for 512 members, 562.1 so)
  }
  if constexpr (VEC <= 2)
    if (k <= 2) return (const void*)k_batch<2, VEC>;
  if (k <= 4) return (const void*)k_batch<4, VEC>;
  if (k <= 8) return (const void*)k_batch<8, VEC>;
  return (const void*)k_batch<16, VEC>;
}

// The kernels for k right-hand sides in accesses of vec doubles.  The rows-only
// variant serves work lists without sorted chunks.
static inline const void* batch_rows_kernel(int k, int vec) {
  return vec == 4 ? batch_rows_kernel_t<4>(k) : vec == 2 ? batch_rows_kernel_t<2>(k) : batch_rows_kernel_t<1>(k);
}
static inline const void* batch_kernel(int k, int vec) {
  return vec == 4 ? batch_kernel_t<4>(k) : vec == 2 ? batch_kernel_t<2>(k) : batch_kernel_t<1>(k);
}

// Doubles per access (at most `most`) that k columns of a member with these operands allow.
static inline int batch_access(int most, int k, const double* B, int64_t ldb, const double* C, int64_t ldc) {
  while (most > 1 && (k % most || ldb % most || ldc % most || ((uintptr_t)B | (uintptr_t)C) % (8 * most))) most /= 2;
  return most;
}

}  // namespace spmv
