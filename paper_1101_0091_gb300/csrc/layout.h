// Layout shared by the kernels and the host code: device status codes, the
// bounded-wait limit, launch constants and the device views of the formats.
#pragma once

#include <stdint.h>

namespace spmv {

// Device status word codes written by kernels (0 = fine).
enum : int { DEV_OK = 0, DEV_WAIT_TIMEOUT = 1 };

// Bounded device waits give up after this many nanoseconds of %globaltimer.
constexpr unsigned long long kWaitLimitNs = 1000000000ull;

// ------------------------------------------------------- layout constants
constexpr int kThreads = 256;        // threads per CTA of the row kernels
constexpr int kStagedRows = 256;     // rows per CRS_STAGED block (one per thread)
constexpr int kLongRow = 64;         // rows longer than this are handled warp-per-row
constexpr int kWarpRowsPerBlock = kThreads / 32;
constexpr int kSellC = 32;           // SELL chunk height
constexpr uint32_t kBlockWarpFlag = 0x80000000u;  // high bit of a row-block entry: warp-per-row block

// Rows of more than short_row entries, longest first, for the kernel that gives them a warp or a CTA
// each: n_cta[k] of the n rows take a CTA.  The other rows take a lane (per column), four entries a round
// of dependent loads, so short_row is kShortRow, or kShortRowWide where too many rows exceed that
// (kAutoOverShare, internal.h; power-law rows of up to 2000 entries, 200,000 / 1,000,000 of them, k = 1, short_row 32 /
// 16 / 12 / 8: 13.2 / 11.2 / 10.3 / 10.9 and 43.2 / 40.0 / 40.0 / 45.8 us).  With k right-hand sides a warp
// has 32 / k lanes per column, so while they are few a row takes a CTA from more than kCtaRow +
// kWarpRow / k entries on (200,000 power-law rows of up to 500 entries, k = 8 / 16: 27.4 -> 23.1, 47.1 ->
// 32.1 us against a warp up to 512 entries); kManyLongRows keep the GPU busy by themselves, and warps waste
// less on their sums (40,000 rows of 200 entries, k = 4: 207.7 us on CTAs, 92 on warps).
constexpr int kShortRow = 12;
constexpr int kShortRowWide = 32;
constexpr int kCtaRow = 32;
constexpr int kWarpRow = 512;
constexpr size_t kManyLongRows = 16384;
constexpr int kMaxK = 16;
struct LongRows {
  const int32_t* rows = nullptr;
  int n = 0, short_row = 0, n_cta[kMaxK + 1] = {};
};

// Products of matrices with a longer row than this are bound by the thread that walks it, where a row has one.
constexpr int kWalkedRow = 64;

// CRS_L1 reads the rows in aligned groups of four entries from this many entries per row on average
// (kWideRowCols for blocks of two or four columns).
constexpr int64_t kWideRow = 8;
constexpr int64_t kWideRowCols = 16;

// Device view of one CRS matrix (values in FP64 and, optionally, FP32).
struct CsrDev {
  int64_t n_rows = 0, n_cols = 0, nnz = 0;
  const int32_t* row_ptr = nullptr;
  const int32_t* col = nullptr;     // padded to a multiple of 4 entries + 4
  const double* val = nullptr;      // padded to a multiple of 4 entries + 4
  const float* val32 = nullptr;     // padded to a multiple of 4 entries + 4
  const uint32_t* blk = nullptr;    // row blocks of CRS_STAGED (n_blk + 1 entries)
  int64_t n_blk = 0;
  int tile = 0;                     // nonzero capacity of a CRS_STAGED tile
  int prefetch = 0;                 // CTAs ahead whose val/col slices are prefetched into L2 (0 = off)
  bool val32_special = false;       // val32 holds a subnormal, infinite or NaN float
  int lane_cols = 4;                // most columns of a block that a lane of CRS_L1 takes (see upload_csr)
  int32_t longest = 0;              // entries of the longest row
  LongRows long_rows;               // listed (n > 0) when AUTO splits the long rows off CRS_L1
};

struct SellDev {
  int64_t n_rows = 0, n_chunks = 0, slots = 0, nnz = 0;
  int sigma = 0;
  int32_t longest = 0;              // slots per row of the longest chunk
  const int32_t* perm = nullptr;
  const int32_t* row_ptr = nullptr;  // of the CRS matrix (row lengths)
  const int64_t* chunk_ptr = nullptr;
  const int32_t* chunk_len = nullptr;
  const int32_t* col = nullptr;
  const double* val = nullptr;
  const float* val32 = nullptr;
  int prefetch = 0;                 // CTAs ahead whose slots are prefetched into L2 (0 = off)
  bool val32_special = false;
};

// Stored triangle of SPMV_SYM.
struct SymDev {
  int64_t n_rows = 0, nnz = 0;
  const int32_t* row_ptr = nullptr;
  const int32_t* col = nullptr;     // padded like CsrDev::col
  const double* val = nullptr;
  const float* val32 = nullptr;
  int prefetch = 0;
  bool val32_special = false;
};

// Halo part of a split: rows listed in `rows`, CRS over them.
struct HaloDev {
  int64_t n_rows = 0, nnz = 0;
  const int32_t* rows = nullptr;
  const int32_t* row_ptr = nullptr;
  const int32_t* col = nullptr;
  const double* val = nullptr;
  const float* val32 = nullptr;
  bool val32_special = false;
};

}  // namespace spmv
