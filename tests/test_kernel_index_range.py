"""Kernels whose entries or slots reach the end of the range that a plan accepts (nnz up to 2^31 - 1): the
kernels' own source, compiled for the host with CUDA's built-ins stubbed, walks arrays of untouched memory
mappings (which hold zeros and cost nothing) with a few entries written where a row ends.  An index that
wraps leaves the mapping, and the child process dies."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1101_0091_gb300", "csrc")

# What the kernels use of device.cuh and of CUDA; a thread of a CTA is a host thread where the CTA synchronises.
SHIM = r"""
#pragma once
#include <cuda_runtime.h>
#include <sys/mman.h>
#include <barrier>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <thread>
#include <vector>
#include "layout.h"
#undef __shared__
#define __shared__ static
#undef __launch_bounds__
#define __launch_bounds__(...)
#undef __device__
#define __device__
#undef __global__
#define __global__
#undef __forceinline__
#define __forceinline__ inline
static thread_local dim3 threadIdx;
static dim3 blockIdx(0), gridDim(1);
static std::barrier<>*cta_barrier, *warp_barrier;
template <typename T> T __ldg(const T* p) { return *p; }
template <typename T> void __stcs(T* p, T x) { *p = x; }
static inline unsigned __activemask() { return 1; }
static inline int __any_sync(unsigned, int x) { return x; }
static inline int atomicAdd(int* p, int x) { return *p += x; }
static inline int __shfl_sync(unsigned, int x, int) { return x; }
static inline int __clz(int x) { return __builtin_clz(x); }
static inline void __syncwarp() { warp_barrier->arrive_and_wait(); }
static inline void __syncthreads() { cta_barrier->arrive_and_wait(); }
namespace spmv {
struct f32n { float v; };
constexpr unsigned kOneWave = 1216;
inline void prefetch_l2(const void*, uint32_t) {}
inline void grid_wait() {}
inline void grid_dependents() {}
inline double to_f64(double v) { return v; }
inline double to_f64(float v) { return v; }
inline double to_f64(f32n v) { return v.v; }
template <typename T> T ldg(const T* p) { return *p; }
template <typename T> T ldcs(const T* p) { return *p; }
template <typename T> void ldg4(const T* p, T (&x)[4]) { for (int i = 0; i < 4; ++i) x[i] = p[i]; }
template <int W, bool = false> void load_cols(const double* b, double (&g)[W]) { for (int q = 0; q < W; ++q) g[q] = b[q]; }
template <int W, bool = false> void store_cols(double* c, const double (&a)[W]) { for (int q = 0; q < W; ++q) c[q] = a[q]; }
inline double warp_sum_xor(double x, int) { return x; }
inline bool rows_on_16_bytes(const double*, int64_t, const double*, int64_t) { return true; }
inline int cols_per_lane(int, bool, int64_t, int, bool) { return 1; }
}  // namespace spmv
template <typename T> T* mapped(int64_t n) {  // n zeros behind an inaccessible 64 GiB and before another
  const size_t guard = size_t(64) << 30, bytes = (sizeof(T) * (size_t)n + 65535) / 65536 * 65536;
  char* p = (char*)mmap(nullptr, guard + bytes + guard, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (p == MAP_FAILED || mprotect(p + guard, bytes, PROT_READ | PROT_WRITE)) { perror("mmap"); exit(77); }
  return (T*)(p + guard);
}
// threads [t0, t1) of one CTA, one after another, or (sync) as host threads with barriers
template <typename F> void cta(int t0, int t1, bool sync, F f) {
  if (!sync) {
    for (int t = t0; t < t1; ++t) { threadIdx = dim3(t); f(); }
    return;
  }
  std::barrier<> all(t1 - t0);
  cta_barrier = warp_barrier = &all;
  std::vector<std::thread> ts;
  for (int t = t0; t < t1; ++t) ts.emplace_back([=] { threadIdx = dim3(t); f(); });
  for (auto& t : ts) t.join();
}
#define CHECK(x, want) if ((x) != (want)) { printf("line %d: %g instead of %g\n", __LINE__, (double)(x), (double)(want)); return 1; }
"""

# Chunk of 32 rows, the first of 2^26 + 5 entries: its slots lie up to 2^31 + 160 behind one another.
SELL = r"""
template <int W> static int run(const double* val, const int32_t* col, int64_t* chunk_ptr, int32_t* chunk_len, int len) {
  static int32_t perm[32], row_ptr[33];
  for (int i = 0; i < 33; ++i) row_ptr[i] = i ? len : 0;
  static double B[2 * 8], C[32 * 8];
  const int k = W == 1 ? 2 : W;
  for (int i = 0; i < 16; ++i) B[i] = i < k ? 1 : 100 + i;
  cta(0, 1, false, [&] {
    spmv::k_sell_cols<double, W, W % 2 == 0, false>(32, 1, perm, row_ptr, chunk_ptr, chunk_len, col, val, B, k, C, k, k / W, 0);
  });
  for (int q = 0; q < W; ++q) CHECK(C[q], 3.0 + 2 * B[k + q]);
  return 0;
}
int main() {
  const int len = (1 << 26) + 5;
  double* val = mapped<double>(32ll * len);
  int32_t* col = mapped<int32_t>(32ll * len);
  val[0] = 3;
  val[32ll * (len - 1)] = 2;
  col[32ll * (len - 1)] = 1;
  static int64_t chunk_ptr[2] = {0, 32ll * len};
  static int32_t chunk_len[1] = {len};
  if (run<1>(val, col, chunk_ptr, chunk_len, len) || run<2>(val, col, chunk_ptr, chunk_len, len) ||
      run<3>(val, col, chunk_ptr, chunk_len, len))
    return 1;
  static int32_t perm[32];
  static double B[2] = {1, 7}, C[32];
  cta(0, 1, false, [&] { spmv::k_sell<double>(1, 1, perm, chunk_ptr, chunk_len, col, val, B, 1, C, 1, 0); });
  CHECK(C[0], 3.0 + 2 * 7);
  return 0;
}
"""

# Rows that end at 2^31 - 1, the largest nnz of a plan.
LANES = r"""
static const double* val;
static const int32_t* col;
static const int last = INT_MAX;
template <typename F> static int row(int len, int ldb, int k, int threads, bool sync, F f) {
  int32_t row_ptr[2] = {last - len, last};
  static double B[2 * 4], C[4];
  for (int i = 0; i < 8; ++i) B[i] = i < ldb ? 0 : 100 + i;
  for (double& c : C) c = 0;
  cta(0, threads, sync, [&] { f(row_ptr, B, C); });
  const int n = len < 40 ? len : 40;  // the mapping ends in 40 entries of value 1, column 1
  for (int q = 0; q < k; ++q) CHECK(C[q], n * B[ldb + q]);
  return 0;
}
int main() {
  double* v = mapped<double>(last + 5ll);
  int32_t* c = mapped<int32_t>(last + 5ll);
  for (int i = 0; i < 40; ++i) v[last - 1ll - i] = c[last - 1ll - i] = 1;
  val = v, col = c;
  int bad = 0;
  for (int len : {1, 2, 3, 4, 5, 6, 7, 8, 9, 31}) {
    bad |= row(len, 1, 1, 1, false, [&](int32_t* rp, double* B, double* C) {
      spmv::k_crs_row<double, true, false>(1, rp, col, val, B, 1, C, 1, 0);
    });
    bad |= row(len, 2, 1, 1, false, [&](int32_t* rp, double* B, double* C) {
      spmv::k_crs_row<double, false, false>(1, rp, col, val, B, 2, C, 1, 0);
    });
    bad |= row(len, 1, 1, 1, false, [&](int32_t* rp, double* B, double* C) {
      spmv::k_crs_row<double, true, true>(1, rp, col, val, B, 1, C, 1, 0);
    });
    bad |= row(len, 1, 1, 1, false, [&](int32_t* rp, double* B, double* C) {
      spmv::k_crs_wide<double, 1>(1, rp, col, val, B, 1, C, 1);
    });
    bad |= row(len, 4, 4, 1, false, [&](int32_t* rp, double* B, double* C) {
      spmv::k_crs_wide<double, 4>(1, rp, col, val, B, 4, C, 4);
    });
    bad |= row(len, 1, 1, 1, false, [&](int32_t* rp, double* B, double* C) {  // a lane row of k_crs_long
      spmv::k_crs_long<double>(nullptr, 0, 0, 1, rp, col, val, B, 1, C, 1, 1, 32, 0);
    });
    bad |= row(len, 2, 2, 2, false, [&](int32_t* rp, double* B, double* C) {
      spmv::k_crs_cols<double, 1, false>(1, rp, col, val, B, 2, C, 2, 2, 0);
    });
  }
  static int32_t zero = 0;
  for (int k : {1, 3})
    for (int len : {40, 70, 300, 1500, 5000})
      for (int n_cta : {0, 1})  // the row on a warp, on a CTA
        bad |= row(len, k, k, n_cta ? 256 : 32, true, [&](int32_t* rp, double* B, double* C) {
          spmv::k_crs_long<double>(&zero, 1, n_cta, 1, rp, col, val, B, k, C, k, k, 12, 0);
        });
  return bad;
}
"""

# Rows that end 64 entries below: as far as the steps of one entry a lane go.
BATCH = r"""
int main() {
  const int last = INT_MAX - 64;
  double* v = mapped<double>(last);
  int32_t* c = mapped<int32_t>(last);
  static double B[4], C[4];
  for (int len : {50, 127, 128, 129, 700}) {
    int32_t rp[2] = {last - len, last};
    int2 list[1] = {{0, last - len}};
    spmv::BatchMat m = {rp, c, v, B, C, 2, 2, 1};
    for (int lanes : {2, 4, 8, 16, 32})
      for (int lane = 0; lane < 32; ++lane) {
        spmv::BatchItem one = {0, 0, 1, len, (int16_t)lanes, (int16_t)spmv::listed_mode(last), 0, 0};
        spmv::batch_row_item<2, 2>(&m, list, one, 2, lane);
        spmv::batch_row_item<2, 1>(&m, list, one, 2, lane);
      }
  }
  return spmv::listed_mode(last - 64) != 2;  // (the sum over the lanes is stubbed: only the reads are checked)
}
"""

headers = pytest.mark.skipif(not os.path.exists("/usr/local/cuda/include/cuda_runtime.h"), reason="no CUDA headers")


def run_on_host(tmp_path, source, harness):
    text = open(os.path.join(CSRC, source)).read()
    text = text.replace('#include "internal.h"', "")
    text = re.sub(r"<<<.*?>>>", "", text, flags=re.S)
    kernels = re.sub(r"template <[^\n]*>\nstatic cudaError_t \w+\(.*?\n}\n", "", text, flags=re.S)
    kernels = re.sub(r"\n(?://[^\n]*\n)*static int sell_cols\(.*?\n}\n", "\n", kernels, flags=re.S)
    kernels = re.sub(r"\ncudaError_t \w+\(.*?\n}\n", "\n", kernels, flags=re.S)
    (tmp_path / "device.cuh").write_text(SHIM)
    shutil.copy(os.path.join(CSRC, "layout.h"), tmp_path)
    (tmp_path / "t.cpp").write_text(kernels + harness)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++20", "-O1", "-fwrapv", "-pthread", "-I", "/usr/local/cuda/include", "-w",
                    str(tmp_path / "t.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    if r.returncode == 77:
        pytest.skip("no address space: " + r.stderr)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)


@headers
def test_sell_slots_behind_2_31(tmp_path):
    run_on_host(tmp_path, "k_sell.cu", SELL)


@headers
def test_crs_rows_that_end_at_2_31(tmp_path):
    run_on_host(tmp_path, "k_lanes.cu", LANES)


@headers
def test_batch_rows_that_end_at_2_31(tmp_path):
    run_on_host(tmp_path, "batch_kernel.cuh", BATCH)
