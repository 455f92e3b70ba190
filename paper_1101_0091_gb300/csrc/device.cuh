// Device helpers shared by the kernels: PTX wrappers for mbarriers and bulk
// copies, a bounded mbarrier wait, value loads, and the exact float->double
// widening used by the FP32-value forms.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "layout.h"

namespace spmv {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Makes the mbarrier initialisation visible to the async (bulk copy) proxy.
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// One-dimensional bulk copy global -> shared (TMA engine, no tensor map).
// Both addresses 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for phase `parity` of the barrier, giving up after limit_ns.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                  unsigned long long limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > limit_ns) return false;
  }
  return true;
}

// FP32-stored values come in two storage types with the same layout:
//  - f32n: every value is zero or a normal float (the plan checks this on the
//    host when it rounds the values).  Widened exactly in the integer pipe from
//    the IEEE 754 formats: with sign s, biased exponent e and 23-bit fraction m,
//    a normal float is 2^(e-127) * 1.m, the same number as the double with
//    exponent e + (1023 - 127) and fraction m << 29; zero keeps its sign.
//    On this GPU the hardware f32->f64 conversion issues on the FP64 pipe that
//    the FMAs already saturate, so this path avoids it.
//  - float: values that include subnormal, infinite or NaN floats; widened by
//    the hardware conversion (exact for every input).
struct f32n {
  float v;
};

__device__ __forceinline__ double widen_f32n(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t a = u & 0x7fffffffu;
  const uint32_t hi = a ? ((u & 0x80000000u) | ((a >> 3) + (896u << 20))) : (u & 0x80000000u);
  const uint32_t lo = a ? (u << 29) : 0u;
  return __hiloint2double((int)hi, (int)lo);
}

// Fire-and-forget bulk prefetch of [p, p + bytes) into L2 (TMA engine).  p and
// bytes must be multiples of 16 and the range inside the allocation.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  if (bytes == 0) return;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Programmatic dependent launch (launch_dependent, internal.h): grid_dependents lets the next kernel of
// the stream be launched as soon as every CTA of this one has got here (or has exited), so that its CTAs
// take the slots that this kernel's last ones leave; grid_wait holds a kernel launched that way until the
// work before it is complete and visible.  Before grid_wait a kernel reads its plan's own arrays only, and
// what earlier work may have written (B, the solvers' vectors and scalars) is read with plain loads: a
// read-only load (ld.global.nc, __ldg, const __restrict__) could be moved above the wait.
//
// grid_dependents comes after grid_wait, never before: ahead of it, products that fit on the chip several
// times over are launched on top of one another, and the last ones crowd onto the SMs that empty first
// (256^2 Laplacian in a CUDA graph 3.9 us, 2.2 now; eigenproblem matrix of 50,001 rows 9.5 us, 6.5 now).  The
// kernels whose CTAs differ most in time, or that fit on the chip at once, call it in front of their
// stores, for the same reason: eigenproblem matrix of 200,003 rows 15.0 -> 11.4 us, 27-point stencil 48^3
// 13.9 -> 9.1, 400^2 Laplacian 4.5 -> 3.5.  Larger grids of even work overlap more of the next launch with
// their last wave and call it at once (131 x 127 x 129 Poisson, k = 3: 77.8 us, in front of the stores 80.0).
// The lines: k_crs_cols at one wave of kOneWave CTAs, k_crs_row at four, between which it does not matter
// (at once / in front of the stores: 800^2 and 1000^2 Laplacians 7.66 / 7.66, 11.1 / 10.9 us; 72^3, 90^3 and 100^3
// Poisson 6.6 / 6.9, 11.1 / 11.2, 17.2 / 17.0).  (k_crs_cols of several columns holds six CTAs, not eight: up to
// 1.3 of its waves count as one.)
constexpr unsigned kOneWave = 152 * 8;  // CTAs of kThreads that the chip holds, eight per SM
__device__ __forceinline__ void grid_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ double to_f64(double v) { return v; }
__device__ __forceinline__ double to_f64(float v) { return (double)v; }
__device__ __forceinline__ double to_f64(f32n v) { return widen_f32n(v.v); }

// Read-only loads through the non-coherent path.
__device__ __forceinline__ double ldg(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ldg(const float* p) { return __ldg(p); }
__device__ __forceinline__ f32n ldg(const f32n* p) { return f32n{__ldg(reinterpret_cast<const float*>(p))}; }
__device__ __forceinline__ int32_t ldg(const int32_t* p) { return __ldg(p); }

// Streaming loads (evict-first): matrix entries are used once per product.
__device__ __forceinline__ double ldcs(const double* p) { return __ldcs(p); }
__device__ __forceinline__ float ldcs(const float* p) { return __ldcs(p); }
__device__ __forceinline__ f32n ldcs(const f32n* p) { return f32n{__ldcs(reinterpret_cast<const float*>(p))}; }
__device__ __forceinline__ int32_t ldcs(const int32_t* p) { return __ldcs(p); }

// Four consecutive entries from a 16-byte (col, float) or 32-byte (double) aligned address.  The doubles
// are a whole sector, which nothing reads again: they take no line of L1.
__device__ __forceinline__ void ldg4(const double* p, double (&x)[4]) {
  asm volatile("ld.global.nc.L1::no_allocate.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(x[0]), "=d"(x[1]), "=d"(x[2]), "=d"(x[3])
               : "l"(p));
}
__device__ __forceinline__ void ldg4(const float* p, float (&x)[4]) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(p));
  x[0] = t.x, x[1] = t.y, x[2] = t.z, x[3] = t.w;
}
__device__ __forceinline__ void ldg4(const f32n* p, f32n (&x)[4]) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(p));
  x[0].v = t.x, x[1].v = t.y, x[2].v = t.z, x[3].v = t.w;
}
__device__ __forceinline__ void ldg4(const int32_t* p, int32_t (&x)[4]) {
  const int4 t = __ldg(reinterpret_cast<const int4*>(p));
  x[0] = t.x, x[1] = t.y, x[2] = t.z, x[3] = t.w;
}

// Whether every row of the blocks B and C starts on 16 bytes.
inline bool rows_on_16_bytes(const double* B, int64_t ldb, const double* C, int64_t ldc) {
  return ldb % 2 == 0 && ldc % 2 == 0 && (((uintptr_t)B | (uintptr_t)C) & 15) == 0;
}

// Columns per lane of k_crs_cols (k_sell_cols has its own rule, sell_cols) for k right-hand sides over
// n_rows rows: up to `even` (4 or 2; 16-byte accesses) where k divides by it and the rows start on 16
// bytes (a16), 3, 5 or 7 in 8-byte accesses where k divides by one of those and `odd` allows it, else 1.
// These products are bound by the FP64 pipe (a warp's FMA occupies an SM for 16 cycles), so a lane per
// column costs little that the pipe does not hide; a masked kernel of 4, 8 or 16 columns on one lane
// issued the masked FMAs as well (k = 3 on a 131 x 127 x 129 Poisson matrix: 107.9 us masked, 79.7 with
// one column per lane, FP64 floor 71).  Several columns per lane read the row's entries fewer times
// (128^3 Poisson, k = 3 / 7 / 15, one -> several: 78.5 -> 76.1, 178.7 -> 170.5, 374.1 -> 362.3 us) as long as the
// threads still fill the GPU: at 60,000 rows, k = 4, four / two / one columns took 23.8 / 16.7 / 14.1 us, k = 5
// five / one 30.7 / 13.5 us, hence kMinColThreads (the GPU holds 311,296 threads).
constexpr int64_t kMinColThreads = 400000;
inline int cols_per_lane(int k, bool a16, int64_t n_rows, int even, bool odd) {
  const int even_widths[] = {4, 2}, odd_widths[] = {7, 5, 3};
  for (int w : even_widths)
    if (a16 && w <= even && k % w == 0 && n_rows * (k / w) >= kMinColThreads) return w;
  if (odd && !(a16 && k % 2 == 0))
    for (int w : odd_widths)
      if (k % w == 0 && n_rows * (k / w) >= kMinColThreads) return w;
  return 1;
}

// W consecutive columns of a block row: 16-byte accesses where the rows start on 16 bytes (A16, even W), else
// 8-byte ones.  (Plain loads: see grid_wait.)
template <int W, bool A16 = (W % 2 == 0)>
__device__ __forceinline__ void load_cols(const double* b, double (&g)[W]) {
  if constexpr (!A16) {
#pragma unroll
    for (int q = 0; q < W; ++q) g[q] = b[q];
  } else {
#pragma unroll
    for (int q = 0; q < W; q += 2) {
      const double2 x = *reinterpret_cast<const double2*>(b + q);
      g[q] = x.x;
      g[q + 1] = x.y;
    }
  }
}
template <int W, bool A16 = (W % 2 == 0)>
__device__ __forceinline__ void store_cols(double* c, const double (&a)[W]) {
  if constexpr (!A16) {
#pragma unroll
    for (int q = 0; q < W; ++q) c[q] = a[q];
  } else {
#pragma unroll
    for (int q = 0; q < W; q += 2) reinterpret_cast<double2*>(c)[q / 2] = make_double2(a[q], a[q + 1]);
  }
}

__device__ __forceinline__ double warp_sum_xor(double x, int width) {
  for (int off = width >> 1; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

}  // namespace spmv
