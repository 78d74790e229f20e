// One configuration's share of the low-rank time integral (see rp_integral.cu):
// y_k += L_nk (-i)^n x_n and sum_k |y_k|^2.  Every kernel that integrates uses
// these, so a configuration's value does not depend on the kernel.
#pragma once

#include <cuda_runtime.h>

#include "rp_device.cuh"

namespace rp {
namespace {

template <typename T>
struct ProjCfg {
  static constexpr int kB = sizeof(T) == 4 ? 32 : 16;     // columns of L per block
  static constexpr int kCfg = sizeof(T) == 4 ? 2 : 1;     // configurations per thread
};
// y += L (zr, zi) for the columns at l: N pairs of columns (FP32) or N columns (FP64).
template <int N>
__device__ __forceinline__ void proj_add(float2 (&yr)[N], float2 (&yi)[N], const float* l, float zr,
                                         float zi) {
  const float2 r2 = make_float2(zr, zr), i2 = make_float2(zi, zi);
#pragma unroll
  for (int k = 0; k < N; k += 2) {
    const float4 v = *reinterpret_cast<const float4*>(l + 2 * k);
    const float2 a = make_float2(v.x, v.y), b = make_float2(v.z, v.w);
    yr[k] = __ffma2_rn(a, r2, yr[k]);
    yi[k] = __ffma2_rn(a, i2, yi[k]);
    yr[k + 1] = __ffma2_rn(b, r2, yr[k + 1]);
    yi[k + 1] = __ffma2_rn(b, i2, yi[k + 1]);
  }
}
template <int N>
__device__ __forceinline__ void proj_add(double (&yr)[N], double (&yi)[N], const double* l,
                                         double zr, double zi) {
#pragma unroll
  for (int k = 0; k < N; k += 2) {
    const double2 v = *reinterpret_cast<const double2*>(l + k);
    yr[k] = fma(v.x, zr, yr[k]);
    yi[k] = fma(v.x, zi, yi[k]);
    yr[k + 1] = fma(v.y, zr, yr[k + 1]);
    yi[k + 1] = fma(v.y, zi, yi[k + 1]);
  }
}
// sum_k |y_k|^2: eight columns in T, their sums in FP64 (the same value however
// the columns are spread over threads).
__device__ __forceinline__ double proj_norm8(const float2* yr, const float2* yi) {
  float2 s = make_float2(0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 4; ++k) s = __ffma2_rn(yi[k], yi[k], __ffma2_rn(yr[k], yr[k], s));
  return (double)(s.x + s.y);
}
__device__ __forceinline__ double proj_norm8(const double* yr, const double* yi) {
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) s = fma(yi[k], yi[k], fma(yr[k], yr[k], s));
  return s;
}
__device__ __forceinline__ double proj_norm(const float2 (&yr)[16], const float2 (&yi)[16]) {
  return (proj_norm8(yr, yi) + proj_norm8(yr + 4, yi + 4)) +
         (proj_norm8(yr + 8, yi + 8) + proj_norm8(yr + 12, yi + 12));
}
__device__ __forceinline__ double proj_norm(const double (&yr)[16], const double (&yi)[16]) {
  return proj_norm8(yr, yi) + proj_norm8(yr + 8, yi + 8);
}
template <typename T>
struct ProjAcc {
  using type = double;
};
template <>
struct ProjAcc<float> {
  using type = float2;
};

// A slice value (re, im) of one configuration: 8 or 16 bytes.
template <typename T>
struct SliceVal {
  using type = double2;
};
template <>
struct SliceVal<float> {
  using type = float2;
};

__device__ __forceinline__ void slice_copy(unsigned dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void slice_copy(unsigned dst, const double* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Slices in flight per thread and configuration: GN - 1 groups of GS.  Loads into
// registers left one load's latency per four terms exposed (18 % of issue slots
// used); the ring costs no registers, and a thread reads only what it copied, so
// nothing waits on other threads.
template <typename T>
__host__ __device__ constexpr int proj_groups() {
  return sizeof(T) == 4 ? 6 : 3;  // of four slices; FP64 spends 16 x longer on a term
}

// Bytes of the ring of a block of `threads` threads with C configurations each.
template <typename T>
__host__ __device__ constexpr size_t proj_ring_bytes(int threads, int C) {
  return (size_t)threads * C * 4 * proj_groups<T>() * 2 * sizeof(T);
}

// Partial sums of C configurations over the n_e slices at p[c] + n stride
// (complex values, stride in T), against the KB columns of L at sl[n * ld].
// ring: this thread's first entry of the block's ring, entries `threads` apart.
template <typename T, int C, int GN = proj_groups<T>(), int GS = 4>
__device__ __forceinline__ void project_block(typename ProjAcc<T>::type (&yr)[C][16],
                                              typename ProjAcc<T>::type (&yi)[C][16],
                                              const T* const (&p)[C], size_t stride, const T* sl,
                                              int ld, int n_e, typename SliceVal<T>::type* ring,
                                              int threads) {
  using V = typename SliceVal<T>::type;
#pragma unroll
  for (int c = 0; c < C; ++c)
#pragma unroll
    for (int k = 0; k < 16; ++k) yr[c][k] = yi[c][k] = typename ProjAcc<T>::type{};
  const unsigned rs = smem_u32(ring);
  const unsigned step = (unsigned)(threads * sizeof(V));
  const T* src[C];
#pragma unroll
  for (int c = 0; c < C; ++c) src[c] = p[c];
  int issued = 0, slot = 0;  // slices copied so far, next ring group
  auto issue = [&]() {
#pragma unroll
    for (int a = 0; a < GS; ++a)
      if (issued + a < n_e) {
#pragma unroll
        for (int c = 0; c < C; ++c) {
          slice_copy(rs + (unsigned)((slot * GS + a) * C + c) * step, src[c]);
          src[c] += stride;
        }
      }
    asm volatile("cp.async.commit_group;" ::: "memory");
    issued += GS;
    slot = slot + 1 == GN ? 0 : slot + 1;
  };
#pragma unroll 1
  for (int g = 0; g < GN - 1; ++g) issue();
  int use = 0;
#pragma unroll 1
  for (int n = 0; n < n_e; n += GS) {
    issue();
    asm volatile("cp.async.wait_group %0;" ::"n"(GN - 1) : "memory");
#pragma unroll
    for (int a = 0; a < GS; ++a) {
      if (n + a < n_e) {  // the same for the whole CTA
        const T* l = sl + (n + a) * ld;
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const V v = ring[((use * GS + a) * C + c) * threads];
          if (GS == 1 ? (n & 1) : (a & 1)) proj_add(yr[c], yi[c], l, v.y, -v.x);
          else proj_add(yr[c], yi[c], l, v.x, v.y);
        }
      }
    }
    use = use + 1 == GN ? 0 : use + 1;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Stages columns k0 .. k0 + KB - 1 of a field's L (n_e rows) as sl[n][KB].
template <typename T, int KB = ProjCfg<T>::kB>
__device__ __forceinline__ void stage_factor(T* sl, const T* __restrict__ Lf, int ldk, int n_e,
                                             int k0, int tid, int nthreads) {
  for (int e = tid; e < n_e * KB; e += nthreads) {
    const int n = e / KB, k = k0 + e % KB;
    sl[e] = k < ldk ? Lf[n * ldk + k] : T(0);
  }
}

}  // namespace
}  // namespace rp
