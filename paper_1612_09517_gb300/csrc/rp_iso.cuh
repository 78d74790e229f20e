// Products and shared-memory layout of the kernels whose threads own KPT = 2^LK
// configurations (rp_chip.cu, rp_term.cu).
#pragma once

#include <cuda_runtime.h>

#include "rp_device.cuh"

namespace rp {
namespace {

// y += g q on (re, im)
__device__ __forceinline__ void madd(Cx<float>& y, float g, const Cx<float>& q) {
  const float2 s = __ffma2_rn(make_float2(g, g), make_float2(q.re, q.im), make_float2(y.re, y.im));
  y.re = s.x;
  y.im = s.y;
}
__device__ __forceinline__ void madd(Cx<double>& y, double g, const Cx<double>& q) {
  y.re = fma(g, q.re, y.re);
  y.im = fma(g, q.im, y.im);
}
// y += g q where g is not shared by other products: two scalar multiply-adds
// (the packed form would first build the pair (g, g)); the same rounding
template <typename T>
__device__ __forceinline__ void madd_s(Cx<T>& y, T g, const Cx<T>& q) {
  y.re = fma(g, q.re, y.re);
  y.im = fma(g, q.im, y.im);
}
// y += i g q
template <typename T>
__device__ __forceinline__ void madd_i(Cx<T>& y, T g, const Cx<T>& q) {
  y.re = fma(-g, q.im, y.re);
  y.im = fma(g, q.re, y.im);
}

// The KPT values of electron state e at a slot: vectors of two FP32 values or
// one FP64 value, [e][group][slot], so a warp's accesses are contiguous.
template <typename T, int LK>
struct Vec {
  static constexpr int KPT = 1 << LK;
  static constexpr int W = sizeof(T) == 4 && LK > 0 ? 2 : 1;  // values per access
  static constexpr int G = KPT / W;                           // accesses
  struct alignas(W * sizeof(Cx<T>)) Pack {
    Cx<T> v[W];
  };
  static __device__ __forceinline__ void get(const Cx<T>* buf, int S, int e, int slot,
                                             Cx<T> (&q)[KPT]) {
    const Pack* p = reinterpret_cast<const Pack*>(buf) + (size_t)(e * G) * S + slot;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const Pack k = p[g * S];
#pragma unroll
      for (int w = 0; w < W; ++w) q[g * W + w] = k.v[w];
    }
  }
  static __device__ __forceinline__ void put(Cx<T>* buf, int S, int e, int slot,
                                             const Cx<T> (&q)[KPT]) {
    Pack* p = reinterpret_cast<Pack*>(buf) + (size_t)(e * G) * S + slot;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      Pack k;
#pragma unroll
      for (int w = 0; w < W; ++w) k.v[w] = q[g * W + w];
      p[g * S] = k;
    }
  }
};

}  // namespace
}  // namespace rp
