// Coherent-state amplitudes of a sample, for the kernels that build psi(0).
#pragma once

#include <stdint.h>

#include "rp_kernels.cuh"

namespace rp {
namespace {

// ---- Philox4x32-10 (Salmon et al., SC'11) and coherent states (Eq. 15) ----

__device__ __forceinline__ void philox4x32_10(uint32_t (&c)[4], uint32_t k0, uint32_t k1) {
  const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
  const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += W0;
      k1 += W1;
    }
    const uint32_t lo0 = M0 * c[0], hi0 = __umulhi(M0, c[0]);
    const uint32_t lo1 = M1 * c[2], hi1 = __umulhi(M1, c[2]);
    const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
  }
}

__device__ __forceinline__ double u53(uint32_t hi, uint32_t lo) {
  return ((double)(hi >> 5) * 67108864.0 + (double)(lo >> 6)) * (1.0 / 9007199254740992.0);
}

// Components c_j (o[2 j], o[2 j + 1], j = 0 .. 2I) of the coherent state of the
// nucleus at layout position p for sample s: Philox draw of the direction
// (counter (input index, s_lo, s_hi, pair), key seed; cos theta = 1 - 2 u1,
// phi = 2 pi u2, Eq. 17) and c_j = sqrt(C(2I, j)) cos^{2I-j}(theta/2)
// sin^j(theta/2) e^{i j phi} (Eq. 15); u receives (u1, u2).
__device__ __forceinline__ void coherent_amp(const LayoutDev& L, int p, uint32_t pair,
                                             unsigned long long s, uint64_t seed, double* o,
                                             double* u) {
  const int k = L.input_index[p];
  uint32_t c[4] = {(uint32_t)k, (uint32_t)(s & 0xFFFFFFFFull), (uint32_t)(s >> 32), pair};
  philox4x32_10(c, (uint32_t)(seed & 0xFFFFFFFFull), (uint32_t)(seed >> 32));
  const double u1 = u53(c[0], c[1]), u2 = u53(c[2], c[3]);
  u[0] = u1;
  u[1] = u2;
  const double ch = sqrt(1.0 - u1), sh = sqrt(u1);  // cos(theta/2), sin(theta/2)
  const int d = L.d[p], twoI = d - 1;
  double binom = 1.0;  // C(2I, j)
  for (int j = 0; j < d; ++j) {
    if (j > 0) binom = binom * (double)(twoI - j + 1) / (double)j;
    double mag = sqrt(binom);
    for (int i = 0; i < twoI - j; ++i) mag *= ch;
    for (int i = 0; i < j; ++i) mag *= sh;
    double sn, cs;
    sincospi(2.0 * (double)j * u2, &sn, &cs);
    o[2 * j] = mag * cs;
    o[2 * j + 1] = mag * sn;
  }
}

}  // namespace
}  // namespace rp
