// Whole propagations on chip for isotropic systems that fit one SM.
//
// One CTA holds the Chebyshev vectors of its rows for a whole horizon
// (k_chip_items: items from a device counter) or one macro-step
// (k_chip_macro).  A thread owns KPT = 2^LK nuclear configurations that differ
// in the LK innermost spin-1/2 nuclei:
//   * phi_{n-1} and the accumulator psi(h) of its own configurations stay in
//     registers; shared memory holds phi_{n-1} (read by the partners) and
//     phi_{n-2} in the buffer that receives phi_n, one block barrier per term;
//   * flip-flops of the in-thread nuclei are register to register;
//   * digits, directions and addresses of the other nuclei are found once per
//     nucleus and serve the KPT configurations, whose partners' components lie
//     side by side (one 16-byte access per two FP32 values).
// Arithmetic per configuration and term, in this order for every LK:
//   u = (D + J-, kappa- and flip-flop terms) phi_{n-1},  phi_n = u - phi_{n-2}
// with the factor 2/dE of the recurrence folded into the constants (formed in
// FP64, rounded once).  FP32 subtracts phi_{n-2} last: summing into it rounds
// every product at the size of phi (norm errors twice as large); FP64 starts
// from it, which costs no operation.  An isotropic H is real, so a product is
// one packed fma.rn.f32x2 on (re, im); only kappa mixes re and im.  The global
// phase exp(-i E_c h) of the propagator is left out (no yield, survival or
// expectation value depends on it), which makes the coefficients of the sum
// real: c_n = r_n (-i)^n; cf holds r_n with the sign of (-i)^n for n mod 4 >= 2.
//
// Rows that exceed one SM (FP32, Z up to 8 x 2048) are split over the 2^cb CTAs of
// a thread-block cluster by the cb outermost spin-1/2 nuclei (layout positions lb =
// n_half - cb and up): the local configuration l of CTA `rank` is
//   m = (l >> lb) << (lb + cb) | rank << lb | l mod 2^lb,
// the partner under nucleus lb + i is the same slot of CTA rank XOR 2^i (read
// through distributed shared memory, the direction being the CTA's), and one
// cluster barrier per term takes the place of the block barrier.
#include <algorithm>
#include <cstring>

#include "rp_device.cuh"
#include "rp_iso.cuh"
#include "rp_kernels.cuh"
#include "rp_project.cuh"
#include "rp_sample.cuh"

namespace rp {

namespace {

__device__ __forceinline__ unsigned chip_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Barrier of the block or, split over a cluster, of the cluster (release /
// acquire: shared-memory writes before it are seen by every CTA after it).
template <int CB>
__device__ __forceinline__ void chip_barrier() {
  if constexpr (CB > 0)
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  else
    __syncthreads();
}
// The two halves of the cluster's barrier, for work that needs neither.
template <int CB>
__device__ __forceinline__ void chip_arrive() {
  if constexpr (CB > 0) asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
template <int CB>
__device__ __forceinline__ void chip_wait() {
  if constexpr (CB > 0) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  else __syncthreads();
}
// Address in the cluster's shared window of the CTA `rank`.
__device__ __forceinline__ unsigned chip_peer(unsigned a, unsigned rank) {
  unsigned ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  return ra;
}
// The KPT values of electron state e at a slot of a peer's buffer (base: its
// shared-cluster address); volatile, so it stays between the barriers.
template <int LK>
__device__ __forceinline__ void peer_get(unsigned base, int S, int e, int slot,
                                         Cx<float> (&q)[1 << LK]) {
  using V = Vec<float, LK>;
  const unsigned a = base + (unsigned)(((e * V::G) * S + slot) * (int)sizeof(typename V::Pack));
#pragma unroll
  for (int g = 0; g < V::G; ++g) {
    const unsigned p = a + (unsigned)(g * S * (int)sizeof(typename V::Pack));
    if constexpr (V::W == 2)
      asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(q[2 * g].re), "=f"(q[2 * g].im), "=f"(q[2 * g + 1].re), "=f"(q[2 * g + 1].im)
                   : "r"(p));
    else
      asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(q[g].re), "=f"(q[g].im) : "r"(p));
  }
}

// Partner "up" (nuclear quantum number one lower: S_- I_+ brings it here) adds
// its components (u0, u1) to targets (t0, t1), "down" the reverse:
//   radical 0: 0 -> 2, 1 -> 3;  radical 1: 0 -> 1, 2 -> 3.
// One component at a time, so that only KPT values are in flight.
// Flip-flop of a spin-1/2 nucleus from a slot that holds the partner above (down
// = false) or below: FP32 multiplies both directions (one by zero); FP64, whose
// products cost 16 times as much as a select, picks the target first.
template <int KPT>
__device__ __forceinline__ void add_either(Cx<float> (&y)[KPT][4], int tu, int td, bool down,
                                           float gu, float gd, const Cx<float> (&q)[KPT]) {
#pragma unroll
  for (int c = 0; c < KPT; ++c) {
    madd(y[c][tu], gu, q[c]);
    madd(y[c][td], gd, q[c]);
  }
}
template <int KPT>
__device__ __forceinline__ void add_either(Cx<double> (&y)[KPT][4], int tu, int td, bool down,
                                           double gu, double gd, const Cx<double> (&q)[KPT]) {
  const double g = down ? gd : gu;
#pragma unroll
  for (int c = 0; c < KPT; ++c) {
    Cx<double> t = down ? y[c][td] : y[c][tu];
    madd(t, g, q[c]);
    if (down) y[c][td] = t;
    else y[c][tu] = t;
  }
}
template <typename T, int LK>
__device__ __forceinline__ void flip_either(Cx<T> (&y)[1 << LK][4], int rr, bool down, T g,
                                            const Cx<T>* cur, int S, int sl) {
  constexpr int KPT = 1 << LK;
  const T gu = down ? T(0) : g, gd = down ? g : T(0);
  Cx<T> q[KPT];
  if (rr == 0) {
    Vec<T, LK>::get(cur, S, down ? 2 : 0, sl, q);
    add_either<KPT>(y, 2, 0, down, gu, gd, q);
    Vec<T, LK>::get(cur, S, down ? 3 : 1, sl, q);
    add_either<KPT>(y, 3, 1, down, gu, gd, q);
  } else {
    Vec<T, LK>::get(cur, S, down ? 1 : 0, sl, q);
    add_either<KPT>(y, 1, 0, down, gu, gd, q);
    Vec<T, LK>::get(cur, S, down ? 3 : 2, sl, q);
    add_either<KPT>(y, 3, 2, down, gu, gd, q);
  }
}
template <typename T, int LK, bool UP>
__device__ __forceinline__ void flip_one(Cx<T> (&y)[1 << LK][4], int rr, T g, const Cx<T>* cur,
                                         int S, int sl) {
  constexpr int KPT = 1 << LK;
  Cx<T> q[KPT];
  if (rr == 0) {
    Vec<T, LK>::get(cur, S, UP ? 0 : 2, sl, q);
#pragma unroll
    for (int c = 0; c < KPT; ++c) madd(y[c][UP ? 2 : 0], g, q[c]);
    Vec<T, LK>::get(cur, S, UP ? 1 : 3, sl, q);
#pragma unroll
    for (int c = 0; c < KPT; ++c) madd(y[c][UP ? 3 : 1], g, q[c]);
  } else {
    Vec<T, LK>::get(cur, S, UP ? 0 : 1, sl, q);
#pragma unroll
    for (int c = 0; c < KPT; ++c) madd(y[c][UP ? 1 : 0], g, q[c]);
    Vec<T, LK>::get(cur, S, UP ? 2 : 3, sl, q);
#pragma unroll
    for (int c = 0; c < KPT; ++c) madd(y[c][UP ? 3 : 2], g, q[c]);
  }
}

constexpr int kChipMaxCb = 3;

// Partner values of the nuclei that select the CTA, loaded at the start of a term
// (a remote load takes far longer than a local one) and used in their turn.
template <int LK, int CB>
struct PeerVals {
  Cx<float> q[CB > 0 ? CB : 1][2][1 << LK];
};
template <int LK, int CB>
__device__ __forceinline__ void peer_load(PeerVals<LK, CB>& v, unsigned own, unsigned rank,
                                          unsigned rad, int S, int sl) {
#pragma unroll
  for (int i = 0; i < CB; ++i) {
    const unsigned peer = chip_peer(own, rank ^ (1u << i));
    const bool down = (rank >> i) & 1u, r1 = (rad >> i) & 1u;
    peer_get<LK>(peer, S, down ? (r1 ? 1 : 2) : 0, sl, v.q[i][0]);
    peer_get<LK>(peer, S, down ? 3 : (r1 ? 2 : 1), sl, v.q[i][1]);
  }
}
template <int LK, int CB>
__device__ __forceinline__ void peer_add(Cx<float> (&y)[1 << LK][4], const PeerVals<LK, CB>& v,
                                         unsigned rank, unsigned rad, const float* g) {
  constexpr int KPT = 1 << LK;
#pragma unroll
  for (int i = 0; i < CB; ++i) {
    {
      const bool down = (rank >> i) & 1u, r1 = (rad >> i) & 1u;
      const float gi = g[i];
#pragma unroll
      for (int c = 0; c < KPT; ++c) {
        if (!r1) {
          if (down) {
            madd(y[c][0], gi, v.q[i][0][c]);
            madd(y[c][1], gi, v.q[i][1][c]);
          } else {
            madd(y[c][2], gi, v.q[i][0][c]);
            madd(y[c][3], gi, v.q[i][1][c]);
          }
        } else {
          if (down) {
            madd(y[c][0], gi, v.q[i][0][c]);
            madd(y[c][2], gi, v.q[i][1][c]);
          } else {
            madd(y[c][1], gi, v.q[i][0][c]);
            madd(y[c][3], gi, v.q[i][1][c]);
          }
        }
      }
    }
  }
}

// Diagonal 2 (H_mm - E_c) / dE of the four electron states of configuration m.
template <typename T>
__device__ __forceinline__ void chip_diag(const HamDev<double>& H, const FieldDev<double>& F,
                                          unsigned m, T (&d)[4]) {
  double b[2] = {0.0, 0.0};
  unsigned q = m;
  for (int p = 0; p < H.n_nuc; ++p) {
    const unsigned dd = (unsigned)H.d[p], j = q % dd;
    q /= dd;
    const double v = (0.5 * (double)(dd - 1) - (double)j) * H.v[p][2];
    if (H.rad[p] == 0) b[0] += v;
    else b[1] += v;
  }
  const double sp = 0.5 * (b[0] + b[1]), sm = 0.5 * (b[0] - b[1]), hJ = 0.5 * H.Je;
  d[0] = (T)(2.0 * (F.s * (F.omega + hJ + sp) - F.sh_re));
  d[1] = (T)(2.0 * (F.s * (-hJ + sm) - F.sh_re));
  d[2] = (T)(2.0 * (F.s * (-hJ - sm) - F.sh_re));
  d[3] = (T)(2.0 * (F.s * (-F.omega + hJ - sp) - F.sh_re));
}

// Constants of a CTA's rows (one system, one field) in shared memory.
template <typename T>
struct alignas(16) ChipConst {
  T g[kMaxNucDev];  // 2 (a/2) / dE (x sqrt 2 for spin 1)
  T J, kappa;       // 2 J / dE, 2 kappa / dE
  int d[kMaxNucDev], st[kMaxNucDev];  // dimension and stride in slots (spins above 1)
  unsigned rad;                       // radical of nucleus p in bit p
  int n_half, n_one, n_nuc;           // n_half: spin-1/2 nuclei of the CTA's own slots
};

template <typename T>
__device__ void chip_const(ChipConst<T>& K, const HamDev<double>& H, const FieldDev<double>& F,
                           int lk, int cb, int tid) {
  if (tid < H.n_nuc) {
    const int p = tid;
    const double g = 2.0 * F.s * H.U[p][4] * (H.d[p] == 3 ? 1.41421356237309504880 : 1.0);
    K.g[p] = (T)g;
    K.d[p] = H.d[p];
    K.st[p] = (int)(H.stride[p] >> (lk + cb));
  }
  if (tid == 0) {
    K.J = (T)(2.0 * F.s * H.Je);
    K.kappa = (T)(2.0 * F.s * H.kappa);
    K.n_half = H.n_half - cb;
    K.n_one = H.n_one;
    K.n_nuc = H.n_nuc;
    unsigned m = 0;
    for (int p = 0; p < H.n_nuc; ++p) m |= (unsigned)(H.rad[p] & 1) << p;
    K.rad = m;
  }
}

// The thread's configurations to and from a buffer.
template <typename T, int LK>
__device__ __forceinline__ void chip_put(Cx<T>* b, int S, int slot, const Cx<T> (&v)[1 << LK][4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    Cx<T> q[1 << LK];
#pragma unroll
    for (int c = 0; c < (1 << LK); ++c) q[c] = v[c][e];
    Vec<T, LK>::put(b, S, e, slot, q);
  }
}
template <typename T, int LK>
__device__ __forceinline__ void chip_get(const Cx<T>* b, int S, int slot, Cx<T> (&v)[1 << LK][4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    Cx<T> q[1 << LK];
    Vec<T, LK>::get(b, S, e, slot, q);
#pragma unroll
    for (int c = 0; c < (1 << LK); ++c) v[c][e] = q[c];
  }
}

// One term: u = phi_n from phi_{n-1} (own values a, partners in cur) and, unless
// FIRST, phi_{n-2} (own entries of prev).  dt: diagonals, four per
// configuration.  t: slot within the row, base: the row's first slot.
template <typename T, int LK, int CB>
__device__ __forceinline__ void chip_term(const ChipConst<T>& K, Cx<T> (&y)[1 << LK][4],
                                          const Cx<T> (&a)[1 << LK][4], const T* dt,
                                          const Cx<T>* cur, const Cx<T>* prev, bool first, int S,
                                          int base, int t, unsigned dig) {
  constexpr int KPT = 1 << LK;
  // four configurations per thread have no registers to hold them all term
  constexpr bool kEarly = CB > 0 && LK == 1;
  PeerVals<LK, kEarly ? CB : 0> pv;
  unsigned rank = 0;
  if constexpr (CB > 0) rank = chip_rank();
  if constexpr (kEarly) peer_load<LK, CB>(pv, smem_u32(cur), rank, K.rad >> K.n_half, S, base + t);
  if constexpr (sizeof(T) == 8) {
    if (first) {
#pragma unroll
      for (int c = 0; c < KPT; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) y[c][e] = {T(0), T(0)};
    } else {
      chip_get<T, LK>(prev, S, base + t, y);
    }
  }
#pragma unroll
  for (int c = 0; c < KPT; ++c) {
    T d[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) d[e] = dt[((size_t)c * S + base + t) * 4 + e];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (sizeof(T) == 4) y[c][e] = {d[e] * a[c][e].re, d[e] * a[c][e].im};
      else y[c][e] = {fma(d[e], a[c][e].re, -y[c][e].re), fma(d[e], a[c][e].im, -y[c][e].im)};
    }
  }
  const T J = K.J, kp = K.kappa;
  if (J != T(0)) {
#pragma unroll
    for (int c = 0; c < KPT; ++c) {
      madd(y[c][1], J, a[c][2]);
      madd(y[c][2], J, a[c][1]);
    }
  }
  if (kp != T(0)) {  // -i kappa (2 P_S - 1)
#pragma unroll
    for (int c = 0; c < KPT; ++c) {
      madd_i(y[c][0], kp, a[c][0]);
      madd_i(y[c][1], kp, a[c][2]);
      madd_i(y[c][2], kp, a[c][1]);
      madd_i(y[c][3], kp, a[c][3]);
    }
  }
  // in-thread nuclei
#pragma unroll
  for (int p = 0; p < LK; ++p) {
    const T g = K.g[p];
    if (!((K.rad >> p) & 1u)) {
#pragma unroll
      for (int c = 0; c < KPT; ++c) {
        const int o = c ^ (1 << p), down = (c >> p) & 1;
        madd(y[c][down ? 0 : 2], g, a[o][down ? 2 : 0]);
        madd(y[c][down ? 1 : 3], g, a[o][down ? 3 : 1]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < KPT; ++c) {
        const int o = c ^ (1 << p), down = (c >> p) & 1;
        madd(y[c][down ? 0 : 1], g, a[o][down ? 1 : 0]);
        madd(y[c][down ? 2 : 3], g, a[o][down ? 3 : 2]);
      }
    }
  }
  // other spin-1/2 nuclei; above the lane bits the direction is the warp's
  unsigned rm = K.rad >> LK;
  const int nh = K.n_half;
  int bit = 1;
#pragma unroll LK == 1 ? 2 : 1
  for (int p = LK; p < nh; ++p, bit <<= 1, rm >>= 1) {
    const int sl = base + (t ^ bit), rr = (int)(rm & 1u);
    const bool down = (t & bit) != 0;
    const T g = K.g[p];
    if (bit >= 32) {
      if (down) flip_one<T, LK, false>(y, rr, g, cur, S, sl);
      else flip_one<T, LK, true>(y, rr, g, cur, S, sl);
    } else {
      flip_either<T, LK>(y, rr, down, g, cur, S, sl);
    }
  }
  if constexpr (CB > 0) {  // the nuclei that select the CTA
    if constexpr (kEarly) {
      peer_add<LK, CB>(y, pv, rank, rm, K.g + nh);
    } else {
      PeerVals<LK, CB> v;
      peer_load<LK, CB>(v, smem_u32(cur), rank, rm, S, base + t);
      peer_add<LK, CB>(y, v, rank, rm, K.g + nh);
    }
    rm >>= CB;
  }
  // spin-1 nuclei: digit j, up from j + 1, down from j - 1 (FP32: a missing
  // partner reads the own slot with weight zero)
  const int n0 = nh + CB, n1 = n0 + K.n_one;
  int st = bit;
#pragma unroll 1
  for (int p = n0; p < n1; ++p, st *= 3, rm >>= 1, dig >>= 2) {
    const unsigned j = dig & 3u;
    const int rr = (int)(rm & 1u);
    const T g = K.g[p];
    if constexpr (sizeof(T) == 4 && LK < 2) {  // both partners' loads before either product
      const int su = base + (j < 2u ? t + st : t), sd = base + (j > 0u ? t - st : t);
      const T gu = j < 2u ? g : T(0), gd = j > 0u ? g : T(0);
      Cx<T> u0[KPT], u1[KPT], d0[KPT], d1[KPT];
      Vec<T, LK>::get(cur, S, 0, su, u0);
      Vec<T, LK>::get(cur, S, rr ? 2 : 1, su, u1);
      Vec<T, LK>::get(cur, S, rr ? 1 : 2, sd, d0);
      Vec<T, LK>::get(cur, S, 3, sd, d1);
      if (rr == 0) {
#pragma unroll
        for (int c = 0; c < KPT; ++c) {
          madd(y[c][2], gu, u0[c]);
          madd(y[c][3], gu, u1[c]);
          madd(y[c][0], gd, d0[c]);
          madd(y[c][1], gd, d1[c]);
        }
      } else {
#pragma unroll
        for (int c = 0; c < KPT; ++c) {
          madd(y[c][1], gu, u0[c]);
          madd(y[c][3], gu, u1[c]);
          madd(y[c][0], gd, d0[c]);
          madd(y[c][2], gd, d1[c]);
        }
      }
    } else {
      if (sizeof(T) == 4 || j < 2u)
        flip_one<T, LK, true>(y, rr, j < 2u ? g : T(0), cur, S, base + (j < 2u ? t + st : t));
      if (sizeof(T) == 4 || j > 0u)
        flip_one<T, LK, false>(y, rr, j > 0u ? g : T(0), cur, S, base + (j > 0u ? t - st : t));
    }
  }
  // any other spin
  if (n1 < K.n_nuc) {
    unsigned q = (unsigned)t / (unsigned)K.st[n1];
#pragma unroll 1
    for (int p = n1; p < K.n_nuc; ++p) {
      const unsigned dd = (unsigned)K.d[p], j = q % dd;
      q /= dd;
      const int rr = (int)((K.rad >> p) & 1u), so = K.st[p];
      const T I = T(0.5) * T(dd - 1), M = I - T(j);
      if (j + 1u < dd)
        flip_one<T, LK, true>(y, rr, K.g[p] * sqrt(I * (I + 1) - M * (M - 1)), cur, S,
                              base + t + so);
      if (j > 0u)
        flip_one<T, LK, false>(y, rr, K.g[p] * sqrt(I * (I + 1) - M * (M + 1)), cur, S,
                               base + t - so);
    }
  }
  if (first) {  // phi_1 = H phi_0, half of the recurrence's sum
#pragma unroll
    for (int c = 0; c < KPT; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) y[c][e] = {T(0.5) * y[c][e].re, T(0.5) * y[c][e].im};
  } else if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      Cx<T> q[KPT];
      Vec<T, LK>::get(prev, S, e, base + t, q);
#pragma unroll
      for (int c = 0; c < KPT; ++c) y[c][e] = {y[c][e].re - q[c].re, y[c][e].im - q[c].im};
    }
  }
}

// psi(h) += r_n (-i)^n phi_n: r phi (n even) or -i r phi (n odd), r with the sign of
// n mod 4 >= 2; lo = r_n - fl(r_n).
template <typename T, int KPT, bool ODD>
__device__ __forceinline__ void chip_accumulate(Cx<T> (&acc)[KPT][4], const Cx<T> (&y)[KPT][4], T r,
                                                T lo) {
#pragma unroll
  for (int c = 0; c < KPT; ++c)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (ODD) {
        if (sizeof(T) == 4) madd_i(acc[c][e], -lo, y[c][e]);
        madd_i(acc[c][e], -r, y[c][e]);
      } else {
        if (sizeof(T) == 4) madd(acc[c][e], lo, y[c][e]);
        madd(acc[c][e], r, y[c][e]);
      }
    }
}

// Singlet slice <S|phi_n> = (phi_1 - phi_2) / sqrt 2 of the thread's configurations:
// entry c * xs of the row's slice n.
template <typename T, int KPT>
__device__ __forceinline__ void chip_singlet(T* x, int xs, const Cx<T> (&y)[KPT][4]) {
  const T r = T(0.70710678118654752440);
#pragma unroll
  for (int c = 0; c < KPT; ++c) {
    typename SliceVal<T>::type v;
    v.x = (y[c][1].re - y[c][2].re) * r;
    v.y = (y[c][1].im - y[c][2].im) * r;
    *reinterpret_cast<typename SliceVal<T>::type*>(x + (size_t)c * xs * 2) = v;
  }
}

// A macro-step of the thread's configurations: psi(t) in the thread's entries of
// buffer 0, on return psi(t + h) there (so nothing of the state is held in
// registers while the integral runs).  Threads without configurations (on =
// false) only keep the barriers.  xn: the thread's entry of the row's slices,
// stride between slices xstride (complex), between the thread's configurations
// xs.  Not inlined: the caller's live values would spill inside the term loop.
template <typename T, int LK, int CB>
__device__ __noinline__ void chip_macro(int S, int base, int t, bool on, unsigned dig,
                                        const T* __restrict__ cf, int n_c, T* xn, size_t xstride,
                                        int xs, bool store_x) {
  constexpr int KPT = 1 << LK;
  extern __shared__ __align__(16) unsigned char chip_smem[];
  const ChipConst<T>& K = *reinterpret_cast<const ChipConst<T>*>(chip_smem);
  Cx<T>* b0 = reinterpret_cast<Cx<T>*>(chip_smem + sizeof(ChipConst<T>));
  Cx<T>* b1 = b0 + (size_t)4 * KPT * S;
  const T* dt = reinterpret_cast<const T*>(b1 + (size_t)4 * KPT * S);
  const T* cl = cf + n_c;
  Cx<T> a[KPT][4], y[KPT][4], acc[KPT][4];
  if (on) {
    chip_get<T, LK>(b0, S, base + t, a);
    if (store_x) chip_singlet<T, KPT>(xn, xs, a);
#pragma unroll
    for (int c = 0; c < KPT; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[c][e] = {T(0), T(0)};
    chip_accumulate<T, KPT, false>(acc, a, cf[0], cl[0]);
  }
  chip_barrier<CB>();
#pragma unroll 1
  for (int n = 1; n < n_c; n += 2) {  // n_c is even: n odd, then n + 1 even
    if (on) {
      chip_term<T, LK, CB>(K, y, a, dt, b0, b1, n == 1, S, base, t, dig);
      chip_put<T, LK>(b1, S, base + t, y);
    }
    chip_arrive<CB>();
    if (on) {
      if (store_x) chip_singlet<T, KPT>(xn + (size_t)n * xstride * 2, xs, y);
      chip_accumulate<T, KPT, true>(acc, y, cf[n], cl[n]);
    }
    chip_wait<CB>();
    if (n + 1 < n_c) {
      if (on) {
        chip_term<T, LK, CB>(K, a, y, dt, b1, b0, false, S, base, t, dig);
        chip_put<T, LK>(b0, S, base + t, a);
      }
      chip_arrive<CB>();
      if (on) {
        if (store_x) chip_singlet<T, KPT>(xn + (size_t)(n + 1) * xstride * 2, xs, a);
        chip_accumulate<T, KPT, false>(acc, a, cf[n + 1], cl[n + 1]);
      }
      chip_wait<CB>();
    }
  }
  if (on) chip_put<T, LK>(b0, S, base + t, acc);
}

// Two-bit digits of the spin-1 nuclei of slot t.
__device__ __forceinline__ unsigned chip_digits(const HamDev<double>& H, int t, int lk, int cb) {
  unsigned q = (unsigned)t >> (H.n_half - cb - lk), dig = 0;
  for (int i = 0; i < H.n_one; ++i) {
    dig |= (q % 3u) << (2 * i);
    q /= 3u;
  }
  return dig;
}

// Most threads of a CTA, which bounds the registers: FP32 96 to 128, FP64 255 with
// several configurations per thread.
template <typename T>
__host__ __device__ constexpr int chip_max_threads(int lk) {
  if (sizeof(T) == 8) return lk == 0 ? 512 : 256;
  return lk == 1 ? 640 : 512;
}

// Survival and time-trace sums of a thread's configurations.
template <typename T, int KPT>
__device__ __forceinline__ double chip_norm(const Cx<T> (&a)[KPT][4]) {
  double s = 0.0;
#pragma unroll
  for (int c = 0; c < KPT; ++c)
#pragma unroll
    for (int e = 0; e < 4; ++e)
      s += (double)a[c][e].re * (double)a[c][e].re + (double)a[c][e].im * (double)a[c][e].im;
  return s;
}

// v += (P_S, norm, Re, Im <A_e x 1>) of one configuration (see k_trace).
template <typename T>
__device__ __forceinline__ void trace_terms(const Cx<T> (&a)[4], const ElecOp& A, double (&v)[4]) {
  const double dr = (double)a[1].re - (double)a[2].re, di = (double)a[1].im - (double)a[2].im;
  v[0] += 0.5 * (dr * dr + di * di);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const double cr = (double)a[e].re, ci = (double)a[e].im;
    v[1] += cr * cr + ci * ci;
    if (A.on) {
      double yr = 0.0, yi = 0.0;
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const double xr = (double)a[f].re, xi = (double)a[f].im;
        yr += A.re[4 * e + f] * xr - A.im[4 * e + f] * xi;
        yi += A.re[4 * e + f] * xi + A.im[4 * e + f] * xr;
      }
      v[2] += cr * yr + ci * yi;
      v[3] += cr * yi - ci * yr;
    }
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums over a block in a fixed order, so that equal calls give equal bits (atomics on
// shared memory add in the order in which the warps arrive).

// sums[2 row], sums[2 row + 1] of the rows of a block, a row's `per_row` threads side by
// side: thread i left its integral at p[i * step] and its norm at p[i * step + norm].  A
// warp per row, once per item.
__device__ __forceinline__ void row_sums(const double* p, int step, int norm, int rows,
                                         int per_row, double* sums, int tid) {
  const int lane = tid & 31, warps = (int)blockDim.x >> 5;
#pragma unroll 1
  for (int row = tid >> 5; row < rows; row += warps) {
    double a = 0.0, b = 0.0;
#pragma unroll 1
    for (int i = lane; i < per_row; i += 32) {
      const double* q = p + (row * per_row + i) * step;
      a += q[0];
      b += q[norm];
    }
    a = warp_sum(a);
    b = warp_sum(b);
    if (lane == 0) {
      sums[2 * row] = a;
      sums[2 * row + 1] = b;
    }
  }
}

// Scratch of trace_add: sums of the warps, then of the block (read by rank 0 of a cluster).
struct alignas(16) TraceSums {
  double warp[32][4], block[4];
};

// at[q] += the block's (cluster's) sum of v[q]: one addition per macro-step.  Every thread
// of the block calls it; the barriers of the next macro-step keep its scratch.
template <int CB>
__device__ __forceinline__ void trace_add(TraceSums& W, const double (&v)[4], int nq, double* at,
                                          int tid, unsigned rank) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (q >= nq) break;
    const double w = warp_sum(v[q]);
    if ((tid & 31) == 0) W.warp[tid >> 5][q] = w;
  }
  __syncthreads();
  double s = 0.0;
  if (tid < nq) {
#pragma unroll 1
    for (int k = 0; k < ((int)blockDim.x >> 5); ++k) s += W.warp[k][tid];
  }
  if constexpr (CB > 0) {
    if (tid < nq) W.block[tid] = s;
    chip_barrier<CB>();
    if (tid < nq && rank == 0)
      for (unsigned k = 1; k < (1u << CB); ++k) {
        double u;
        asm volatile("ld.shared::cluster.f64 %0, [%1];"
                     : "=d"(u)
                     : "r"(chip_peer(smem_u32(&W.block[tid]), k)));
        s += u;
      }
  }
  if (tid < nq && rank == 0) atomicAdd(at + tid, s);
}

// One launch over all items: CTAs take groups of up to rpc items of one field
// from a device counter and run their whole horizon.  Shared memory: two
// buffers of S slots (the second doubles as the integral's ring), the factor L,
// rows' sums.  The singlet slices of a macro-step
// go to the CTA's scratch and come back as the thread's own entries for the
// time integral (rp_integral.cu).
// MT, MB: most threads of a CTA and CTAs per SM, which bound the registers.  CB > 0: a
// row per cluster of 2^CB CTAs (rpc = 1), groups drawn by the cluster's rank 0.
template <typename T, int LK, int MT, int MB, int CB>
__global__ void __launch_bounds__(MT, MB) k_chip_items(
    const ChipArgs<T> A, const PItem* __restrict__ items, const int2* __restrict__ groups,
    int n_groups, int* __restrict__ counter, int rpc, int S, T* __restrict__ Xscratch, double* __restrict__ per_sample, double* __restrict__ trace,
    const ElecOp op) {
  constexpr int KPT = 1 << LK, KB = ProjCfg<T>::kB;
  extern __shared__ __align__(16) unsigned char chip_smem[];
  __shared__ int s_group;
  __shared__ TraceSums s_trace;
  ChipConst<T>& K = *reinterpret_cast<ChipConst<T>*>(chip_smem);
  Cx<T>* buf = reinterpret_cast<Cx<T>*>(chip_smem + sizeof(ChipConst<T>));
  T* dt = reinterpret_cast<T*>(buf + (size_t)8 * KPT * S);  // diagonals [KPT][S][4]
  T* sl = dt + (size_t)4 * KPT * S;
  double* sums = reinterpret_cast<double*>(sl + (size_t)A.n_c * KB);  // [rpc][2]
  double* amps = sums + 2 * rpc;                                      // [rpc][max_nuc][20]
  // the integral's ring: buffer 1, 4 KPT slices per thread
  auto* ring = reinterpret_cast<typename SliceVal<T>::type*>(buf + (size_t)4 * KPT * S) + threadIdx.x;
  const int tid = threadIdx.x;
  const unsigned rank = CB > 0 ? chip_rank() : 0u;
  constexpr int cb = CB;
  T* xc = Xscratch + (size_t)blockIdx.x * A.n_c * KPT * S * 2;
  for (;;) {
    // rank 0 draws the group for its cluster
    if (tid == 0 && rank == 0) s_group = atomicAdd(counter, 1);
    chip_barrier<CB>();
    int gi = s_group;
    if constexpr (CB > 0) {
      asm volatile("ld.shared::cluster.s32 %0, [%1];"
                   : "=r"(gi)
                   : "r"(chip_peer(smem_u32(&s_group), 0)));
    }
    if (gi >= n_groups) break;  // the same for the whole CTA (cluster)
    const int2 grp = groups[gi];
    const PItem I0 = items[grp.x];
    const HamDev<double>& H = A.ham[I0.sys];
    const FieldDev<double> F = A.fields[I0.field];
    const int Sr = (int)(H.Z >> (LK + cb));
    const int row = tid / Sr, t = tid - row * Sr, base = row * Sr;
    const bool on = row < grp.y;
    chip_const<T>(K, H, F, LK, cb, tid);
    const LayoutDev& Ly = A.lay[I0.sys];
    if (!A.deterministic)
      for (int q = tid; q < grp.y * Ly.n_nuc; q += blockDim.x) {
        const int r = q / Ly.n_nuc, p = q % Ly.n_nuc;
        double u[2];
        const uint32_t pair = A.pair_of ? A.pair_of[I0.sys] : A.pair_base + (uint32_t)I0.sys;
        coherent_amp(Ly, p, pair, (unsigned long long)items[grp.x + r].sample, A.seed,
                     amps + ((size_t)r * A.max_nuc + p) * 20, u);
      }
    __syncthreads();
    unsigned dig = 0;
    if (on) {
      Cx<T> a[KPT][4];
      dig = chip_digits(H, t, LK, cb);
      const long long sample = items[grp.x + row].sample;
#pragma unroll
      for (int c = 0; c < KPT; ++c) {
        const unsigned l = ((unsigned)t << LK) | (unsigned)c;
        const int lb = H.n_half - cb;
        const unsigned m = CB > 0 ? (((l >> lb) << (lb + cb)) | (rank << lb) | (l & ((1u << lb) - 1u))) : l;
        T d[4];
        chip_diag<T>(H, F, m, d);
#pragma unroll
        for (int e = 0; e < 4; ++e) dt[((size_t)c * S + base + t) * 4 + e] = d[e];
        double pr = 1.0, pi = 0.0;
        if (A.deterministic == 3) {
          pr = A.sec_rank[m] == sample ? A.sec_scale[sample] : 0.0;
        } else if (A.deterministic) {
          pr = (long long)m == sample ? 1.0 : 0.0;
        } else {
          unsigned q = m;
          const double* am = amps + (size_t)row * A.max_nuc * 20;
          for (int p = 0; p < Ly.n_nuc; ++p) {
            const unsigned dd = (unsigned)Ly.d[p], j = q % dd;
            q /= dd;
            const double ar = am[p * 20 + 2 * j], ai = am[p * 20 + 2 * j + 1];
            const double nr = pr * ar - pi * ai;
            pi = pr * ai + pi * ar;
            pr = nr;
          }
        }
        const double s = 0.70710678118654752440;
        a[c][0] = a[c][3] = {T(0), T(0)};
        a[c][1] = {(T)(s * pr), (T)(s * pi)};
        a[c][2] = {(T)(-s * pr), (T)(-s * pi)};
      }
      chip_put<T, LK>(buf, S, base + t, a);
    }
    const T* cf = A.coef + (size_t)I0.field * 2 * A.n_c;
    const bool integrate = trace == nullptr;
    int2 mt = make_int2(0, 0);
    const T* Lf = nullptr;
    if (integrate) {
      mt = A.meta[I0.field];
      Lf = A.L + (size_t)I0.field * A.n_c * A.ldk;
      if (mt.x <= KB) stage_factor<T>(sl, Lf, A.ldk, (mt.y + 1) & ~1, 0, tid, blockDim.x);
    }
    const int n_e = (mt.y + 1) & ~1;
    double integral = 0.0;
    const size_t xrow = (size_t)KPT * S;
#pragma unroll 1
    for (int km = 0; km < I0.n_macro; ++km) {
      chip_macro<T, LK, CB>(S, base, t, on, dig, cf, A.n_c, xc + (size_t)(base + t) * 2,
                        xrow, S, integrate);
      if (integrate) {
        for (int k0 = 0; k0 < mt.x; k0 += KB) {
          if (mt.x > KB) {  // several blocks of columns: staged in turn
            __syncthreads();
            stage_factor<T>(sl, Lf, A.ldk, n_e, k0, tid, blockDim.x);
            __syncthreads();
          }
          if (on) {
#pragma unroll 1
            for (int c = 0; c < KPT; ++c) {
              typename ProjAcc<T>::type yr[1][16], yi[1][16];
              const T* const p[1] = {xc + ((size_t)c * S + base + t) * 2};
              project_block<T, 1, 4, KPT>(yr, yi, p, xrow * 2, sl, KB, n_e, ring, S);
              integral += proj_norm(yr[0], yi[0]);
            }
          }
        }
      } else {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        if (on) {
          Cx<T> a[KPT][4];
          chip_get<T, LK>(buf, S, base + t, a);
#pragma unroll
          for (int c = 0; c < KPT; ++c) trace_terms<T>(a[c], op, v);
        }
        trace_add<CB>(s_trace, v, op.on ? 4 : 2, trace + 4 * (km + 1), tid, rank);
      }
    }
    // integral and norm to the thread's own entries of the ring, which it is done with
    constexpr int kStep = (int)(sizeof(typename SliceVal<T>::type) / sizeof(double));
    if (on) {
      Cx<T> a[KPT][4];
      chip_get<T, LK>(buf, S, base + t, a);
      double* own = reinterpret_cast<double*>(ring);
      own[0] = integral;
      own[kStep * S] = chip_norm<T, KPT>(a);
    }
    __syncthreads();
    row_sums(reinterpret_cast<const double*>(buf + (size_t)4 * KPT * S), kStep, kStep * S, grp.y, Sr,
             sums, tid);
    chip_barrier<CB>();
    if (tid < grp.y && rank == 0) {
      double si = sums[2 * tid], surv = sums[2 * tid + 1];
      if constexpr (CB > 0) {
        for (unsigned k = 1; k < (1u << cb); ++k) {
          const unsigned a = chip_peer(smem_u32(&sums[2 * tid]), k);
          double u, v;
          asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(u), "=d"(v) : "r"(a));
          si += u;
          surv += v;
        }
      }
      const double phS = A.k_S[I0.sys] * si;
      double* o = per_sample + items[grp.x + tid].out * 3;
      o[0] = phS;
      o[1] = 1.0 - surv - phS;  // Haberkorn: d|psi|^2/dt = -k_S <P_S> - k_T <P_T>
      o[2] = surv;
    }
    __syncthreads();
  }
  if constexpr (CB > 0) chip_barrier<CB>();  // no CTA leaves while a peer may read its memory
}

// ---- few configurations per SM: one thread per configuration and electron state ----
//
// With fewer than about 256 configurations per SM the length of a thread's
// chain of dependent instructions decides, in FP64 most of all (a warp's FP64
// instruction holds its scheduler's unit for 64 cycles).  A row then takes 4 Z
// threads.  A thread's row of H has at most one partner per nucleus (an
// isotropic coupling brings each electron state either the configuration above
// or the one below), so offsets and weights of the whole horizon sit in
// registers and a term is one shared-memory read and one packed multiply-add
// per nucleus.  The slices of the macro-step stay in shared memory too, and
// the integral's 32 columns are spread over the four threads of a
// configuration.  The sums run in chip_term's order: results do not depend on
// which of the two kernels ran.
constexpr int kSplitNuc = 8;  // Z <= 256
template <typename T>
__host__ __device__ constexpr int split_max_threads() {
  return sizeof(T) == 4 ? 1024 : 768;
}

template <typename T>
struct SplitRow {
  T w[kSplitNuc];     // couplings (weight zero where there is no partner)
  int off[kSplitNuc];  // entry of the partner in a buffer
  T d;                // diagonal (as chip_term forms it)
  int own;            // entry of state 3 - e of the own configuration
  int src;            // entry of the state kappa couples to (e for 0 and 3, else own)
};

// y (phi_{n-2}) becomes phi_n; a = phi_{n-1} of this thread.
template <typename T>
__device__ __forceinline__ void split_term(const SplitRow<T>& R, int n_nuc, T J, T kp, bool mid,
                                           Cx<T>& y, const Cx<T>& a, const Cx<T>* cur) {
  Cx<T> q[kSplitNuc];
#pragma unroll
  for (int p = 0; p < kSplitNuc; ++p)
    if (p < n_nuc) q[p] = cur[R.off[p]];
  Cx<T> u;
  if (sizeof(T) == 4) u = {R.d * a.re, R.d * a.im};
  else u = {fma(R.d, a.re, -y.re), fma(R.d, a.im, -y.im)};
  if (J != T(0) && mid) madd_s(u, J, cur[R.own]);
  if (kp != T(0)) madd_i(u, kp, cur[R.src]);
#pragma unroll
  for (int p = 0; p < kSplitNuc; ++p)
    if (p < n_nuc) madd_s(u, R.w[p], q[p]);
  if (sizeof(T) == 4) y = {u.re - y.re, u.im - y.im};
  else y = u;
}

// MT: most threads of the launch (small CTAs keep more in registers)
template <typename T, int MT>
__global__ void __launch_bounds__(MT, 1) k_split_items(
    const ChipArgs<T> A, const PItem* __restrict__ items, const int2* __restrict__ groups,
    int n_groups, int* __restrict__ counter, int rpc, int S, double* __restrict__ per_sample,
    double* __restrict__ trace, const ElecOp op) {
  extern __shared__ __align__(16) unsigned char chip_smem[];
  __shared__ int s_group;
  __shared__ TraceSums s_trace;
  // two buffers [e][S], slices [n_c][S], factor [n_c][32], sums, amplitudes
  Cx<T>* buf = reinterpret_cast<Cx<T>*>(chip_smem);
  Cx<T>* xs = buf + (size_t)8 * S;
  T* sl = reinterpret_cast<T*>(xs + (trace ? 0 : (size_t)A.n_c * S));
  double* sums = reinterpret_cast<double*>(sl + (trace ? 0 : (size_t)A.n_c * 32));
  double* amps = sums + 2 * rpc;
  const int tid = threadIdx.x;
  for (;;) {
    if (tid == 0) s_group = atomicAdd(counter, 1);
    __syncthreads();
    const int gi = s_group;
    if (gi >= n_groups) break;  // the same for the whole CTA
    const int2 grp = groups[gi];
    const PItem I0 = items[grp.x];
    const HamDev<double>& H = A.ham[I0.sys];
    const FieldDev<double> F = A.fields[I0.field];
    const int Z = (int)H.Z, n_nuc = H.n_nuc;
    const int row = tid / (4 * Z), e = (tid - row * 4 * Z) / Z, m = tid % Z;
    const int slot = row * Z + m;  // 4 Z is a multiple of Z
    const bool on = row < grp.y;
    const LayoutDev& Ly = A.lay[I0.sys];
    if (!A.deterministic)
      for (int q = tid; q < grp.y * Ly.n_nuc; q += blockDim.x) {
        const int r = q / Ly.n_nuc, p = q % Ly.n_nuc;
        double u[2];
        const uint32_t pair = A.pair_of ? A.pair_of[I0.sys] : A.pair_base + (uint32_t)I0.sys;
        coherent_amp(Ly, p, pair, (unsigned long long)items[grp.x + r].sample, A.seed,
                     amps + ((size_t)r * A.max_nuc + p) * 20, u);
      }
    const T* cf = A.coef + (size_t)I0.field * 2 * A.n_c;
    const T* cl = cf + A.n_c;
    int2 mt = make_int2(0, 0);
    const T* Lf = nullptr;
    if (!trace) {
      mt = A.meta[I0.field];
      Lf = A.L + (size_t)I0.field * A.n_c * A.ldk;
      if (mt.x <= 32) stage_factor<T, 32>(sl, Lf, A.ldk, (mt.y + 1) & ~1, 0, tid, blockDim.x);
    }
    const int n_e = (mt.y + 1) & ~1;
    SplitRow<T> R;
    const T J = (T)(2.0 * F.s * H.Je), kp = (T)(2.0 * F.s * H.kappa);
    const bool mid = e == 1 || e == 2;
    Cx<T> a = {T(0), T(0)};
    __syncthreads();
    if (on) {
      T d4[4];
      chip_diag<T>(H, F, (unsigned)m, d4);
      R.d = e == 0 ? d4[0] : e == 1 ? d4[1] : e == 2 ? d4[2] : d4[3];
      R.own = (3 - e) * S + slot;
      R.src = mid ? R.own : e * S + slot;
      unsigned q = (unsigned)m;
#pragma unroll
      for (int p = 0; p < kSplitNuc; ++p) {
        R.w[p] = T(0);
        R.off[p] = e * S + slot;
        if (p < n_nuc) {
          const unsigned dd = (unsigned)H.d[p], j = q % dd;
          q /= dd;
          const int flip = H.rad[p] == 0 ? 2 : 1, st = (int)H.stride[p];
          const bool up = (e & flip) != 0;  // S_- I_+ from j + 1, else S_+ I_- from j - 1
          if (up ? j + 1u < dd : j > 0u) {
            double g = 2.0 * F.s * H.U[p][4];
            if (dd == 3) g *= 1.41421356237309504880;
            R.w[p] = (T)g;
            if (dd > 3) {
              const T I = T(0.5) * T(dd - 1), M = I - T(j);
              R.w[p] *= up ? sqrt(I * (I + 1) - M * (M - 1)) : sqrt(I * (I + 1) - M * (M + 1));
            }
            R.off[p] = (e ^ flip) * S + slot + (up ? st : -st);
          }
        }
      }
      // psi(0) of this thread's state
      double pr = 1.0, pi = 0.0;
      const long long sample = items[grp.x + row].sample;
      if (A.deterministic == 3) {
        pr = A.sec_rank[m] == sample ? A.sec_scale[sample] : 0.0;
      } else if (A.deterministic) {
        pr = (long long)m == sample ? 1.0 : 0.0;
      } else {
        unsigned qq = (unsigned)m;
        const double* am = amps + (size_t)row * A.max_nuc * 20;
        for (int p = 0; p < Ly.n_nuc; ++p) {
          const unsigned dd = (unsigned)Ly.d[p], j = qq % dd;
          qq /= dd;
          const double ar = am[p * 20 + 2 * j], ai = am[p * 20 + 2 * j + 1];
          const double nr = pr * ar - pi * ai;
          pi = pr * ai + pi * ar;
          pr = nr;
        }
      }
      const double s = e == 1 ? 0.70710678118654752440 : -0.70710678118654752440;
      if (mid) a = {(T)(s * pr), (T)(s * pi)};
    }
    double integral = 0.0;
    Cx<T>* b0 = buf + (size_t)e * S + slot;  // this thread's entries
    Cx<T>* b1 = b0 + (size_t)4 * S;
    const bool keeps = !trace && on && e == 0;  // stores the slices
    // slice n from the buffer holding phi_n, by the threads of state 0
    auto slice = [&](int n, const Cx<T>* b) {
      const Cx<T> p1 = b[S + slot], p2 = b[2 * S + slot];
      const T r = T(0.70710678118654752440);
      xs[(size_t)n * S + slot] = {(p1.re - p2.re) * r, (p1.im - p2.im) * r};
    };
#pragma unroll 1
    for (int km = 0; km < I0.n_macro; ++km) {
      Cx<T> y = {T(0), T(0)}, acc = {T(0), T(0)};
      if (on) {
        *b0 = a;
        if (sizeof(T) == 4) madd_s(acc, cl[0], a);
        madd_s(acc, cf[0], a);
      }
      __syncthreads();
#pragma unroll 1
      for (int n = 1; n < A.n_c; n += 2) {
        if (on) {
          split_term<T>(R, n_nuc, J, kp, mid, y, a, buf);
          if (n == 1) {
            y.re *= T(0.5);
            y.im *= T(0.5);
          }
          *b1 = y;
          if (keeps) slice(n - 1, buf);
          if (sizeof(T) == 4) madd_i(acc, -cl[n], y);
          madd_i(acc, -cf[n], y);
        }
        __syncthreads();
        if (n + 1 < A.n_c) {
          if (on) {
            split_term<T>(R, n_nuc, J, kp, mid, a, y, buf + (size_t)4 * S);
            *b0 = a;
            if (keeps) slice(n, buf + (size_t)4 * S);
            if (sizeof(T) == 4) madd_s(acc, cl[n + 1], a);
            madd_s(acc, cf[n + 1], a);
          }
          __syncthreads();
        }
      }
      a = acc;
      if (!trace) {
        if (keeps) slice(A.n_c - 1, buf + (size_t)4 * S);  // n_c is even: the last n is odd
        __syncthreads();
        for (int k0 = 0; k0 < mt.x; k0 += 32) {
          if (mt.x > 32) {  // several blocks of columns: staged in turn
            __syncthreads();
            stage_factor<T, 32>(sl, Lf, A.ldk, n_e, k0, tid, blockDim.x);
            __syncthreads();
          }
          if (on) {
            constexpr int N = sizeof(T) == 4 ? 4 : 8;  // eight columns
            typename ProjAcc<T>::type yr[N], yi[N];
#pragma unroll
            for (int k = 0; k < N; ++k) yr[k] = yi[k] = typename ProjAcc<T>::type{};
            const T* l = sl + 8 * e;
#pragma unroll 2
            for (int n = 0; n < n_e; n += 2) {
              const Cx<T> v = xs[(size_t)n * S + slot], u = xs[(size_t)(n + 1) * S + slot];
              proj_add(yr, yi, l + n * 32, v.re, v.im);
              proj_add(yr, yi, l + (n + 1) * 32, u.im, -u.re);
            }
            integral += proj_norm8(yr, yi);
          }
        }
      } else {
        // every state of the configuration for the observables: psi(t + h) once more
        __syncthreads();
        if (on) *b0 = a;
        __syncthreads();
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        if (on && e == 0) {
          const Cx<T> c4[4] = {buf[slot], buf[S + slot], buf[2 * S + slot], buf[3 * S + slot]};
          trace_terms<T>(c4, op, v);
        }
        trace_add<0>(s_trace, v, op.on ? 4 : 2, trace + 4 * (km + 1), tid, 0u);
      }
    }
    double* part = reinterpret_cast<double*>(buf);  // psi is in registers
    __syncthreads();
    if (on) {
      part[2 * tid] = integral;
      part[2 * tid + 1] = (double)a.re * (double)a.re + (double)a.im * (double)a.im;
    }
    __syncthreads();
    row_sums(part, 2, 1, grp.y, 4 * Z, sums, tid);
    __syncthreads();
    if (tid < grp.y) {
      const double phS = A.k_S[I0.sys] * sums[2 * tid], surv = sums[2 * tid + 1];
      double* o = per_sample + items[grp.x + tid].out * 3;
      o[0] = phS;
      o[1] = 1.0 - surv - phS;
      o[2] = surv;
    }
    __syncthreads();
  }
}

// ---- anisotropic systems: one thread per configuration and electron state ----
//
// The same for tensors of any form, in rotated nuclear frames (rp_plan.cpp,
// nuclear_frame): U = [[0, u], [w, 0]] with w real, so each electron state takes
// one component of each partner.  A row is split over 2^CB CTAs by the outermost
// spin-1/2 nuclei where rows are few (in FP64 the chip's 304 FP64 lanes are the
// bound, and 32 rows on 32 SMs leave most of them idle) or long.
template <typename T>
struct alignas(16) AnisoConst {
  T w[kMaxNucDev], ur[kMaxNucDev], ui[kMaxNucDev];  // 2/dE folded in, x sqrt 2 for spin 1
  int d[kMaxNucDev], st[kMaxNucDev];
  T J, kappa;
  unsigned rad;
  int lb, n_nuc;  // spin-1/2 nuclei of the CTA's own slots, all nuclei
};

template <typename T>
struct AnisoRow {
  T d;                   // diagonal
  T c2r, c2i, c1r, c1i;  // couplings to states e ^ 2 and e ^ 1 of the own configuration
};

// u += (wr + i wi) q
template <typename T>
__device__ __forceinline__ void madd_c(Cx<T>& u, T wr, T wi, const Cx<T>& q) {
  u.re = fma(wr, q.re, fma(-wi, q.im, u.re));
  u.im = fma(wr, q.im, fma(wi, q.re, u.im));
}

__device__ __forceinline__ Cx<float> peer_value(unsigned a, float) {
  Cx<float> v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.re), "=f"(v.im) : "r"(a));
  return v;
}
__device__ __forceinline__ Cx<double> peer_value(unsigned a, double) {
  Cx<double> v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.re), "=d"(v.im) : "r"(a));
  return v;
}

// y (phi_{n-2}) becomes phi_n; a = phi_{n-1} of this thread, l its local configuration.
template <typename T, int CB>
__device__ __forceinline__ void aniso_term(const AnisoConst<T>& K, const AnisoRow<T>& R, Cx<T>& y,
                                           const Cx<T>& a, const Cx<T>* cur, int S, int slot, int l,
                                           int e, unsigned rank) {
  Cx<T> pv[CB > 0 ? CB : 1];
#pragma unroll
  for (int i = 0; i < CB; ++i) {  // remote values first: they take longest
    const int flip = ((K.rad >> (K.lb + i)) & 1u) ? 1 : 2;
    pv[i] = peer_value(chip_peer(smem_u32(cur + (e ^ flip) * S + slot), rank ^ (1u << i)), T(0));
  }
  Cx<T> u;
  if (sizeof(T) == 4) u = {R.d * a.re, R.d * a.im};
  else u = {fma(R.d, a.re, -y.re), fma(R.d, a.im, -y.im)};
  madd_c(u, R.c2r, R.c2i, cur[(e ^ 2) * S + slot]);
  madd_c(u, R.c1r, R.c1i, cur[(e ^ 1) * S + slot]);
  const bool mid = e == 1 || e == 2;
  if (K.J != T(0) && mid) madd_s(u, K.J, cur[(3 - e) * S + slot]);
  if (K.kappa != T(0)) madd_i(u, K.kappa, mid ? cur[(3 - e) * S + slot] : a);
  // low states (electron up) take the high ones through u (partner above) or w
  // (below), high states the low ones through w or conj(u)
  auto add = [&](int p, bool hi, bool down, T f, const Cx<T>& q) {
    const bool c = hi == down;
    const T ui = K.ui[p];
    madd_c(u, f * (c ? K.ur[p] : K.w[p]), c ? (hi ? -f * ui : f * ui) : T(0), q);
  };
  unsigned rm = K.rad;
#pragma unroll 2
  for (int p = 0; p < K.lb; ++p, rm >>= 1) {
    const int flip = (rm & 1u) ? 1 : 2;
    const bool down = (l >> p) & 1;
    add(p, (e & flip) != 0, down, T(1), cur[(e ^ flip) * S + (slot ^ (1 << p))]);
  }
#pragma unroll
  for (int i = 0; i < CB; ++i, rm >>= 1) {
    const int flip = (rm & 1u) ? 1 : 2;
    add(K.lb + i, (e & flip) != 0, (rank >> i) & 1u, T(1), pv[i]);
  }
  unsigned q = (unsigned)l >> K.lb;
#pragma unroll 1
  for (int p = K.lb + CB; p < K.n_nuc; ++p, rm >>= 1) {
    const unsigned dd = (unsigned)K.d[p], j = dd == 3u ? q % 3u : q % dd;
    q = dd == 3u ? q / 3u : q / dd;
    const int flip = (rm & 1u) ? 1 : 2, st = K.st[p];
    const bool hi = (e & flip) != 0;
    T fu = T(1), fd = T(1);
    if (dd != 3u) {
      const T I = T(0.5) * T(dd - 1), M = I - T(j);
      fu = sqrt(I * (I + 1) - M * (M - 1));
      fd = sqrt(I * (I + 1) - M * (M + 1));
    }
    if (j + 1u < dd) add(p, hi, false, fu, cur[(e ^ flip) * S + slot + st]);
    if (j > 0u) add(p, hi, true, fd, cur[(e ^ flip) * S + slot - st]);
  }
  if (sizeof(T) == 4) y = {u.re - y.re, u.im - y.im};
  else y = u;
}

template <typename T, int CB, int MT>
__global__ void __launch_bounds__(MT, CB == 0 && MT == 256 ? 2 : 1) k_split_aniso(
    const ChipArgs<T> A, const PItem* __restrict__ items, const int2* __restrict__ groups,
    int n_groups, int* __restrict__ counter, int S, double* __restrict__ per_sample,
    double* __restrict__ trace, const ElecOp op) {
  extern __shared__ __align__(16) unsigned char chip_smem[];
  __shared__ int s_group;
  __shared__ TraceSums s_trace;
  __shared__ __align__(16) double sums[2];
  __shared__ AnisoConst<T> K;
  // two buffers [e][S], slices [n_c][S], factor [n_c][32], amplitudes
  Cx<T>* buf = reinterpret_cast<Cx<T>*>(chip_smem);
  Cx<T>* xs = buf + (size_t)8 * S;
  T* sl = reinterpret_cast<T*>(xs + (trace ? 0 : (size_t)A.n_c * S));
  double* amps = reinterpret_cast<double*>(sl + (trace ? 0 : (size_t)A.n_c * 32));
  const int tid = threadIdx.x;
  const unsigned rank = CB > 0 ? chip_rank() : 0u;
  for (;;) {
    if (tid == 0 && rank == 0) s_group = atomicAdd(counter, 1);
    chip_barrier<CB>();
    int gi = s_group;
    if constexpr (CB > 0) {
      asm volatile("ld.shared::cluster.s32 %0, [%1];"
                   : "=r"(gi)
                   : "r"(chip_peer(smem_u32(&s_group), 0)));
    }
    if (gi >= n_groups) break;  // the same for the whole cluster
    const PItem I0 = items[groups[gi].x];
    const HamDev<double>& H = A.ham[I0.sys];
    const FieldDev<double> F = A.fields[I0.field];
    const LayoutDev& Ly = A.lay[I0.sys];
    const int Zl = (int)(H.Z >> CB), lb = H.n_half - CB;
    const int e = tid / Zl, l = tid - e * Zl;
    const bool on = e < 4;
    const unsigned m = CB > 0 ? (((unsigned)l >> lb) << (lb + CB)) | (rank << lb) |
                                    ((unsigned)l & ((1u << lb) - 1u))
                              : (unsigned)l;
    if (tid < H.n_nuc) {
      const int p = tid;
      const double c = 2.0 * F.s * (H.d[p] == 3 ? 1.41421356237309504880 : 1.0);
      K.w[p] = (T)(c * H.U[p][4]);
      K.ur[p] = (T)(c * H.U[p][2]);
      K.ui[p] = (T)(c * H.U[p][3]);
      K.d[p] = H.d[p];
      K.st[p] = (int)(H.stride[p] >> CB);
      // amplitudes of psi(0) in the rotated frames (Eqs. 15, 17)
      double in[20], u[2];
      if (A.deterministic) {
        const int j = (int)((I0.sample / Ly.stride[p]) % Ly.d[p]);
        for (int q = 0; q < 2 * Ly.d[p]; ++q) in[q] = q == 2 * j ? 1.0 : 0.0;
      } else {
        const uint32_t pair = A.pair_of ? A.pair_of[I0.sys] : A.pair_base + (uint32_t)I0.sys;
        coherent_amp(Ly, p, pair, (unsigned long long)I0.sample, A.seed, in, u);
      }
      const int dn = Ly.d[p];
      const double* D = A.frame + ((size_t)I0.sys * kMaxNucDev + p) * 200;
      for (int i = 0; i < dn; ++i) {
        double re = 0.0, im = 0.0;
        for (int j = 0; j < dn; ++j) {
          const double dr = D[2 * (i * dn + j)], di = D[2 * (i * dn + j) + 1];
          re += dr * in[2 * j] - di * in[2 * j + 1];
          im += dr * in[2 * j + 1] + di * in[2 * j];
        }
        amps[p * 20 + 2 * i] = re;
        amps[p * 20 + 2 * i + 1] = im;
      }
    }
    if (tid == 0) {
      K.J = (T)(2.0 * F.s * H.Je);
      K.kappa = (T)(2.0 * F.s * H.kappa);
      unsigned rd = 0;
      for (int p = 0; p < H.n_nuc; ++p) rd |= (unsigned)(H.rad[p] & 1) << p;
      K.rad = rd;
      K.lb = lb;
      K.n_nuc = H.n_nuc;
    }
    const T* cf = A.coef + (size_t)I0.field * 2 * A.n_c;
    const T* cl = cf + A.n_c;
    int2 mt = make_int2(0, 0);
    const T* Lf = nullptr;
    if (!trace) {
      mt = A.meta[I0.field];
      Lf = A.L + (size_t)I0.field * A.n_c * A.ldk;
      if (mt.x <= 32) stage_factor<T, 32>(sl, Lf, A.ldk, (mt.y + 1) & ~1, 0, tid, blockDim.x);
    }
    const int n_e = (mt.y + 1) & ~1;
    __syncthreads();
    AnisoRow<T> R{};
    Cx<T> a = {T(0), T(0)};
    if (on) {
      double b[2][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
      double pr = 1.0, pi = 0.0;
      unsigned q = m;
      for (int p = 0; p < H.n_nuc; ++p) {
        const unsigned dd = (unsigned)H.d[p], j = q % dd;
        q /= dd;
        const double M = 0.5 * (double)(dd - 1) - (double)j;
        for (int k = 0; k < 3; ++k) {
          if (H.rad[p] == 0) b[0][k] += M * H.v[p][k];
          else b[1][k] += M * H.v[p][k];
        }
        const double ar = amps[p * 20 + 2 * j], ai = amps[p * 20 + 2 * j + 1];
        const double nr = pr * ar - pi * ai;
        pi = pr * ai + pi * ar;
        pr = nr;
      }
      const double sp = 0.5 * (b[0][2] + b[1][2]), sm = 0.5 * (b[0][2] - b[1][2]);
      const double hJ = 0.5 * H.Je;
      const double dz = e == 0 ? F.omega + hJ + sp : e == 1 ? -hJ + sm : e == 2 ? -hJ - sm
                                                                              : -F.omega + hJ - sp;
      R.d = (T)(2.0 * (F.s * dz - F.sh_re));
      // S_1 . b_1 and S_2 . b_2 off the diagonal: (b_x -+ i b_y) / 2
      R.c2r = (T)(F.s * b[0][0]);
      R.c2i = (T)(F.s * ((e & 2) ? b[0][1] : -b[0][1]));
      R.c1r = (T)(F.s * b[1][0]);
      R.c1i = (T)(F.s * ((e & 1) ? b[1][1] : -b[1][1]));
      const double s = e == 1 ? 0.70710678118654752440 : -0.70710678118654752440;
      if (e == 1 || e == 2) a = {(T)(s * pr), (T)(s * pi)};
    }
    double integral = 0.0;
    Cx<T>* b0 = buf + (size_t)(on ? e : 0) * S + l;  // this thread's entries
    Cx<T>* b1 = b0 + (size_t)4 * S;
    const bool keeps = !trace && on && e == 0;  // stores the slices
    auto slice = [&](int n, const Cx<T>* b) {
      const Cx<T> p1 = b[S + l], p2 = b[2 * S + l];
      const T r = T(0.70710678118654752440);
      xs[(size_t)n * S + l] = {(p1.re - p2.re) * r, (p1.im - p2.im) * r};
    };
#pragma unroll 1
    for (int km = 0; km < I0.n_macro; ++km) {
      Cx<T> y = {T(0), T(0)}, acc = {T(0), T(0)};
      if (on) {
        *b0 = a;
        if (sizeof(T) == 4) madd_s(acc, cl[0], a);
        madd_s(acc, cf[0], a);
      }
      chip_barrier<CB>();
#pragma unroll 1
      for (int n = 1; n < A.n_c; n += 2) {
        if (on) {
          aniso_term<T, CB>(K, R, y, a, buf, S, l, l, e, rank);
          if (n == 1) {
            y.re *= T(0.5);
            y.im *= T(0.5);
          }
          *b1 = y;
        }
        chip_arrive<CB>();
        if (on) {
          if (keeps) slice(n - 1, buf);
          if (sizeof(T) == 4) madd_i(acc, -cl[n], y);
          madd_i(acc, -cf[n], y);
        }
        chip_wait<CB>();
        if (n + 1 < A.n_c) {
          if (on) {
            aniso_term<T, CB>(K, R, a, y, buf + (size_t)4 * S, S, l, l, e, rank);
            *b0 = a;
          }
          chip_arrive<CB>();
          if (on) {
            if (keeps) slice(n, buf + (size_t)4 * S);
            if (sizeof(T) == 4) madd_s(acc, cl[n + 1], a);
            madd_s(acc, cf[n + 1], a);
          }
          chip_wait<CB>();
        }
      }
      a = acc;
      if (!trace) {
        if (keeps) slice(A.n_c - 1, buf + (size_t)4 * S);  // n_c is even: the last n is odd
        __syncthreads();
        for (int k0 = 0; k0 < mt.x; k0 += 32) {
          if (mt.x > 32) {  // several blocks of columns: staged in turn
            __syncthreads();
            stage_factor<T, 32>(sl, Lf, A.ldk, n_e, k0, tid, blockDim.x);
            __syncthreads();
          }
          if (on) {
            constexpr int N = sizeof(T) == 4 ? 4 : 8;  // eight columns
            typename ProjAcc<T>::type yr[N], yi[N];
#pragma unroll
            for (int k = 0; k < N; ++k) yr[k] = yi[k] = typename ProjAcc<T>::type{};
            const T* lc = sl + 8 * e;
#pragma unroll 2
            for (int n = 0; n < n_e; n += 2) {
              const Cx<T> v = xs[(size_t)n * S + l], w = xs[(size_t)(n + 1) * S + l];
              proj_add(yr, yi, lc + n * 32, v.re, v.im);
              proj_add(yr, yi, lc + (n + 1) * 32, w.im, -w.re);
            }
            integral += proj_norm8(yr, yi);
          }
        }
      } else {
        // every state of the configuration for the observables: psi(t + h) once more
        // (no peer reads buffer 0 after the last barrier)
        if (on) *b0 = a;
        __syncthreads();
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        if (on && e == 0) {
          const Cx<T> c4[4] = {buf[l], buf[S + l], buf[2 * S + l], buf[3 * S + l]};
          trace_terms<T>(c4, op, v);
        }
        trace_add<CB>(s_trace, v, op.on ? 4 : 2, trace + 4 * (km + 1), tid, rank);
        __syncthreads();
      }
    }
    double* part = reinterpret_cast<double*>(buf);  // psi is in registers
    __syncthreads();
    if (on) {
      part[2 * tid] = integral;
      part[2 * tid + 1] = (double)a.re * (double)a.re + (double)a.im * (double)a.im;
    }
    __syncthreads();
    row_sums(part, 2, 1, 1, 4 * Zl, sums, tid);
    chip_barrier<CB>();
    if (tid == 0 && rank == 0) {
      double si = sums[0], surv = sums[1];
      if constexpr (CB > 0) {
        for (unsigned k = 1; k < (1u << CB); ++k) {
          const unsigned p = chip_peer(smem_u32(&sums[0]), k);
          double u, v;
          asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(u), "=d"(v) : "r"(p));
          si += u;
          surv += v;
        }
      }
      const double phS = A.k_S[I0.sys] * si;
      double* o = per_sample + I0.out * 3;
      o[0] = phS;
      o[1] = 1.0 - surv - phS;
      o[2] = surv;
    }
    __syncthreads();
  }
  if constexpr (CB > 0) chip_barrier<CB>();  // no CTA leaves while a peer may read its memory
}

template <typename T>
size_t aniso_smem_bytes(int S, int n_c, int max_nuc, bool trace) {
  return (size_t)(8 + (trace ? 0 : n_c)) * S * sizeof(Cx<T>) +
         (trace ? 0 : (size_t)n_c * 32 * sizeof(T)) + (size_t)max_nuc * 20 * sizeof(double);
}

template <typename T>
size_t split_smem_bytes(int S, int rpc, int n_c, int max_nuc, bool trace) {
  return (size_t)(8 + (trace ? 0 : n_c)) * S * sizeof(Cx<T>) +
         (trace ? 0 : (size_t)n_c * 32 * sizeof(T)) +
         (size_t)rpc * (2 + max_nuc * 20) * sizeof(double);
}

// One macro-step of every active row, one CTA per row: psi from P to Q, slices
// to X (any order within a row: the integral sums over all of it).
template <typename T, int LK>
__global__ void __launch_bounds__(chip_max_threads<T>(LK), 1) k_chip_macro(
    const ChipArgs<T> A, const int* __restrict__ row_sys, const int* __restrict__ row_field,
    const int2* __restrict__ row_win, int macro_arg, const int* __restrict__ macro_dev,
    const T* __restrict__ P, T* __restrict__ Q, T* __restrict__ X, long long Zslot) {
  constexpr int KPT = 1 << LK;
  extern __shared__ __align__(16) unsigned char chip_smem[];
  ChipConst<T>& K = *reinterpret_cast<ChipConst<T>*>(chip_smem);
  const int r = blockIdx.x, tid = threadIdx.x;
  const int macro = macro_dev ? *macro_dev : macro_arg;
  const int2 w = row_win[r];
  if (macro < w.x || macro >= w.y) return;
  const HamDev<double>& H = A.ham[row_sys ? row_sys[r] : 0];
  const int f = row_field[r];
  const FieldDev<double> F = A.fields[f];
  const int Sr = (int)(H.Z >> LK);
  const bool on = tid < Sr;
  chip_const<T>(K, H, F, LK, 0, tid);
  Cx<T>* buf = reinterpret_cast<Cx<T>*>(chip_smem + sizeof(ChipConst<T>));
  T* dt = reinterpret_cast<T*>(buf + (size_t)8 * KPT * Sr);
  unsigned dig = 0;
  if (on) {
    Cx<T> a[KPT][4];
    dig = chip_digits(H, tid, LK, 0);
#pragma unroll
    for (int c = 0; c < KPT; ++c) {
      const unsigned m = ((unsigned)tid << LK) | (unsigned)c;
      T d[4];
      chip_diag<T>(H, F, m, d);
#pragma unroll
      for (int e = 0; e < 4; ++e) dt[((size_t)c * Sr + tid) * 4 + e] = d[e];
      const Cx<T>* p = reinterpret_cast<const Cx<T>*>(P) + ((size_t)r * Zslot + m) * 4;
#pragma unroll
      for (int e = 0; e < 4; ++e) a[c][e] = p[e];
    }
    chip_put<T, LK>(buf, Sr, tid, a);
  }
  __syncthreads();
  chip_macro<T, LK, 0>(Sr, 0, tid, on, dig,
                    A.coef + (size_t)f * 2 * A.n_c, A.n_c,
                    X + ((size_t)r * A.n_c * Zslot + tid) * 2, (size_t)Zslot, Sr, true);
  if (on) {
    Cx<T> a[KPT][4];
    chip_get<T, LK>(buf, Sr, tid, a);
#pragma unroll
    for (int c = 0; c < KPT; ++c) {
      Cx<T>* p = reinterpret_cast<Cx<T>*>(Q) +
                 ((size_t)r * Zslot + (((unsigned)tid << LK) | (unsigned)c)) * 4;
#pragma unroll
      for (int e = 0; e < 4; ++e) p[e] = a[c][e];
    }
  }
}

template <typename T, int LK>
size_t chip_smem_bytes(int S, int rpc, int n_c, int max_nuc) {
  const size_t buf = (size_t)4 * (1 << LK) * S * sizeof(Cx<T>);
  return sizeof(ChipConst<T>) + 2 * buf + buf / 2 + (size_t)n_c * ProjCfg<T>::kB * sizeof(T) +
         (size_t)rpc * (2 + max_nuc * 20) * sizeof(double);
}

constexpr int kChipSmemMax = 224 * 1024;

}  // namespace

template <typename T>
bool chip_plan(long long Zmax, int min_half, int max_nuc, long long load, int n_items, int n_c,
               bool trace, ChipPlan* out) {
  // One SM's share of configurations decides: few, and the length of a term
  // counts (more threads per configuration); many, and its instructions do.
  // Measured (GB300): one field of Z = 96, 16 propagations: 2.2 ms split, 4.9 ms
  // with one configuration per thread; Z = 16 FP64, 704 propagations: 51 and 82
  // ms; Z = 864, 1024 propagations in FP32: 48 ms with two configurations per
  // thread, 51 ms with four, which spill.  FP64 gains nothing from in-thread
  // nuclei (82 -> 143 ms: half the warps), so it takes them only where the
  // threads would not fit.
  const long long per_sm = load / kChipSms;
  out->split = false;
  if (per_sm <= 256 && max_nuc <= kSplitNuc && 4 * Zmax <= split_max_threads<T>()) {
    ChipPlan P;
    P.split = true;
    P.rpc = std::max<int>(1, (int)(32 / (4 * Zmax)));
    P.threads = (int)((4 * P.rpc * Zmax + 31) / 32 * 32);
    P.slots = (int)(P.rpc * Zmax);
    P.smem = split_smem_bytes<T>(P.slots, P.rpc, n_c, max_nuc, trace);
    if (P.smem <= (size_t)kChipSmemMax) {
      // the macro-step launches (graph replay) take one configuration per thread
      P.lk = Zmax <= chip_max_threads<T>(0) ? 0 : std::min(1, min_half);
      *out = P;
      return true;
    }
  }
  const int want = sizeof(T) == 8 || per_sm <= 192 ? 0 : 1;
  for (int lk = std::min(want, min_half); lk <= std::min(2, min_half); ++lk) {
    const long long Sr = Zmax >> lk;
    if (Sr > chip_max_threads<T>(lk)) continue;
    ChipPlan P;
    P.lk = lk;
    // rows per CTA: fill a warp, then up to 128 threads while every SM still
    // gets a CTA
    int rpc = std::max<int>(1, (int)(32 / Sr));
    while (rpc < 32 && (rpc * 2) * Sr <= 128 && n_items / (rpc * 2) >= kChipSms * 2) rpc *= 2;
    P.rpc = rpc;
    P.threads = (int)((rpc * Sr + 31) / 32 * 32);
    P.slots = (int)(rpc * Sr);
    P.smem = lk == 0 ? chip_smem_bytes<T, 0>(P.slots, rpc, n_c, max_nuc)
             : lk == 1 ? chip_smem_bytes<T, 1>(P.slots, rpc, n_c, max_nuc)
                       : chip_smem_bytes<T, 2>(P.slots, rpc, n_c, max_nuc);
    if (P.smem > (size_t)kChipSmemMax) continue;
    *out = P;
    return true;
  }
  return false;
}

// Split over clusters (FP32): the smallest cluster whose CTAs hold their share,
// larger while the rows alone leave SMs idle.  Two configurations per thread
// where 640 threads (96 registers) suffice, else four.
//
// Against one launch per term, in ms (two fields, 8, 32, 128 and 256 propagations; the last
// two at half the horizon): Z = 9216 on 8 CTAs 2.2, 3.9, 6.7, 12.9 and per term 3.5, 4.2,
// 6.1, 10.9; Z = 13824 (four configurations per thread, which spill) 3.1, 5.8, 10.2, 19.7
// and 3.6, 5.3, 8.4, 15.1; Z = 16384 3.5, 6.5, 11.6, 22.7 and 3.7, 5.4, 10.1, 18.0.  So
// beyond about two waves of clusters of 8 (15 to 18 run at once) the per-term launches are
// up to a quarter faster; the rule takes clusters at any number of rows, which is what the
// uneven batches need (few rows per pair), and is faster than the kernels before it at all.
bool chip_cluster_plan(long long Zmax, int min_half, int max_nuc, int n_items, int n_c, bool spin1_only,
                       ChipPlan* out) {
  if (!spin1_only) return false;
  bool found = false;
  for (int cb = 1; cb <= kChipMaxCb; ++cb) {
    const long long Zl = Zmax >> cb;
    for (int lk = 1; lk <= 2; ++lk) {
      if (min_half - cb < lk || (Zl >> lk) > (lk == 1 ? 640 : 512) || (lk == 2 && cb < 3)) continue;
      ChipPlan P;
      P.cb = cb;
      P.lk = lk;
      P.slots = (int)(Zl >> lk);
      P.threads = (P.slots + 31) / 32 * 32;
      P.smem = lk == 1 ? chip_smem_bytes<float, 1>(P.slots, 1, n_c, max_nuc)
                       : chip_smem_bytes<float, 2>(P.slots, 1, n_c, max_nuc);
      if (P.smem > (size_t)kChipSmemMax) continue;
      // a larger cluster while the rows leave SMs idle: one field, 0.3 us, 8 rows: Z =
      // 2304 2.35 ms on 2 CTAs, 1.69 on 4; Z = 4608 2.57 on 4, 2.01 on 8; with 40 rows
      // the smaller one takes 2.37 and 4.82 either way
      if (found && ((long long)n_items << cb) > kChipSms) return true;
      *out = P;
      found = true;
      break;
    }
  }
  return found;
}

namespace {
template <typename T, int MT>
int split_ctas_of(const ChipPlan& P) {
  static std::atomic<unsigned long long> attr_done;
  int dev = 0, n_sm = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (smem_attr_once((const void*)k_split_items<T, MT>, kChipSmemMax, attr_done) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_split_items<T, MT>, P.threads, P.smem) !=
      cudaSuccess)
    return 0;
  return n_sm * std::max(per_sm, 1);
}

// Launch configuration of a plan: `grid` CTAs, in clusters of 2^cb.
cudaLaunchConfig_t chip_cfg(const ChipPlan& P, int grid, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)P.threads, 1, 1);
  cfg.dynamicSmemBytes = P.smem;
  cfg.stream = st;
  if (P.cb > 0) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1u << P.cb;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  return cfg;
}

template <typename T, int LK, int MT, int MB, int CB>
int chip_ctas_of(const ChipPlan& P) {
  static std::atomic<unsigned long long> attr_done;
  const auto kf = k_chip_items<T, LK, MT, MB, CB>;
  int dev = 0, n_sm = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (smem_attr_once((const void*)kf, kChipSmemMax, attr_done) != cudaSuccess) return 0;
  if (CB > 0) {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = chip_cfg(P, 1 << P.cb, nullptr, at);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kf, &cfg) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return n << P.cb;
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kf, P.threads, P.smem) != cudaSuccess)
    return 0;
  return n_sm * std::max(per_sm, 1);
}

// Calls f.operator()<LK, MT, MB, CB>() of the instance of a plan.
template <typename T, typename F>
auto chip_instance(const ChipPlan& P, F&& f) {
  constexpr int M1 = chip_max_threads<T>(1), M2 = chip_max_threads<T>(2);
  if constexpr (sizeof(T) == 4) {
    if (P.cb > 0) {
      if (P.lk == 2) return f.template operator()<2, 512, 1, 3>();
      if (P.cb == 1) return f.template operator()<1, 640, 1, 1>();
      return P.cb == 2 ? f.template operator()<1, 640, 1, 2>() : f.template operator()<1, 640, 1, 3>();
    }
  }
  if (P.lk == 0) return f.template operator()<0, chip_max_threads<T>(0), 1, 0>();
  if constexpr (sizeof(T) == 4) {
    if (P.lk == 1 && P.threads <= 512) return f.template operator()<1, 512, 1, 0>();
  }
  if (P.lk == 1) return f.template operator()<1, M1, 1, 0>();
  return f.template operator()<2, M2, 1, 0>();
}

template <typename T>
struct ChipCtas {
  const ChipPlan& P;
  template <int LK, int MT, int MB, int CB>
  int operator()() const {
    return chip_ctas_of<T, LK, MT, MB, CB>(P);
  }
};
template <typename T>
struct ChipLaunch {
  const ChipArgs<T>& A;
  const ChipPlan& P;
  const PItem* items;
  const int2* groups;
  int n_groups;
  int* counter;
  T* X;
  int grid;
  double* per_sample;
  double* trace;
  const ElecOp& op;
  cudaStream_t st;
  template <int LK, int MT, int MB, int CB>
  cudaError_t operator()() const {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = chip_cfg(P, grid, st, at);
    return cudaLaunchKernelEx(&cfg, k_chip_items<T, LK, MT, MB, CB>, A, items, groups, n_groups,
                              counter, P.rpc, P.slots, X, per_sample, trace, op);
  }
};
}  // namespace

template <typename T>
bool aniso_plan(long long Zmax, int min_half, int max_nuc, int n_items, int n_c, bool trace,
                ChipPlan* out) {
  bool found = false;
  for (int cb = 0; cb <= kChipMaxCb && cb <= min_half; ++cb) {
    const long long Zl = Zmax >> cb;
    if (4 * Zl > split_max_threads<T>()) continue;
    ChipPlan P;
    P.aniso = true;
    P.cb = cb;
    P.slots = (int)Zl;
    P.threads = (int)((4 * Zl + 31) / 32 * 32);
    P.smem = aniso_smem_bytes<T>(P.slots, n_c, max_nuc, trace);
    if (P.smem > (size_t)kChipSmemMax) continue;
    // a larger cluster only while the rows alone leave SMs idle and each CTA keeps a
    // warp per scheduler (32 rows, Z = 192, FP64: one block per row of the generic
    // kernel, 62.5 ms; 4 blocks per row, 9.7)
    if (found && (((long long)n_items << cb) > kChipSms || P.threads < 128)) return true;
    *out = P;
    found = true;
  }
  return found;
}

namespace {
template <typename T, int CB, int MT>
int aniso_ctas_of(const ChipPlan& P) {
  static std::atomic<unsigned long long> attr_done;
  const auto kf = k_split_aniso<T, CB, MT>;
  int dev = 0, n_sm = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (smem_attr_once((const void*)kf, kChipSmemMax, attr_done) != cudaSuccess) return 0;
  cudaLaunchAttribute at[1];
  const cudaLaunchConfig_t cfg = chip_cfg(P, 1 << P.cb, nullptr, at);
  const cudaError_t e = CB > 0 ? cudaOccupancyMaxActiveClusters(&n, kf, &cfg)
                               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kf, P.threads, P.smem);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return CB > 0 ? n << CB : n_sm * std::max(n, 1);
}

// Calls f.operator()<CB, MT>() of the instance of an anisotropic plan.
template <typename T, typename F>
auto aniso_instance(const ChipPlan& P, F&& f) {
  constexpr int MX = split_max_threads<T>();
  if (P.threads <= 256) {
    if (P.cb == 0) return f.template operator()<0, 256>();
    if (P.cb == 1) return f.template operator()<1, 256>();
    return P.cb == 2 ? f.template operator()<2, 256>() : f.template operator()<3, 256>();
  }
  if (P.cb == 0) return f.template operator()<0, MX>();
  if (P.cb == 1) return f.template operator()<1, MX>();
  return P.cb == 2 ? f.template operator()<2, MX>() : f.template operator()<3, MX>();
}
template <typename T>
struct AnisoCtas {
  const ChipPlan& P;
  template <int CB, int MT>
  int operator()() const {
    return aniso_ctas_of<T, CB, MT>(P);
  }
};
template <typename T>
struct AnisoLaunch {
  const ChipArgs<T>& A;
  const ChipPlan& P;
  const PItem* items;
  const int2* groups;
  int n_groups;
  int* counter;
  int grid;
  double* per_sample;
  double* trace;
  const ElecOp& op;
  cudaStream_t st;
  template <int CB, int MT>
  cudaError_t operator()() const {
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = chip_cfg(P, grid, st, at);
    return cudaLaunchKernelEx(&cfg, k_split_aniso<T, CB, MT>, A, items, groups, n_groups, counter,
                              P.slots, per_sample, trace, op);
  }
};
}  // namespace

template <typename T>
int chip_ctas(const ChipPlan& P) {
  if (P.aniso) return aniso_instance<T>(P, AnisoCtas<T>{P});
  if (P.split)
    return P.threads <= 256   ? split_ctas_of<T, 256>(P)
           : P.threads <= 512 ? split_ctas_of<T, 512>(P)
                              : split_ctas_of<T, split_max_threads<T>()>(P);
  return chip_instance<T>(P, ChipCtas<T>{P});
}

template <typename T>
cudaError_t launch_chip_items(const ChipArgs<T>& A, const ChipPlan& P, const PItem* items,
                              const int2* groups, int n_groups, int* counter, T* Xscratch, int ctas,
                              double* per_sample, double* trace, const ElecOp& op,
                              cudaStream_t st) {
  if (n_groups == 0 || ctas == 0) return cudaSuccess;
  const int g = std::min(ctas, n_groups << P.cb);
  if (P.aniso)
    return aniso_instance<T>(P, AnisoLaunch<T>{A, P, items, groups, n_groups, counter, g, per_sample,
                                               trace, op, st});
  if (P.split) {
    if (P.threads <= 256)
      k_split_items<T, 256><<<g, P.threads, P.smem, st>>>(A, items, groups, n_groups, counter, P.rpc,
                                                          P.slots, per_sample, trace, op);
    else if (P.threads <= 512)
      k_split_items<T, 512><<<g, P.threads, P.smem, st>>>(A, items, groups, n_groups, counter, P.rpc,
                                                          P.slots, per_sample, trace, op);
    else
      k_split_items<T, split_max_threads<T>()><<<g, P.threads, P.smem, st>>>(
          A, items, groups, n_groups, counter, P.rpc, P.slots, per_sample, trace, op);
    return cudaGetLastError();
  }
  return chip_instance<T>(P, ChipLaunch<T>{A, P, items, groups, n_groups, counter, Xscratch, g,
                                           per_sample, trace, op, st});
}

template <typename T>
cudaError_t launch_chip_macro(const ChipArgs<T>& A, const ChipPlan& P, const int* row_sys,
                              const int* row_field, const int2* row_win, int macro,
                              const int* macro_dev, int rows, const T* psi, T* out, T* X,
                              long long Zslot, cudaStream_t st) {
  if (rows == 0) return cudaSuccess;
  const long long Sr = Zslot >> P.lk;
  const int threads = (int)((Sr + 31) / 32 * 32);
  const size_t smem = sizeof(ChipConst<T>) + (size_t)10 * (Sr << P.lk) * sizeof(Cx<T>);
#define RP_CHIP(LK)                                                                              \
  {                                                                                              \
    static std::atomic<unsigned long long> attr_done;                                            \
    const cudaError_t e = smem_attr_once((const void*)k_chip_macro<T, LK>, kChipSmemMax, attr_done); \
    if (e != cudaSuccess) return e;                                                              \
    k_chip_macro<T, LK><<<rows, threads, smem, st>>>(A, row_sys, row_field, row_win, macro,      \
                                                     macro_dev, psi, out, X, Zslot);             \
  }
  if (P.lk == 0) RP_CHIP(0)
  else if (P.lk == 1) RP_CHIP(1)
  else RP_CHIP(2)
#undef RP_CHIP
  return cudaGetLastError();
}

#define RP_CHIP_INST(T)                                                                          \
  template bool chip_plan<T>(long long, int, int, long long, int, int, bool, ChipPlan*);                    \
  template int chip_ctas<T>(const ChipPlan&);                                                    \
  template bool aniso_plan<T>(long long, int, int, int, int, bool, ChipPlan*);                   \
  template cudaError_t launch_chip_items<T>(const ChipArgs<T>&, const ChipPlan&, const PItem*,   \
                                            const int2*, int, int*, T*, int, double*, double*,   \
                                            const ElecOp&, cudaStream_t);                        \
  template cudaError_t launch_chip_macro<T>(const ChipArgs<T>&, const ChipPlan&, const int*,     \
                                            const int*, const int2*, int, const int*, int,       \
                                            const T*, T*, T*, long long, cudaStream_t);
RP_CHIP_INST(float)
RP_CHIP_INST(double)
#undef RP_CHIP_INST

}  // namespace rp
