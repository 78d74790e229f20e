// One Chebyshev term per launch for systems that do not fit on chip.
//
// A block takes a tile of 256 KPT consecutive configurations of one row; a
// thread owns KPT = 2^LK consecutive ones.  The state vectors are kept in four
// planes (one per electron state), so an isotropic flip-flop, which needs two
// of a partner's four components, reads two contiguous planes and nothing else
// (with the four components side by side every partner cost a whole 32-byte
// sector; the step kernel is bound by that traffic and its latency).
//   * partners under the LK innermost spin-1/2 nuclei are in the thread's registers;
//   * under the other spin-1/2 nuclei whose stride lies inside the tile, in shared
//     memory;
//   * under all others, in global memory (mostly L2), the direction being the
//     same for the whole block, one wide load per component and thread.
// Constants have 2/dE folded in (formed in FP64, rounded once); phi_n = u -
// phi_{n-2} with u the sum of all products (see rp_chip.cu for the order and the
// dropped global phase, which makes the sum's coefficients r_n (-i)^n).
//
// Anisotropic nuclei are taken in a rotated nuclear frame (rp_plan.cpp,
// nuclear_frame) in which the 2 x 2 electron matrix U of each nucleus has no
// diagonal and one real entry: 12 multiply-adds per nucleus and configuration
// instead of 32.
#include <algorithm>
#include <atomic>
#include <cstring>

#include "rp_device.cuh"
#include "rp_iso.cuh"
#include "rp_kernels.cuh"

namespace rp {

namespace {

constexpr int kTermThreads = 256;


// KPT complex values at p (16- or 32-byte aligned for KPT > 1).
template <typename T, int KPT>
__device__ __forceinline__ void gload(const T* p, Cx<T> (&q)[KPT]) {
  static_assert(KPT <= 2, "one or two configurations per thread");
  if constexpr (sizeof(T) * KPT == 16) {  // two FP64 values
    asm("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
        : "=d"(q[0].re), "=d"(q[0].im), "=d"(q[1].re), "=d"(q[1].im)
        : "l"(p));
  } else if constexpr (sizeof(T) * KPT == 8) {  // 16 bytes
    if constexpr (sizeof(T) == 4) {
      const float4 v = *reinterpret_cast<const float4*>(p);
      q[0] = {v.x, v.y};
      q[1] = {v.z, v.w};
    } else {
      const double2 v = *reinterpret_cast<const double2*>(p);
      q[0] = {v.x, v.y};
    }
  } else {
    const float2 v = *reinterpret_cast<const float2*>(p);
    q[0] = {v.x, v.y};
  }
}
template <typename T, int KPT>
__device__ __forceinline__ void gstore(T* p, const Cx<T> (&q)[KPT]) {
  if constexpr (sizeof(T) * KPT == 16) {
    asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(q[0].re), "d"(q[0].im),
                 "d"(q[1].re), "d"(q[1].im)
                 : "memory");
  } else if constexpr (sizeof(T) * KPT == 8) {
    if constexpr (sizeof(T) == 4)
      *reinterpret_cast<float4*>(p) = make_float4(q[0].re, q[0].im, q[1].re, q[1].im);
    else
      *reinterpret_cast<double2*>(p) = make_double2(q[0].re, q[0].im);
  } else {
    *reinterpret_cast<float2*>(p) = make_float2(q[0].re, q[0].im);
  }
}

// Sums of an anisotropic term: FP32 keeps the products with Re and Im of the
// couplings apart (u = A + i B, so neither needs the swapped pair of q); FP64
// adds them at once.
template <typename T, int KPT>
struct TermSum;
template <int KPT>
struct TermSum<float, KPT> {
  Cx<float> A[KPT][4], B[KPT][4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int c = 0; c < KPT; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) A[c][e] = B[c][e] = {0.f, 0.f};
  }
  __device__ __forceinline__ void real(int c, int e, float g, const Cx<float>& q) {
    madd(A[c][e], g, q);
  }
  __device__ __forceinline__ void imag(int c, int e, float g, const Cx<float>& q) {
    madd(B[c][e], g, q);
  }
  __device__ __forceinline__ Cx<float> get(int c, int e) const {
    return {A[c][e].re - B[c][e].im, A[c][e].im + B[c][e].re};
  }
};
template <int KPT>
struct TermSum<double, KPT> {
  Cx<double> A[KPT][4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int c = 0; c < KPT; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) A[c][e] = {0.0, 0.0};
  }
  __device__ __forceinline__ void real(int c, int e, double g, const Cx<double>& q) {
    madd(A[c][e], g, q);
  }
  __device__ __forceinline__ void imag(int c, int e, double g, const Cx<double>& q) {
    madd_i(A[c][e], g, q);
  }
  __device__ __forceinline__ Cx<double> get(int c, int e) const { return A[c][e]; }
};

// Values of the partners of the thread's configurations, one electron state at a time.
template <typename T, int LK>
struct SmemPartner {
  const Cx<T>* tile;
  int slot;
  __device__ __forceinline__ void get(int e, Cx<T> (&q)[1 << LK]) const {
    Vec<T, LK>::get(tile, kTermThreads, e, slot, q);
  }
};
template <typename T, int LK>
struct GlobalPartner {
  const T* p;  // plane 0 at the partner of the thread's first configuration
  size_t plane;
  __device__ __forceinline__ void get(int e, Cx<T> (&q)[1 << LK]) const {
    gload<T, 1 << LK>(p + (size_t)e * plane, q);
  }
};

// ---- isotropic products ----
template <typename T, int KPT, typename P>
__device__ __forceinline__ void iso_one(Cx<T> (&y)[KPT][4], const P& src, int rr, bool up, T g) {
  Cx<T> q[KPT];
  const int s0 = up ? 0 : (rr == 0 ? 2 : 1), s1 = up ? (rr == 0 ? 1 : 2) : 3;
  Cx<T> p[KPT];
  src.get(s0, q);
  src.get(s1, p);
#pragma unroll
  for (int c = 0; c < KPT; ++c) {
    if (rr == 0) {
      if (up) {
        madd(y[c][2], g, q[c]);
        madd(y[c][3], g, p[c]);
      } else {
        madd(y[c][0], g, q[c]);
        madd(y[c][1], g, p[c]);
      }
    } else {
      if (up) {
        madd(y[c][1], g, q[c]);
        madd(y[c][3], g, p[c]);
      } else {
        madd(y[c][0], g, q[c]);
        madd(y[c][2], g, p[c]);
      }
    }
  }
}
__device__ __forceinline__ void pick(Cx<float>& up, Cx<float>& dn, bool down, float g,
                                     const Cx<float>& q) {
  madd(up, down ? 0.f : g, q);
  madd(dn, down ? g : 0.f, q);
}
__device__ __forceinline__ void pick(Cx<double>& up, Cx<double>& dn, bool down, double g,
                                     const Cx<double>& q) {
  Cx<double> t = down ? dn : up;
  madd(t, g, q);
  if (down) dn = t;
  else up = t;
}
// direction differs between the lanes of a warp
template <typename T, int KPT, typename P>
__device__ __forceinline__ void iso_lane(Cx<T> (&y)[KPT][4], const P& src, int rr, bool down, T g) {
  Cx<T> q[KPT], p[KPT];
  src.get(down ? (rr == 0 ? 2 : 1) : 0, q);
  src.get(down ? 3 : (rr == 0 ? 1 : 2), p);
#pragma unroll
  for (int c = 0; c < KPT; ++c) {
    if (rr == 0) {
      pick(y[c][2], y[c][0], down, g, q[c]);
      pick(y[c][3], y[c][1], down, g, p[c]);
    } else {
      pick(y[c][1], y[c][0], down, g, q[c]);
      pick(y[c][3], y[c][2], down, g, p[c]);
    }
  }
}

// ---- anisotropic products: U = [[0, u], [w, 0]] (u complex, w real) on the electron of
// radical rr, U for the partner above (up), U^dagger for the one below ----
template <typename T, int KPT, typename P>
__device__ __forceinline__ void aniso_one(TermSum<T, KPT>& S, const P& src, int rr, bool up, T ur,
                                          T ui, T w) {
  // lower states (electron up) l take h, higher states h take l:
  //   up:   y_l += u q_h, y_h += w q_l;   down: y_l += w q_h, y_h += conj(u) q_l
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int l0 = k, l1 = 2 * k;  // rr = 0: (k, k + 2); rr = 1: (2 k, 2 k + 1)
    Cx<T> q[KPT], p[KPT];
    if (rr == 0) {
      src.get(l0, q);
      src.get(l0 + 2, p);
    } else {
      src.get(l1, q);
      src.get(l1 + 1, p);
    }
#pragma unroll
    for (int c = 0; c < KPT; ++c) {
      if (rr == 0) {
        if (up) {
          S.real(c, l0, ur, p[c]);
          S.imag(c, l0, ui, p[c]);
          S.real(c, l0 + 2, w, q[c]);
        } else {
          S.real(c, l0, w, p[c]);
          S.real(c, l0 + 2, ur, q[c]);
          S.imag(c, l0 + 2, -ui, q[c]);
        }
      } else {
        if (up) {
          S.real(c, l1, ur, p[c]);
          S.imag(c, l1, ui, p[c]);
          S.real(c, l1 + 1, w, q[c]);
        } else {
          S.real(c, l1, w, p[c]);
          S.real(c, l1 + 1, ur, q[c]);
          S.imag(c, l1 + 1, -ui, q[c]);
        }
      }
    }
  }
}
// direction differs between the lanes: (lr + i li) to the lower, (hr + i hi) to the higher state
template <typename T, int KPT, typename P>
__device__ __forceinline__ void aniso_lane(TermSum<T, KPT>& S, const P& src, int rr, T lr, T li,
                                           T hr, T hi) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int l0 = k, l1 = 2 * k;
    Cx<T> q[KPT], p[KPT];
    if (rr == 0) {
      src.get(l0, q);
      src.get(l0 + 2, p);
    } else {
      src.get(l1, q);
      src.get(l1 + 1, p);
    }
#pragma unroll
    for (int c = 0; c < KPT; ++c) {
      if (rr == 0) {
        S.real(c, l0, lr, p[c]);
        S.imag(c, l0, li, p[c]);
        S.real(c, l0 + 2, hr, q[c]);
        S.imag(c, l0 + 2, hi, q[c]);
      } else {
        S.real(c, l1, lr, p[c]);
        S.imag(c, l1, li, p[c]);
        S.real(c, l1 + 1, hr, q[c]);
        S.imag(c, l1 + 1, hi, q[c]);
      }
    }
  }
}

template <typename T, bool ANISO>
struct TermCfg;
template <typename T>
struct TermCfg<T, false> {
  static constexpr int NB = 2;
};
template <typename T>
struct TermCfg<T, true> {
  static constexpr int NB = 6;
};

// Blocks per SM that bound the registers.
template <typename T, int LK, bool ANISO>
constexpr int term_min_blocks() {
  if (sizeof(T) == 8) return ANISO ? 1 : 2;
  return ANISO && LK == 1 ? 3 : 4;
}

template <typename T, int LK, bool ANISO>
__global__ void __launch_bounds__(kTermThreads, (term_min_blocks<T, LK, ANISO>()))
    k_term(const TermArgs<T> A, const T* __restrict__ cur, const T* __restrict__ prev,
           T* __restrict__ next, T* __restrict__ acc, T* __restrict__ X, int macro_arg,
           const int* __restrict__ macro_dev, int n, int mode, int nacc) {
  constexpr int KPT = 1 << LK, NB = TermCfg<T, ANISO>::NB;
  extern __shared__ __align__(16) unsigned char term_smem[];
  __shared__ T s_out[6];
  __shared__ TermField<T> C;
  __shared__ TermSys<T> Y;
  Cx<T>* tile = reinterpret_cast<Cx<T>*>(term_smem);  // [e][group][thread]
  const int r = blockIdx.y, tid = threadIdx.x;
  {
    const int macro = macro_dev ? *macro_dev : macro_arg;
    const int2 w = A.row_win[r];
    if (macro < w.x || macro >= w.y) return;  // the whole block: one row
  }
  const int f = A.row_field[r];
  const unsigned m0 = blockIdx.x * (kTermThreads * KPT);
  const unsigned m = m0 + (unsigned)tid * KPT;
  const TermSys<T>& Yg = A.sys[A.row_sys ? A.row_sys[r] : 0];
  const unsigned Z = (unsigned)Yg.Z;
  if (m0 >= Z) return;
  const bool on = m < Z;  // Z is a multiple of KPT
  const size_t plane = (size_t)A.plane * 2, row0 = (size_t)r * 4 * plane;
  const T* c = cur + row0 + (size_t)m * 2;
  Cx<T> a[KPT][4];
  if (on) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      Cx<T> q[KPT];
      gload<T, KPT>(c + (size_t)e * plane, q);
#pragma unroll
      for (int k = 0; k < KPT; ++k) a[k][e] = q[k];
      Vec<T, LK>::put(tile, kTermThreads, e, tid, q);
    }
  }
  {
    const int4* s0 = reinterpret_cast<const int4*>(A.field + f);
    int4* d0 = reinterpret_cast<int4*>(&C);
    for (int i = tid; i < (int)(sizeof(C) / 16); i += kTermThreads) d0[i] = s0[i];
    const int4* s1 = reinterpret_cast<const int4*>(&Yg);
    int4* d1 = reinterpret_cast<int4*>(&Y);
    for (int i = tid; i < (int)(sizeof(Y) / 16); i += kTermThreads) d1[i] = s1[i];
  }
  if (tid < 32) {
    // nuclear fields of the nuclei outside the table (digits equal in the block)
    T b[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};  // x1, y1, z1, x2, y2, z2
    if (tid >= Yg.p_out && tid < Yg.n_nuc) {
      const unsigned d = (unsigned)Yg.d[tid], j = (unsigned)((m0 / (unsigned)Yg.stride[tid]) % d);
      const T M = T(0.5) * T(d - 1) - T(j);
      const int o = ((Yg.rad >> tid) & 1u) ? 3 : 0;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const T v = M * Yg.v[tid][i];
        if (o == 0) b[i] = v;
        else b[3 + i] = v;
      }
    }
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) b[i] += __shfl_xor_sync(0xffffffffu, b[i], s);
    if (tid == 0) {  // the table's combinations
      s_out[0] = T(0.5) * (b[2] + b[5]);
      s_out[1] = T(0.5) * (b[2] - b[5]);
      s_out[2] = T(0.5) * b[0];
      s_out[3] = T(0.5) * b[1];
      s_out[4] = T(0.5) * b[3];
      s_out[5] = T(0.5) * b[4];
    }
  }
  __syncthreads();
  if (!on) {  // no barrier below
    // the tensor-core integral reads whole 16-configuration chunks: keep the
    // padding past Z at zero (a refilled row may hold a larger system's slices)
    if (X && A.xblk) {
      for (int k = 0; k < KPT; ++k)
        if (m + k < (Z + kXChunk - 1) / kXChunk * kXChunk) {
          T* p = xblk_addr(X, r, n, m + k, A.Zslot, A.n_c);
          p[0] = p[4] = T(0);
          if (mode == MODE_FIRST) {
            p = xblk_addr(X, r, 0, m + k, A.Zslot, A.n_c);
            p[0] = p[4] = T(0);
          }
        }
    }
    return;
  }
  Cx<T> y[KPT][4];
  // nuclear fields: table entry of m mod tm plus the block's part, scaled by 2/dE
  T bt[NB][KPT];
  {
    const T* bp = A.btab + Y.tab + (m % (unsigned)Y.tm);
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
      for (int k = 0; k < KPT; ++k) bt[i][k] = C.s2 * (bp[(size_t)i * Y.tm + k] + s_out[i]);
  }
  const bool early = sizeof(T) == 8 && mode != MODE_FIRST;  // FP64 starts from phi_{n-2}
  if (early) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      Cx<T> q[KPT];
      gload<T, KPT>(prev + row0 + (size_t)m * 2 + (size_t)e * plane, q);
#pragma unroll
      for (int k = 0; k < KPT; ++k) y[k][e] = q[k];
    }
  }
#pragma unroll
  for (int k = 0; k < KPT; ++k) {
    const T d[4] = {C.D[0] + bt[0][k], C.D[1] + bt[1][k], C.D[1] - bt[1][k], C.D[2] - bt[0][k]};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (early) y[k][e] = {fma(d[e], a[k][e].re, -y[k][e].re), fma(d[e], a[k][e].im, -y[k][e].im)};
      else y[k][e] = {d[e] * a[k][e].re, d[e] * a[k][e].im};
    }
  }
  if (C.J != T(0)) {
#pragma unroll
    for (int k = 0; k < KPT; ++k) {
      madd(y[k][1], C.J, a[k][2]);
      madd(y[k][2], C.J, a[k][1]);
    }
  }
  if (C.kappa != T(0)) {  // -i kappa (2 P_S - 1)
#pragma unroll
    for (int k = 0; k < KPT; ++k) {
      madd_i(y[k][0], C.kappa, a[k][0]);
      madd_i(y[k][1], C.kappa, a[k][2]);
      madd_i(y[k][2], C.kappa, a[k][1]);
      madd_i(y[k][3], C.kappa, a[k][3]);
    }
  }
  const int nh = Y.n_half, p_in = Y.p_in;
  const unsigned rad = Y.rad;
  if constexpr (!ANISO) {
#pragma unroll
    for (int p = 0; p < LK; ++p) {
      const T g = C.g[p];
      const int rr = (int)((rad >> p) & 1u);
#pragma unroll
      for (int k = 0; k < KPT; ++k) {
        const int o = k ^ (1 << p), down = (k >> p) & 1;
        if (rr == 0) {
          madd(y[k][down ? 0 : 2], g, a[o][down ? 2 : 0]);
          madd(y[k][down ? 1 : 3], g, a[o][down ? 3 : 1]);
        } else {
          madd(y[k][down ? 0 : 1], g, a[o][down ? 1 : 0]);
          madd(y[k][down ? 2 : 3], g, a[o][down ? 3 : 2]);
        }
      }
    }
#pragma unroll 1
    for (int p = LK; p < p_in; ++p) {
      const int bit = 1 << (p - LK);
      const SmemPartner<T, LK> src{tile, tid ^ bit};
      const int rr = (int)((rad >> p) & 1u);
      const bool down = (tid & bit) != 0;
      if (bit >= 32) iso_one<T, KPT>(y, src, rr, !down, C.g[p]);
      else iso_lane<T, KPT>(y, src, rr, down, C.g[p]);
    }
#pragma unroll 2
    for (int p = p_in; p < nh; ++p) {
      const GlobalPartner<T, LK> src{cur + row0 + (size_t)(m ^ (1u << p)) * 2, plane};
      iso_one<T, KPT>(y, src, (int)((rad >> p) & 1u), !((m >> p) & 1u), C.g[p]);
    }
    unsigned qd = m >> nh;
#pragma unroll 2
    for (int p = nh; p < Y.n_nuc; ++p) {
      const unsigned d = (unsigned)Y.d[p], j = d == 3u ? qd % 3u : qd % d;
      qd = d == 3u ? qd / 3u : qd / d;
      const int rr = (int)((rad >> p) & 1u);
      const size_t st = (size_t)Y.stride[p] * 2;
      T gu = C.g[p], gd = gu;
      if (d != 3u) {
        const T I = T(0.5) * T(d - 1), M = I - T(j);
        gu *= sqrt(I * (I + 1) - M * (M - 1));
        gd *= sqrt(I * (I + 1) - M * (M + 1));
      }
      if (j + 1u < d) iso_one<T, KPT>(y, GlobalPartner<T, LK>{c + st, plane}, rr, true, gu);
      if (j > 0u) iso_one<T, KPT>(y, GlobalPartner<T, LK>{c - st, plane}, rr, false, gd);
    }
  } else {
    TermSum<T, KPT> S;
    S.clear();
    // own configuration: the x and y parts of S_1 . b_1 and S_2 . b_2
#pragma unroll
    for (int k = 0; k < KPT; ++k) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const T s1 = (e & 2) ? T(1) : T(-1), s2 = (e & 1) ? T(1) : T(-1);
        S.real(k, e, bt[2][k], a[k][e ^ 2]);
        S.imag(k, e, s1 * bt[3][k], a[k][e ^ 2]);
        S.real(k, e, bt[4][k], a[k][e ^ 1]);
        S.imag(k, e, s2 * bt[5][k], a[k][e ^ 1]);
      }
    }
#pragma unroll
    for (int p = 0; p < LK; ++p) {
      const T ur = C.ur[p], ui = C.ui[p], w = C.g[p];
      const int rr = (int)((rad >> p) & 1u);
#pragma unroll
      for (int k = 0; k < KPT; ++k) {
        const int o = k ^ (1 << p), down = (k >> p) & 1;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (rr == 0) {
            if (down) {
              S.real(k, i, w, a[o][i + 2]);
              S.real(k, i + 2, ur, a[o][i]);
              S.imag(k, i + 2, -ui, a[o][i]);
            } else {
              S.real(k, i, ur, a[o][i + 2]);
              S.imag(k, i, ui, a[o][i + 2]);
              S.real(k, i + 2, w, a[o][i]);
            }
          } else {
            if (down) {
              S.real(k, 2 * i, w, a[o][2 * i + 1]);
              S.real(k, 2 * i + 1, ur, a[o][2 * i]);
              S.imag(k, 2 * i + 1, -ui, a[o][2 * i]);
            } else {
              S.real(k, 2 * i, ur, a[o][2 * i + 1]);
              S.imag(k, 2 * i, ui, a[o][2 * i + 1]);
              S.real(k, 2 * i + 1, w, a[o][2 * i]);
            }
          }
        }
      }
    }
#pragma unroll 1
    for (int p = LK; p < p_in; ++p) {
      const int bit = 1 << (p - LK);
      const SmemPartner<T, LK> src{tile, tid ^ bit};
      const int rr = (int)((rad >> p) & 1u);
      const bool down = (tid & bit) != 0;
      const T ur = C.ur[p], ui = C.ui[p], w = C.g[p];
      if (bit >= 32)
        aniso_one<T, KPT>(S, src, rr, !down, ur, ui, w);
      else
        aniso_lane<T, KPT>(S, src, rr, down ? w : ur, down ? T(0) : ui, down ? ur : w,
                           down ? -ui : T(0));
    }
#pragma unroll 1
    for (int p = p_in; p < nh; ++p) {
      const GlobalPartner<T, LK> src{cur + row0 + (size_t)(m ^ (1u << p)) * 2, plane};
      aniso_one<T, KPT>(S, src, (int)((rad >> p) & 1u), !((m >> p) & 1u), C.ur[p], C.ui[p], C.g[p]);
    }
    unsigned qd = m >> nh;
#pragma unroll 1
    for (int p = nh; p < Y.n_nuc; ++p) {
      const unsigned d = (unsigned)Y.d[p], j = d == 3u ? qd % 3u : qd % d;
      qd = d == 3u ? qd / 3u : qd / d;
      const int rr = (int)((rad >> p) & 1u);
      const size_t st = (size_t)Y.stride[p] * 2;
      T fu = T(1), fd = T(1);
      if (d != 3u) {
        const T I = T(0.5) * T(d - 1), M = I - T(j);
        fu = sqrt(I * (I + 1) - M * (M - 1));
        fd = sqrt(I * (I + 1) - M * (M + 1));
      }
      if (j + 1u < d)
        aniso_one<T, KPT>(S, GlobalPartner<T, LK>{c + st, plane}, rr, true, fu * C.ur[p],
                          fu * C.ui[p], fu * C.g[p]);
      if (j > 0u)
        aniso_one<T, KPT>(S, GlobalPartner<T, LK>{c - st, plane}, rr, false, fd * C.ur[p],
                          fd * C.ui[p], fd * C.g[p]);
    }
#pragma unroll
    for (int k = 0; k < KPT; ++k)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const Cx<T> v = S.get(k, e);
        y[k][e].re += v.re;
        y[k][e].im += v.im;
      }
  }
  // phi_n, accumulator psi(h) += r_n (-i)^n phi_n, singlet slice
  const T* cf = A.coef + (size_t)f * 2 * A.n_c;
  const T* cl = cf + A.n_c;
  const size_t off = row0 + (size_t)m * 2;
  const T h = T(0.70710678118654752440);
  // s += c_j phi_j, j odd: -i r, even: r
  auto add_term = [&](Cx<T> (&s)[KPT], const Cx<T> (&v)[KPT], int j) {
    const T r_ = cf[j], l_ = cl[j];
    if (j & 1) {
#pragma unroll
      for (int k = 0; k < KPT; ++k) {
        if (sizeof(T) == 4) madd_i(s[k], -l_, v[k]);
        madd_i(s[k], -r_, v[k]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < KPT; ++k) {
        if (sizeof(T) == 4) madd(s[k], l_, v[k]);
        madd(s[k], r_, v[k]);
      }
    }
  };
  Cx<T> x[KPT], x0[KPT];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    Cx<T> v[KPT], own[KPT];
    // phi_{n-1} of the own configurations, from the tile
    if (nacc >= 2 || mode == MODE_FIRST) Vec<T, LK>::get(tile, kTermThreads, e, tid, own);
    if (mode == MODE_FIRST) {
#pragma unroll
      for (int k = 0; k < KPT; ++k) v[k] = {T(0.5) * y[k][e].re, T(0.5) * y[k][e].im};
    } else if (sizeof(T) == 4) {
      Cx<T> q[KPT];
      gload<T, KPT>(prev + off + (size_t)e * plane, q);
#pragma unroll
      for (int k = 0; k < KPT; ++k) v[k] = {y[k][e].re - q[k].re, y[k][e].im - q[k].im};
      if (nacc >= 3) {
        Cx<T> s[KPT];
        gload<T, KPT>(acc + off + (size_t)e * plane, s);
        add_term(s, q, n - 2);
        add_term(s, own, n - 1);
        add_term(s, v, n);
        gstore<T, KPT>(acc + off + (size_t)e * plane, s);
      }
    } else {
#pragma unroll
      for (int k = 0; k < KPT; ++k) v[k] = y[k][e];
    }
    if (mode != MODE_LAST) gstore<T, KPT>(next + off + (size_t)e * plane, v);
    if (nacc == 1 || nacc == 2) {
      Cx<T> s[KPT];
      if (mode == MODE_FIRST) {
#pragma unroll
        for (int k = 0; k < KPT; ++k) s[k] = {T(0), T(0)};
      } else {
        gload<T, KPT>(acc + off + (size_t)e * plane, s);
      }
      if (nacc == 2) add_term(s, own, n - 1);
      add_term(s, v, n);
      gstore<T, KPT>(acc + off + (size_t)e * plane, s);
    }
    if (e == 1) {
#pragma unroll
      for (int k = 0; k < KPT; ++k) {
        x[k] = v[k];
        x0[k] = own[k];
      }
    }
    if (e == 2) {
#pragma unroll
      for (int k = 0; k < KPT; ++k) {
        x[k] = {(x[k].re - v[k].re) * h, (x[k].im - v[k].im) * h};
        x0[k] = {(x0[k].re - own[k].re) * h, (x0[k].im - own[k].im) * h};
      }
    }
  }
  if (X && A.xblk) {
#pragma unroll
    for (int k = 0; k < KPT; ++k) {
      T* p = xblk_addr(X, r, n, m + k, A.Zslot, A.n_c);
      p[0] = x[k].re;
      p[4] = x[k].im;
      if (mode == MODE_FIRST) {
        p = xblk_addr(X, r, 0, m + k, A.Zslot, A.n_c);
        p[0] = x0[k].re;
        p[4] = x0[k].im;
      }
    }
  } else if (X) {
    T* xr = X + ((size_t)r * A.n_c * A.Zslot + m) * 2;
    gstore<T, KPT>(xr + (size_t)n * A.Zslot * 2, x);
    if (mode == MODE_FIRST) gstore<T, KPT>(xr, x0);
  }
}

// ---- the same in FP32 where every system has the nine spin-1/2 nuclei of a tile ----
//
// Digits and directions of all nuclei outside the tile are then the block's.  Warp 0
// lists their partners once (addresses and weights); each thread copies its own 16 bytes
// per component into its own shared-memory slots some entries ahead of their use
// (cp.async, no barrier: nobody else reads them).  phi_{n-2} and the accumulator follow
// as the list's last entries.  An anisotropic partner has two entries; the second goes
// straight to registers (a copy passes the L1 twice, which all copies would fill).  The
// tile's nuclei are unrolled and the fields of the nuclei outside it come from a table,
// so a thread spends its instructions on products.
//
// Bounds: HBM (isotropic), issue slots and L1 (anisotropic).  Z = 2^20, 14 rows (1.9 GB
// of vectors): 355 us per term in the general form, 353 with the copies alone (65 % of
// issue slots used, half of them by integer work), 300 as it is: at 3.9 vector passes
// 6.1 TB/s of a measured 6.8.  Anisotropic, Z = 2359296, 6 rows, whole call: 243, 232
// and 187 ms, 177 with the second entries direct (the same for every second isotropic
// partner: 305 us).
constexpr int kRingThreads = kTermThreads, kRingTileBits = 9;
constexpr int kRingParts = 2 * kMaxNucDev;

template <bool ANISO>
struct RingCfg {
  static constexpr int RS = 4;              // copies (two components each) in flight
  static constexpr int HE = ANISO ? 2 : 1;  // entries per partner
  static constexpr int NB = ANISO ? 6 : 2;
  static constexpr size_t smem = (size_t)kRingThreads * 16 * (4 + 2 * RS);
};

__device__ __forceinline__ void cp16(unsigned d, const float* p) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(p) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// components of entry h of a partner: those its products read
template <bool ANISO>
__device__ __forceinline__ void ring_comps(int rr, bool up, int h, int& c0, int& c1) {
  if (ANISO) {
    c0 = rr ? 2 * h : h;
    c1 = rr ? c0 + 1 : c0 + 2;
  } else {
    c0 = up ? 0 : (rr ? 1 : 2);
    c1 = up ? (rr ? 2 : 1) : 3;
  }
}
__device__ __forceinline__ void unpack(const float4& v, Cx<float> (&q)[2]) {
  q[0] = {v.x, v.y};
  q[1] = {v.z, v.w};
}

// Sums of one thread's two configurations (see TermSum for A and B).
template <bool ANISO>
struct RingSum {
  Cx<float> A[2][4], B[ANISO ? 2 : 1][ANISO ? 4 : 1];
  // isotropic flip-flop with a partner of known direction: q, p hold its components
  __device__ __forceinline__ void iso(bool up, int rr, float g, const Cx<float> (&q)[2],
                                      const Cx<float> (&p)[2]) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (up) {
        if (rr) madd(A[k][1], g, q[k]);
        else madd(A[k][2], g, q[k]);
        madd(A[k][3], g, p[k]);
      } else {
        madd(A[k][0], g, q[k]);
        if (rr) madd(A[k][2], g, p[k]);
        else madd(A[k][1], g, p[k]);
      }
    }
  }
  // the same with a weight for each direction, one of them zero
  __device__ __forceinline__ void iso2(int rr, float gu, float gd, const Cx<float> (&q)[2],
                                       const Cx<float> (&p)[2]) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      madd(A[k][0], gd, q[k]);
      madd(A[k][3], gu, p[k]);
      if (rr) {
        madd(A[k][1], gu, q[k]);
        madd(A[k][2], gd, p[k]);
      } else {
        madd(A[k][2], gu, q[k]);
        madd(A[k][1], gd, p[k]);
      }
    }
  }
  // states l (electron up) and h of a pair: l += (ur + i ui or w) q_h, h += (w or conj) q_l
  __device__ __forceinline__ void pair(bool up, int l, int h, float ur, float ui, float w,
                                       const Cx<float> (&q)[2], const Cx<float> (&p)[2]) {
    if constexpr (ANISO) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (up) {
          madd(A[k][l], ur, p[k]);
          madd(B[k][l], ui, p[k]);
          madd(A[k][h], w, q[k]);
        } else {
          madd(A[k][l], w, p[k]);
          madd(A[k][h], ur, q[k]);
          madd(B[k][h], -ui, q[k]);
        }
      }
    }
  }
  __device__ __forceinline__ void pair2(int l, int h, float lr, float li, float hr, float hi,
                                        const Cx<float> (&q)[2], const Cx<float> (&p)[2]) {
    if constexpr (ANISO) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        madd(A[k][l], lr, p[k]);
        madd(B[k][l], li, p[k]);
        madd(A[k][h], hr, q[k]);
        madd(B[k][h], hi, q[k]);
      }
    }
  }
  // A[e] += i g v
  __device__ __forceinline__ void imag(int k, int e, float g, const Cx<float>& v) {
    if constexpr (ANISO) madd(B[k][e], g, v);
    else madd_i(A[k][e], g, v);
  }
  __device__ __forceinline__ Cx<float> get(int k, int e) const {
    if constexpr (ANISO) return {A[k][e].re - B[k][e].im, A[k][e].im + B[k][e].re};
    else return A[k][e];
  }
};

template <bool ANISO>
__global__ void __launch_bounds__(kRingThreads, ANISO ? 3 : 4) k_term_ring(
    const TermArgs<float> A, const float* __restrict__ cur, const float* __restrict__ prev,
    float* __restrict__ next, float* __restrict__ acc, float* __restrict__ X, int macro_arg,
    const int* __restrict__ macro_dev, int n, int mode, int nacc) {
  using Cfg = RingCfg<ANISO>;
  constexpr int RS = Cfg::RS, HE = Cfg::HE, NB = Cfg::NB;
  extern __shared__ __align__(16) unsigned char term_smem[];
  __shared__ longlong2 s_ptr[kRingParts * HE + 4];  // addresses of an entry at m = 0
  __shared__ float4 s_w[kRingParts];                // g, ur, ui, code (radical | 2 up)
  __shared__ float4 s_in[kRingTileBits];            // the same of the tile's nuclei
  __shared__ int s_np;
  const int r = blockIdx.y, tid = threadIdx.x;
  {
    const int macro = macro_dev ? *macro_dev : macro_arg;
    const int2 w = A.row_win[r];
    if (macro < w.x || macro >= w.y) return;  // the whole block: one row
  }
  const TermField<float>& C = A.field[A.row_field[r]];
  const TermSys<float>& Y = A.sys[A.row_sys ? A.row_sys[r] : 0];
  const unsigned m0 = blockIdx.x << kRingTileBits, m = m0 + 2u * tid;
  if (m0 >= (unsigned)Y.Z) return;  // Z is a multiple of the tile
  const size_t plane = (size_t)A.plane * 2, row0 = (size_t)r * 4 * plane;
  const float* c = cur + row0 + (size_t)m * 2;
  float4* tile = reinterpret_cast<float4*>(term_smem);  // [e][thread]
  const unsigned ring0 = (unsigned)__cvta_generic_to_shared(tile + 4 * kRingThreads + tid);
  constexpr unsigned kComp = kRingThreads * 16, kSlot = 2 * kComp;
  const unsigned rad = Y.rad;
  const int n_pro = min(RS, Y.n_half - kRingTileBits);
#pragma unroll
  for (int q = 0; q < RS; ++q) {  // spin-1/2 nuclei next to the tile need no list
    if (q >= n_pro) break;
    const int p = kRingTileBits + q;
    int c0, c1;
    ring_comps<ANISO>((int)((rad >> p) & 1u), !((m0 >> p) & 1u), 0, c0, c1);
    const float* src = cur + row0 + (size_t)(m ^ (1u << p)) * 2;
    cp16(ring0 + q * kSlot, src + c0 * plane);
    cp16(ring0 + q * kSlot + kComp, src + c1 * plane);
    cp_commit();
  }
  RingSum<ANISO> S;
  Cx<float> a[2][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float4 v = *reinterpret_cast<const float4*>(c + e * plane);
    tile[e * kRingThreads + tid] = v;
    a[0][e] = {v.x, v.y};
    a[1][e] = {v.z, v.w};
  }
  if (tid < 32) {
    // partners outside the tile, the upper one of a nucleus before the lower one
    bool hu = false, hd = false;
    float fu = 1.f, fd = 1.f;
    if (tid >= kRingTileBits && tid < Y.n_nuc) {
      const unsigned d = (unsigned)Y.d[tid], j = (m0 / (unsigned)Y.stride[tid]) % d;
      hu = j + 1u < d;
      hd = j > 0u;
      if (d > 3u) {
        const float I = 0.5f * (float)(d - 1), M = I - (float)j;
        fu = sqrtf(I * (I + 1) - M * (M - 1));
        fd = sqrtf(I * (I + 1) - M * (M + 1));
      }
    }
    const unsigned bu = __ballot_sync(0xffffffffu, hu), bd = __ballot_sync(0xffffffffu, hd);
    const unsigned below = (1u << tid) - 1u;
    int at = __popc(bu & below) + __popc(bd & below);
    if (tid < Y.n_nuc) {
      const int rr = (int)((rad >> tid) & 1u);
      const float g = C.g[tid], ur = ANISO ? C.ur[tid] : 0.f, ui = ANISO ? C.ui[tid] : 0.f;
      if (tid < kRingTileBits) s_in[tid] = make_float4(g, ur, ui, __int_as_float(rr));
      const long long st = 2 * (long long)Y.stride[tid];
      auto put = [&](bool up, float f) {
        s_w[at] = make_float4(f * g, f * ur, f * ui, __int_as_float(rr | (up ? 2 : 0)));
#pragma unroll
        for (int h = 0; h < HE; ++h) {
          int c0, c1;
          ring_comps<ANISO>(rr, up, h, c0, c1);
          const float* b = cur + row0 + (up ? st : -st);
          s_ptr[at * HE + h] = make_longlong2((long long)(b + c0 * plane), (long long)(b + c1 * plane));
        }
        ++at;
      };
      if (hu) put(true, fu);
      if (hd) put(false, fd);
    }
    const int np = __popc(bu) + __popc(bd);
    if (tid < 4) {  // phi_{n-2} and the accumulator, two components each
      const float* b = (tid & 1 ? acc : prev) + row0 + (size_t)(tid & 2) * plane;
      const bool need = mode != MODE_FIRST && (!(tid & 1) || nacc);
      s_ptr[np * HE + tid] = make_longlong2(need ? (long long)b : 0, (long long)(b + plane));
    }
    if (tid == 0) s_np = np;
  }
  // nuclear fields: table entries of the tile and of the nuclei outside it, times 2/dE
  float bt[NB][2];
  {
    const float* bp = A.btab + Y.tab + 2 * tid;
    const float* op = A.btab + Y.otab + (size_t)blockIdx.x * NB;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const float2 v = *reinterpret_cast<const float2*>(bp + ((size_t)i << kRingTileBits));
      const float o = op[i];
      bt[i][0] = C.s2 * (v.x + o);
      bt[i][1] = C.s2 * (v.y + o);
    }
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float d[4] = {C.D[0] + bt[0][k], C.D[1] + bt[1][k], C.D[1] - bt[1][k], C.D[2] - bt[0][k]};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      S.A[k][e] = {d[e] * a[k][e].re, d[e] * a[k][e].im};
      if constexpr (ANISO) {
        // the x and y parts of S_1 . b_1 and S_2 . b_2
        const float s1 = (e & 2) ? 1.f : -1.f, s2 = (e & 1) ? 1.f : -1.f;
        madd(S.A[k][e], bt[2][k], a[k][e ^ 2]);
        madd(S.A[k][e], bt[4][k], a[k][e ^ 1]);
        S.B[k][e] = {s1 * bt[3][k] * a[k][e ^ 2].re, s1 * bt[3][k] * a[k][e ^ 2].im};
        madd(S.B[k][e], s2 * bt[5][k], a[k][e ^ 1]);
      }
    }
  }
  const float Jx = C.J, kp = C.kappa;
  if (Jx != 0.f) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      madd(S.A[k][1], Jx, a[k][2]);
      madd(S.A[k][2], Jx, a[k][1]);
    }
  }
  if (kp != 0.f) {  // -i kappa (2 P_S - 1)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      S.imag(k, 0, kp, a[k][0]);
      S.imag(k, 1, kp, a[k][2]);
      S.imag(k, 2, kp, a[k][1]);
      S.imag(k, 3, kp, a[k][3]);
    }
  }
  __syncthreads();  // no barrier below
  {                 // nucleus 0: the thread's other configuration
    const float4 w = s_in[0];
    const int rr = __float_as_int(w.w) & 1;
    if constexpr (ANISO) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        auto one = [&](int l_, int h_) {
          madd(S.A[0][l_], w.y, a[1][h_]);
          madd(S.B[0][l_], w.z, a[1][h_]);
          madd(S.A[0][h_], w.x, a[1][l_]);
          madd(S.A[1][l_], w.x, a[0][h_]);
          madd(S.A[1][h_], w.y, a[0][l_]);
          madd(S.B[1][h_], -w.z, a[0][l_]);
        };
        if (rr) one(2 * h, 2 * h + 1);
        else one(h, h + 2);
      }
    } else {
      // configuration 0 has the partner above, 1 the one below
      if (rr) {
        madd(S.A[0][1], w.x, a[1][0]);
        madd(S.A[0][3], w.x, a[1][2]);
        madd(S.A[1][0], w.x, a[0][1]);
        madd(S.A[1][2], w.x, a[0][3]);
      } else {
        madd(S.A[0][2], w.x, a[1][0]);
        madd(S.A[0][3], w.x, a[1][1]);
        madd(S.A[1][0], w.x, a[0][2]);
        madd(S.A[1][1], w.x, a[0][3]);
      }
    }
  }
#pragma unroll
  for (int p = 1; p < kRingTileBits; ++p) {
    const int bit = 1 << (p - 1);
    const float4 w = s_in[p];
    const int rr = __float_as_int(w.w) & 1;
    const bool down = (tid & bit) != 0;  // the warp's for bit >= 32
    const float4* t = tile + (tid ^ bit);
    Cx<float> q[2], pp[2];
    if constexpr (ANISO) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        auto one = [&](int l, int hs) {
          unpack(t[l * kRingThreads], q);
          unpack(t[hs * kRingThreads], pp);
          if (bit >= 32)
            S.pair(!down, l, hs, w.y, w.z, w.x, q, pp);
          else
            S.pair2(l, hs, down ? w.x : w.y, down ? 0.f : w.z, down ? w.y : w.x, down ? -w.z : 0.f,
                    q, pp);
        };
        if (rr) one(2 * h, 2 * h + 1);
        else one(h, h + 2);
      }
    } else {
      int c0, c1;
      ring_comps<false>(rr, !down, 0, c0, c1);
      unpack(t[c0 * kRingThreads], q);
      unpack(t[c1 * kRingThreads], pp);
      if (bit >= 32) S.iso(!down, rr, w.x, q, pp);
      else S.iso2(rr, down ? 0.f : w.x, down ? w.x : 0.f, q, pp);
    }
  }
  // partners outside the tile
  const int np = s_np;
  unsigned slot = ring0;
  auto copy = [&](int q, unsigned at) {
    if (q < np + 4) {
      const longlong2 pp = s_ptr[q < np ? q * HE : np * HE + (q - np)];
      if (pp.x) {
        cp16(at, reinterpret_cast<const float*>(pp.x) + (size_t)m * 2);
        cp16(at + kComp, reinterpret_cast<const float*>(pp.y) + (size_t)m * 2);
      }
    }
    cp_commit();
  };
  for (int q = n_pro; q < RS; ++q) copy(q, ring0 + q * kSlot);
  int ahead = RS;
  auto take = [&](Cx<float> (&q)[2], Cx<float> (&p)[2]) {  // this entry's two components
    cp_wait<RS - 1>();
    float4 u, v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(u.x), "=f"(u.y), "=f"(u.z), "=f"(u.w)
                 : "r"(slot)
                 : "memory");
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(slot + kComp)
                 : "memory");
    unpack(u, q);
    unpack(v, p);
  };
  auto refill = [&]() {
    copy(ahead++, slot);
    slot += kSlot;
    if (slot == ring0 + RS * kSlot) slot = ring0;
  };
#pragma unroll 1
  for (int i = 0; i < np; ++i) {
    const float4 w = s_w[i];
    const int code = __float_as_int(w.w);
    Cx<float> q[2], p[2];
    if constexpr (ANISO) {
      // the second entry straight to registers, loaded one entry's work ahead
      const longlong2 pp = s_ptr[2 * i + 1];
      const float4 du = __ldg(reinterpret_cast<const float4*>(pp.x) + m / 2),
                   dv = __ldg(reinterpret_cast<const float4*>(pp.y) + m / 2);
      auto half = [&](bool up, int h) {
        if (code & 1) S.pair(up, 2 * h, 2 * h + 1, w.y, w.z, w.x, q, p);
        else S.pair(up, h, h + 2, w.y, w.z, w.x, q, p);
      };
      take(q, p);
      if (code & 2) half(true, 0);
      else half(false, 0);
      refill();
      unpack(du, q);
      unpack(dv, p);
      if (code & 2) half(true, 1);
      else half(false, 1);
    } else {
      take(q, p);
      if (code & 2) {
        if (code & 1) S.iso(true, 1, w.x, q, p);
        else S.iso(true, 0, w.x, q, p);
      } else {
        if (code & 1) S.iso(false, 1, w.x, q, p);
        else S.iso(false, 0, w.x, q, p);
      }
      refill();
    }
  }
  // phi_n = u - phi_{n-2}, the accumulator's pending terms, the singlet slice
  const size_t off = row0 + (size_t)m * 2;
  const float* cf = A.coef + (size_t)A.row_field[r] * 2 * A.n_c;
  const float* cl = cf + A.n_c;
  // s += c_j phi_j, j odd: -i r, even: r
  auto add_term = [&](Cx<float> (&s)[2], const Cx<float> (&v)[2], int j, float hi, float lo) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (j & 1) {
        madd_i(s[k], -lo, v[k]);
        madd_i(s[k], -hi, v[k]);
      } else {
        madd(s[k], lo, v[k]);
        madd(s[k], hi, v[k]);
      }
    }
  };
  float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f, h2 = 0.f, l2 = 0.f;  // of n, n - 1, n - 2
  if (nacc >= 1) h0 = cf[n], l0 = cl[n];
  if (nacc >= 2) h1 = cf[n - 1], l1 = cl[n - 1];
  if (nacc >= 3) h2 = cf[n - 2], l2 = cl[n - 2];
  const float hs = 0.70710678118654752440f;
  Cx<float> x[2], x0[2];
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    Cx<float> pv[2][2], sv[2][2];
    if (mode != MODE_FIRST) {
      take(pv[0], pv[1]);
      refill();
      if (nacc) take(sv[0], sv[1]);
      refill();
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int e = 2 * hh + t;
      Cx<float> v[2], own[2];
      if (nacc >= 2) unpack(tile[e * kRingThreads + tid], own);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const Cx<float> u = S.get(k, e);
        if (mode == MODE_FIRST) v[k] = {0.5f * u.re, 0.5f * u.im};
        else v[k] = {u.re - pv[t][k].re, u.im - pv[t][k].im};
      }
      if (mode != MODE_LAST) gstore<float, 2>(next + off + e * plane, v);
      if (nacc) {
        Cx<float> s[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) s[k] = mode == MODE_FIRST ? Cx<float>{0.f, 0.f} : sv[t][k];
        if (nacc >= 3) add_term(s, pv[t], n - 2, h2, l2);
        if (nacc >= 2) add_term(s, own, n - 1, h1, l1);
        add_term(s, v, n, h0, l0);
        gstore<float, 2>(acc + off + e * plane, s);
      }
      if (e == 1 || e == 2) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (e == 1) {
            x[k] = v[k];
            if (mode == MODE_FIRST) x0[k] = own[k];
          } else {
            x[k] = {(x[k].re - v[k].re) * hs, (x[k].im - v[k].im) * hs};
            if (mode == MODE_FIRST) x0[k] = {(x0[k].re - own[k].re) * hs, (x0[k].im - own[k].im) * hs};
          }
        }
      }
    }
  }
  if (X && A.xblk) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      float* p = xblk_addr(X, r, n, m + k, A.Zslot, A.n_c);
      p[0] = x[k].re;
      p[4] = x[k].im;
      if (mode == MODE_FIRST) {
        p = xblk_addr(X, r, 0, m + k, A.Zslot, A.n_c);
        p[0] = x0[k].re;
        p[4] = x0[k].im;
      }
    }
  } else if (X) {
    float* xr = X + ((size_t)r * A.n_c * A.Zslot + m) * 2;
    gstore<float, 2>(xr + (size_t)n * A.Zslot * 2, x);
    if (mode == MODE_FIRST) gstore<float, 2>(xr, x0);
  }
}

// The table of nuclear fields of the configurations i < tm: (z1 + z2)/2,
// (z1 - z2)/2, x1/2, y1/2, x2/2, y2/2 of b_r = sum_k M_k A_k e_z over the
// nuclei whose digit varies within the table (p < p_out).  FP64 sums.
template <typename T>
__global__ void __launch_bounds__(256) k_term_table(const HamDev<double>* __restrict__ ham,
                                                    const TermSys<T>* __restrict__ sys, int nb,
                                                    T* __restrict__ btab) {
  const HamDev<double>& H = ham[blockIdx.y];
  const TermSys<T>& Y = sys[blockIdx.y];
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Y.tm) return;
  double b[2][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
  long long q = i;
  for (int p = 0; p < Y.p_out; ++p) {
    const int d = H.d[p], j = (int)(q % d);
    q /= d;
    const double M = 0.5 * (double)(d - 1) - (double)j;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (H.rad[p] == 0) b[0][k] += M * H.v[p][k];
      else b[1][k] += M * H.v[p][k];
    }
  }
  T* o = btab + Y.tab + i;
  o[0] = (T)(0.5 * (b[0][2] + b[1][2]));
  o[Y.tm] = (T)(0.5 * (b[0][2] - b[1][2]));
  if (nb == 6) {
    o[2 * Y.tm] = (T)(0.5 * b[0][0]);
    o[3 * Y.tm] = (T)(0.5 * b[0][1]);
    o[4 * Y.tm] = (T)(0.5 * b[1][0]);
    o[5 * Y.tm] = (T)(0.5 * b[1][1]);
  }
}

// The same of the nuclei outside a tile (p >= p_out), for each tile.
template <typename T>
__global__ void __launch_bounds__(256) k_term_outer(const HamDev<double>* __restrict__ ham,
                                                    const TermSys<T>* __restrict__ sys, int nb,
                                                    T* __restrict__ btab) {
  const HamDev<double>& H = ham[blockIdx.y];
  const TermSys<T>& Y = sys[blockIdx.y];
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Y.Z / Y.tm) return;
  double b[2][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
  long long q = i;
  for (int p = Y.p_out; p < H.n_nuc; ++p) {
    const int d = H.d[p], j = (int)(q % d);
    q /= d;
    const double M = 0.5 * (double)(d - 1) - (double)j;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (H.rad[p] == 0) b[0][k] += M * H.v[p][k];
      else b[1][k] += M * H.v[p][k];
    }
  }
  T* o = btab + Y.otab + i * nb;
  o[0] = (T)(0.5 * (b[0][2] + b[1][2]));
  o[1] = (T)(0.5 * (b[0][2] - b[1][2]));
  if (nb == 6) {
    o[2] = (T)(0.5 * b[0][0]);
    o[3] = (T)(0.5 * b[0][1]);
    o[4] = (T)(0.5 * b[1][0]);
    o[5] = (T)(0.5 * b[1][1]);
  }
}

template <bool ANISO>
cudaError_t launch_ring(const TermArgs<float>& A, const float* cur, const float* prev, float* next,
                        float* acc, float* X, int macro, const int* macro_dev, int rows, int n,
                        int mode, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done;
  const auto kf = k_term_ring<ANISO>;
  const cudaError_t e = smem_attr_once((const void*)kf, (int)RingCfg<ANISO>::smem, attr_done);
  if (e != cudaSuccess) return e;
  const unsigned tiles = (unsigned)((A.Zslot + (1 << kRingTileBits) - 1) >> kRingTileBits);
  kf<<<dim3(tiles, rows), kRingThreads, RingCfg<ANISO>::smem, st>>>(
      A, cur, prev, next, acc, X, macro, macro_dev, n, mode, term_nacc(false, n, mode));
  return cudaGetLastError();
}

template <typename T, int LK, bool ANISO>
cudaError_t launch_term_of(const TermArgs<T>& A, const T* cur, const T* prev, T* next, T* acc, T* X,
                           int macro, const int* macro_dev, int rows, int n, int mode,
                           cudaStream_t st) {
  const int nacc = term_nacc(sizeof(T) == 8, n, mode);
  constexpr int KPT = 1 << LK;
  const unsigned tiles = (unsigned)((A.Zslot + kTermThreads * KPT - 1) / (kTermThreads * KPT));
  const size_t smem = (size_t)kTermThreads * KPT * 4 * sizeof(Cx<T>);
  k_term<T, LK, ANISO><<<dim3(tiles, rows), kTermThreads, smem, st>>>(A, cur, prev, next, acc, X,
                                                                      macro, macro_dev, n, mode, nacc);
  return cudaGetLastError();
}

}  // namespace

// Two configurations per thread where every system has a spin-1/2 nucleus: with
// four the registers leave 16 warps per SM, which the latency of the partner
// loads does not allow (Z = 2^20: 376 us per term against 355).
template <typename T>
int term_lk(bool aniso, int min_half) {
  return min_half >= 1 ? 1 : 0;
}
int term_tile(int lk) { return kTermThreads << lk; }

template <typename T>
cudaError_t launch_term_table(const HamDev<double>* ham, const TermSys<T>* sys, int n_sys,
                              long long tm_max, long long tiles_max, bool aniso, T* btab,
                              cudaStream_t st) {
  if (n_sys == 0) return cudaSuccess;
  if (tiles_max > 0)
    k_term_outer<T><<<dim3((unsigned)((tiles_max + 255) / 256), n_sys), 256, 0, st>>>(
        ham, sys, aniso ? 6 : 2, btab);
  k_term_table<T><<<dim3((unsigned)((tm_max + 255) / 256), n_sys), 256, 0, st>>>(
      ham, sys, aniso ? 6 : 2, btab);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_term(const TermArgs<T>& A, int lk, bool aniso, const T* cur, const T* prev,
                        T* next, T* acc, T* X, int macro, const int* macro_dev, int rows, int n,
                        int mode, cudaStream_t st) {
  if (rows == 0) return cudaSuccess;
  if constexpr (sizeof(T) == 4) {
    if (A.ring)
      return aniso ? launch_ring<true>(A, cur, prev, next, acc, X, macro, macro_dev, rows, n, mode, st)
                   : launch_ring<false>(A, cur, prev, next, acc, X, macro, macro_dev, rows, n, mode, st);
  }
  if (aniso)
    return lk == 1 ? launch_term_of<T, 1, true>(A, cur, prev, next, acc, X, macro, macro_dev, rows, n, mode, st)
                   : launch_term_of<T, 0, true>(A, cur, prev, next, acc, X, macro, macro_dev, rows, n, mode, st);
  if (lk == 1)
    return launch_term_of<T, 1, false>(A, cur, prev, next, acc, X, macro, macro_dev, rows, n, mode, st);
  return launch_term_of<T, 0, false>(A, cur, prev, next, acc, X, macro, macro_dev, rows, n, mode, st);
}

#define RP_TERM_INST(T)                                                                         \
  template int term_lk<T>(bool, int);                                                           \
  template cudaError_t launch_term_table<T>(const HamDev<double>*, const TermSys<T>*, int,       \
                                            long long, long long, bool, T*, cudaStream_t);       \
  template cudaError_t launch_term<T>(const TermArgs<T>&, int, bool, const T*, const T*, T*, T*, \
                                      T*, int, const int*, int, int, int, cudaStream_t);
RP_TERM_INST(float)
RP_TERM_INST(double)
#undef RP_TERM_INST

}  // namespace rp
