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
  if constexpr (sizeof(T) * KPT == 16) {  // 32 bytes
    if constexpr (sizeof(T) == 4) {
      asm("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
          : "=f"(q[0].re), "=f"(q[0].im), "=f"(q[1].re), "=f"(q[1].im), "=f"(q[2].re),
            "=f"(q[2].im), "=f"(q[3].re), "=f"(q[3].im)
          : "l"(p));
    } else {
      asm("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
          : "=d"(q[0].re), "=d"(q[0].im), "=d"(q[1].re), "=d"(q[1].im)
          : "l"(p));
    }
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
    if constexpr (sizeof(T) == 4) {
      asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(q[0].re),
                   "f"(q[0].im), "f"(q[1].re), "f"(q[1].im), "f"(q[2].re), "f"(q[2].im),
                   "f"(q[3].re), "f"(q[3].im)
                   : "memory");
    } else {
      asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(q[0].re), "d"(q[0].im),
                   "d"(q[1].re), "d"(q[1].im)
                   : "memory");
    }
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

template <typename T, int LK, bool ANISO>
cudaError_t launch_term_of(const TermArgs<T>& A, const T* cur, const T* prev, T* next, T* acc, T* X,
                           int macro, const int* macro_dev, int rows, int n, int mode,
                           cudaStream_t st) {
  // the accumulator takes the pending terms together: three at a time in FP32
  // (phi_n, phi_{n-1} and phi_{n-2} are at hand), which cuts a term from 5.25 to
  // 3.9 vector passes on average; FP64 is bound by arithmetic and adds each
  const int nacc = mode == MODE_FIRST ? 2
                   : sizeof(T) == 8   ? 1
                   : mode == MODE_LAST ? (n - 2) % 3 + 1
                                       : ((n - 1) % 3 == 0 ? 3 : 0);
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
                              long long tm_max, bool aniso, T* btab, cudaStream_t st) {
  if (n_sys == 0) return cudaSuccess;
  k_term_table<T><<<dim3((unsigned)((tm_max + 255) / 256), n_sys), 256, 0, st>>>(
      ham, sys, aniso ? 6 : 2, btab);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_term(const TermArgs<T>& A, int lk, bool aniso, const T* cur, const T* prev,
                        T* next, T* acc, T* X, int macro, const int* macro_dev, int rows, int n,
                        int mode, cudaStream_t st) {
  if (rows == 0) return cudaSuccess;
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
                                            long long, bool, T*, cudaStream_t);                  \
  template cudaError_t launch_term<T>(const TermArgs<T>&, int, bool, const T*, const T*, T*, T*, \
                                      T*, int, const int*, int, int, int, cudaStream_t);
RP_TERM_INST(float)
RP_TERM_INST(double)
#undef RP_TERM_INST

}  // namespace rp
