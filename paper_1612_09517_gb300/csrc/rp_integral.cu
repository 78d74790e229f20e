// The exact time integral of a macro-step (Eqs. 20, 22) by a low-rank factor
// of its weights, and the device-side planning of that factor.
//
// int_0^h |<S|psi(t + tau)>|^2 dtau = sum_nm W_nm <x_n|x_m> with the singlet
// slices x_n = <S|phi_n> and W_nm = i^(n-m) w_nm, w real, symmetric and
// positive semidefinite:
//   w_nm = eps_n eps_m int_0^h exp(-kbar tau) J_n(dE tau) J_m(dE tau) dtau.
// The functions J_n(dE tau) on [0, h] are band-limited, so w has numerical rank
// about dE h / pi + 12 (28-32 of n_c = 88).  With w = L L^T (pivoted Cholesky),
//   integral = sum_z sum_k |y_k(z)|^2,  y_k(z) = sum_n L_nk (-i)^n x_n(z),
// which costs 2 rank n_c real multiply-adds per configuration instead of the
// 2 n_c^2 of the complex Gram matrix <x_n|x_m> (5.3k instead of 16k at the
// default n_c), needs no Gram accumulators, and sums squares only.
#include <algorithm>
#include <cmath>

#include "rp_device.cuh"
#include "rp_kernels.cuh"
#include "rp_project.cuh"

namespace rp {

namespace {

constexpr int kPlanThreads = 256;

// Nodes of the quadrature of w: the integrand is entire of exponential type
// dE h on [-1, 1] times exp(-kbar h (t + 1) / 2); q-point Gauss-Legendre is
// exact to degree 2 q - 1, and the Chebyshev coefficients J_j(x) fall below
// 1e-17 for j > x + 12 x^(1/3) + 12 (x <= 88).  Strong decay within one step
// (kbar h > 8) takes n_c + x + 48 nodes.
__host__ __device__ inline int plan_nodes(double x, double b, int n_c) {
  if (b > 8.0) return n_c + (int)ceil(x) + 48;
  const int q = (int)ceil(0.5 * (x + 12.0 * cbrt(x) + sqrt(80.0 * b) + 24.0));
  return (q + 7) & ~7;
}

size_t plan_smem_bytes(int q, int n_c) {
  const size_t area = std::max((size_t)q * (n_c + 2), (size_t)n_c * n_c);
  return (area + (size_t)n_c * (n_c + 1) + 2 * (size_t)n_c + q + 1) * sizeof(double);
}

// One CTA per field.  J_n at the nodes by Miller's backward recurrence (one
// thread per node, started where J is below 1e-25, so no rescaling), w from the
// nodes, then w = L L^T by left-looking Cholesky with diagonal pivoting until
// the largest remaining diagonal is below stop x trace (each remaining entry of
// w is then below that too).  L_nk carries the sign of (-i)^n (see k_project);
// meta[f] = (rank, number of leading terms n whose entries of w exceed the
// bound).  W, if not NULL, receives the complex weights W_nm.  FP64 throughout:
// bound by the FP64 units (about 0.3 M multiply-adds per field).
template <typename T>
__global__ void __launch_bounds__(kPlanThreads) k_plan_integral(
    const IntegralIn* __restrict__ in, int n_c, double stop, T* __restrict__ L, int ldk,
    int2* __restrict__ meta, double* __restrict__ W) {
  extern __shared__ __align__(16) double pl_smem[];
  __shared__ double s_red[2];
  __shared__ int s_piv;
  const int f = blockIdx.x, tid = threadIdx.x;
  const IntegralIn I = in[f];
  const double x = I.dE * I.h, b = I.kbar * I.h;
  const int q = plan_nodes(x, b, n_c);
  const int ldf = n_c + 2, ldw = n_c + 1;
  const size_t area = max((size_t)q * ldf, (size_t)n_c * n_c);
  double* F = pl_smem;              // [q][ldf]: sqrt(weight) eps_n J_n at the nodes, later L [k][n]
  double* w = F + area;             // [n_c][ldw]
  double* d = w + (size_t)n_c * ldw;  // remaining diagonal
  double* d0 = d + n_c;             // diagonal of w
  double* inv = d0 + n_c;           // 1 / k
  for (int k = tid; k <= q; k += kPlanThreads) inv[k] = k > 0 ? 1.0 / (double)k : 0.0;
  __syncthreads();
  if (tid < q) {
    // Gauss-Legendre node and weight by Newton's iteration on P_q
    double z = cospi(((double)tid + 0.75) / ((double)q + 0.5)), dp = 1.0;
    for (int it = 0; it < 8; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= q; ++k) {
        const double a = inv[k];
        const double p2 = (2.0 - a) * z * p1 - (1.0 - a) * p0;
        p0 = p1;
        p1 = p2;
      }
      dp = (double)q * (z * p1 - p0) / (z * z - 1.0);
      const double dz = p1 / dp;
      z -= dz;
      if (fabs(dz) < 1e-15) break;
    }
    const double tau = 0.5 * I.h * (z + 1.0);
    const double wt = 0.5 * I.h * exp(-I.kbar * tau) * 2.0 / ((1.0 - z * z) * dp * dp);
    const double xx = I.dE * tau;
    double* Fr = F + (size_t)tid * ldf;
    for (int n = 0; n < n_c; ++n) Fr[n] = 0.0;
    double scale = sqrt(wt);
    if (xx < 1e-6) {  // the next terms are below 1e-19
      Fr[0] = 1.0 - 0.25 * xx * xx;
      Fr[1] = 0.5 * xx;
      Fr[2] = 0.125 * xx * xx;
    } else {
      const int m = ((int)ceil(xx + 11.0 * cbrt(xx)) + 22) & ~1;
      const double t = 2.0 / xx;
      double jp1 = 0.0, jn = 1e-150, norm = 2.0 * jn;  // m is even
      for (int n = m; n >= 1; --n) {
        const double jm1 = (double)n * t * jn - jp1;
        jp1 = jn;
        jn = jm1;
        const int k = n - 1;
        if (k < n_c) Fr[k] = jn;
        if ((k & 1) == 0) norm += k == 0 ? jn : 2.0 * jn;
      }
      scale /= norm;
    }
    for (int n = 0; n < n_c; ++n) Fr[n] *= (n == 0 ? scale : 2.0 * scale);
  }
  __syncthreads();
  // w = F^T F on 4 x 4 tiles of the upper triangle
  const int nt = n_c / 4, tiles = nt * (nt + 1) / 2;
  for (int t = tid; t < tiles; t += kPlanThreads) {
    int ti = 0, r = t;
    while (r >= nt - ti) {
      r -= nt - ti;
      ++ti;
    }
    const int tj = ti + r;
    double a[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) a[i][j] = 0.0;
    for (int p = 0; p < q; ++p) {
      const double* Fp = F + (size_t)p * ldf;
      double u[4], v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        u[i] = Fp[4 * ti + i];
        v[i] = Fp[4 * tj + i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) a[i][j] = fma(u[i], v[j], a[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int n = 4 * ti + i, m = 4 * tj + j;
        w[n * ldw + m] = a[i][j];
        w[m * ldw + n] = a[i][j];
      }
  }
  __syncthreads();
  if (W) {
    double* Wf = W + (size_t)f * n_c * n_c * 2;
    for (int e = tid; e < n_c * n_c; e += kPlanThreads) {
      const int n = e / n_c, m = e % n_c, ph = (n - m) & 3;
      const double v = w[n * ldw + m];
      Wf[2 * e] = ph == 0 ? v : (ph == 2 ? -v : 0.0);
      Wf[2 * e + 1] = ph == 1 ? v : (ph == 3 ? -v : 0.0);
    }
  }
  if (!L) return;
  for (int n = tid; n < n_c; n += kPlanThreads) d[n] = d0[n] = w[n * ldw + n];
  __syncthreads();
  if (tid == 0) {
    double tr = 0.0;
    for (int n = 0; n < n_c; ++n) tr += d[n];
    s_red[0] = tr;
  }
  __syncthreads();
  const double tr = s_red[0], lim = stop * tr;
  int rank = 0;
  for (; rank < n_c; ++rank) {
    if (tid < 32) {  // pivot: the largest remaining diagonal
      double best = -1.0;
      int at = 0;
      for (int n = tid; n < n_c; n += 32)
        if (d[n] > best) {
          best = d[n];
          at = n;
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oa = __shfl_xor_sync(0xffffffffu, at, o);
        if (ob > best || (ob == best && oa < at)) {
          best = ob;
          at = oa;
        }
      }
      if (tid == 0) {
        s_piv = at;
        s_red[1] = best;
      }
    }
    __syncthreads();
    const int p = s_piv;
    const double dpv = s_red[1];
    if (!(dpv > lim)) break;  // the same for the whole CTA
    if (tid < n_c) {
      double c = w[tid * ldw + p];
      for (int j = 0; j < rank; ++j) c = fma(-F[(size_t)j * n_c + tid], F[(size_t)j * n_c + p], c);
      const double l = c / sqrt(dpv);
      F[(size_t)rank * n_c + tid] = l;
      d[tid] = tid == p ? 0.0 : d[tid] - l * l;
    }
    __syncthreads();
  }
  __syncthreads();
  T* Lf = L + (size_t)f * n_c * ldk;
  for (int e = tid; e < n_c * ldk; e += kPlanThreads) {
    const int n = e / ldk, k = e % ldk;
    const double v = k < rank ? F[(size_t)k * n_c + n] : 0.0;
    Lf[e] = (T)((n & 2) ? -v : v);
  }
  if (tid == 0) {
    // a term with diagonal d enters the integral through entries up to sqrt(d)
    int ne = n_c;
    while (ne > 2 && d0[ne - 1] * tr <= lim * lim) --ne;
    meta[f] = make_int2(rank, ne);
  }
}

// integral[r] += sum_z sum_k |y_k(z)|^2 for the rows active in this macro-step,
// y_k(z) = sum_n L_nk (-i)^n x_n(z): (-i)^n x is (re, im), (im, -re) and their
// negatives for n mod 4 = 0, 1, 2, 3, and L carries the sign of n mod 4 >= 2.
// A thread holds the KB partial sums y_k of kCfg configurations in registers;
// L of the row's field is staged in shared memory and read as broadcasts, the
// slices x_n stream once per KB-column block of L (one block for the default
// plans in FP32, two in FP64) through a ring of asynchronous copies.  FP32 works
// on pairs (y_k, y_{k+1}) by fma.rn.f32x2.  The squares of one configuration
// are summed in T and added in FP64.
// CLUSTER: the CTAs of a row form a thread-block cluster and its first one adds their sums
// in order.
constexpr int kProjThreads = 128;

template <typename T, bool CLUSTER>
__global__ void __launch_bounds__(kProjThreads) k_project(
    const SysTab<T> S, const T* __restrict__ X, const T* __restrict__ L, int ldk,
    const int2* __restrict__ meta, const int* __restrict__ row_field,
    const int2* __restrict__ row_win, int macro_arg, const int* __restrict__ macro_dev, int n_c,
    long long z_per_cta, double* __restrict__ integral) {
  using Acc = typename ProjAcc<T>::type;
  constexpr int KB = ProjCfg<T>::kB, C = ProjCfg<T>::kCfg;
  extern __shared__ __align__(16) unsigned char proj_smem[];
  __shared__ double red[kProjThreads];
  T* sl = reinterpret_cast<T*>(proj_smem);  // [n_c][KB], then the ring of slices
  auto* ring = reinterpret_cast<typename SliceVal<T>::type*>(sl + (size_t)n_c * KB) + threadIdx.x;
  const int r = blockIdx.y;
  const int macro = macro_dev ? *macro_dev : macro_arg;
  {
    const int2 w = row_win[r];
    if (macro < w.x || macro >= w.y) return;
  }
  const long long Z = S.ham[S.row_sys ? S.row_sys[r] : 0].Z;
  const long long Zs = S.Zslot;
  const long long z0 = (long long)blockIdx.x * z_per_cta;
  const long long z1 = min(Z, z0 + z_per_cta);
  if (!CLUSTER && z0 >= z1) return;
  const int f = row_field[r];
  const int2 mt = meta[f];
  const int n_e = (mt.y + 1) & ~1;  // n_c is even
  const T* Lf = L + (size_t)f * n_c * ldk;
  const T* Xr = X + (size_t)r * n_c * Zs * 2;
  const int tid = threadIdx.x;
  double sum = 0.0;
  for (int k0 = 0; k0 < mt.x; k0 += KB) {
    __syncthreads();
    stage_factor<T>(sl, Lf, ldk, n_e, k0, tid, kProjThreads);
    __syncthreads();
    for (long long c0 = z0; c0 < z1; c0 += kProjThreads * C) {
      // configurations past the end read the last one and are not counted
      const T* p[C];
      bool on[C];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const long long z = c0 + c * kProjThreads + tid;
        on[c] = z < z1;
        p[c] = Xr + (on[c] ? z : z1 - 1) * 2;
      }
      Acc yr[C][16], yi[C][16];
      if (!on[0]) break;  // nothing left for this thread (no barrier until the next block)
      project_block<T, C>(yr, yi, p, (size_t)Zs * 2, sl, KB, n_e, ring, kProjThreads);
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (on[c]) sum += proj_norm(yr[c], yi[c]);
    }
  }
  const double tot = block_sum<kProjThreads>(sum, red);
  if constexpr (CLUSTER) {
    __shared__ double part;
    if (tid == 0) part = tot;
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    if (blockIdx.x == 0 && tid == 0) {  // the cluster's rank 0
      double s = integral[r];
      for (unsigned k = 0; k < gridDim.x; ++k) {
        unsigned a;
        double v;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(&part)), "r"(k));
        asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
        s += v;
      }
      integral[r] = s;
    }
    // no CTA leaves while the first one may read its sum
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  } else if (tid == 0) {
    atomicAdd(integral + r, tot);
  }
}

// The same in FP64 for rows of at most 96 configurations.  A warp's FP64 instruction holds
// its scheduler for 64 cycles however many of its lanes work, so a row of 16 configurations
// on one warp leaves three of the four schedulers idle.  Here a warp takes eight columns of
// every configuration, 32 at a time.  64 rows, one macro-step, in us (k_project, this):
// Z = 16 154 and 53, 64 158 and 101, 96 159 and 148, 125 163 and 204; the Gram matrix of the
// slices took 81 at Z = 16.
constexpr int kFewConfigs = 96;
constexpr int kFewCols = 32;  // eight per warp

__global__ void __launch_bounds__(kProjThreads) k_project_few(
    const SysTab<double> S, const double* __restrict__ X, const double* __restrict__ L, int ldk,
    const int2* __restrict__ meta, const int* __restrict__ row_field,
    const int2* __restrict__ row_win, int macro_arg, const int* __restrict__ macro_dev, int n_c,
    double* __restrict__ integral) {
  extern __shared__ __align__(16) unsigned char proj_smem[];
  __shared__ double red[kProjThreads];
  double* sl = reinterpret_cast<double*>(proj_smem);  // [n_c][kFewCols]
  const int r = blockIdx.x, tid = threadIdx.x;
  const int macro = macro_dev ? *macro_dev : macro_arg;
  {
    const int2 w = row_win[r];
    if (macro < w.x || macro >= w.y) return;
  }
  const int Z = (int)S.ham[S.row_sys ? S.row_sys[r] : 0].Z;
  const size_t Zs = (size_t)S.Zslot;
  const int f = row_field[r];
  const int2 mt = meta[f];
  const int n_e = (mt.y + 1) & ~1;  // n_c is even
  const double2* Xr = reinterpret_cast<const double2*>(X) + (size_t)r * n_c * Zs;
  const double* l = sl + 8 * (tid >> 5);
  double sum = 0.0;
  for (int k0 = 0; k0 < mt.x; k0 += kFewCols) {
    __syncthreads();
    stage_factor<double, kFewCols>(sl, L + (size_t)f * n_c * ldk, ldk, n_e, k0, tid, kProjThreads);
    __syncthreads();
    for (int z = tid & 31; z < Z; z += 32) {
      double yr[8], yi[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) yr[k] = yi[k] = 0.0;
#pragma unroll 2
      for (int n = 0; n < n_e; n += 2) {
        const double2 u = Xr[n * Zs + z], v = Xr[(n + 1) * Zs + z];
        proj_add(yr, yi, l + n * kFewCols, u.x, u.y);
        proj_add(yr, yi, l + (n + 1) * kFewCols, v.y, -v.x);
      }
      sum += proj_norm8(yr, yi);
    }
  }
  const double tot = block_sum<kProjThreads>(sum, red);
  if (tid == 0) atomicAdd(integral + r, tot);
}

}  // namespace

int integral_ldk(int n_c) { return (n_c + 7) & ~7; }

template <typename T>
cudaError_t launch_plan_integral(const IntegralIn* in, const IntegralIn* host_in, int n_fields,
                                 int n_c, T* L, int2* meta, double* W, cudaStream_t st) {
  if (n_fields == 0) return cudaSuccess;
  int q = 8;
  for (int f = 0; f < n_fields; ++f)
    q = std::max(q, plan_nodes(host_in[f].dE * host_in[f].h, host_in[f].kbar * host_in[f].h, n_c));
  if (q > kPlanThreads) return cudaErrorInvalidValue;
  const size_t smem = plan_smem_bytes(q, n_c);
  static std::atomic<unsigned long long> attr_done;
  const cudaError_t e = smem_attr_once((const void*)k_plan_integral<T>,
                                       (int)plan_smem_bytes(2 * 88 + 48, 88), attr_done);
  if (e != cudaSuccess) return e;
  // w's own rounding is 1e-16 of its trace; the FP32 plans' tolerance is 1e-9
  const double stop = sizeof(T) == 4 ? 1e-12 : 1e-16;
  k_plan_integral<T><<<n_fields, kPlanThreads, smem, st>>>(in, n_c, stop, L, integral_ldk(n_c),
                                                           meta, W);
  return cudaGetLastError();
}

template <typename T>
size_t proj_smem_bytes(int n_c) {
  return (size_t)n_c * ProjCfg<T>::kB * sizeof(T) +
         proj_ring_bytes<T>(kProjThreads, ProjCfg<T>::kCfg);
}

template <typename T>
cudaError_t launch_project(const SysTab<T>& S, const T* X, const T* L, const int2* meta,
                           const int* row_field, const int2* row_win, int macro,
                           const int* macro_dev, int rows, int n_c, double* integral,
                           cudaStream_t st) {
  if (rows == 0) return cudaSuccess;
  if constexpr (sizeof(T) == 8) {
    if (S.Zslot <= kFewConfigs) {
      k_project_few<<<rows, kProjThreads, (size_t)n_c * kFewCols * sizeof(double), st>>>(
          S, X, L, integral_ldk(n_c), meta, row_field, row_win, macro, macro_dev, n_c, integral);
      return cudaGetLastError();
    }
  }
  const long long tile = (long long)kProjThreads * ProjCfg<T>::kCfg;
  const long long tiles = (S.Zslot + tile - 1) / tile;
  const size_t smem = proj_smem_bytes<T>(n_c);
  static std::atomic<unsigned long long> attr_done[2];
  auto go = [&](auto kf, unsigned ctas, unsigned cluster, long long per, int k) {
    const cudaError_t e = smem_attr_once((const void*)kf, (int)proj_smem_bytes<T>(88), attr_done[k]);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas, (unsigned)rows, 1);
    cfg.blockDim = dim3(kProjThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kf, S, X, L, integral_ldk(n_c), meta, row_field, row_win, macro,
                              macro_dev, n_c, per * tile, integral);
  };
  // A row of up to 1024 configurations is one cluster's, a tile per CTA: its sum runs in a
  // fixed order, and equal calls give equal bits.  (One CTA per row does so too: whole
  // calls of kernel = 2, Z = 864, FP64, 32 rows, 62 ms against 39.)
  if (S.Zslot <= 1024) {
    unsigned c = 1;
    while (c < tiles) c *= 2;
    return c == 1 ? go(k_project<T, false>, 1u, 1u, 1, 0) : go(k_project<T, true>, c, c, 1, 1);
  }
  // a CTA takes up to 8 tiles of configurations (its L costs one tile's loads),
  // fewer where the rows alone would not give every SM several CTAs
  const long long per = std::min<long long>(8, std::max<long long>(1, tiles * rows / (kChipSms * 12)));
  return go(k_project<T, false>, (unsigned)((tiles + per - 1) / per), 1u, per, 0);
}

#define RP_INTEGRAL_INST(T)                                                                       \
  template cudaError_t launch_plan_integral<T>(const IntegralIn*, const IntegralIn*, int, int, T*, \
                                               int2*, double*, cudaStream_t);                      \
  template cudaError_t launch_project<T>(const SysTab<T>&, const T*, const T*, const int2*,        \
                                         const int*, const int2*, int, const int*, int, int,       \
                                         double*, cudaStream_t);
RP_INTEGRAL_INST(float)
RP_INTEGRAL_INST(double)
#undef RP_INTEGRAL_INST

}  // namespace rp
