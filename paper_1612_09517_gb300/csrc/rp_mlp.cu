// Forward pass of the control-variate network on the tensor cores.
//
// The weights are BF16 numbers; an FP32 activation is the exact sum of three (8 + 8 +
// 8 mantissa bits), so a layer is three tcgen05.mma kind::f16 products per weight tile
// with FP32 accumulators: every product is exact, as in an FP32 multiply-add of the
// same numbers.  The tensor core's FP32 sums are not rounded to nearest, and the error
// grows with the number of MMAs into one accumulator: after 32 inputs (2 MMAs of each
// part, the low parts first) the accumulator is drained into FP32 sums in registers while the other buffer fills.
//
// One CTA takes 128 feature rows through all layers: activations never leave the chip.
// 512 threads hold the sums of one row and a quarter of the outputs each, apply bias
// and SiLU and write the split activations as the next layer's A operand (256 threads
// with half a row each spilled: with the issuing warp they have 168 registers); one
// thread of another warp streams weight tiles (16 inputs x all outputs, one bulk copy each, four in
// flight) and issues the MMAs.  All waits are bounded.
//
// Bounds: within a CTA the layers of a tile are a chain (products, drain, SiLU, next
// operand); the tensor cores are busy about a quarter of the time.  65536 rows x 8
// fields, 46 inputs, 3 x 256: 9.3 ms as FP32 CUDA-core products with a pass over memory
// per layer and activation, 2.1 ms here.  Draining every 64 inputs instead of 32 takes
// 1.9 ms, but the variance of g is then off by 1.1e-6 (5e-7 as it is, 6e-7 in FP32).
#include <algorithm>
#include <atomic>

#include "rp_device.cuh"
#include "rp_mlp.cuh"
#include "rp_tc.cuh"

namespace rp {

namespace {

constexpr int kRows = 128;
constexpr int kWorkers = 512;           // four threads per row
constexpr int kMlpThreads = kWorkers + 32;
constexpr int kTileK = 16, kTiles = 4;  // inputs per weight tile, tiles in flight
constexpr int kGroup = 2;               // weight tiles per accumulator

// outputs padded to the tile of an instance, inputs of the first layer to whole tiles
inline int pad_hidden(int h) { return h <= 64 ? 64 : h <= 128 ? 128 : 256; }
__host__ __device__ inline int pad_in(int d) { return (d + kTileK - 1) / kTileK * kTileK; }

// Instruction descriptor of kind::f16: D FP32, A and B BF16, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(unsigned d, uint64_t a, uint64_t b, uint32_t idesc,
                                         unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ bool wait(unsigned bar, unsigned parity) {
  return mbar_wait<(1ll << 20)>(bar, parity);
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
  return v;
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void worker_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kWorkers) : "memory");
}

// Weight tile t of the stream: [input / 8][output / 8][8 outputs][8 inputs]; after the
// tiles the biases of the hidden layers and the output layer's weights, FP32, HP each.
__global__ void k_mlp_pack(const MlpNet N, int HP, __nv_bfloat16* __restrict__ out, long long total) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) {
    const int j = (int)(i - total), l = j / HP, o = j % HP;
    if (l > N.layers) return;
    float v = 0.f;
    if (o < N.hidden)
      v = l < N.layers ? N.params[N.b_off[l] + o] : __bfloat162float(N.wbf[N.w_off[l] + o]);
    reinterpret_cast<float*>(out + total)[j] = v;
    return;
  }
  const int tile = HP * kTileK, t = (int)(i / tile), w = (int)(i % tile);
  const int t0 = pad_in(N.d_in) / kTileK, th = HP / kTileK;
  const int l = t < t0 ? 0 : 1 + (t - t0) / th, c = t < t0 ? t : (t - t0) % th;
  const int k = c * kTileK + w / (HP * 8) * 8 + w % 8, o = w % (HP * 8) / 8;
  const int in = l == 0 ? N.d_in : N.hidden;
  out[i] = k < in && o < N.hidden ? N.wbf[N.w_off[l] + (long long)o * in + k] : __float2bfloat16(0.f);
}

// Eight activations of a row to the A operand (parts `part` bytes apart): v = hi + mid +
// lo exactly, barring underflow of the low parts.
__device__ __forceinline__ void put8(unsigned char* A, unsigned part, int row, int k8,
                                     float (&v)[8]) {
  unsigned char* d = A + (unsigned)k8 * (kRows * 16) + (unsigned)row * 16;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    unsigned w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
      w[i] = *reinterpret_cast<const unsigned*>(&h);
      v[2 * i] -= __low2float(h);
      v[2 * i + 1] -= __high2float(h);
    }
    *reinterpret_cast<uint4*>(d + q * part) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

template <int HP>
__global__ void __launch_bounds__(kMlpThreads, 1) k_mlp(
    const MlpNet N, const __nv_bfloat16* __restrict__ packed, int n, const float* __restrict__ x,
    const double* __restrict__ fields, int n_fields, double inv_scale, float* __restrict__ out,
    double* __restrict__ acc, int* __restrict__ err, unsigned part) {
  constexpr int CPT = HP / 4;  // outputs per thread
  constexpr unsigned kTileBytes = HP * kTileK * 2;
  extern __shared__ __align__(1024) unsigned char mlp_smem[];
  // full[tile], empty[tile], ready[accumulator], drained[accumulator]
  __shared__ __align__(8) unsigned long long bars[2 * kTiles + 4];
  __shared__ unsigned tmem_slot;
  __shared__ float part_g[3][kRows];
  unsigned char* A = mlp_smem;  // three parts of [input / 8][row][8 inputs]
  const unsigned a_base = smem_u32(mlp_smem), w_base = a_base + 3 * part;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto full = [&](int i) { return smem_u32(&bars[i]); };
  auto empty = [&](int i) { return smem_u32(&bars[kTiles + i]); };
  auto ready = [&](int i) { return smem_u32(&bars[2 * kTiles + i]); };
  auto drained = [&](int i) { return smem_u32(&bars[2 * kTiles + 2 + i]); };
  if (tid == 0) {
    for (int i = 0; i < 2 * kTiles + 4; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bars[i])),
                   "r"(i >= 2 * kTiles + 2 ? kWorkers : 1)
                   : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(2 * HP)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = tmem_slot;

  const int nf = fields ? n_fields : 1, blocks = (n + kRows - 1) / kRows;
  const int units = blocks * nf;
  const int mine = ((int)blockIdx.x < units) ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int K0 = pad_in(N.d_in);
  const int per_unit = K0 / kTileK + (N.layers - 1) * (HP / kTileK);
  const float* aux = reinterpret_cast<const float*>(packed + (size_t)per_unit * (HP * kTileK));
  const long long total = (long long)mine * per_unit;  // weight tiles this CTA takes
  long long loaded = 0, used = 0;                      // of the copying thread
  int groups = 0;                                      // accumulators filled so far
  int failed = 0;
  auto load_next = [&]() {
    bulk_load(w_base + (unsigned)(loaded % kTiles) * kTileBytes,
              packed + (size_t)(loaded % per_unit) * (HP * kTileK), kTileBytes,
              full((int)(loaded % kTiles)));
    ++loaded;
  };
  if (tid == kWorkers)
    while (loaded < total && loaded < kTiles) load_next();

  const int row = (warp & 3) * 32 + lane, quarter = (warp >> 2) & 3;  // of a worker
  for (int iu = 0; iu < mine; ++iu) {
    const int u = (int)blockIdx.x + iu * (int)gridDim.x;
    const int f = u % nf, i0 = u / nf * kRows;
    const bool valid = i0 + row < n;
    if (warp < kWorkers / 32) {
      // features as the first A operand, zero beyond d_in and beyond the rows
      const float* xi = x + (size_t)(i0 + row) * N.d_in;
      const float xb = fields ? (float)(fields[f] * inv_scale) : 0.f;
      for (int k8 = quarter; k8 < K0 / 8; k8 += 4) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int k = 8 * k8 + j;
          v[j] = 0.f;
          if (valid && k < N.d_in) v[j] = fields && k == N.d_in - 1 ? xb : xi[k];
        }
        put8(A, part, row, k8, v);
      }
    }
    for (int l = 0; l < N.layers; ++l) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (__syncthreads_or(failed)) goto done;  // all threads
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int nt = (l == 0 ? K0 : HP) / kTileK, ng = (nt + kGroup - 1) / kGroup;
      if (warp == kWorkers / 32) {
        if (lane == 0) {
          const uint32_t id = idesc_bf16(kRows, HP);
          for (int g = 0; g < ng; ++g) {
            const int b = (groups + g) & 1, use = (groups + g) >> 1;  // earlier uses of it
            const int t0 = g * kGroup, t1 = min(nt, t0 + kGroup);
            if (use > 0 && !wait(drained(b), (unsigned)(use - 1) & 1u)) failed = 1;
            for (int t = t0; t < t1 && !failed; ++t) {
              const long long w = used + (t - t0);
              if (!wait(full((int)(w % kTiles)), (unsigned)(w / kTiles) & 1u)) failed = 1;
            }
            if (failed) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // the low parts first: only sums with the high part round at full size
#pragma unroll
            for (int q = 2; q >= 0; --q)
              for (int t = t0; t < t1; ++t) {
                const int s = (int)((used + (t - t0)) % kTiles);
                mma_bf16(tmem + (unsigned)(b * HP),
                         umma_desc(a_base + (unsigned)q * part + (unsigned)t * (2 * kRows * 16),
                                   kRows * 16, 128),
                         umma_desc(w_base + (unsigned)s * kTileBytes, HP * 16, 128), id,
                         t == t0 && q == 2 ? 0u : 1u);
              }
            for (int t = t0; t < t1; ++t) mma_commit(empty((int)((used + (t - t0)) % kTiles)));
            mma_commit(ready(b));
            // tiles of the previous group are free once its MMAs are done
            for (long long p = loaded - kTiles; p < used && loaded < total; ++p) {
              if (!wait(empty((int)(p % kTiles)), (unsigned)(p / kTiles) & 1u)) {
                failed = 1;
                break;
              }
              load_next();
            }
            used += t1 - t0;
          }
        }
        groups += ng;
        failed = __shfl_sync(0xffffffffu, failed, 0);
        continue;
      }
      float z[CPT];
      for (int g = 0; g < ng; ++g) {
        const int b = (groups + g) & 1;
        if (!failed && !wait(ready(b), (unsigned)((groups + g) >> 1) & 1u)) failed = 1;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const unsigned col = tmem + (((unsigned)(warp & 3) * 32u) << 16) + (unsigned)(b * HP + quarter * CPT);
#pragma unroll
        for (int i = 0; i < CPT; i += 16) {
          float v[16];
          tmem_ld16(col + (unsigned)i, v);
#pragma unroll
          for (int j = 0; j < 16; ++j) z[i + j] = g == 0 ? v[j] : z[i + j] + v[j];
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(drained(b));
      }
      groups += ng;
      // bias, SiLU, then the next layer's operand (every MMA of this layer is done) or
      // the output layer's products
      // (outputs beyond hidden have zero weights and bias: SiLU gives zero)
      const bool last = l == N.layers - 1;
      const float4* bias = reinterpret_cast<const float4*>(aux + l * HP + quarter * CPT);
      const float4* wo = reinterpret_cast<const float4*>(aux + N.layers * HP + quarter * CPT);
      float g = 0.f;
#pragma unroll
      for (int i = 0; i < CPT; i += 8) {
        const float4 b0 = __ldg(bias + i / 4), b1 = __ldg(bias + i / 4 + 1);
        float v[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float a = z[i + j] + v[j];
          v[j] = a / (1.f + __expf(-a));
        }
        if (!last) {
          put8(A, part, row, (quarter * CPT + i) / 8, v);
        } else {
          const float4 w0 = __ldg(wo + i / 4), w1 = __ldg(wo + i / 4 + 1);
          const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
          for (int j = 0; j < 8; ++j) g = fmaf(v[j], w[j], g);
        }
      }
      if (last) {
        if (quarter > 0) part_g[quarter - 1][row] = g;
        worker_sync();
        if (quarter == 0) {
          g += part_g[0][row] + part_g[1][row] + part_g[2][row] + __ldg(N.params + N.b_off[N.layers]);
          if (!fields) {
            if (valid) out[i0 + row] = g;
          } else {
            const double v = valid ? (double)g : 0.0;
            const double s1 = warp_sum(v), s2 = warp_sum(v * v);
            if (lane == 0) {
              atomicAdd(acc + 2 * f, s1);
              atomicAdd(acc + 2 * f + 1, s2);
            }
          }
        }
        worker_sync();  // part_g is free again
      }
    }
  }
done:
  if (failed) atomicExch(err, 1);
  // copies and MMAs in flight land before shared and tensor memory are given back
  if (tid == kWorkers) {
    if (used > 0 && !wait(empty((int)((used - 1) % kTiles)), (unsigned)((used - 1) / kTiles) & 1u))
      atomicExch(err, 1);
    for (long long t = used; t < loaded; ++t)
      if (!wait(full((int)(t % kTiles)), (unsigned)(t / kTiles) & 1u)) atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * HP));
}

template <int HP>
cudaError_t launch_mlp_of(const MlpNet& net, const __nv_bfloat16* packed, int n, const float* x,
                          const double* fields, int n_fields, double inv_scale, float* out,
                          double* acc, int* err, cudaStream_t st) {
  static std::atomic<unsigned long long> attr_done;
  const auto kf = k_mlp<HP>;
  const int ka = std::max(HP, pad_in(net.d_in));
  const unsigned part = (unsigned)ka * kRows * 2;
  // at least 116 KB: one CTA per SM, which owns the tensor memory it asks for
  const int smem = std::max((int)(3 * part + kTiles * HP * kTileK * 2), 116 * 1024);
  cudaError_t e = smem_attr_once((const void*)kf, 3 * 2 * kRows * 256 + kTiles * 256 * kTileK * 2, attr_done);
  if (e != cudaSuccess) return e;
  int dev = 0, n_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const long long units = (long long)((n + kRows - 1) / kRows) * (fields ? n_fields : 1);
  kf<<<(unsigned)std::min<long long>(units, n_sm), kMlpThreads, smem, st>>>(
      net, packed, n, x, fields, n_fields, inv_scale, out, acc, err, part);
  return cudaGetLastError();
}

}  // namespace

bool mlp_fused(const MlpNet& net) {
  return net.hidden <= kMlpMaxHidden && net.layers <= kMlpMaxLayers && pad_in(net.d_in) <= 256;
}
static long long mlp_tile_values(const MlpNet& net) {
  const int HP = pad_hidden(net.hidden);
  return (long long)HP * (pad_in(net.d_in) + (net.layers - 1) * HP);
}
size_t mlp_packed_values(const MlpNet& net) {  // FP32 values count twice
  return (size_t)mlp_tile_values(net) + 2 * (size_t)(net.layers + 1) * pad_hidden(net.hidden);
}
cudaError_t launch_mlp_pack(const MlpNet& net, __nv_bfloat16* packed, cudaStream_t st) {
  const int HP = pad_hidden(net.hidden);
  const long long total = mlp_tile_values(net), threads = total + (net.layers + 1) * HP;
  k_mlp_pack<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(net, HP, packed, total);
  return cudaGetLastError();
}
cudaError_t launch_mlp(const MlpNet& net, const __nv_bfloat16* packed, int n, const float* x,
                       const double* fields, int n_fields, double inv_scale, float* out,
                       double* acc, int* err, cudaStream_t st) {
  if (n <= 0 || (fields && n_fields <= 0)) return cudaSuccess;
  switch (pad_hidden(net.hidden)) {
    case 64: return launch_mlp_of<64>(net, packed, n, x, fields, n_fields, inv_scale, out, acc, err, st);
    case 128: return launch_mlp_of<128>(net, packed, n, x, fields, n_fields, inv_scale, out, acc, err, st);
    default: return launch_mlp_of<256>(net, packed, n, x, fields, n_fields, inv_scale, out, acc, err, st);
  }
}

}  // namespace rp
