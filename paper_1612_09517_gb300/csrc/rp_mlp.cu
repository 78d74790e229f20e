// Forward pass of the control-variate network on the tensor cores.
//
// The tensor core's FP32 sums are truncated, not rounded to nearest, and a truncated sum is
// too small in magnitude: every layer's result shrinks, which no averaging over samples
// removes.  So the large products are summed without any rounding.  The activations of a
// row and the weights of an output are each cut at 2^-8 of their largest magnitude,
//   a = a1 + a2 + a3,  w = w1 + w2,
// a1 and w1 whole multiples (at most 128 in magnitude) of a power of two of the row or
// output.  A sum of up to 256 products a1 w1 then has at most 23 bits: exact in FP32 in any
// order.  It has an accumulator of its own.  a2, a3 (BF16) and w2 hold what is left, and
// the products with them, 2^-8 of the sum and smaller, go to a second accumulator, where
// truncation is far below the FP32 rounding of the result.  Before the cut each input takes
// the power of two of its largest weight, which its weights give up: the cut then keeps
// what contributes, also where inputs differ by orders of magnitude (a field of 500 field
// scales: rms error 2.6e-6 without, 2.1e-7 with it).  w1 + w2 is the BF16 weight
// exactly, a1 + a2 + a3 the FP32 activation to 2^-26 of the row's largest.  Errors of g,
// E[g] and its variance against 64 bits, 4096 samples, 3 x 256, means over six networks:
// 2.2e-7 (rms), 2.2e-8 and 2.8e-8; the layer-by-layer pass in rounded FP32 has 6.4e-7,
// 1.6e-8 and 3.3e-8; one accumulator drained every 32 inputs had 2.9e-7, 7.7e-8, 3.1e-7.
// (Rows and outputs whose largest is below 2^-119 or from 2^126 on are not cut: a1 is then
// the upper eight bits of a, w1 zero.)
//
// A row with an infinity or NaN among its activations would turn every product of the split
// into NaN, where an infinity passes an FP32 multiply-add.  The tensor cores get zeros for
// its finite values, and the sums of the infinite and NaN ones are formed beside them.
//
// One CTA takes 128 feature rows through all layers: activations never leave the chip.
// 512 threads hold the sums of one row and a quarter of the outputs each, apply bias
// and SiLU and write the split activations as the next layer's A operand (256 threads
// with half a row each spilled: with the issuing warp they have 168 registers); one
// thread of another warp streams weight tiles (w1 and w2 of 16 inputs x all outputs in
// turn, one bulk copy each, 32 KB in flight) and issues the MMAs.  All waits are bounded.
//
// Bounds: within a CTA the layers of a tile are a chain (products, SiLU, next operand).
// 65536 rows x 8 fields, 46 inputs, 3 x 256: 9.3 ms as FP32 CUDA-core products with a pass
// over memory per layer and activation, 2.2 ms with the drained accumulator and here (2.1
// without the scales).
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
constexpr int kTileK = 16;  // inputs per weight tile
constexpr int kRing = 32 * 1024;  // bytes of weight tiles in flight

// Outputs padded to the tile of an instance, inputs of the first layer to whole tiles
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
// Eight columns of each accumulator.
__device__ __forceinline__ void tmem_ld8x2(unsigned a, unsigned b, float (&v)[8], float (&w)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
        "=f"(v[7]), "=f"(w[0]), "=f"(w[1]), "=f"(w[2]), "=f"(w[3]), "=f"(w[4]), "=f"(w[5]),
        "=f"(w[6]), "=f"(w[7])
      : "r"(a), "r"(b)
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
__device__ __forceinline__ void worker_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kWorkers) : "memory");
}

// The power of two that cuts numbers of magnitude up to `top`: multiples of it reach 128 at
// `top`.  Zero where nothing is cut: tops whose powers leave the range of FP32.
struct Cut {
  float grid, inv;
};
// top: the bits of the magnitude, which compare as integers, NaN above infinity
__device__ __forceinline__ unsigned mag(float v) { return __float_as_uint(v) & 0x7fffffffu; }
__device__ __forceinline__ Cut cut_of(unsigned top) {
  const int e = (int)(top >> 23) - 126;  // 2^(e-1) <= top < 2^e
  if (e < -118 || e > 126) return {0.f, 0.f};
  return {__uint_as_float((unsigned)(e + 120) << 23), __uint_as_float((unsigned)(134 - e) << 23)};
}
// v less its multiple of the grid (to nearest), which goes to `high`; both exact.
__device__ __forceinline__ float cut_high(const Cut& c, float v, float& high) {
  const float q = fmaf(v, c.inv, 12582912.f) - 12582912.f;  // 1.5 2^23: rounds to an integer
  high = q * c.grid;
  return fmaf(-q, c.grid, v);
}

// The packed weights: tiles in the order of the stream, tile t as [part][input / 8]
// [output / 8][8 outputs][8 inputs], part 0 w1 and 1 w2; then, in FP32, the biases of the
// hidden layers and the output layer's weights, HP each, and the scales, 256 per layer.
// Input k of layer l has the power of two of its largest weight, relative to that of the
// layer and at least 2^-60.  Each block finds the scales of its layer and takes 32 of its
// outputs, one per warp.
constexpr int kMaxIn = 256, kPackThreads = 1024;
__global__ void __launch_bounds__(kPackThreads) k_mlp_pack(const MlpNet N, int HP,
                                                           __nv_bfloat16* __restrict__ out,
                                                           long long total) {
  __shared__ unsigned tops[kMaxIn], all;
  __shared__ float sc[kMaxIn];
  const int tid = threadIdx.x, lane = tid & 31, per = HP / 32;
  const int l = (int)blockIdx.x / per, o = (int)blockIdx.x % per * 32 + (tid >> 5);
  const int in = l == 0 ? N.d_in : N.hidden, pad = l == 0 ? pad_in(N.d_in) : HP;
  float* aux = reinterpret_cast<float*>(out + total);
  if (tid < kMaxIn) tops[tid] = 0u;
  if (tid == 0) all = 0u;
  __syncthreads();
  {
    const int k = tid % kMaxIn;
    unsigned m = 0u;  // magnitudes compare as integers
    if (k < in) {
      const __nv_bfloat16* w = N.wbf + N.w_off[l] + k;
#pragma unroll 16
      for (int q = tid / kMaxIn; q < N.hidden; q += kPackThreads / kMaxIn)
        m = max(m, mag(__bfloat162float(w[(long long)q * in])));
      atomicMax(&tops[k], m);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) atomicMax(&all, m);
  }
  __syncthreads();
  if (tid < kMaxIn) {
    const int e = max((int)(tops[tid] >> 23) - (int)(all >> 23), -60);
    sc[tid] = __uint_as_float((unsigned)(127 + e) << 23);
    if (blockIdx.x % per == 0) aux[(N.layers + 1) * HP + l * kMaxIn + tid] = sc[tid];
  }
  // biases, and the output layer's weights from the blocks of the last hidden layer
  if (lane == 0) {
    const bool on = o < N.hidden;
    aux[l * HP + o] = on ? N.params[N.b_off[l] + o] : 0.f;
    if (l == N.layers - 1) aux[N.layers * HP + o] = on ? __bfloat162float(N.wbf[N.w_off[N.layers] + o]) : 0.f;
  }
  __syncthreads();
  const int t0 = l == 0 ? 0 : (pad_in(N.d_in) + (l - 1) * HP) / kTileK;  // first tile of the layer
  const __nv_bfloat16* w = N.wbf + N.w_off[l] + (long long)o * in;
  const bool on = o < N.hidden;
  float v[kMaxIn / 32];
  unsigned top = 0u;
#pragma unroll
  for (int i = 0; i < kMaxIn / 32; ++i) {
    const int k = i * 32 + lane;
    v[i] = on && k < in ? __bfloat162float(w[k]) / sc[k] : 0.f;  // powers of two: exact
    top = max(top, mag(v[i]));
  }
  const Cut c = cut_of(__reduce_max_sync(0xffffffffu, top));
#pragma unroll
  for (int i = 0; i < kMaxIn / 32; ++i) {
    const int k = i * 32 + lane;
    if (k >= pad) break;
    float high;
    const float low = cut_high(c, v[i], high);
    __nv_bfloat16* d = out + (size_t)(2 * (t0 + k / kTileK)) * HP * kTileK +
                       (k % kTileK) / 8 * (HP * 8) + o * 8 + k % 8;
    d[0] = __float2bfloat16(high);
    d[(size_t)HP * kTileK] = __float2bfloat16(low);
  }
}

// Eight activations of a row that is not cut: eight bits each (truncated: rounding could
// reach infinity), or what is not finite of a row that holds such values (`odd`).
__device__ __noinline__ void put8_uncut(unsigned char* d, unsigned part, bool odd, float4 lo, float4 hi) {
  const float v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
  __nv_bfloat16 h[3][8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const unsigned b = __float_as_uint(v[i]);
    float r = v[i];
    if (odd) {
      const bool finite = (b & 0x7f800000u) != 0x7f800000u;
      h[0][i] = __ushort_as_bfloat16(finite ? 0 : (b & 0x7fffffu) ? 0x7fff : (unsigned short)(b >> 16));
      r = 0.f;
    } else {
      h[0][i] = __ushort_as_bfloat16((unsigned short)(b >> 16));
      r -= __bfloat162float(h[0][i]);
    }
    h[1][i] = __float2bfloat16(r);
    h[2][i] = __float2bfloat16(r - __bfloat162float(h[1][i]));
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) *reinterpret_cast<uint4*>(d + q * part) = *reinterpret_cast<const uint4*>(h[q]);
}

// Eight activations of a row to the three parts of the A operand (`part` bytes apart).
__device__ __forceinline__ void put8(unsigned char* A, unsigned part, int row, int k8, const Cut& c,
                                     bool odd, float (&v)[8]) {
  unsigned char* d = A + (unsigned)k8 * (kRows * 16) + (unsigned)row * 16;
  if (c.inv == 0.f) {
    put8_uncut(d, part, odd, make_float4(v[0], v[1], v[2], v[3]), make_float4(v[4], v[5], v[6], v[7]));
    return;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    unsigned w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float x = v[2 * i], y = v[2 * i + 1];
      if (q == 0) {
        v[2 * i] = cut_high(c, x, x);
        v[2 * i + 1] = cut_high(c, y, y);
      }
      const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
      w[i] = *reinterpret_cast<const unsigned*>(&h);
      if (q > 0) {
        v[2 * i] = x - __low2float(h);
        v[2 * i + 1] = y - __high2float(h);
      }
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
  constexpr int kTiles = kRing / (int)kTileBytes;  // 4 to 16
  extern __shared__ __align__(128) unsigned char mlp_smem[];
  // full[tile], empty[tile], then: a layer's products are done
  __shared__ __align__(8) unsigned long long bars[2 * kTiles + 1];
  __shared__ unsigned tmem_slot;
  // largest magnitudes of the quarters of a row; at the end their shares of g
  __shared__ __align__(4) unsigned quarters[4][kRows];
  __shared__ double moments[4][2];
  unsigned char* A = mlp_smem;  // three parts of [input / 8][row][8 inputs]
  const unsigned a_base = smem_u32(mlp_smem), w_base = a_base + 3 * part;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto full = [&](int i) { return smem_u32(&bars[i]); };
  auto empty = [&](int i) { return smem_u32(&bars[kTiles + i]); };
  const unsigned ready = smem_u32(&bars[2 * kTiles]);
  if (tid == 0) {
    for (int i = 0; i < 2 * kTiles + 1; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[i])) : "memory");
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
  const int per_unit = 2 * (K0 / kTileK + (N.layers - 1) * (HP / kTileK));
  const float* aux = reinterpret_cast<const float*>(packed + (size_t)per_unit * (HP * kTileK));
  const float* scales = aux + (N.layers + 1) * HP;
  const long long total = (long long)mine * per_unit;  // weight tiles this CTA takes
  long long loaded = 0, used = 0;                      // of the copying thread
  unsigned phase = 0;                                  // of `ready`
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
  // the cut of a worker's row from the largest magnitude of its quarter
  bool odd = false;  // the row holds infinities or NaN
  auto row_cut = [&](unsigned top) {
    quarters[quarter][row] = top;
    worker_sync();
    top = max(max(quarters[0][row], quarters[1][row]), max(quarters[2][row], quarters[3][row]));
    odd = top >= 0x7f800000u;
    return cut_of(top);
  };
  for (int iu = 0; iu < mine; ++iu) {
    const int u = (int)blockIdx.x + iu * (int)gridDim.x;
    const int f = u % nf, i0 = u / nf * kRows;
    const bool valid = i0 + row < n;
    if (warp < kWorkers / 32) {
      // features as the first A operand, zero beyond d_in and beyond the rows
      const float* xi = x + (size_t)(i0 + row) * N.d_in;
      const float xb = fields ? (float)(fields[f] * inv_scale) : 0.f;
      auto features = [&](int k8, float (&v)[8]) {
        const float4* m = reinterpret_cast<const float4*>(scales) + 2 * k8;
        const float4 m0 = __ldg(m), m1 = __ldg(m + 1);
        const float mm[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int k = 8 * k8 + j;
          v[j] = 0.f;
          if (valid && k < N.d_in) v[j] = (fields && k == N.d_in - 1 ? xb : xi[k]) * mm[j];
        }
      };
      float v[8];
      unsigned top = 0u;
      for (int k8 = quarter; k8 < K0 / 8; k8 += 4) {
        features(k8, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) top = max(top, mag(v[j]));
      }
      const Cut c = row_cut(top);
      for (int k8 = quarter; k8 < K0 / 8; k8 += 4) {
        features(k8, v);
        put8(A, part, row, k8, c, odd, v);
      }
    }
    for (int l = 0; l < N.layers; ++l) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (__syncthreads_or(failed)) goto done;  // all threads
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int nt = (l == 0 ? K0 : HP) / kTileK;
      if (warp == kWorkers / 32) {
        if (lane == 0) {
          const uint32_t id = idesc_bf16(kRows, HP);
          // the slot that tile p was in, once the MMAs that read it are done
          auto refill = [&](long long before) {
            while (!failed && loaded < total && loaded - kTiles < before) {
              const long long p = loaded - kTiles;
              if (wait(empty((int)(p % kTiles)), (unsigned)(p / kTiles) & 1u)) load_next();
              else failed = 1;
            }
          };
          for (int t = 0; t < 2 * nt && !failed; ++t) {
            const int s = (int)(used % kTiles), low = t & 1;
            if (!wait(full(s), (unsigned)(used / kTiles) & 1u)) {
              failed = 1;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t b = umma_desc(w_base + (unsigned)s * kTileBytes, HP * 16, 128);
            // a1 w1 to the first accumulator, all other products to the second
#pragma unroll
            for (int q = 2; q >= 0; --q) {
              const bool exact = q == 0 && !low;
              mma_bf16(tmem + (exact ? 0u : (unsigned)HP),
                       umma_desc(a_base + (unsigned)q * part + (unsigned)(t >> 1) * (2 * kRows * 16),
                                 kRows * 16, 128),
                       b, id, t == 0 && (exact || q == 2) ? 0u : 1u);
            }
            mma_commit(empty(s));
            ++used;
            refill(used - 1);
          }
          if (!failed) {
            mma_commit(ready);
            refill(used);
          }
        }
        failed = __shfl_sync(0xffffffffu, failed, 0);
        continue;
      }
      if (!failed && !wait(ready, phase)) failed = 1;
      phase ^= 1u;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // sums, bias, SiLU, then the next layer's operand (every MMA of this layer is done) or
      // the output layer's products
      // (outputs beyond hidden have zero weights and bias: SiLU gives zero)
      const bool last = l == N.layers - 1;
      const float4* bias = reinterpret_cast<const float4*>(aux + l * HP + quarter * CPT);
      const float4* wo = reinterpret_cast<const float4*>(aux + N.layers * HP + quarter * CPT);
      const float4* next = reinterpret_cast<const float4*>(scales + (l + 1) * kMaxIn + quarter * CPT);
      const unsigned col = tmem + (((unsigned)(warp & 3) * 32u) << 16) + (unsigned)(quarter * CPT);
      // sums of an odd row: its values that are not finite lie in the first part of the
      // operand, the other two have room for the sums of this thread's outputs
      auto odd_sums = [&](int o) {  // of outputs o .. o + 3
        return reinterpret_cast<float4*>(A + (unsigned)(1 + ((o >> 2) & 1)) * part +
                                         (unsigned)(o / 8) * (kRows * 16) + (unsigned)row * 16);
      };
      if (odd) {
        const int in = l == 0 ? N.d_in : N.hidden;
#pragma unroll 1
        for (int o = quarter * CPT; o < (quarter + 1) * CPT; ++o) {
          float sum = 0.f;
          const __nv_bfloat16* w = N.wbf + N.w_off[l] + (long long)o * in;
#pragma unroll 1
          for (int k = 0; o < N.hidden && k < in; ++k) {
            const float a = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(
                A + (unsigned)(k / 8) * (kRows * 16) + (unsigned)row * 16 + (unsigned)(k % 8) * 2));
            if (a != 0.f) sum = fmaf(a, __bfloat162float(w[k]), sum);
          }
          reinterpret_cast<float*>(odd_sums(o))[o & 3] = sum;
        }
      }
      float z[CPT];
      unsigned top = 0u;
#pragma unroll
      for (int i = 0; i < CPT; i += 8) {
        float v[8], w[8];
        tmem_ld8x2(col + (unsigned)i, col + (unsigned)(HP + i), v, w);
#pragma unroll
        for (int j = 0; j < 8; j += 4) {
          const float4 b = __ldg(bias + (i + j) / 4);
          const float4 m = last ? make_float4(1.f, 1.f, 1.f, 1.f) : __ldg(next + (i + j) / 4);
          const float bb[4] = {b.x, b.y, b.z, b.w}, mm[4] = {m.x, m.y, m.z, m.w};
          if (odd) {
            const float4 q = *odd_sums(quarter * CPT + i + j);
            v[j] = q.x, v[j + 1] = q.y, v[j + 2] = q.z, v[j + 3] = q.w;
            w[j] = w[j + 1] = w[j + 2] = w[j + 3] = 0.f;
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float a = (v[j + k] + w[j + k]) + bb[k];
            z[i + j + k] = a / (1.f + __expf(-a)) * mm[k];
            top = max(top, mag(z[i + j + k]));
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (!last) {
        const Cut c = row_cut(top);
#pragma unroll
        for (int i = 0; i < CPT; i += 8) {
          float v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = z[i + j];
          put8(A, part, row, (quarter * CPT + i) / 8, c, odd, v);
        }
        continue;
      }
      float g = 0.f;
#pragma unroll
      for (int i = 0; i < CPT; i += 4) {
        const float4 w = __ldg(wo + i / 4);
        g = fmaf(z[i + 3], w.w, fmaf(z[i + 2], w.z, fmaf(z[i + 1], w.y, fmaf(z[i], w.x, g))));
      }
      quarters[quarter][row] = __float_as_uint(g);
      worker_sync();
      if (quarter == 0) {
        g = __uint_as_float(quarters[0][row]) + __uint_as_float(quarters[1][row]) +
            __uint_as_float(quarters[2][row]) + __uint_as_float(quarters[3][row]) +
            __ldg(N.params + N.b_off[N.layers]);
        if (!fields) {
          if (valid) out[i0 + row] = g;
        } else {
          const double v = valid ? (double)g : 0.0;
          const double s1 = warp_sum(v), s2 = warp_sum(v * v);
          if (lane == 0) {
            moments[warp][0] = s1;
            moments[warp][1] = s2;
          }
        }
      }
      worker_sync();  // `quarters` is free again, the moments are there
      if (fields && tid < 2)
        atomicAdd(acc + 2 * f + tid,
                  (moments[0][tid] + moments[1][tid]) + (moments[2][tid] + moments[3][tid]));
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
  const int smem = std::max((int)(3 * part) + kRing, 116 * 1024);
  cudaError_t e = smem_attr_once((const void*)kf, 3 * 2 * kRows * 256 + kRing, attr_done);
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
  return net.hidden <= kMlpMaxHidden && net.layers <= kMlpMaxLayers && pad_in(net.d_in) <= kMaxIn;
}
static long long mlp_tile_values(const MlpNet& net) {
  const int HP = pad_hidden(net.hidden);
  return 2ll * HP * (pad_in(net.d_in) + (net.layers - 1) * HP);
}
size_t mlp_packed_values(const MlpNet& net) {  // FP32 values count twice
  return (size_t)mlp_tile_values(net) +
         2 * ((size_t)(net.layers + 1) * pad_hidden(net.hidden) + (size_t)net.layers * kMaxIn);
}
cudaError_t launch_mlp_pack(const MlpNet& net, __nv_bfloat16* packed, cudaStream_t st) {
  const int HP = pad_hidden(net.hidden);
  k_mlp_pack<<<net.layers * HP / 32, kPackThreads, 0, st>>>(net, HP, packed, mlp_tile_values(net));
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
