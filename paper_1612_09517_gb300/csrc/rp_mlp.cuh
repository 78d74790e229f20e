// Forward pass of the control-variate network in one kernel (rp_mlp.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace rp {

constexpr int kMlpMaxHidden = 256;  // widest hidden layer of the fused pass
constexpr int kMlpMaxLayers = 8;

struct MlpNet {
  const __nv_bfloat16* wbf;  // all weights, flat
  const float* params;       // FP32 parameters, flat (biases)
  long long w_off[kMlpMaxLayers + 1], b_off[kMlpMaxLayers + 1];
  int d_in, hidden, layers;
};

// Whether the fused pass takes the network, and the values of packed weights it needs.
bool mlp_fused(const MlpNet& net);
size_t mlp_packed_values(const MlpNet& net);

// Hidden-layer weights in the order the kernel's copies read them.
cudaError_t launch_mlp_pack(const MlpNet& net, __nv_bfloat16* packed, cudaStream_t st);

// g of n feature rows x (n x d_in).  fields NULL: x as it is, g to out (n floats).  Else
// the last feature is fields[f] * inv_scale for each of n_fields fields, and acc[2 f],
// acc[2 f + 1] receive the sums of g and g^2 (FP64, added).  err: a device word, zero
// before, nonzero after a bounded wait gave up.
cudaError_t launch_mlp(const MlpNet& net, const __nv_bfloat16* packed, int n, const float* x,
                       const double* fields, int n_fields, double inv_scale, float* out,
                       double* acc, int* err, cudaStream_t st);

}  // namespace rp
