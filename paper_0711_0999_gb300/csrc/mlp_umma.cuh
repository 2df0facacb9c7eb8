// Tensor-core kernels of the warm-start network (17 -> 4 x 256 tanh -> 2),
// used by mlp.cu; not part of the C ABI.
#pragma once

#include "common.cuh"

namespace nedmft {

constexpr int kMlpIn = 17, kMlpHid = 256, kMlpOut = 2, kMlpLayers = 5;

// Offset of layer l's weights in the parameter array (its biases follow them).
constexpr size_t mlp_w_off(int l) {
  const int dims[kMlpLayers + 1] = {kMlpIn, kMlpHid, kMlpHid, kMlpHid, kMlpHid, kMlpOut};
  size_t o = 0;
  for (int i = 0; i < l; ++i) o += (size_t)dims[i] * dims[i + 1] + dims[i + 1];
  return o;
}

// Where the network's inputs come from: n x 17 features, or the pairs (a, b)
// = (s / nc, s % nc) of a contour's rows: a table of six values per row, the
// tanh of the relative time per pair, and the five features all pairs share.
struct MlpInput {
  const float* x = nullptr;      // n x 17
  const float* row = nullptr;    // nc x 6
  const float* rel = nullptr;    // nc x nc
  int nc = 0;
  float u = 0.f, e = 0.f, dt = 0.f;
};

// Bytes of the packed weights, and of everything a gradient keeps for n samples.
size_t mlp_forward_scratch();
size_t mlp_grad_scratch(int n);

// y[s] = network(input s), s < n; accumulate: y[s] = (first ? 0 : y[s]) + scale network(input s).
// Packs the weights when `pack` (scratch then holds them for later calls).
int mlp_forward(const float* params, const MlpInput& in, size_t n, float* y, bool accumulate, bool first, float scale,
                bool pack, char* scratch, cudaStream_t st);
// Mean squared error and its gradient.
int mlp_gradient(const float* params, const float* x, const float* target, int n, float* grad, float* loss,
                 char* scratch, cudaStream_t st);
int mlp_set_wait_ns(uint64_t ns, cudaStream_t st);

}  // namespace nedmft
