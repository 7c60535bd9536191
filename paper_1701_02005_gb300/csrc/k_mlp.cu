// MLP of the learned wall model: 40 -> 128 -> 128 -> 128 -> 128 -> 5, erf-based
// GELU on the hidden layers, linear output.  The network runs on the tensor
// cores (k_mlp_tc.cu: BF16 weights and activation operands, FP32 accumulation;
// the gradients of the mean-squared error of the normalised outputs with the
// same BF16-operand GEMMs, batch sums through per-CTA partials in a fixed order:
// deterministic); training keeps FP32 master weights and applies Adam (Kingma &
// Ba 2015).
// (No counterpart in the paper.)
#include <cuda_bf16.h>

#include "pnp_common.cuh"
#include "pnp_wall.cuh"

namespace pnp {

MlpDims mlp_dims() {
  MlpDims d{};
  const int ins[kMlpLayers] = {kMlpIn, kMlpHidden, kMlpHidden, kMlpHidden, kMlpHidden};
  const int outs[kMlpLayers] = {kMlpHidden, kMlpHidden, kMlpHidden, kMlpHidden, kMlpOut};
  size_t off = 0;
  for (int l = 0; l < kMlpLayers; ++l) {
    d.in[l] = ins[l];
    d.out[l] = outs[l];
    d.woff[l] = off;
    off += (size_t)ins[l] * outs[l];
    d.boff[l] = off;
    off += outs[l];
  }
  d.nparam = off;
  return d;
}

__global__ void k_mlp_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                           float* __restrict__ v, size_t n, float lr, float b1, float b2, float eps, float c1,
                           float c2) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const float gt = g[t];
  const float mt = b1 * m[t] + (1.f - b1) * gt;
  const float vt = b2 * v[t] + (1.f - b2) * gt * gt;
  m[t] = mt;
  v[t] = vt;
  p[t] -= lr * (mt / c1) / (sqrtf(vt / c2) + eps);
}

cudaError_t mlp_adam(const MlpBufs& b, size_t nparam, float lr, float beta1, float beta2, float eps, int t,
                     cudaStream_t s) {
  const float c1 = 1.f - powf(beta1, (float)t), c2 = 1.f - powf(beta2, (float)t);
  k_mlp_adam<<<(unsigned)((nparam + 255) / 256), 256, 0, s>>>(b.param, b.grad, b.m, b.v, nparam, lr, beta1, beta2,
                                                              eps, c1, c2);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return mlp_make_images(b.param, b.wimg, s);
}

}  // namespace pnp
