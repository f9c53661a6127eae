// The LSTM cell's arithmetic (gates i, f, g, o; App. "Agent Design"), shared by the
// step-by-step cell kernels and the whole-segment cluster kernels. Fused multiply-adds are
// written out, so that both form every value by the same operations whatever the compiler
// would contract in either.
#pragma once

#include "common.cuh"

namespace ddppo {

__device__ __forceinline__ float lstm_sigm(float x) { return 1.0f / (1.0f + expf(-x)); }

// pre-activations z* -> gates i, f, g, o, new cell state c and output h; cp is the masked
// previous cell state
__device__ __forceinline__ void lstm_cell_fwd(float zi, float zf, float zg, float zo, float cp,
                                              float& i, float& f, float& g, float& o, float& c,
                                              float& h) {
  i = lstm_sigm(zi);
  f = lstm_sigm(zf);
  g = tanhf(zg);
  o = lstm_sigm(zo);
  c = __fmaf_rn(i, g, __fmul_rn(f, cp));
  h = o * tanhf(c);
}

// gate gradients of one cell: dh is the gradient of h, dc_in the carried gradient of c
// (added when carry), cp the masked previous cell state; dc_out the gradient carried on
__device__ __forceinline__ void lstm_cell_bwd(float i, float f, float g, float o, float c, float cp,
                                              float dh, bool carry, float dc_in, float& dzi,
                                              float& dzf, float& dzg, float& dzo, float& dc_out) {
  const float tc = tanhf(c);
  float dc = __fmul_rn(__fmul_rn(dh, o), __fmaf_rn(-tc, tc, 1.f));
  if (carry) dc = __fadd_rn(dc, dc_in);
  dzi = dc * g * i * (1.f - i);
  dzf = dc * cp * f * (1.f - f);
  dzg = dc * i * __fmaf_rn(-g, g, 1.f);
  dzo = dh * tc * o * (1.f - o);
  dc_out = dc * f;
}

}  // namespace ddppo
