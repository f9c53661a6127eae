// Generalised advantage estimation (Sec. 4 "Training": gamma 0.99, GAE tau 0.95) as a
// reverse scan of affine maps.
//
// A_t = delta_t + c_t A_{t+1} with delta_t = r_t + gamma (1-d_t) V_{t+1} - V_t and
// c_t = gamma lam (1-d_t) is an affine recurrence. A CTA stages a [T, 32-env] tile of
// (delta, c) into shared memory with coalesced loads. Its 16 warps split T; lane = env, so
// every shared-memory access is one row of 32 banks. Each warp composes the maps of its
// steps, the warps' maps meet in shared memory, and each warp replays its steps from the
// value entering them, storing one coalesced row a step.
//
// Bound: HBM for many envs (17 bytes a sample), a launch's latency for one rollout of 64.
// A warp per env with the lanes splitting T read shared memory 32 values deep in one bank;
// a call then took 13.2 us at 128 steps x 64 envs, 24.8 at 256 x 64 and 51 at 128 x 16384.
// Here 8.8, 9.9 and 10.9 (an empty call: 8.5).
#include "common.cuh"

namespace ddppo {

constexpr int kGaeWarps = 16;

__global__ void __launch_bounds__(kGaeWarps * 32) gae_kernel(const float* __restrict__ r,
                                                             const uint8_t* __restrict__ d,
                                                             const float* __restrict__ v, int T, int E,
                                                             float gamma, float lam,
                                                             float* __restrict__ adv,
                                                             float* __restrict__ ret) {
  DDPPO_PDL_ENTRY();
  extern __shared__ float sh[];
  float* sdelta = sh;           // [T][32]
  float* sc = sh + T * 32;      // [T][32]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
#pragma unroll 8
  for (int t = w; t < T; t += kGaeWarps) {
    float de = 0.f, c = 0.f;
    if (e < E) {
      const float nd = d[(size_t)t * E + e] ? 0.f : 1.f;
      de = r[(size_t)t * E + e] + gamma * nd * v[(size_t)(t + 1) * E + e] - v[(size_t)t * E + e];
      c = gamma * lam * nd;
    }
    sdelta[t * 32 + lane] = de;
    sc[t * 32 + lane] = c;
  }
  __syncthreads();
  const int L = (T + kGaeWarps - 1) / kGaeWarps;
  const int t0 = min(T, w * L), t1 = min(T, t0 + L);
  // the composition of this warp's maps, A_t0 = P + Q A_t1, takes the place of row t0 in the
  // tile (no shared memory beside the tile: T up to the whole of it); row t0 stays here
  float P = 0.f, Q = 1.f, d0 = 0.f, c0 = 0.f;
#pragma unroll 4
  for (int t = t1 - 1; t >= t0; --t) {
    d0 = sdelta[t * 32 + lane];
    c0 = sc[t * 32 + lane];
    P = d0 + c0 * P;
    Q = c0 * Q;
  }
  if (t0 < t1) {
    sdelta[t0 * 32 + lane] = P;
    sc[t0 * 32 + lane] = Q;
  }
  __syncthreads();
  if (e >= E || t0 >= t1) return;
  float A = 0.f;
  for (int t = (T - 1) / L * L; t > t0; t -= L) A = sdelta[t * 32 + lane] + sc[t * 32 + lane] * A;
#pragma unroll 4
  for (int t = t1 - 1; t >= t0; --t) {
    const float de = t == t0 ? d0 : sdelta[t * 32 + lane];
    const float c = t == t0 ? c0 : sc[t * 32 + lane];
    A = de + c * A;
    adv[(size_t)t * E + e] = A;
    ret[(size_t)t * E + e] = A + v[(size_t)t * E + e];
  }
}

int launch_gae(const float* r, const uint8_t* d, const float* v, int T, int E, float gamma,
               float lam, float* adv, float* ret, cudaStream_t s) {
  const size_t smem = (size_t)T * 32 * 2 * sizeof(float);
  if (smem > 227 * 1024) {
    set_error("gae: T too large for one shared-memory tile");
    return DDPPO_E_CONFIG;
  }
  if (smem > 48 * 1024)
    DDPPO_CHECK_CUDA(cudaFuncSetAttribute(gae_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)smem));
  if (E == 0 || T == 0) return DDPPO_OK;
  ::ddppo::launch_k(gae_kernel, (E + 31) / 32, kGaeWarps * 32, smem, s, r, d, v, T, E, gamma, lam, adv, ret);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

}  // namespace ddppo
