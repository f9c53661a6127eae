// Learning-step kernels: the PPO clipped-surrogate loss (Eq. 2) with value and entropy
// terms fused with its exact gradient, the global gradient norm, Adam (Kingma & Ba 2015),
// the per-epoch env permutation for minibatches, and the optional advantage
// normalisation. Every reduction is block partials followed by one fixed-order pass.
#include <algorithm>
#include <atomic>

#include "cluster.cuh"
#include "rl.cuh"

namespace ddppo {

__device__ __forceinline__ float wsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// block reduction of NV values per thread into part[blockIdx.x * NV + k] (256 threads)
template <int NV>
__device__ void block_partials(float (&v)[NV], float* part) {
  __shared__ float sh[NV][8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const float s = wsum(v[k]);
    if (lane == 0) sh[k][w] = s;
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    float s = 0.f;
    for (int q = 0; q < 8; ++q) s += sh[threadIdx.x][q];
    part[blockIdx.x * NV + threadIdx.x] = s;
  }
}

// per sample i:
//   logp = log_softmax(logits)[a], rho = exp(logp - logp_old)
//   pol_i = -min(rho A, clip(rho) A); v_i = 0.5 (R - V)^2; H_i = -sum p log p
//   d logp = -rho A when the unclipped term is the active minimum (ties split evenly
//   between the two branches, which sum to the same when rho is inside the clip range)
//   dlogits_j = [dlogp (1[j=a] - p_j) + c_e p_j (log p_j + H_i)] / n ; dV = c_v (V - R) / n
struct LossIn {
  int n;
  const float* logits; const float* values; const int32_t* actions; const float* logp_old;
  const float* adv; const float* ret;
  float clip, cv, ce;
};
__device__ __forceinline__ void loss_sample(const LossIn& q, int i, float* dlogits, float* dvalues,
                                            float (&acc)[5]) {
  const float clip = q.clip, ce = q.ce;
  float lg[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) lg[k] = q.logits[(size_t)i * 4 + k];
  int a = q.actions[i];
  const float A = q.adv[i], old = q.logp_old[i], V = q.values[i], R = q.ret[i];
  const float mx = fmaxf(fmaxf(lg[0], lg[1]), fmaxf(lg[2], lg[3]));
  float z = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) z += expf(lg[k] - mx);
  const float lse = mx + logf(z);
  float lp[4], p[4], H = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    lp[k] = lg[k] - lse;
    p[k] = expf(lp[k]);
    H -= p[k] * lp[k];
  }
  a = a < 0 ? 0 : (a > 3 ? 3 : a);
  const float lpa = a == 0 ? lp[0] : a == 1 ? lp[1] : a == 2 ? lp[2] : lp[3];
  const float rho = expf(lpa - old);
  const float s1 = rho * A;
  const float rc = fminf(fmaxf(rho, 1.f - clip), 1.f + clip);
  const float s2 = rc * A;
  const bool inside = rho >= 1.f - clip && rho <= 1.f + clip;
  const float dlp = (inside || s1 < s2) ? -rho * A : 0.f;
  const float inv = 1.0f / (float)q.n;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    dlogits[(size_t)i * 4 + k] = inv * (dlp * ((k == a ? 1.f : 0.f) - p[k]) + ce * p[k] * (lp[k] + H));
  dvalues[i] = inv * q.cv * (V - R);
  acc[0] += -fminf(s1, s2);
  acc[1] += 0.5f * (R - V) * (R - V);
  acc[2] += H;
  acc[3] += fabsf(rho - 1.f) > clip ? 1.f : 0.f;
  acc[4] += old - lpa;
}
__device__ __forceinline__ void loss_stats(const float (&s)[5], int n, float cv, float ce, float* stats) {
  const float inv = 1.0f / (float)n;
  const float pol = s[0] * inv, vl = s[1] * inv, ent = s[2] * inv;
  stats[0] = pol + cv * vl - ce * ent;
  stats[1] = pol;
  stats[2] = vl;
  stats[3] = ent;
  stats[4] = s[3] * inv;
  stats[5] = s[4] * inv;
  stats[6] = 0.f;
  stats[7] = 0.f;
}

__global__ void __launch_bounds__(256) ppo_loss_kernel(LossIn q, float* dlogits, float* dvalues, float* part) {
  DDPPO_PDL_ENTRY();
  float acc[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < q.n; i += gridDim.x * blockDim.x)
    loss_sample(q, i, dlogits, dvalues, acc);
  block_partials<5>(acc, part);
}

// The whole loss in one launch and without scratch: one cluster, whose CTAs' partial sums
// meet in the shared memory of its first CTA (in rank order). Bound: latency -- one sample
// a thread up to 4096 samples (3.1 us of kernel). One block over all samples and a second
// launch for its sums took 13.4 us a call at 4096 samples, 30.9 at 16384 and 223 at 131072;
// here 10.8, 11.4 and 11.6 (an empty call: 8.5).
__global__ void __launch_bounds__(1024) ppo_loss_cluster_kernel(LossIn q, float* dlogits, float* dvalues,
                                                                float* stats) {
  DDPPO_PDL_ENTRY();
  __shared__ float warp_part[32][5];
  __shared__ float cta_part[16][5];  // of the first CTA: one row per rank
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint32_t rank = cluster_rank();
  cluster_arrive();  // waited for below: the first CTA runs before anything is stored there
  float acc[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < q.n; i += gridDim.x * blockDim.x)
    loss_sample(q, i, dlogits, dvalues, acc);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const float t = wsum(acc[k]);
    if (lane == 0) warp_part[w][k] = t;
  }
  __syncthreads();
  cluster_wait();
  if (threadIdx.x < 5) {
    float t = 0.f;
    for (int j = 0; j < nw; ++j) t += warp_part[j][threadIdx.x];
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(map_rank(smem_addr(&cta_part[rank][threadIdx.x]), 0u)),
                 "f"(t)
                 : "memory");
  }
  __syncwarp();
  cluster_sync();
  if (rank != 0 || threadIdx.x != 0) return;
  float s[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    s[k] = 0.f;
    for (int j = 0; j < (int)gridDim.x; ++j) s[k] += cta_part[j][k];
  }
  loss_stats(s, q.n, q.cv, q.ce, stats);
}

// the sum over nb blocks of NV partials each (part[b * NV + k]) by one block of kFinal
// threads, in a fixed order: thread i adds partials i, i + kFinal, ... in turn, then a fixed
// halving tree over the threads. Every thread reads its partials before the first barrier.
constexpr int kFinal = 256;
template <int NV>
__device__ void final_sums(const float* part, int nb, float (&out)[NV]) {
  __shared__ float sh[NV][kFinal];
  float acc[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) acc[k] = 0.f;
  for (int b = threadIdx.x; b < nb; b += kFinal)
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] += __ldcg(part + b * NV + k);
#pragma unroll
  for (int k = 0; k < NV; ++k) sh[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int w = kFinal / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
#pragma unroll
      for (int k = 0; k < NV; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) out[k] = sh[k][0];
}

__global__ void __launch_bounds__(kFinal) ppo_loss_final(int nb, int n, const float* part, float cv,
                                                        float ce, float* stats) {
  DDPPO_PDL_ENTRY();
  float s[5];
  final_sums<5>(part, nb, s);
  if (threadIdx.x != 0) return;
  loss_stats(s, n, cv, ce, stats);
}

// one cluster of 1, 2, 4 or 8 CTAs (16 where the device allows that many), 256 threads each
// up to one sample a thread, then 1024
static int launch_loss_cluster(const LossIn& q, float* dlogits, float* dvalues, float* stats, cudaStream_t s) {
  static std::atomic<int> largest[64];  // 0: not asked yet
  int dev = 0;
  DDPPO_CHECK_CUDA(cudaGetDevice(&dev));
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(1024);
  cfg.attrs = attr;
  int most = dev < 64 ? largest[dev].load() : 8;
  if (!most) {
    cfg.gridDim = dim3(16);
    cfg.numAttrs = 1;
    attr[0].val.clusterDim.x = 16;
    int num = 0;
    most = 8;
    if (cudaFuncSetAttribute(ppo_loss_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
            cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&num, ppo_loss_cluster_kernel, &cfg) == cudaSuccess && num > 0)
      most = 16;
    else
      (void)cudaGetLastError();
    largest[dev].store(most);
  }
  int ctas = 1;
  while (ctas < most && ctas * 256 < q.n) ctas *= 2;
  attr[0].val.clusterDim.x = (unsigned)ctas;
  cfg.gridDim = dim3((unsigned)ctas);
  cfg.blockDim = dim3(q.n > ctas * 256 ? 1024 : 256);
  cfg.stream = s;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  DDPPO_CHECK_CUDA(cudaLaunchKernelEx(&cfg, ppo_loss_cluster_kernel, q, dlogits, dvalues, stats));
  return DDPPO_OK;
}

int launch_ppo_loss(int n, const float* logits, const float* values, const int32_t* actions,
                    const float* logp_old, const float* adv, const float* ret, float clip, float cv,
                    float ce, float* stats, float* dlogits, float* dvalues, float* part,
                    size_t part_elems, cudaStream_t s) {
  if (n <= 0) return DDPPO_OK;
  const LossIn q{n, logits, values, actions, logp_old, adv, ret, clip, cv, ce};
  // one cluster up to 8 samples for each of its 16384 threads (at 131072 samples 11.6 us a
  // call, no more than the two launches of the form below take for few), and where there is
  // no scratch
  if (!part || n <= 131072) return launch_loss_cluster(q, dlogits, dvalues, stats, s);
  const int nb = std::min((n + 255) / 256, 1024);
  if ((size_t)nb * 5 > part_elems) { set_error("ppo_loss: scratch too small"); return DDPPO_E_CONFIG; }
  return launch_ppo_loss_blocks(n, logits, values, actions, logp_old, adv, ret, clip, cv, ce, stats, dlogits,
                                dvalues, part, nb, s);
}

int launch_ppo_loss_blocks(int n, const float* logits, const float* values, const int32_t* actions,
                           const float* logp_old, const float* adv, const float* ret, float clip,
                           float cv, float ce, float* stats, float* dlogits, float* dvalues,
                           float* part, int nb, cudaStream_t s) {
  if (n <= 0) return DDPPO_OK;
  const LossIn q{n, logits, values, actions, logp_old, adv, ret, clip, cv, ce};
  ::ddppo::launch_k(ppo_loss_kernel, nb, 256, 0, s, q, dlogits, dvalues, part);
  DDPPO_CHECK_LAUNCH();
  ::ddppo::launch_k(ppo_loss_final, 1, kFinal, 0, s, nb, n, part, cv, ce, stats);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

// ---- sum of squares / sums, two-stage ----
__global__ void __launch_bounds__(256) sumsq_partial(const float* __restrict__ x, size_t n,
                                                     float* part, int square, const float* shift) {
  DDPPO_PDL_ENTRY();
  float v[1] = {0.f};
  const float mu = shift ? shift[0] : 0.f;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float d = x[i] - mu;
    v[0] += square ? d * d : d;
  }
  block_partials<1>(v, part);
}
__global__ void __launch_bounds__(kFinal) sum_final(int nb, const float* __restrict__ part, float* out,
                                                   int mode, float scale) {
  DDPPO_PDL_ENTRY();
  float t[1];
  final_sums<1>(part, nb, t);
  if (threadIdx.x != 0) return;
  const float s = t[0];
  if (mode == 1) out[0] = s * scale;         // mean
  else out[0] = sqrtf(s * scale);            // population std
}

static int reduce_blocks(size_t n) {
  size_t b = (n + 255) / 256;
  if (b > 1024) b = 1024;
  if (b < 1) b = 1;
  return (int)b;
}

// ---- the optimizer step ----
// Both kernels walk the parameters four at a time, 16-byte accesses where the gradient
// allows them (the other arrays are the library's). The update moves 28 bytes a parameter:
// 8.5 M parameters (237 MB) take 34 us, in which 176 MB pass through memory -- the last of what
// it writes is still in L2 when it ends; with scalar accesses and the bias corrections' two
// double-precision powers in every block it took 84 us.
__device__ __forceinline__ float4 ld4(const float* p, bool aligned) {
  if (aligned) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[1], p[2], p[3]);
}

// block partials of sum (scale g)^2; the last block to finish adds them in final_sums' order
__global__ void __launch_bounds__(kFinal) opt_scalars_kernel(const float* __restrict__ g, float scale,
                                                             size_t n, int aligned, float b1,
                                                             float b2, const int64_t* t_dev,
                                                             int64_t t_off, float* opt,
                                                             float* norm_copy, int* cnt,
                                                             float* part) {
  DDPPO_PDL_ENTRY();
  __shared__ int last;
  // the bias corrections beside the first block's loads
  if (blockIdx.x == 0 && (threadIdx.x == 0 || threadIdx.x == 32)) {
    const double step = (double)(t_off + (t_dev ? *t_dev : 0));
    opt[threadIdx.x ? 2 : 1] = (float)(1.0 - pow((double)(threadIdx.x ? b2 : b1), step));
  }
  float v[1] = {0.f};
  const size_t n4 = n / 4;
#pragma unroll 4
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    const float4 x = ld4(g + 4 * i, aligned != 0);
    const float a = scale * x.x, b = scale * x.y, c = scale * x.z, d = scale * x.w;
    v[0] += a * a;
    v[0] += b * b;
    v[0] += c * c;
    v[0] += d * d;
  }
  if (blockIdx.x == 0 && threadIdx.x < n - 4 * n4) {
    const float a = scale * g[4 * n4 + threadIdx.x];
    v[0] += a * a;
  }
  block_partials<1>(v, part);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(cnt, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  float t[1];
  final_sums<1>(part, gridDim.x, t);
  if (threadIdx.x != 0) return;
  opt[0] = sqrtf(t[0]);
  if (norm_copy) *norm_copy = opt[0];
  *cnt = 0;
}

int launch_opt_scalars(const float* g, float scale, size_t n, float b1, float b2,
                       const int64_t* t_dev, int64_t t_off, float* opt, float* norm_copy, int* cnt,
                       float* part, size_t part_elems, cudaStream_t s) {
  const int nb = reduce_blocks(n);
  if ((size_t)nb > part_elems) { set_error("grad_norm: scratch too small"); return DDPPO_E_CONFIG; }
  ::ddppo::launch_k(opt_scalars_kernel, nb, kFinal, 0, s, g, scale, n, ((uintptr_t)g & 15) == 0 ? 1 : 0,
                    b1, b2, t_dev, t_off, opt, norm_copy, cnt, part);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

struct AdamArgs {
  float coef, bc1, bc2, lr, b1, b2, eps;
};
__device__ __forceinline__ void adam_one(const AdamArgs& a, float g, float& p, float& m, float& v) {
  const float gi = g * a.coef;
  m = a.b1 * m + (1.f - a.b1) * gi;
  v = a.b2 * v + (1.f - a.b2) * gi * gi;
  p -= a.lr * (m / a.bc1) / (sqrtf(v / a.bc2) + a.eps);
}
__global__ void __launch_bounds__(256) adam_kernel(float* __restrict__ p, const float* __restrict__ g,
                                                   float scale, float* __restrict__ m,
                                                   float* __restrict__ v, size_t n, int aligned,
                                                   const float* __restrict__ opt, float max_norm,
                                                   float lr, float b1, float b2, float eps) {
  DDPPO_PDL_ENTRY();
  AdamArgs a{1.f, opt[1], opt[2], lr, b1, b2, eps};
  if (max_norm > 0.f) a.coef = fminf(1.f, max_norm / (opt[0] + 1e-6f));
  const size_t n4 = n / 4;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    const float4 gv = ld4(g + 4 * i, aligned != 0);
    float4 pv = *reinterpret_cast<float4*>(p + 4 * i), mv = *reinterpret_cast<float4*>(m + 4 * i),
           vv = *reinterpret_cast<float4*>(v + 4 * i);
    adam_one(a, scale * gv.x, pv.x, mv.x, vv.x);
    adam_one(a, scale * gv.y, pv.y, mv.y, vv.y);
    adam_one(a, scale * gv.z, pv.z, mv.z, vv.z);
    adam_one(a, scale * gv.w, pv.w, mv.w, vv.w);
    *reinterpret_cast<float4*>(p + 4 * i) = pv;
    *reinterpret_cast<float4*>(m + 4 * i) = mv;
    *reinterpret_cast<float4*>(v + 4 * i) = vv;
  }
  if (blockIdx.x == 0 && threadIdx.x < n - 4 * n4) {
    const size_t i = 4 * n4 + threadIdx.x;
    adam_one(a, scale * g[i], p[i], m[i], v[i]);
  }
}

int launch_adam(float* p, const float* g, float scale, float* m, float* v, size_t n,
                const float* opt, float max_norm, float lr, float b1, float b2, float eps,
                cudaStream_t s) {
  size_t b = (n / 4 + 255) / 256;
  b = std::max<size_t>(1, std::min<size_t>(b, 152 * 8));
  ::ddppo::launch_k(adam_kernel, (unsigned)b, 256, 0, s, p, g, scale, m, v, n,
                    ((uintptr_t)g & 15) == 0 ? 1 : 0, opt, max_norm, lr, b1, b2, eps);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

// ---- env permutation: Fisher-Yates over the counter hash (seed, env 0, update, stream 7) ----
__device__ __forceinline__ uint64_t sm64r(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__global__ void perm_kernel(uint64_t seed, const int64_t* __restrict__ update_dev, int64_t epoch,
                            int E, int32_t* perm) {
  DDPPO_PDL_ENTRY();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int64_t update = *update_dev;
  for (int i = 0; i < E; ++i) perm[i] = i;
  uint64_t k = sm64r(seed);
  k = sm64r(k + 0);
  k = sm64r(k + (uint64_t)update);
  for (int i = E - 1; i >= 1; --i) {
    const uint64_t idx = ((uint64_t)epoch * E + i) & 0xFFFFFFFFFFull;
    const uint64_t h = sm64r(k + ((7ull << 40) | idx));
    const int j = (int)(((h >> 32) * (uint64_t)(i + 1)) >> 32);
    const int32_t t = perm[i];
    perm[i] = perm[j];
    perm[j] = t;
  }
}
int launch_permutation(uint64_t seed, const int64_t* update_dev, int64_t epoch, int E,
                       int32_t* perm, cudaStream_t s) {
  ::ddppo::launch_k(perm_kernel, 1, 32, 0, s, seed, update_dev, epoch, E, perm);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

// ---- advantage normalisation: (A - mean) / (std + 1e-5), population std ----
__global__ void normalize_kernel(const float* __restrict__ x, float* __restrict__ y, size_t n,
                                 const float* __restrict__ mean, const float* __restrict__ sd) {
  DDPPO_PDL_ENTRY();
  const float mu = mean[0], inv = 1.0f / (sd[0] + 1e-5f);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    y[i] = (x[i] - mu) * inv;
}
int launch_normalize_adv(const float* adv, float* out, size_t n, float* scal2, float* part,
                         size_t part_elems, cudaStream_t s) {
  const int nb = reduce_blocks(n);
  if ((size_t)nb > part_elems) { set_error("normalize: scratch too small"); return DDPPO_E_CONFIG; }
  ::ddppo::launch_k(sumsq_partial, nb, 256, 0, s, adv, n, part, 0, nullptr);
  DDPPO_CHECK_LAUNCH();
  ::ddppo::launch_k(sum_final, 1, kFinal, 0, s, nb, part, scal2, 1, 1.0f / (float)n);
  DDPPO_CHECK_LAUNCH();
  ::ddppo::launch_k(sumsq_partial, nb, 256, 0, s, adv, n, part, 1, scal2);
  DDPPO_CHECK_LAUNCH();
  ::ddppo::launch_k(sum_final, 1, kFinal, 0, s, nb, part, scal2 + 1, 2, 1.0f / (float)n);
  DDPPO_CHECK_LAUNCH();
  ::ddppo::launch_k(normalize_kernel, reduce_blocks(n), 256, 0, s, adv, out, n, scal2, scal2 + 1);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

}  // namespace ddppo
