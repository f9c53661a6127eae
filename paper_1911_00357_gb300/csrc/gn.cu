// GroupNorm with groups of two channels (C/2 groups per image), the normalisation of the
// ResNet encoder's convolutions (Sec. 4 replaces BatchNorm by GroupNorm). Activations are
// NHWC fp32 [N, HW, C].
//
// The statistics and the backward reductions split every image over S blocks (a grid of
// S x N) so that a small batch -- the 64 frames of one rollout step -- still covers every
// SM. Each thread owns V consecutive channels (V = 4, or 2 when C % 4 != 0) of one pixel
// row and loads them as one vector. Blocks write per-channel partial sums; the last block
// of an image to finish (a per-image arrival counter, re-armed by that block) combines the
// S partials in block order, so every result is deterministic. The element-wise passes
// (normalise + residual + ReLU, and the input gradient) are vectorised the same way.
#include <algorithm>

#include "gn_ring.cuh"
#include "nn_kernels.cuh"
#include "tc_common.cuh"

namespace ddppo {

namespace {

constexpr int kThreads = kGnThreads;

template <int V>
__device__ __forceinline__ void ldv(const float* p, float (&v)[V]) {
  if constexpr (V == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else {
    const float2 t = *reinterpret_cast<const float2*>(p);
    v[0] = t.x; v[1] = t.y;
  }
}
template <int V>
__device__ __forceinline__ void stv(float* p, const float (&v)[V]) {
  if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
}
__device__ __forceinline__ uint32_t pack_bf2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
template <int V>
__device__ __forceinline__ void stv_bf(__nv_bfloat16* p, const float (&v)[V]) {
  if constexpr (V == 4) *reinterpret_cast<uint2*>(p) = make_uint2(pack_bf2(v[0], v[1]), pack_bf2(v[2], v[3]));
  else *reinterpret_cast<uint32_t*>(p) = pack_bf2(v[0], v[1]);
}

// E4M3 codes of v / sc (saturating), V consecutive bytes
template <int V>
__device__ __forceinline__ void stv_e4m3(uint8_t* p, const float (&v)[V], float sc) {
  uint32_t w = 0;
#pragma unroll
  for (int j = 0; j < V; ++j) w |= (uint32_t)e4m3_sat(v[j] / sc) << (8 * j);
  if (V == 4) *reinterpret_cast<uint32_t*>(p) = w;
  else *reinterpret_cast<uint16_t*>(p) = (uint16_t)w;
}

// the block's largest m folded into *amax (one atomic per block; every thread calls it)
__device__ __forceinline__ void block_amax(float m, unsigned* amax) {
  __shared__ float wm[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float b = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) b = fmaxf(b, wm[w]);
    atomicMax(amax, __float_as_uint(b));
  }
}
template <int V>
__device__ __forceinline__ void stv_op(void* p, size_t i, const float (&v)[V], bool bf) {
  if (bf) stv_bf<V>((__nv_bfloat16*)p + i, v);
  else stv<V>((float*)p + i, v);
}

// threads of the block: R = C / V per pixel row, P rows per pass
__host__ __device__ inline int rows_per_pass(int C, int V) { return gn_rows_per_pass(C, V); }

// sums the per-thread pair (a[v], b[v]) over the P rows of the block for every channel,
// in row order; results for channel c at out[2c], out[2c + 1]. sh holds blockDim x 2V.
template <int V>
__device__ __forceinline__ void block_pair_sums(const float (&a)[V], const float (&b)[V], float* sh,
                                                int C, float* out) {
  const int R = C / V, P = blockDim.x / R;
  for (int v = 0; v < V; ++v) {
    sh[threadIdx.x * 2 * V + v] = a[v];
    sh[threadIdx.x * 2 * V + V + v] = b[v];
  }
  __syncthreads();
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    const int cv = c / V, v = c % V;
    float sa = 0.f, sb = 0.f;
    for (int r = 0; r < P; ++r) {
      const float* q = sh + (size_t)(r * R + cv) * 2 * V;
      sa += q[v];
      sb += q[V + v];
    }
    out[2 * c] = sa;
    out[2 * c + 1] = sb;
  }
}

// true in exactly one block per image: the last to arrive after writing its partials
__device__ __forceinline__ bool last_of_image(int* cnt, int S, int* flag) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *flag = atomicAdd(cnt, 1) == S - 1;
  __syncthreads();
  if (!*flag) return false;
  __threadfence();
  return true;
}

// ---- the arithmetic every form shares, with its fused multiply-adds written out: all forms
//      give the same bits whatever the compiler would contract in each ----
__device__ __forceinline__ void sum_shifted(float x, float K, float& s1, float& s2) {
  const float d = x - K;
  s1 += d;
  s2 = __fmaf_rn(d, d, s2);
}
__device__ __forceinline__ float normalised(float x, float mu, float rs, float gm, float bt) {
  return __fmaf_rn(__fmul_rn(x - mu, rs), gm, bt);
}
__device__ __forceinline__ void sum_grad(float d, float x, float mu, float rs, float& sg, float& sgx) {
  sg += d;
  sgx = __fmaf_rn(d, __fmul_rn(x - mu, rs), sgx);
}
// group mean of two gamma-weighted channel sums
__device__ __forceinline__ float group_mean(float a, float g0, float b, float g1, float inv) {
  return __fmul_rn(__fmaf_rn(a, g0, __fmul_rn(b, g1)), inv);
}
__device__ __forceinline__ float input_grad(float d, float x, float mu, float rs, float gm, float m1,
                                            float m2) {
  const float xh = __fmul_rn(x - mu, rs);
  return __fmul_rn(rs, __fmaf_rn(-xh, m2, __fmaf_rn(d, gm, -m1)));
}
// where the mask of the ReLU that followed the normalisation comes from
enum : int { MASK_NONE = 0, MASK_Z, MASK_POS, MASK_Y };
__host__ __device__ __forceinline__ int mask_kind(const GNBack& b, int V) {
  return b.relu_from_z ? MASK_Z : (V == 4 && b.pos) ? MASK_POS : b.relu_y ? MASK_Y : MASK_NONE;
}
// d masked by that ReLU; o the element offset, c0 its channel
template <int V>
__device__ __forceinline__ void mask_relu(const GNBack& b, size_t o, int c0, const float (&x)[V],
                                          const float* mu, const float* rs, float (&d)[V]) {
  const int kind = mask_kind(b, V);
  if (kind == MASK_Z) {
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (!(normalised(x[v], mu[v], rs[v], b.gamma[c0 + v], b.beta[c0 + v]) > 0.f)) d[v] = 0.f;
  } else if (kind == MASK_POS) {
    const unsigned m = b.pos[o / 4];
#pragma unroll
    for (int v = 0; v < V; ++v) d[v] = (m >> v) & 1u ? d[v] : 0.f;
  } else if (kind == MASK_Y) {
    float y[V];
    ldv<V>(b.relu_y + o, y);
#pragma unroll
    for (int v = 0; v < V; ++v) d[v] = y[v] > 0.f ? d[v] : 0.f;
  }
}
__device__ __forceinline__ bool masks_given(const GNBack& b) { return b.relu_y || b.pos; }

// ---- statistics: shifted sums about the image's first pixel, combined in double ----
// the block's per-channel (sum d, sum d^2), d = z - z[first pixel], over its pixel rows
// [pb, pe) of image zi, written to pp[2c], pp[2c + 1]
template <int V>
__device__ __forceinline__ void block_shifted_sums(const float* __restrict__ zi, int pb, int pe, int C,
                                                   float* sh, float* pp) {
  const int R = C / V, P = blockDim.x / R;
  const int cv = threadIdx.x % R, pr = threadIdx.x / R, c0 = cv * V;
  float K[V], s1[V], s2[V];
  ldv<V>(zi + c0, K);
#pragma unroll
  for (int v = 0; v < V; ++v) s1[v] = s2[v] = 0.f;
#pragma unroll 8
  for (int p = pb + pr; p < pe; p += P) {
    float x[V];
    ldv<V>(zi + (size_t)p * C + c0, x);
#pragma unroll
    for (int v = 0; v < V; ++v) sum_shifted(x[v], K[v], s1[v], s2[v]);
  }
  block_pair_sums<V>(s1, s2, sh, C, pp);
}

// An image's pixel count as the statistics use it: 1 / HW, and 1 / (2 HW) where HW is a power
// of two (the product is then the quotient), else 0. The device's double-precision division
// takes some 2000 cycles, and every block ended in two of them.
struct PixelCount {
  int HW;
  double inv, inv2;
};

// statistics of one group from its two channels' shifted sums a, b about k0, k1
__device__ __forceinline__ void group_stats(const double (&a)[2], const double (&b)[2], float k0, float k1,
                                            const PixelCount& px, float eps, float* mean, float* rstd) {
  const double m0 = (double)k0 + a[0] * px.inv, m1 = (double)k1 + a[1] * px.inv;
  const double q0 = b[0] - a[0] * a[0] * px.inv, q1 = b[1] - a[1] * a[1] * px.inv;
  const double dm = m0 - m1, sum = q0 + q1 + 0.5 * px.HW * dm * dm;
  double var = px.inv2 != 0.0 ? sum * px.inv2 : sum / (2.0 * px.HW);
  if (var < 0.0) var = 0.0;
  *mean = (float)(0.5 * (m0 + m1));
  *rstd = 1.0f / sqrtf((float)var + eps);
}

// the image's group means and 1 / sqrt(var + eps) from its S x C x 2 partials, read
// through L2 into sh and combined in block order (double); results to mean[g], rstd[g]
__device__ __forceinline__ void combine_groups(const float* pim, const float* __restrict__ zi, int S,
                                               int C, const PixelCount& px, float eps, float* sh,
                                               float* mean, float* rstd) {
  for (int i = threadIdx.x; i < S * C * 2; i += blockDim.x) sh[i] = __ldcg(pim + i);
  __syncthreads();
  const int G = C / 2;
  for (int g = threadIdx.x; g < G; g += blockDim.x) {
    double a[2], b[2];
    for (int j = 0; j < 2; ++j) {
      const int c = 2 * g + j;
      a[j] = b[j] = 0.0;
      for (int t = 0; t < S; ++t) {
        a[j] += (double)sh[(t * C + c) * 2];
        b[j] += (double)sh[(t * C + c) * 2 + 1];
      }
    }
    group_stats(a, b, zi[2 * g], zi[2 * g + 1], px, eps, mean + g, rstd + g);
  }
}

template <int V>
__global__ void __launch_bounds__(kThreads) gn_stats_kernel(const float* __restrict__ z, PixelCount px, int C,
                                                            int S, float eps, float* __restrict__ part,
                                                            int* __restrict__ cnt, float* __restrict__ mean,
                                                            float* __restrict__ rstd) {
  DDPPO_PDL_ENTRY();
  extern __shared__ float sh[];
  __shared__ int flag;
  const int HW = px.HW, n = blockIdx.y, sb = blockIdx.x;
  const int chunk = (HW + S - 1) / S, pb = sb * chunk, pe = min(HW, pb + chunk);
  const float* zi = z + (size_t)n * HW * C;
  block_shifted_sums<V>(zi, pb, pe, C, sh, part + ((size_t)n * S + sb) * C * 2);
  if (!last_of_image(cnt + n, S, &flag)) return;
  const int G = C / 2;
  combine_groups(part + (size_t)n * S * C * 2, zi, S, C, px, eps, sh, mean + (size_t)n * G,
                 rstd + (size_t)n * G);
  if (threadIdx.x == 0) cnt[n] = 0;  // re-arm for the next launch on this stream
}

// ---- out = act(gn(z) + res) ----
// one vector of V channels x of z (r of the residual, d of zd) at element offset o; mu/rs (and
// mud/rsd) point at the group statistics of its first channel; returns max |out| (E4M3 copy)
// RES, ZD: the residual / the normalised shortcut is present (compile-time: the registers of
// what is absent are what a fourth block per SM needs)
template <int V, bool ZD>
struct ChannelParams {  // of the thread's V channels: gamma, beta, and the shortcut's
  float gm[V], bt[V], gd[V], bd[V];
  __device__ __forceinline__ ChannelParams(const GNApply& a, int c0) {
    ldv<V>(a.gamma + c0, gm);
    ldv<V>(a.beta + c0, bt);
    if (ZD) {
      ldv<V>(a.gamma_d + c0, gd);
      ldv<V>(a.beta_d + c0, bd);
    }
  }
};
template <int V, bool RES, bool ZD>
__device__ __forceinline__ float finish_vec(const GNApply& a, const ChannelParams<V, ZD>& q, size_t o,
                                            float (&x)[V], const float (&r)[V], const float (&d)[V],
                                            const float* mu, const float* rs, const float* mud,
                                            const float* rsd, float f8s) {
#pragma unroll
  for (int v = 0; v < V; ++v) x[v] = normalised(x[v], mu[v / 2], rs[v / 2], q.gm[v], q.bt[v]);
  if (RES) {
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] += r[v];
  }
  if (ZD) {
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] += normalised(d[v], mud[v / 2], rsd[v / 2], q.gd[v], q.bd[v]);
  }
  if (a.relu) {
#pragma unroll
    for (int v = 0; v < V; ++v) x[v] = fmaxf(x[v], 0.f);
  }
  if (a.out) stv<V>(a.out + o, x);
  if (a.out_bf) stv_bf<V>(a.out_bf + o, x);
  if (V == 4 && a.pos) {
    unsigned m = 0;
#pragma unroll
    for (int v = 0; v < V; ++v) m |= x[v] > 0.f ? 1u << v : 0u;
    a.pos[o / 4] = (uint8_t)m;
  }
  float f8m = 0.f;
  if (a.out_f8) {
    stv_e4m3<V>(a.out_f8 + o, x, f8s);
#pragma unroll
    for (int v = 0; v < V; ++v) f8m = fmaxf(f8m, fabsf(x[v]));
  }
  return f8m;
}
// Rows pr, pr + P, ... below `end` of an image (element offset ib, the thread's channel c0),
// kRows at a time: all loads of a group are issued before its stores. (The outputs may
// alias the inputs as far as the compiler knows, so it moves no load above a store: one row
// at a time, every row waited for its own loads, 37 us for a 32x32 x 32 image. 4096 such
// images with a residual: 334 us, 4.8 TB/s, against 367 us.)
// sz, sd: the rows of z and of zd (else the residual) staged in shared memory, pitch Cs (null:
// read from global memory).
constexpr int kRows = 4;
// blocks an SM of gn_image_kernel: four with kRows rows in flight where the images are many
// waves; six with one row where they fit in one (700 images of 1024 x 32 with a residual: 65 us,
// 78 in two waves of four)
constexpr int kImageCtas = 4, kFewCtas = 6;
template <int V, bool RES, bool ZD, int ROWS>
__device__ __forceinline__ float normalise_rows(const GNApply& a, size_t ib, int pr, int end, int P, int C,
                                                int c0, const float* sz, const float* sd, int Cs,
                                                const float* mu, const float* rs, const float* mud,
                                                const float* rsd, float f8s) {
  const ChannelParams<V, ZD> q(a, c0);
  float f8m = 0.f;
  for (int p0 = pr; p0 < end; p0 += ROWS * P) {
    float x[ROWS][V], r[ROWS][V], d[ROWS][V];
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
      const int p = p0 + u * P;
      if (p >= end) break;
      const size_t o = ib + (size_t)p * C + c0;
      ldv<V>(sz ? sz + (size_t)p * Cs : a.z + o, x[u]);
      if (RES) ldv<V>(sd && !ZD ? sd + (size_t)p * Cs : a.resid + o, r[u]);
      if (ZD) ldv<V>(sd ? sd + (size_t)p * Cs : a.zd + o, d[u]);
    }
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
      const int p = p0 + u * P;
      if (p >= end) break;
      f8m = fmaxf(f8m, finish_vec<V, RES, ZD>(a, q, ib + (size_t)p * C + c0, x[u], r[u], d[u], mu, rs, mud,
                                              rsd, f8s));
    }
  }
  return f8m;
}

template <int V, int ROWS, int ROWS2 = ROWS>  // ROWS2: with a second or third input
__device__ __forceinline__ float normalise_rows_any(const GNApply& a, size_t ib, int pr, int end, int P, int C,
                                                    int c0, const float* sz, const float* sd, int Cs,
                                                    const float* mu, const float* rs, const float* mud,
                                                    const float* rsd, float f8s) {
  if (a.zd && a.resid) return normalise_rows<V, true, true, ROWS2>(a, ib, pr, end, P, C, c0, sz, sd, Cs, mu, rs, mud, rsd, f8s);
  if (a.zd) return normalise_rows<V, false, true, ROWS2>(a, ib, pr, end, P, C, c0, sz, sd, Cs, mu, rs, mud, rsd, f8s);
  if (a.resid) return normalise_rows<V, true, false, ROWS2>(a, ib, pr, end, P, C, c0, sz, sd, Cs, mu, rs, mud, rsd, f8s);
  return normalise_rows<V, false, false, ROWS>(a, ib, pr, end, P, C, c0, sz, sd, Cs, mu, rs, mud, rsd, f8s);
}

template <int V>
__global__ void __launch_bounds__(kThreads) gn_apply_kernel(GNApply a, int HW, int C) {
  DDPPO_PDL_ENTRY();
  const int R = C / V, G = C / 2;
  const int n = blockIdx.y;
  const int per = HW * R;
  const size_t ib = (size_t)n * HW * C;
  const float f8s = a.out_f8 ? *a.f8_scale : 1.f;
  float f8m = 0.f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < per; i += gridDim.x * blockDim.x) {
    const int c0 = (i % R) * V;
    const size_t gq = (size_t)n * G + c0 / 2, o = ib + (size_t)i * V;
    const float* mud = a.zd ? a.mean_d + gq : nullptr;
    const float* rsd = a.zd ? a.rstd_d + gq : nullptr;
    float x[V], r[V], d[V];
    ldv<V>(a.z + o, x);
    if (a.resid) ldv<V>(a.resid + o, r);
    if (a.zd) ldv<V>(a.zd + o, d);
    if (a.zd) {
      const ChannelParams<V, true> q(a, c0);
      f8m = fmaxf(f8m, a.resid ? finish_vec<V, true, true>(a, q, o, x, r, d, a.mean + gq, a.rstd + gq, mud, rsd, f8s)
                               : finish_vec<V, false, true>(a, q, o, x, r, d, a.mean + gq, a.rstd + gq, mud, rsd, f8s));
    } else {
      const ChannelParams<V, false> q(a, c0);
      f8m = fmaxf(f8m, a.resid ? finish_vec<V, true, false>(a, q, o, x, r, d, a.mean + gq, a.rstd + gq, mud, rsd, f8s)
                               : finish_vec<V, false, false>(a, q, o, x, r, d, a.mean + gq, a.rstd + gq, mud, rsd, f8s));
    }
  }
  if (a.out_f8) block_amax(f8m, a.f8_amax);
}

// ---- statistics and normalisation in one launch ----
// Every block of the (S, N) grid is resident (cooperative launch). Each block sums its
// pixel rows as the statistics kernel does (z, and zd when present); the S blocks of an
// image then meet at a per-image barrier: an arrival counter, and a departure counter
// whose last increment re-arms both for the next launch. The wait is bounded: on a
// run-out the sticky timeout flag is set and the block returns without writing. After
// the barrier each block combines the image's partials in block order exactly as the
// statistics kernel's last block does (so the statistics are bit-identical for the same
// S), block 0 of the image stores them for the backward, and every block normalises the
// rows it just summed (still in L2): z is read from HBM once, and one launch replaces two.
constexpr unsigned GN_SPIN_LIMIT = 1u << 22;

__device__ __forceinline__ bool image_barrier(int* arrive, int* depart, int S, int32_t* err,
                                              int* s_ok) {
  __threadfence();  // this thread's partial sums are visible device-wide before the arrival
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(arrive, 1);
    int ok = 0;
    for (unsigned i = 0; i < GN_SPIN_LIMIT; ++i) {
      if (*(volatile int*)arrive >= S) { ok = 1; break; }
      if (err && (*(volatile int32_t*)err & ERRF_TIMEOUT)) break;
      __nanosleep(64);
    }
    if (!ok && err) atomicOr(err, ERRF_TIMEOUT);
    __threadfence();
    // every block has stopped reading `arrive` once the departures reach S
    if (atomicAdd(depart, 1) == S - 1) {
      atomicExch(arrive, 0);
      atomicExch(depart, 0);
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

constexpr int kFusedBlocks = 5;  // per SM; the split of an image over blocks, and with it the
                                // order of its sums, follows from it
template <int V>
__global__ void __launch_bounds__(kThreads, kFusedBlocks) gn_fused_kernel(GNApply a, PixelCount px, int C, int S, float eps,
                                                            float* __restrict__ part,
                                                            float* __restrict__ part_d, int* arrive,
                                                            int* depart, int32_t* err) {
  DDPPO_PDL_ENTRY();
  extern __shared__ float sh[];
  __shared__ int s_ok;
  const int HW = px.HW, n = blockIdx.y, sb = blockIdx.x, G = C / 2;
  const int chunk = (HW + S - 1) / S, pb = sb * chunk, pe = min(HW, pb + chunk);
  const size_t ib = (size_t)n * HW * C;
  float* st = sh + max((int)blockDim.x * 2 * V, S * C * 2);  // [4][G]: mean, rstd, mean_d, rstd_d
  block_shifted_sums<V>(a.z + ib, pb, pe, C, sh, part + ((size_t)n * S + sb) * C * 2);
  if (a.zd) {
    __syncthreads();
    block_shifted_sums<V>(a.zd + ib, pb, pe, C, sh, part_d + ((size_t)n * S + sb) * C * 2);
  }
  if (!image_barrier(arrive + n, depart + n, S, err, &s_ok)) return;
  combine_groups(part + (size_t)n * S * C * 2, a.z + ib, S, C, px, eps, sh, st, st + G);
  if (a.zd) {
    __syncthreads();
    combine_groups(part_d + (size_t)n * S * C * 2, a.zd + ib, S, C, px, eps, sh, st + 2 * G,
                   st + 3 * G);
  }
  __syncthreads();
  if (sb == 0) {
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
      const_cast<float*>(a.mean)[(size_t)n * G + g] = st[g];
      const_cast<float*>(a.rstd)[(size_t)n * G + g] = st[G + g];
      if (a.zd) {
        const_cast<float*>(a.mean_d)[(size_t)n * G + g] = st[2 * G + g];
        const_cast<float*>(a.rstd_d)[(size_t)n * G + g] = st[3 * G + g];
      }
    }
  }
  const int R = C / V, P = blockDim.x / R;
  const int cv = threadIdx.x % R, pr = threadIdx.x / R, c0 = cv * V;
  const float f8s = a.out_f8 ? *a.f8_scale : 1.f;
  // with a residual two rows in flight: 95 us for 256 images of 4096 x 32, four rows 104
  const float f8m = normalise_rows_any<V, kRows, 2>(a, ib, pb + pr, pe, P, C, c0, nullptr, nullptr, 0, st + c0 / 2, st + G + c0 / 2,
                          st + 2 * G + c0 / 2, st + 3 * G + c0 / 2, f8s);
  if (a.out_f8) block_amax(f8m, a.f8_amax);
}

// ---- one block per image: statistics and normalisation without any grid barrier ----
// The block sums the whole image (the statistics kernel's S = 1 arithmetic), combines in
// shared memory, and normalises the image it just read (an L2 hit). An ordinary launch:
// nothing waits on another block, so it needs no co-residency.
__device__ __forceinline__ void combine_groups_one(const float* p, const float* __restrict__ zi,
                                                   int C, const PixelCount& px, float eps, float* mean,
                                                   float* rstd) {
  for (int g = threadIdx.x; g < C / 2; g += blockDim.x) {
    const double a[2] = {(double)p[4 * g], (double)p[4 * g + 2]};
    const double b[2] = {(double)p[4 * g + 1], (double)p[4 * g + 3]};
    group_stats(a, b, zi[2 * g], zi[2 * g + 1], px, eps, mean + g, rstd + g);
  }
}

template <int V, bool RES, bool ZD, int CTAS>
__global__ void __launch_bounds__(kThreads, CTAS) gn_image_kernel(GNApply a, PixelCount px, int C, float eps) {
  DDPPO_PDL_ENTRY();
  extern __shared__ float sh[];
  const int HW = px.HW, n = blockIdx.x, G = C / 2;
  const size_t ib = (size_t)n * HW * C;
  float* pz = sh + (int)blockDim.x * 2 * V;  // [C][2] partial sums of z, then of zd
  float* pd = pz + 2 * C;
  float* st = pd + 2 * C;                    // [4][G]: mean, rstd, mean_d, rstd_d
  block_shifted_sums<V>(a.z + ib, 0, HW, C, sh, pz);
  if (ZD) {
    __syncthreads();
    block_shifted_sums<V>(a.zd + ib, 0, HW, C, sh, pd);
  }
  __syncthreads();
  combine_groups_one(pz, a.z + ib, C, px, eps, st, st + G);
  if (ZD) combine_groups_one(pd, a.zd + ib, C, px, eps, st + 2 * G, st + 3 * G);
  __syncthreads();
  for (int g = threadIdx.x; g < G; g += blockDim.x) {
    const_cast<float*>(a.mean)[(size_t)n * G + g] = st[g];
    const_cast<float*>(a.rstd)[(size_t)n * G + g] = st[G + g];
    if (ZD) {
      const_cast<float*>(a.mean_d)[(size_t)n * G + g] = st[2 * G + g];
      const_cast<float*>(a.rstd_d)[(size_t)n * G + g] = st[3 * G + g];
    }
  }
  const int R = C / V, P = blockDim.x / R;
  const int cv = threadIdx.x % R, pr = threadIdx.x / R, c0 = cv * V;
  const float f8s = a.out_f8 ? *a.f8_scale : 1.f;
  const float f8m = normalise_rows<V, RES, ZD, CTAS == kImageCtas ? kRows : 1>(a, ib, pr, HW, P, C, c0, nullptr, nullptr, 0, st + c0 / 2, st + G + c0 / 2,
                          st + 2 * G + c0 / 2, st + 3 * G + c0 / 2, f8s);
  if (a.out_f8) block_amax(f8m, a.f8_amax);
}

// the instance for the inputs that are present
template <int V, int CTAS>
void (*image_kernel(const GNApply& a))(GNApply, PixelCount, int, float) {
  if (a.resid) return a.zd ? gn_image_kernel<V, true, true, CTAS> : gn_image_kernel<V, true, false, CTAS>;
  return a.zd ? gn_image_kernel<V, false, true, CTAS> : gn_image_kernel<V, false, false, CTAS>;
}

// ---- backward reductions: g = dy (masked by the ReLU that followed), xhat = (z - mu) rstd;
//      per image and channel sum(g) and sum(g xhat); group means of gamma-weighted sums ----
template <int V>
__global__ void __launch_bounds__(kThreads) gn_bwd_reduce_kernel(GNBack b, int HW, int C, int S,
                                                                 float* __restrict__ part,
                                                                 int* __restrict__ cnt) {
  DDPPO_PDL_ENTRY();
  extern __shared__ float sh[];
  __shared__ int flag;
  const int R = C / V, P = blockDim.x / R, G = C / 2;
  const int n = blockIdx.y, sb = blockIdx.x;
  const int cv = threadIdx.x % R, pr = threadIdx.x / R, c0 = cv * V;
  const int chunk = (HW + S - 1) / S, pb = sb * chunk, pe = min(HW, pb + chunk);
  const size_t ib = (size_t)n * HW * C;
  float mu[V], rs[V], sg[V], sgx[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    mu[v] = b.mean[(size_t)n * G + (c0 + v) / 2];
    rs[v] = b.rstd[(size_t)n * G + (c0 + v) / 2];
    sg[v] = sgx[v] = 0.f;
  }
#pragma unroll 8
  for (int p = pb + pr; p < pe; p += P) {
    const size_t o = ib + (size_t)p * C + c0;
    float d[V], x[V];
    ldv<V>(b.z + o, x);
    ldv<V>(b.dy + o, d);
    mask_relu<V>(b, o, c0, x, mu, rs, d);
#pragma unroll
    for (int v = 0; v < V; ++v) sum_grad(d[v], x[v], mu[v], rs[v], sg[v], sgx[v]);
  }
  float* pp = part + ((size_t)n * S + sb) * C * 2;
  block_pair_sums<V>(sg, sgx, sh, C, pp);
  if (!last_of_image(cnt + n, S, &flag)) return;
  // per-channel totals (block order), then the group means of gamma-weighted sums
  const float* pim = part + (size_t)n * S * C * 2;
  for (int i = threadIdx.x; i < S * C * 2; i += blockDim.x) sh[i] = __ldcg(pim + i);
  __syncthreads();
  float* tot = sh + S * C * 2;  // [C][2]
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    float a = 0.f, e = 0.f;
    for (int t = 0; t < S; ++t) {
      a += sh[(t * C + c) * 2];
      e += sh[(t * C + c) * 2 + 1];
    }
    tot[2 * c] = a;
    tot[2 * c + 1] = e;
    b.dbeta_part[(size_t)n * C + c] = a;
    b.dgamma_part[(size_t)n * C + c] = e;
  }
  __syncthreads();
  const float inv = 1.0f / (float)(2 * HW);
  for (int g = threadIdx.x; g < G; g += blockDim.x) {
    const float g0 = b.gamma[2 * g], g1 = b.gamma[2 * g + 1];
    b.m1[(size_t)n * G + g] = group_mean(tot[4 * g], g0, tot[4 * g + 2], g1, inv);
    b.m2[(size_t)n * G + g] = group_mean(tot[4 * g + 1], g0, tot[4 * g + 3], g1, inv);
  }
  if (threadIdx.x == 0) cnt[n] = 0;
}

// ---- dz = rstd (g gamma - m1 - xhat m2); optionally g itself (the masked gradient) ----
template <int V>
__global__ void __launch_bounds__(kThreads) gn_bwd_apply_kernel(GNBack b, int HW, int C) {
  DDPPO_PDL_ENTRY();
  const int R = C / V, G = C / 2;
  const int n = blockIdx.y;
  const int per = HW * R;
  const size_t ib = (size_t)n * HW * C;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < per; i += gridDim.x * blockDim.x) {
    const int c0 = (i % R) * V;
    const size_t o = ib + (size_t)i * V;
    float d[V], x[V], gm[V], r[V], mu[V], rs[V];
    const size_t gi = (size_t)n * G + c0 / 2;
    ldv<V>(b.z + o, x);
    ldv<V>(b.gamma + c0, gm);
    ldv<V>(b.dy + o, d);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      mu[v] = b.mean[gi + v / 2];
      rs[v] = b.rstd[gi + v / 2];
    }
    mask_relu<V>(b, o, c0, x, mu, rs, d);
    if (b.g_out && masks_given(b)) stv<V>(b.g_out + o, d);
#pragma unroll
    for (int v = 0; v < V; ++v)
      r[v] = input_grad(d[v], x[v], mu[v], rs[v], gm[v], b.m1[gi + v / 2], b.m2[gi + v / 2]);
    if (b.dz32) stv<V>(b.dz32 + o, r);
    if (b.dzop) stv_op<V>(b.dzop, o, r, b.op_bf16);
  }
}

// ---- backward, one block per image: the reduction (the reduce kernel's S = 1 arithmetic),
//      the group means in shared memory, then the input gradient of the image just read ----
template <int V>
__global__ void __launch_bounds__(kThreads, 4) gn_bwd_image_kernel(GNBack b, int HW, int C) {
  DDPPO_PDL_ENTRY();
  extern __shared__ float sh[];
  const int R = C / V, P = blockDim.x / R, G = C / 2;
  const int n = blockIdx.x;
  const int cv = threadIdx.x % R, pr = threadIdx.x / R, c0 = cv * V;
  const size_t ib = (size_t)n * HW * C;
  float* part = sh + blockDim.x * 2 * V;  // [C][2]: sum g, sum g xhat
  float* m12 = part + 2 * C;              // [2][G]: m1, m2
  float mu[V], rs[V], sg[V], sgx[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    mu[v] = b.mean[(size_t)n * G + (c0 + v) / 2];
    rs[v] = b.rstd[(size_t)n * G + (c0 + v) / 2];
    sg[v] = sgx[v] = 0.f;
  }
#pragma unroll 8
  for (int p = pr; p < HW; p += P) {
    const size_t o = ib + (size_t)p * C + c0;
    float d[V], x[V];
    ldv<V>(b.z + o, x);
    ldv<V>(b.dy + o, d);
    mask_relu<V>(b, o, c0, x, mu, rs, d);
#pragma unroll
    for (int v = 0; v < V; ++v) sum_grad(d[v], x[v], mu[v], rs[v], sg[v], sgx[v]);
  }
  block_pair_sums<V>(sg, sgx, sh, C, part);
  __syncthreads();
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    b.dbeta_part[(size_t)n * C + c] = 0.f + part[2 * c];
    b.dgamma_part[(size_t)n * C + c] = 0.f + part[2 * c + 1];
  }
  const float inv = 1.0f / (float)(2 * HW);
  for (int g = threadIdx.x; g < G; g += blockDim.x) {
    const float g0 = b.gamma[2 * g], g1 = b.gamma[2 * g + 1];
    const float t0 = 0.f + part[4 * g], t1 = 0.f + part[4 * g + 1];
    const float t2 = 0.f + part[4 * g + 2], t3 = 0.f + part[4 * g + 3];
    m12[g] = group_mean(t0, g0, t2, g1, inv);
    m12[G + g] = group_mean(t1, g0, t3, g1, inv);
  }
  __syncthreads();
  float gm[V];
  ldv<V>(b.gamma + c0, gm);
  // kRows rows at a time, loads before stores (as normalise_rows)
  for (int p0 = pr; p0 < HW; p0 += kRows * P) {
    float x[kRows][V], d[kRows][V];
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const size_t o = ib + (size_t)(p0 + u * P) * C + c0;
      if (p0 + u * P >= HW) break;
      ldv<V>(b.z + o, x[u]);
      ldv<V>(b.dy + o, d[u]);
      mask_relu<V>(b, o, c0, x[u], mu, rs, d[u]);
    }
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const size_t o = ib + (size_t)(p0 + u * P) * C + c0;
      if (p0 + u * P >= HW) break;
      if (b.g_out && masks_given(b)) stv<V>(b.g_out + o, d[u]);
      float r[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int g = (c0 + v) / 2;
        r[v] = input_grad(d[u][v], x[u][v], mu[v], rs[v], gm[v], m12[g], m12[G + g]);
      }
      if (b.dz32) stv<V>(b.dz32 + o, r);
      if (b.dzop) stv_op<V>(b.dzop, o, r, b.op_bf16);
    }
  }
}

// ---- slices: few images, one block per image and run of Cs channels ----
// Groups are two channels, so a run of channels needs nothing from the others: a block stages
// its run of an image (HW x Cs fp32, with the residual or dy; copied asynchronously by the
// threads that use it) in shared memory and does both passes from there. With few images
// (the act batch, small updates) narrow runs spread an image over the SMs without a barrier,
// and one launch replaces two. Runs are at least 8 channels (one 32-byte sector); the copies
// ask L2 for the whole line, which the neighbouring runs' blocks use.
//
// The sums are those of the one-block-per-image form: thread (row class pr, vector cv) adds
// rows pr, pr + P, ... with P = 256 / (C / 4) of the whole image's layout, so the bits are
// the same for every run width.
//
// Bound: latency (an image's loads, its chain of sums, the reduction, its stores).
// Measured: the act batch's 17 normalisations 8.1 us each against 10.7 (statistics 7.3, apply
// 3.3) in two launches; the backward of 64 frames 10.2 against 16.2, of 300 frames 21.7
// against 30.3.
__device__ __forceinline__ void copy16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__global__ void __launch_bounds__(kThreads) gn_slice_kernel(GNApply a, PixelCount px, int C, int Cs, float eps) {
  DDPPO_PDL_ENTRY();
  extern __shared__ __align__(16) float sm[];
  const int R = Cs / 4, P = blockDim.x / R, G = C / 2, Gs = Cs / 2, HW = px.HW, n = blockIdx.y;
  const int cv = threadIdx.x % R, pr = threadIdx.x / R, cb = blockIdx.x * Cs, c0 = cb + cv * 4;
  const size_t ib = (size_t)n * HW * C;
  float* sz = sm;                               // [HW][Cs]
  const bool two = a.zd || a.resid;
  float* sd = sz + (two ? (size_t)HW * Cs : 0);  // [HW][Cs] of zd or of the residual
  float* sh = sd + (size_t)HW * Cs;             // [threads][8] partial sums
  float* pz = sh + blockDim.x * 8;              // [Cs][2] of z, then of zd
  float* pd = pz + 2 * Cs;
  float* st = pd + 2 * Cs;                      // [4][Gs]: mean, rstd, mean_d, rstd_d
  for (int p = pr; p < HW; p += P) copy16(sz + (size_t)p * Cs + cv * 4, a.z + ib + (size_t)p * C + c0);
  if (two) {
    const float* src = a.zd ? a.zd : a.resid;
    for (int p = pr; p < HW; p += P) copy16(sd + (size_t)p * Cs + cv * 4, src + ib + (size_t)p * C + c0);
  }
  float K[4], Kd[4] = {0.f, 0.f, 0.f, 0.f};
  ldv<4>(a.z + ib + c0, K);
  if (a.zd) ldv<4>(a.zd + ib + c0, Kd);
  copies_done();  // each thread reads back only what it copied
  for (int j = 0; j < (a.zd ? 2 : 1); ++j) {
    const float* src = (j ? sd : sz) + cv * 4;
    float s1[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int p = pr; p < HW; p += P) {
      float x[4];
      ldv<4>(src + (size_t)p * Cs, x);
#pragma unroll
      for (int v = 0; v < 4; ++v) sum_shifted(x[v], j ? Kd[v] : K[v], s1[v], s2[v]);
    }
    if (j) __syncthreads();
    block_pair_sums<4>(s1, s2, sh, Cs, j ? pd : pz);
  }
  __syncthreads();
  combine_groups_one(pz, a.z + ib + cb, Cs, px, eps, st, st + Gs);
  if (a.zd) combine_groups_one(pd, a.zd + ib + cb, Cs, px, eps, st + 2 * Gs, st + 3 * Gs);
  __syncthreads();
  for (int g = threadIdx.x; g < Gs; g += blockDim.x) {
    const size_t o = (size_t)n * G + cb / 2 + g;
    const_cast<float*>(a.mean)[o] = st[g];
    const_cast<float*>(a.rstd)[o] = st[Gs + g];
    if (a.zd) {
      const_cast<float*>(a.mean_d)[o] = st[2 * Gs + g];
      const_cast<float*>(a.rstd_d)[o] = st[3 * Gs + g];
    }
  }
  const float f8s = a.out_f8 ? *a.f8_scale : 1.f;
  const float f8m = normalise_rows_any<4, kRows>(a, ib, pr, HW, P, C, c0, sz + cv * 4, sd + cv * 4, Cs, st + cv * 2,
                          st + Gs + cv * 2, st + 2 * Gs + cv * 2, st + 3 * Gs + cv * 2, f8s);
  if (a.out_f8) block_amax(f8m, a.f8_amax);
}

__global__ void __launch_bounds__(kThreads) gn_bwd_slice_kernel(GNBack b, int HW, int C, int Cs) {
  DDPPO_PDL_ENTRY();
  extern __shared__ __align__(16) float sm[];
  const int R = Cs / 4, P = blockDim.x / R, G = C / 2, Gs = Cs / 2, n = blockIdx.y;
  const int cv = threadIdx.x % R, pr = threadIdx.x / R, cb = blockIdx.x * Cs, c0 = cb + cv * 4;
  const size_t ib = (size_t)n * HW * C;
  float* sz = sm;                        // [HW][Cs]
  float* sy = sz + (size_t)HW * Cs;      // [HW][Cs] of dy, masked in the first pass
  float* sh = sy + (size_t)HW * Cs;      // [threads][8] partial sums
  float* part = sh + blockDim.x * 8;     // [Cs][2]: sum g, sum g xhat
  float* m12 = part + 2 * Cs;            // [2][Gs]: m1, m2
  for (int p = pr; p < HW; p += P) {
    const size_t o = ib + (size_t)p * C + c0;
    copy16(sz + (size_t)p * Cs + cv * 4, b.z + o);
    copy16(sy + (size_t)p * Cs + cv * 4, b.dy + o);
  }
  float mu[4], rs[4], gm[4], sg[4] = {0.f, 0.f, 0.f, 0.f}, sgx[4] = {0.f, 0.f, 0.f, 0.f};
  ldv<4>(b.gamma + c0, gm);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    mu[v] = b.mean[(size_t)n * G + (c0 + v) / 2];
    rs[v] = b.rstd[(size_t)n * G + (c0 + v) / 2];
  }
  copies_done();  // each thread reads back only what it copied
  const bool masked = b.relu_from_z || masks_given(b);
  for (int p0 = pr; p0 < HW; p0 += kRows * P) {
    float d[kRows][4], x[kRows][4];
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const int p = p0 + u * P;
      if (p >= HW) break;
      ldv<4>(sz + (size_t)p * Cs + cv * 4, x[u]);
      ldv<4>(sy + (size_t)p * Cs + cv * 4, d[u]);
      mask_relu<4>(b, ib + (size_t)p * C + c0, c0, x[u], mu, rs, d[u]);
    }
#pragma unroll
    for (int u = 0; u < kRows; ++u) {
      const int p = p0 + u * P;
      if (p >= HW) break;
      if (masked) stv<4>(sy + (size_t)p * Cs + cv * 4, d[u]);
      if (b.g_out && masks_given(b)) stv<4>(b.g_out + ib + (size_t)p * C + c0, d[u]);
#pragma unroll
      for (int v = 0; v < 4; ++v) sum_grad(d[u][v], x[u][v], mu[v], rs[v], sg[v], sgx[v]);
    }
  }
  block_pair_sums<4>(sg, sgx, sh, Cs, part);
  __syncthreads();
  for (int c = threadIdx.x; c < Cs; c += blockDim.x) {
    b.dbeta_part[(size_t)n * C + cb + c] = 0.f + part[2 * c];
    b.dgamma_part[(size_t)n * C + cb + c] = 0.f + part[2 * c + 1];
  }
  const float inv = 1.0f / (float)(2 * HW);
  for (int g = threadIdx.x; g < Gs; g += blockDim.x) {
    const float g0 = b.gamma[cb + 2 * g], g1 = b.gamma[cb + 2 * g + 1];
    const float t0 = 0.f + part[4 * g], t1 = 0.f + part[4 * g + 1];
    const float t2 = 0.f + part[4 * g + 2], t3 = 0.f + part[4 * g + 3];
    m12[g] = group_mean(t0, g0, t2, g1, inv);
    m12[Gs + g] = group_mean(t1, g0, t3, g1, inv);
  }
  __syncthreads();
  const float m1[2] = {m12[cv * 2], m12[cv * 2 + 1]}, m2[2] = {m12[Gs + cv * 2], m12[Gs + cv * 2 + 1]};
#pragma unroll 4
  for (int p = pr; p < HW; p += P) {
    const size_t o = ib + (size_t)p * C + c0;
    float d[4], x[4], r[4];
    ldv<4>(sz + (size_t)p * Cs + cv * 4, x);
    ldv<4>(sy + (size_t)p * Cs + cv * 4, d);
#pragma unroll
    for (int v = 0; v < 4; ++v) r[v] = input_grad(d[v], x[v], mu[v], rs[v], gm[v], m1[v / 2], m2[v / 2]);
    if (b.dz32) stv<4>(b.dz32 + o, r);
    if (b.dzop) stv_op<4>(b.dzop, o, r, b.op_bf16);
  }
}

// ---- backward of many images: each streamed twice through a shared-memory ring ----
// The backward reads z and dy twice. One block per image keeps four images per SM in work,
// 160 MB of a 32x32 x 32 batch, more than L2 holds: the second reading came from memory
// again. Here two blocks per SM take images in turn. One warp copies units (z, dy and the mask
// bits of kRingRows P pixels, up to 16.5 KB) into a ring with bulk copies, an image's units for
// the sums and then the same again for the gradient; eight warps consume them. The images
// in work (2 x 152) stay in L2 -- 912 images of 1024 x 32 read 260 MB from memory, 239 MB of z
// and dy once -- and copies are in flight whatever the consumers wait for.
// Sums in the one-block-per-image order: bit-identical.
// Measured on the encoder's 21 launches over 4096 frames: 4.14 ms, against 5.2 ms with one
// block per image and the same masks (6.3 ms when the masks were read from the stored fp32
// outputs). Two blocks and two rows a thread: 4 rows 4.8 ms, three blocks 4.4, one row 4.7,
// one block of 4 rows 4.1.
constexpr int kRingThreads = 288, kRingCtas = 2, kRingMax = 6;
constexpr int kRingHalf = kRingRows * 4 * 1024, kRingUnit = 2 * kRingHalf + kRingRows * 256;
__device__ __forceinline__ void consumers_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

template <int MASK>
__global__ void __launch_bounds__(kRingThreads, kRingCtas)
    gn_bwd_ring_kernel(GNBack b, int HW, int C, int N, int units, int32_t* err) {
  DDPPO_PDL_ENTRY();
  extern __shared__ __align__(128) uint8_t ring[];
  __shared__ uint64_t full[kRingMax], empty[kRingMax];
  __shared__ int abort_flag;
  __shared__ uint32_t n_issued;
  volatile int* abort = &abort_flag;
  const int R = C / 4, P = kThreads / R, G = C / 2, rows = kRingRows * P;
  const size_t image = (size_t)HW * C;
  float* sh = reinterpret_cast<float*>(ring + (size_t)units * kRingUnit);  // [256][8]
  float* part = sh + kThreads * 8;  // [C][2]: sum g, sum g xhat
  float* m12 = part + 2 * C;        // [2][G]: m1, m2
  if (threadIdx.x == 0) {
    for (int i = 0; i < units; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kThreads / 32);
    }
    abort_flag = 0;
    n_issued = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int slot = 0;
  uint32_t phase = 0;
  auto next = [&]() {
    if (++slot == units) { slot = 0; phase ^= 1u; }
  };
  if (threadIdx.x >= kThreads) {
    if (threadIdx.x == kThreads) {
      uint32_t it = 0;
      for (int n = blockIdx.x; n < N && !*abort; n += gridDim.x)
        for (int p2 = 0; p2 < 2 * HW && !*abort;) {
          const int p = p2 < HW ? p2 : p2 - HW, cnt = min(rows, HW - p);
          const size_t o = n * image + (size_t)p * C;
          const uint32_t bytes = (uint32_t)(cnt * C) * 4u, pb = MASK == MASK_POS ? bytes / 16 : 0u;
          if (!mbar_wait(&empty[slot], phase ^ 1u, abort, err)) break;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&full[slot])),
                       "r"(2 * bytes + pb)
                       : "memory");
          uint8_t* u = ring + (size_t)slot * kRingUnit;
          bulk_copy(u, b.z + o, bytes, &full[slot]);
          bulk_copy(u + kRingHalf, b.dy + o, bytes, &full[slot]);
          if (MASK == MASK_POS) bulk_copy(u + 2 * kRingHalf, b.pos + o / 4, pb, &full[slot]);
          ++it;
          next();
          p2 += cnt;
        }
      n_issued = it;
    }
  } else {
    const int cv = threadIdx.x % R, pr = threadIdx.x / R, c0 = cv * 4;
    const bool active = pr < P;
    bool ok = true;
    float gm[4], bt[4];
    ldv<4>(b.gamma + c0, gm);
    if (MASK == MASK_Z) ldv<4>(b.beta + c0, bt);
    // statistics of the next image, fetched while the current one is worked on
    float2 nmu = make_float2(0.f, 0.f), nrs = nmu;
    auto fetch = [&](int n) {
      if (n >= N) return;
      nmu = *reinterpret_cast<const float2*>(b.mean + (size_t)n * G + 2 * cv);
      nrs = *reinterpret_cast<const float2*>(b.rstd + (size_t)n * G + 2 * cv);
    };
    fetch(blockIdx.x);
    const float inv = 1.0f / (float)(2 * HW);
    // one unit: the thread's rows, dy masked; the slot is free once they are in registers
    auto take = [&](int p, float (&x)[kRingRows][4], float (&d)[kRingRows][4], const float (&mu)[4], const float (&rs)[4]) {
      ok = mbar_wait(&full[slot], phase, abort, err) && ok;
      const float* sz = reinterpret_cast<const float*>(ring + (size_t)slot * kRingUnit) + pr * C + c0;
      const uint8_t* sp = ring + (size_t)slot * kRingUnit + 2 * kRingHalf + (pr * C + c0) / 4;
#pragma unroll
      for (int u = 0; u < kRingRows; ++u) {
        if (!active || p + u * P + pr >= HW) break;
        ldv<4>(sz + u * P * C, x[u]);
        ldv<4>(sz + u * P * C + kRingHalf / 4, d[u]);
        if (MASK == MASK_Z) {
#pragma unroll
          for (int v = 0; v < 4; ++v)
            if (!(normalised(x[u][v], mu[v], rs[v], gm[v], bt[v]) > 0.f)) d[u][v] = 0.f;
        } else if (MASK == MASK_POS) {
          const unsigned m = sp[u * P * C / 4];
#pragma unroll
          for (int v = 0; v < 4; ++v) d[u][v] = (m >> v) & 1u ? d[u][v] : 0.f;
        }
      }
      __syncwarp();
      if ((threadIdx.x & 31) == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&empty[slot])) : "memory");
      next();
    };
    for (int n = blockIdx.x; n < N; n += gridDim.x) {
      const float mu[4] = {nmu.x, nmu.x, nmu.y, nmu.y}, rs[4] = {nrs.x, nrs.x, nrs.y, nrs.y};
      fetch(n + gridDim.x);
      float sg[4] = {0.f, 0.f, 0.f, 0.f}, sgx[4] = {0.f, 0.f, 0.f, 0.f};
      for (int p = 0; p < HW; p += rows) {
        float x[kRingRows][4], d[kRingRows][4];
        take(p, x, d, mu, rs);
#pragma unroll
        for (int u = 0; u < kRingRows; ++u) {
          if (!active || p + u * P + pr >= HW) break;
#pragma unroll
          for (int v = 0; v < 4; ++v) sum_grad(d[u][v], x[u][v], mu[v], rs[v], sg[v], sgx[v]);
        }
      }
      // per-channel sums over the P row classes, in class order (block_pair_sums' arithmetic)
      if (active) {
        stv<4>(sh + threadIdx.x * 8, sg);
        stv<4>(sh + threadIdx.x * 8 + 4, sgx);
      }
      consumers_sync();
      for (int c = threadIdx.x; c < C; c += kThreads) {
        const float* q = sh + (c >> 2) * 8 + (c & 3);
        float sa = 0.f, sb = 0.f;
        for (int r = 0; r < P; ++r) {
          sa += q[(size_t)r * R * 8];
          sb += q[(size_t)r * R * 8 + 4];
        }
        part[2 * c] = sa;
        part[2 * c + 1] = sb;
        if (ok) {
          b.dbeta_part[(size_t)n * C + c] = 0.f + sa;
          b.dgamma_part[(size_t)n * C + c] = 0.f + sb;
        }
      }
      consumers_sync();
      for (int g = threadIdx.x; g < G; g += kThreads) {
        const float g0 = b.gamma[2 * g], g1 = b.gamma[2 * g + 1];
        const float t0 = 0.f + part[4 * g], t1 = 0.f + part[4 * g + 1];
        const float t2 = 0.f + part[4 * g + 2], t3 = 0.f + part[4 * g + 3];
        m12[g] = group_mean(t0, g0, t2, g1, inv);
        m12[G + g] = group_mean(t1, g0, t3, g1, inv);
      }
      consumers_sync();
      const float m1[2] = {m12[2 * cv], m12[2 * cv + 1]}, m2[2] = {m12[G + 2 * cv], m12[G + 2 * cv + 1]};
      for (int p = 0; p < HW; p += rows) {
        float x[kRingRows][4], d[kRingRows][4];
        take(p, x, d, mu, rs);
#pragma unroll
        for (int u = 0; u < kRingRows; ++u) {
          if (!active || !ok || p + u * P + pr >= HW) break;
          const size_t o = n * image + (size_t)(p + u * P + pr) * C + c0;
          if (MASK == MASK_POS && b.g_out) stv<4>(b.g_out + o, d[u]);
          float r[4];
#pragma unroll
          for (int v = 0; v < 4; ++v)
            r[v] = input_grad(d[u][v], x[u][v], mu[v], rs[v], gm[v], m1[v / 2], m2[v / 2]);
          if (b.dz32) stv<4>(b.dz32 + o, r);
          if (b.dzop) stv_op<4>(b.dzop, o, r, b.op_bf16);
        }
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (abort_flag) {  // the copies still in flight land (bounded) before the block ends
    if (threadIdx.x == 0) {
      const uint32_t first = n_issued > (uint32_t)units ? n_issued - units : 0u;
      for (uint32_t it = first; it < n_issued; ++it) mbar_drain_wait(&full[it % units], (it / units) & 1u);
    }
    __syncthreads();
  }
}

size_t ring_smem(int units, int C) {
  return (size_t)units * kRingUnit + ((size_t)kThreads * 8 + 3 * (size_t)C) * sizeof(float);
}
// ring depth (0: not covered): what two blocks per SM leave room for (228 KB, 1 KB of it
// reserved per block)
int ring_units(const GNBack& b, int HW, int C) {
  const int kind = mask_kind(b, 4);
  if (C % 4 || C > 512 || kind == MASK_Y) return 0;
  // other widths take the one-block-per-image form, whose threads load their own mask byte
  if (kind == MASK_POS && !ring_mask_copies_ok(HW, C)) return 0;
  const size_t room = (size_t)228 * 1024 / kRingCtas - 2048 - ring_smem(0, C);
  return (int)std::min<size_t>(kRingMax, room / kRingUnit);
}

PixelCount pixel_count(int HW) {
  return PixelCount{HW, 1.0 / HW, (HW & (HW - 1)) == 0 ? 1.0 / (2.0 * HW) : 0.0};
}

int num_sms_cached() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
      sms = 1;
  }
  return sms;
}

bool gn_shape_ok(int C) { return C >= 2 && C % 2 == 0 && C / (C % 4 == 0 ? 4 : 2) <= kThreads; }

// blocks per image: enough for ~8 blocks per SM overall, at least one pixel pass each
int gn_split(int N, int HW, int C, const GnScratch& w) {
  // images of at most 32K elements (128 KB): one block each -- a block sums such an image
  // faster than S blocks combine their partials (measured: the 64-image act batch); and any
  // image size once there are at least 4 images per SM (one block each already fills the GPU)
  if ((long)HW * C <= 32768 || N >= 4 * num_sms_cached()) return 1;
  const int V = C % 4 == 0 ? 4 : 2;
  const int P = rows_per_pass(C, V);
  const int want = (8 * num_sms_cached() + N - 1) / N;
  int S = std::min(want, (HW + P - 1) / P);
  S = std::min(S, 64);
  S = std::min(S, std::max(1, 4096 / C));  // the combine stages S x C x 2 floats in shared memory
  S = std::max(S, 1);
  while (S > 1 && (size_t)N * S * C * 2 > w.part_elems) --S;
  return S;
}

unsigned apply_blocks(int N, int HW, int C, int V) {
  const long per = (long)HW * (C / V);
  const int want = (8 * num_sms_cached() + N - 1) / N;
  long bx = (per + kThreads - 1) / kThreads;
  bx = std::min<long>(bx, std::max(want, 1));
  return (unsigned)std::max<long>(bx, 1);
}

// bytes of shared memory of a slice block (tensors: staged arrays)
size_t slice_smem(int HW, int Cs, int threads, int tensors) {
  return ((size_t)tensors * HW * Cs + (size_t)threads * 8 + 6 * (size_t)Cs) * sizeof(float);
}

// channels per slice block (0: the slice form does not apply): the widest run of whole warps
// whose staging leaves room for three blocks per SM and whose blocks still fill the GPU
// twice, else the narrowest that fits
int slice_channels(int N, int HW, int C, int tensors) {
  if (C % 8 || C / 4 > kThreads) return 0;
  const int P = rows_per_pass(C, 4), sms = num_sms_cached();
  int best = 0;
  for (int Cs = C; Cs >= 8; Cs -= 8) {
    const int th = P * (Cs / 4);
    if (C % Cs || th % 32) continue;
    const size_t smem = slice_smem(HW, Cs, th, tensors);
    if (smem > 110 * 1024) continue;
    best = Cs;
    if (smem <= 74 * 1024 && (long)N * (C / Cs) >= 2l * sms) break;
  }
  return best;
}

template <class K>
int smem_attr(K kern, bool* done) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && !done[dev]) {
    DDPPO_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024));
    done[dev] = true;
  }
  return DDPPO_OK;
}

int threads_for(int C, int V) {
  const int R = C / V;
  return R * rows_per_pass(C, V);
}

}  // namespace

size_t gn_part_elems(int max_images, int max_C) {
  return (size_t)(max_images + 8 * num_sms_cached() + 64) * max_C * 2;
}

// dynamic shared memory of the one-launch kernel for S blocks per image
static size_t fused_smem(int S, int C, int V) {
  const int th = threads_for(C, V);
  return ((size_t)std::max(th * 2 * V, S * C * 2) + 2 * (size_t)C) * sizeof(float);
}

// blocks per image of the one-launch form: gn_split's choice, lowered until all S x N
// blocks are resident at once; 0 when even S = 1 is not (the two-launch form then keeps
// gn_split's choice). The statistics launch of the two-launch form uses the same S, so
// the two forms give bit-identical statistics.
static int gn_split_one_launch(int N, int HW, int C, const GnScratch& w) {
  if (!w.cnt2) return 0;
  const int V = C % 4 == 0 ? 4 : 2;
  void (*kern)(GNApply, PixelCount, int, int, float, float*, float*, int*, int*, int32_t*) =
      V == 4 ? gn_fused_kernel<4> : gn_fused_kernel<2>;
  const int th = threads_for(C, V);
  const int sms = num_sms_cached();
  for (int S = gn_split(N, HW, C, w); S >= 1; --S) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, th, fused_smem(S, C, V)) != cudaSuccess)
      return 0;
    if ((long)S * N <= (long)std::min(occ, kFusedBlocks) * sms) return S;
  }
  return 0;
}

// whether a forward of these sizes (tensors: z, and a residual or shortcut beside it) needs the
// scratch: not where one block sums an image or a slice of its channels and normalises it
bool gn_fwd_scratch(int N, int HW, int C, int tensors, const GnScratch& w) {
  return gn_split(N, HW, C, w) != 1 || (N < 4 * num_sms_cached() && !slice_channels(N, HW, C, tensors));
}

int launch_gn_stats(const float* z, int N, int HW, int C, float eps, float* mean, float* rstd,
                    const GnScratch& w, cudaStream_t s) {
  if (!N || !HW) return DDPPO_OK;
  if (!gn_shape_ok(C) || N > w.max_images || N > 65535) {
    set_error("gn: unsupported channel count or too many images for the scratch");
    return DDPPO_E_CONFIG;
  }
  const int V = C % 4 == 0 ? 4 : 2;
  const int S1 = gn_split_one_launch(N, HW, C, w);
  const int S = S1 ? S1 : gn_split(N, HW, C, w);
  const int th = threads_for(C, V);
  const size_t smem = std::max((size_t)th * 2 * V, (size_t)S * C * 2) * sizeof(float);
  const dim3 grid(S, N);
  if (V == 4) ::ddppo::launch_k(gn_stats_kernel<4>, grid, th, smem, s, z, pixel_count(HW), C, S, eps, w.part, w.cnt, mean, rstd);
  else ::ddppo::launch_k(gn_stats_kernel<2>, grid, th, smem, s, z, pixel_count(HW), C, S, eps, w.part, w.cnt, mean, rstd);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

int launch_gn_fused(const GNApply& a, int N, int HW, int C, float eps, const GnScratch& w,
                    int32_t* err, cudaStream_t s, bool* launched) {
  *launched = false;
  if (!N || !HW) { *launched = true; return DDPPO_OK; }
  if (!gn_shape_ok(C) || N > w.max_images || N > 65535) return DDPPO_OK;
  const int V = C % 4 == 0 ? 4 : 2;
  const int th = threads_for(C, V);
  void (*kern)(GNApply, PixelCount, int, int, float, float*, float*, int*, int*, int32_t*) =
      V == 4 ? gn_fused_kernel<4> : gn_fused_kernel<2>;
  const int nt = a.zd ? 2 : 1;
  if (gn_split(N, HW, C, w) == 1) {
    // one block sums an image, or a run of its channels where the run fits shared memory
    if (const int Cs = N < 4 * num_sms_cached() ? slice_channels(N, HW, C, a.zd || a.resid ? 2 : 1) : 0) {
      static bool done[64] = {};
      DDPPO_TRY(smem_attr(gn_slice_kernel, done));
      const int ths = rows_per_pass(C, 4) * (Cs / 4);
      ::ddppo::launch_k(gn_slice_kernel, dim3(C / Cs, N), ths, slice_smem(HW, Cs, ths, a.zd || a.resid ? 2 : 1), s, a, pixel_count(HW), C, Cs, eps);
      DDPPO_CHECK_LAUNCH();
      *launched = true;
      return DDPPO_OK;
    }
    // many images (at least 4 per SM: the update's minibatches): one block per image; few: the statistics launch then a normalise launch that spreads
    // each image over many blocks
    if (N < 4 * num_sms_cached()) return DDPPO_OK;
    const size_t smem = ((size_t)th * 2 * V + 6 * (size_t)C) * sizeof(float);
    const PixelCount px = pixel_count(HW);
    const auto kern = V != 4 ? image_kernel<2, kImageCtas>(a)
                      : N <= kFewCtas * num_sms_cached() ? image_kernel<4, kFewCtas>(a)
                                                         : image_kernel<4, kImageCtas>(a);
    ::ddppo::launch_k(kern, N, th, smem, s, a, px, C, eps);
    DDPPO_CHECK_LAUNCH();
    *launched = true;
    return DDPPO_OK;
  }
  // every block resident at once, and the partials of z (and zd) in the scratch;
  // otherwise two launches
  const int S = gn_split_one_launch(N, HW, C, w);
  if (S < 1 || (size_t)nt * N * S * C * 2 > w.part_elems) return DDPPO_OK;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(S, N);
  cfg.blockDim = dim3(th);
  cfg.dynamicSmemBytes = fused_smem(S, C, V);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  float* part_d = w.part + (size_t)N * S * C * 2;
  DDPPO_CHECK_CUDA(cudaLaunchKernelEx(&cfg, kern, a, pixel_count(HW), C, S, eps, w.part, part_d, w.cnt, w.cnt2, err));
  *launched = true;
  return DDPPO_OK;
}

int launch_gn_apply(const GNApply& a, int N, int HW, int C, cudaStream_t s) {
  if (!N || !HW) return DDPPO_OK;
  if (!gn_shape_ok(C) || N > 65535) { set_error("gn: unsupported shape"); return DDPPO_E_CONFIG; }
  const int V = C % 4 == 0 ? 4 : 2;
  const dim3 grid(apply_blocks(N, HW, C, V), N);
  if (V == 4) ::ddppo::launch_k(gn_apply_kernel<4>, grid, kThreads, 0, s, a, HW, C);
  else ::ddppo::launch_k(gn_apply_kernel<2>, grid, kThreads, 0, s, a, HW, C);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

int launch_gn_bwd(const GNBack& b, int N, int HW, int C, const GnScratch& w, int32_t* err,
                  cudaStream_t s) {
  if (!N || !HW) return DDPPO_OK;
  if (!gn_shape_ok(C) || N > w.max_images || N > 65535) {
    set_error("gn: unsupported channel count or too many images for the scratch");
    return DDPPO_E_CONFIG;
  }
  const int V = C % 4 == 0 ? 4 : 2;
  const int S = gn_split(N, HW, C, w);
  const int th = threads_for(C, V);
  if (const int Cs = S == 1 && N < 4 * num_sms_cached() ? slice_channels(N, HW, C, 2) : 0) {
    static bool done[64] = {};
    DDPPO_TRY(smem_attr(gn_bwd_slice_kernel, done));
    const int ths = rows_per_pass(C, 4) * (Cs / 4);
    ::ddppo::launch_k(gn_bwd_slice_kernel, dim3(C / Cs, N), ths, slice_smem(HW, Cs, ths, 2), s, b, HW, C, Cs);
    DDPPO_CHECK_LAUNCH();
    return DDPPO_OK;
  }
  if (S == 1 && N >= 4 * num_sms_cached()) {
    // many small images: one block per image, reduction and input gradient in one launch
    if (const int units = ring_units(b, HW, C)) {
      static bool done[3][64] = {};
      const int kind = mask_kind(b, 4);
      auto kern = kind == MASK_Z ? gn_bwd_ring_kernel<MASK_Z>
                  : kind == MASK_POS ? gn_bwd_ring_kernel<MASK_POS> : gn_bwd_ring_kernel<MASK_NONE>;
      DDPPO_TRY(smem_attr(kern, done[kind]));
      ::ddppo::launch_k(kern, std::min(N, kRingCtas * num_sms_cached()), kRingThreads, ring_smem(units, C), s, b,
                        HW, C, N, units, err);
      DDPPO_CHECK_LAUNCH();
      return DDPPO_OK;
    }
    const size_t smem1 = ((size_t)th * 2 * V + 3 * (size_t)C) * sizeof(float);
    if (V == 4) ::ddppo::launch_k(gn_bwd_image_kernel<4>, N, th, smem1, s, b, HW, C);
    else ::ddppo::launch_k(gn_bwd_image_kernel<2>, N, th, smem1, s, b, HW, C);
    DDPPO_CHECK_LAUNCH();
    return DDPPO_OK;
  }
  const size_t smem = std::max((size_t)th * 2 * V, (size_t)(S + 1) * C * 2) * sizeof(float);
  const dim3 grid(S, N);
  if (V == 4) ::ddppo::launch_k(gn_bwd_reduce_kernel<4>, grid, th, smem, s, b, HW, C, S, w.part, w.cnt);
  else ::ddppo::launch_k(gn_bwd_reduce_kernel<2>, grid, th, smem, s, b, HW, C, S, w.part, w.cnt);
  DDPPO_CHECK_LAUNCH();
  const dim3 ga(apply_blocks(N, HW, C, V), N);
  if (V == 4) ::ddppo::launch_k(gn_bwd_apply_kernel<4>, ga, kThreads, 0, s, b, HW, C);
  else ::ddppo::launch_k(gn_bwd_apply_kernel<2>, ga, kThreads, 0, s, b, HW, C);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

// ---- GroupNorm apply + ReLU + 3x3 / stride-2 / pad-1 max pool (4 channels per thread) ----
// A thread walks down a column of windows: of a window's three input rows the first is the
// last of the window above, kept normalised, so it loads six pixels and not nine, all in
// flight at once. Each window compares in (ky, kx) order. Bound: HBM -- z once, the pooled
// outputs once (3.0 GB for 4096 images of 64x64x32). Nine loads a window one after another
// took 959 us there; this form 595 (5.0 TB/s).
__global__ void __launch_bounds__(kThreads) gn_relu_maxpool_kernel(GNApply a, int H, int W, int C, int rows,
                                                                   float* __restrict__ pool,
                                                                   __nv_bfloat16* __restrict__ pool_bf,
                                                                   uint8_t* __restrict__ arg) {
  DDPPO_PDL_ENTRY();
  const int Hq = (H - 1) / 2 + 1, Wq = (W - 1) / 2 + 1, C4 = C / 4, G = C / 2;
  const int n = blockIdx.y, p0 = blockIdx.x * rows, p1 = min(Hq, p0 + rows);
  const float* zi = a.z + (size_t)n * H * W * C;
  const float f8s = a.out_f8 ? *a.f8_scale : 1.f;
  float f8m = 0.f;
  for (int i = threadIdx.x; i < Wq * C4; i += kThreads) {
    const int q = i / C4, c0 = (i - q * C4) * 4;
    float gm[4], bt[4], mu[4], rs[4];
    ldv<4>(a.gamma + c0, gm);
    ldv<4>(a.beta + c0, bt);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      mu[v] = a.mean[(size_t)n * G + (c0 + v) / 2];
      rs[v] = a.rstd[(size_t)n * G + (c0 + v) / 2];
    }
    const int x0 = 2 * q - 1;
    const bool in[3] = {x0 >= 0, true, x0 + 2 < W};
    // normalised rows of the column's three pixels; pixels outside count as -infinity
    const auto load = [&](int iy, float (&x)[3][4]) {
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (in[k] && iy >= 0 && iy < H) ldv<4>(zi + ((size_t)iy * W + x0 + k) * C + c0, x[k]);
    };
    const auto norm = [&](int iy, float (&x)[3][4]) {
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int v = 0; v < 4; ++v)
          x[k][v] = in[k] && iy >= 0 && iy < H ? fmaxf(normalised(x[k][v], mu[v], rs[v], gm[v], bt[v]), 0.f)
                                               : -INFINITY;
    };
    float top[3][4];
    load(2 * p0 - 1, top);
    norm(2 * p0 - 1, top);
#pragma unroll 1
    for (int p = p0; p < p1; ++p) {
      float mid[3][4], bot[3][4];
      load(2 * p, mid);
      load(2 * p + 1, bot);
      norm(2 * p, mid);
      norm(2 * p + 1, bot);
      float best[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      int bi[4] = {0, 0, 0, 0};
#pragma unroll
      for (int k = 0; k < 9; ++k)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const float y = k < 3 ? top[k % 3][v] : k < 6 ? mid[k % 3][v] : bot[k % 3][v];
          if (y > best[v]) { best[v] = y; bi[v] = k; }
        }
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int v = 0; v < 4; ++v) top[k][v] = bot[k][v];
      const size_t o = (((size_t)n * Hq + p) * Wq + q) * C + c0;
      stv<4>(pool + o, best);
      if (pool_bf) stv_bf<4>(pool_bf + o, best);
      if (a.out_f8) {
        stv_e4m3<4>(a.out_f8 + o, best, f8s);
#pragma unroll
        for (int v = 0; v < 4; ++v) f8m = fmaxf(f8m, best[v]);
      }
      *reinterpret_cast<uchar4*>(arg + o) = make_uchar4(bi[0], bi[1], bi[2], bi[3]);
    }
  }
  if (a.out_f8) block_amax(f8m, a.f8_amax);
}

int launch_gn_relu_maxpool(const GNApply& a, int N, int H, int W, int C, float* pool,
                           __nv_bfloat16* pool_bf, uint8_t* arg, cudaStream_t s) {
  if (!N) return DDPPO_OK;
  const int Hq = (H - 1) / 2 + 1, Wq = (W - 1) / 2 + 1;
  if (C % 4 || N > 65535 || (int64_t)Hq * Wq * C >= (1ll << 31)) {
    set_error("gn_relu_maxpool: unsupported shape");
    return DDPPO_E_CONFIG;
  }
  // few images: their rows over several blocks (each normalises the row above its first again)
  const int rows = std::max(1, (int)std::min<long>(Hq, (long)N * Hq / (8l * num_sms_cached())));
  ::ddppo::launch_k(gn_relu_maxpool_kernel, dim3((Hq + rows - 1) / rows, N), kThreads, 0, s, a, H, W, C, rows, pool,
                    pool_bf, arg);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

}  // namespace ddppo
