// SIMT GEMM (the plain FP32 form, and the fallback shape path of the BF16 form) with
// deterministic split-K, plus the dispatcher that routes bf16 operands to tcgen05.
#include "gemm.cuh"
#include "nn_kernels.cuh"

namespace ddppo {

// 4 neighbouring operands, element i present where i < n (vec: 4-element aligned rows)
__device__ __forceinline__ float4 ld4(const float* p, int n, bool vec) {
  if (vec && n >= 4) return __ldg((const float4*)p);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (n > 0) v.x = __ldg(p);
  if (n > 1) v.y = __ldg(p + 1);
  if (n > 2) v.z = __ldg(p + 2);
  if (n > 3) v.w = __ldg(p + 3);
  return v;
}
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p, int n, bool vec) {
  if (vec && n >= 4) {
    const uint2 u = __ldg((const uint2*)p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
  }
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (n > 0) v.x = __bfloat162float(p[0]);
  if (n > 1) v.y = __bfloat162float(p[1]);
  if (n > 2) v.z = __bfloat162float(p[2]);
  if (n > 3) v.w = __bfloat162float(p[3]);
  return v;
}

constexpr int SB_K = 16;
constexpr int kSplitSteps = 2;  // steps of SB_K a K split has at least

// One operand's BR x SB_K tile: registers while the previous tile is multiplied, then shared
// memory [k][row]. K-contiguous rows are transposed on the way; rows stored [K][R] are not.
template <int BR, typename T>
struct SimtTile {
  static constexpr int kUnits = BR * SB_K / 4;        // groups of 4 elements
  static constexpr int kPer = (kUnits + 255) / 256;   // per thread
  float4 v[kPer];
  __device__ __forceinline__ void load(const T* p, int ld, int r0, int R, int k0, int kend, bool t, bool vec) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int u = threadIdx.x + 256 * i;
      v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (kUnits % 256 && u >= kUnits) continue;
      if (t) {
        const int k = k0 + u / (BR / 4), r = r0 + u % (BR / 4) * 4;
        if (k < kend) v[i] = ld4(p + (size_t)k * ld + r, R - r, vec);
      } else {
        const int r = r0 + (u >> 2), k = k0 + (u & 3) * 4;
        if (r < R) v[i] = ld4(p + (size_t)r * ld + k, kend - k, vec);
      }
    }
  }
  __device__ __forceinline__ void store(float (*sh)[BR + 4], bool t) const {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int u = threadIdx.x + 256 * i;
      if (kUnits % 256 && u >= kUnits) continue;
      if (t) {
        *(float4*)&sh[u / (BR / 4)][u % (BR / 4) * 4] = v[i];
      } else {
        const int r = u >> 2, k = (u & 3) * 4;
        sh[k][r] = v[i].x;
        sh[k + 1][r] = v[i].y;
        sh[k + 2][r] = v[i].z;
        sh[k + 3][r] = v[i].w;
      }
    }
  }
};

enum { SIMT_VEC_A = 1, SIMT_VEC_B = 2, SIMT_VEC_C = 4 };
struct SimtArgs {
  int M, N, K, lda, ldb, ldc, c_bf16, relu, kchunk, a_t, b_t, vec;
  const void* A;
  const void* B;
  float* C;
  float beta;
  const float* bias;
  float* partial;
};

// C tile BM x BN a CTA; a thread owns TM/4 groups of 4 rows (BM / (TM/4) apart) by 4
// neighbouring columns, so an operand read is one 16-byte shared load and TM x 4 FMAs use
// TM/4 + 1 of them. Each output's sum runs over k in ascending order, one FMA a step.
// Bound: FP32 FMA issue; the next tile's global loads are in flight while this one is
// multiplied (two shared buffers, one barrier a tile). A 64x64 tile with scalar loads and
// 8 shared loads per 16 FMAs took 29 us a launch over the 60 GEMMs of the small FP32 update
// (3.3 ms of update in all); this form 8.7.
template <int BM, int BN, int TM, typename T>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const SimtArgs q) {
  DDPPO_PDL_ENTRY();
  constexpr int TX = BN / 4, G = TM / 4, MS = BM / G;
  static_assert(TX * (BM / TM) == 256, "one micro-tile a thread");
  __shared__ __align__(16) float As[2][SB_K][BM + 4];
  __shared__ __align__(16) float Bs[2][SB_K][BN + 4];
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int M = q.M, N = q.N;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;  // M tiles on x: M can exceed 65535 tiles
  const int kbeg = blockIdx.z * q.kchunk, kend = min(q.K, kbeg + q.kchunk);
  const T* A = (const T*)q.A;
  const T* B = (const T*)q.B;
  const bool va = q.vec & SIMT_VEC_A, vb = q.vec & SIMT_VEC_B, at = q.a_t, bt = q.b_t;
  float acc[TM][4] = {};
  SimtTile<BM, T> ta;
  SimtTile<BN, T> tb;
  ta.load(A, q.lda, m0, M, kbeg, kend, at, va);
  tb.load(B, q.ldb, n0, N, kbeg, kend, bt, vb);
  int buf = 0;
  for (int k0 = kbeg; k0 < kend; k0 += SB_K, buf ^= 1) {
    ta.store(As[buf], at);
    tb.store(Bs[buf], bt);
    __syncthreads();  // also: every thread is done with the other buffer's previous tile
    if (k0 + SB_K < kend) {
      ta.load(A, q.lda, m0, M, k0 + SB_K, kend, at, va);
      tb.load(B, q.ldb, n0, N, k0 + SB_K, kend, bt, vb);
    }
#pragma unroll
    for (int kk = 0; kk < SB_K; ++kk) {
      const float4 b = *(const float4*)&Bs[buf][kk][tx * 4];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float4 a = *(const float4*)&As[buf][kk][g * MS + ty * 4];
        const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float* c = acc[g * 4 + i];
          c[0] = fmaf(av[i], b.x, c[0]);
          c[1] = fmaf(av[i], b.y, c[1]);
          c[2] = fmaf(av[i], b.z, c[2]);
          c[3] = fmaf(av[i], b.w, c[3]);
        }
      }
    }
  }
  const int n = n0 + tx * 4;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + i / 4 * MS + ty * 4 + i % 4;
    if (m >= M) continue;
    if (q.partial) {
      float* p = q.partial + ((size_t)blockIdx.z * M + m) * N + n;
      if ((q.vec & SIMT_VEC_C) && n + 3 < N) {
        *(float4*)p = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (n + j < N) p[j] = acc[i][j];
      }
      continue;
    }
    const size_t o = (size_t)m * q.ldc + n;
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = acc[i][j];
      if (n + j >= N) continue;
      if (q.beta != 0.f) v[j] += q.beta * q.C[o + j];
      if (q.bias) v[j] += q.bias[n + j];
      if (q.relu) v[j] = fmaxf(v[j], 0.f);
    }
    if ((q.vec & SIMT_VEC_C) && n + 3 < N) {
      *(float4*)(q.C + o) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (n + j >= N) continue;
        if (q.c_bf16) ((__nv_bfloat16*)q.C)[o + j] = __float2bfloat16_rn(v[j]);
        else q.C[o + j] = v[j];
      }
    }
  }
}

// C = beta*C + sum_z partial[z] (+ bias) (ReLU), summed in split order. V neighbouring
// columns a thread: 1 for few outputs (latency: as many threads as there are outputs), 4 for
// many (a quarter of the blocks). Several loads
// in flight, added in order: at 64 frames the encoder's 12 reductions took 49 us a step with
// one output a thread, 34 now; the FP32 update's 48 small ones 154 us in blocks of 256 and
// dependent loads, 139 now.
template <int V>
__device__ __forceinline__ void add_partial(float (&v)[V], const float (&u)[V]) {
#pragma unroll
  for (int j = 0; j < V; ++j) v[j] += u[j];
}
template <int V>
__device__ __forceinline__ void load_partial(float (&u)[V], const float* p) {
  if constexpr (V == 4) {
    const float4 t = *(const float4*)p;
    u[0] = t.x; u[1] = t.y; u[2] = t.z; u[3] = t.w;
  } else {
    u[0] = *p;
  }
}
template <int V>
__global__ void __launch_bounds__(256) splitk_reduce_kernel(int M, int N, int splits,
                                                            const float* __restrict__ partial,
                                                            float* __restrict__ C, int ldc, int c_bf16,
                                                            float beta, const float* __restrict__ bias,
                                                            int relu) {
  DDPPO_PDL_ENTRY();
  const size_t idx = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * V, mn = (size_t)M * N;
  if (idx >= mn) return;
  const int m = (int)(idx / N), n = (int)(idx % N);
  const float* p = partial + idx;
  float v[V] = {};
  int z = 0;
  constexpr int F = V == 4 ? 4 : 8;
  for (; z + F <= splits; z += F, p += F * mn) {
    float u[F][V];
#pragma unroll
    for (int i = 0; i < F; ++i) load_partial<V>(u[i], p + i * mn);
#pragma unroll
    for (int i = 0; i < F; ++i) add_partial<V>(v, u[i]);
  }
#pragma unroll 3
  for (; z < splits; ++z, p += mn) {
    float u[V];
    load_partial<V>(u, p);
    add_partial<V>(v, u);
  }
  const size_t o = (size_t)m * ldc + n;
#pragma unroll
  for (int j = 0; j < V; ++j) {
    if (beta != 0.f) v[j] += beta * C[o + j];
    if (bias) v[j] += bias[n + j];
    if (relu) v[j] = fmaxf(v[j], 0.f);
    if (c_bf16) ((__nv_bfloat16*)C)[o + j] = __float2bfloat16_rn(v[j]);
    else if (V == 1) C[o] = v[0];
  }
  if constexpr (V == 4)
    if (!c_bf16) *(float4*)(C + o) = make_float4(v[0], v[1], v[2], v[3]);
}

// 4-element groups of a row are aligned for the vector load or store of `bytes` an element
static bool rows_of_4(const void* p, int ld, int bytes) {
  return ld % 4 == 0 && ((uintptr_t)p & (uintptr_t)(4 * bytes - 1)) == 0;
}

template <int BM, int BN, int TM>
static int launch_simt(SimtArgs& q, bool op_bf16, const GemmWorkspace& ws, int& splits, cudaStream_t s) {
  const int gm = (q.M + BM - 1) / BM, gn = (q.N + BN - 1) / BN;
  const int tiles = gm * gn, target = 2 * ws.num_sms;
  splits = 1;
  // too few tiles for the chip: split K, at least two steps of SB_K a split (8 steps: 11.7
  // us instead of 6.9 for the update's 64x64-tiled launches)
  if (tiles < target && q.K >= 4 * SB_K * kSplitSteps) {
    splits = min((target + tiles - 1) / tiles, q.K / (SB_K * kSplitSteps));
    const size_t per = (size_t)q.M * q.N;
    if (per > 0) splits = (int)min((size_t)splits, ws.partial_elems / per);
    if (splits < 2) splits = 1;
  }
  q.kchunk = (q.K + splits - 1) / splits;
  q.kchunk = (q.kchunk + SB_K - 1) / SB_K * SB_K;
  splits = (q.K + q.kchunk - 1) / q.kchunk;
  q.partial = nullptr;
  if (splits > 1) DDPPO_TRY(ws.sums(s, &q.partial));
  if (q.partial ? rows_of_4(q.partial, q.N, 4) : (!q.c_bf16 && rows_of_4(q.C, q.ldc, 4))) q.vec |= SIMT_VEC_C;
  if (op_bf16)
    ::ddppo::launch_k(gemm_simt_kernel<BM, BN, TM, __nv_bfloat16>, dim3(gm, gn, splits), 256, 0, s, q);
  else
    ::ddppo::launch_k(gemm_simt_kernel<BM, BN, TM, float>, dim3(gm, gn, splits), 256, 0, s, q);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

static int gemm_simt(const GemmDesc& d, bool op_bf16, const GemmWorkspace& ws, cudaStream_t s) {
  const int eb = op_bf16 ? 2 : 4;
  SimtArgs q{};
  q.M = d.M; q.N = d.N; q.K = d.K; q.lda = d.lda; q.ldb = d.ldb; q.ldc = d.ldc;
  q.c_bf16 = d.c_bf16; q.relu = d.relu; q.a_t = d.a_t; q.b_t = d.b_t;
  q.A = d.A; q.B = d.B; q.C = (float*)d.C; q.beta = d.beta; q.bias = d.bias;
  if (rows_of_4(d.A, d.lda, eb)) q.vec |= SIMT_VEC_A;
  if (rows_of_4(d.B, d.ldb, eb)) q.vec |= SIMT_VEC_B;
  int splits;
  // one tile shape leaves half its FMAs on padding for 32 channels: 128x32 and 32x128 there
  // (9.5 us a launch; 64x64: 14.3). 128x64 saves shared reads where it still gives two CTAs
  // an SM (19.7 us; 64x64: 20.2)
  if (d.N <= 32) DDPPO_TRY((launch_simt<128, 32, 4>(q, op_bf16, ws, splits, s)));
  else if (d.M <= 32) DDPPO_TRY((launch_simt<32, 128, 4>(q, op_bf16, ws, splits, s)));
  else if (((d.M + 127) / 128) * (int64_t)((d.N + 63) / 64) >= 2 * ws.num_sms) DDPPO_TRY((launch_simt<128, 64, 8>(q, op_bf16, ws, splits, s)));
  else DDPPO_TRY((launch_simt<64, 64, 4>(q, op_bf16, ws, splits, s)));
  if (q.partial)
    DDPPO_TRY(launch_splitk_reduce(d.M, d.N, splits, q.partial, q.C, d.ldc, d.c_bf16, d.beta, d.bias, d.relu, s));
  return DDPPO_OK;
}

int launch_splitk_reduce(int M, int N, int splits, const float* partial, float* C, int ldc,
                         int c_bf16, float beta, const float* bias, int relu, cudaStream_t s) {
  const size_t n = (size_t)M * N;
  // four columns a thread where that still leaves the chip (152 SMs) a block each
  if (n >= 152 * 1024 && N % 4 == 0 && rows_of_4(partial, N, 4) && (c_bf16 || rows_of_4(C, ldc, 4)))
    ::ddppo::launch_k(splitk_reduce_kernel<4>, (unsigned)((n / 4 + 255) / 256), 256, 0, s, M, N, splits, partial, C,
                      ldc, c_bf16, beta, bias, relu);
  else
    ::ddppo::launch_k(splitk_reduce_kernel<1>, (unsigned)((n + 127) / 128), 128, 0, s, M, N, splits, partial, C,
                      ldc, c_bf16, beta, bias, relu);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

// E4M3 operands on the tensor cores. The kernel's layouts are byte layouts (a 128-byte
// operand row is 64 bf16 or 128 E4M3 values, and one MMA consumes 32 bytes of K either
// way), so the contraction runs on the 16-bit view of its operands: K, the leading
// dimensions and a convolution's channels count E4M3 pairs, and only the MMA kind and the
// epilogue's scale differ from the bf16 form.
static int gemm_fp8(const GemmDesc& d, const GemmWorkspace& ws, cudaStream_t s) {
  if (d.convw || d.a_t || d.b_t || (d.K % 2) || (d.lda % 2) || (d.ldb % 2) ||
      (d.conv && (d.conv->C % 2))) {
    set_error("gemm: E4M3 operands must be K-major with even K, leading dimensions and channels");
    return DDPPO_E_CONFIG;
  }
  GemmDesc p = d;
  p.K = d.K / 2;
  p.lda = d.lda / 2;
  p.ldb = d.ldb / 2;
  ConvShape cp;
  if (d.conv) {
    cp = *d.conv;
    cp.C = d.conv->C / 2;
    p.conv = &cp;
    if (!gemm_conv_supported(cp, p.A)) {
      set_error("gemm: E4M3 convolution needs 64 | C (or C = 64 on the halo path)");
      return DDPPO_E_CONFIG;
    }
  } else if (!gemm_tc_supported(p)) {
    set_error("gemm: E4M3 operands need 16-byte aligned rows and K >= 32");
    return DDPPO_E_CONFIG;
  }
  return gemm_tc(p, ws, s);
}

// the single-channel convolution kernel covers this contraction: an implicit convolution
// of a 1-channel input into fp32 rows of Cout (no bias, ReLU or bf16 output)
static bool conv_c1_ok(const GemmDesc& d) {
  return d.conv && d.conv->C == 1 && conv_c1_tc_supported(d.conv->k, d.conv->Cout) &&
         d.N == d.conv->Cout && d.ldc == d.N && !d.c_bf16 && !d.bias && !d.relu && !d.fp8 &&
         d.ldb >= d.conv->k * d.conv->k;
}

// the stem's weight gradient: N is the padded tap count of the GEMM-layout gradient
static bool wgrad_stem_ok(const GemmDesc& d, bool op_bf16, const GemmWorkspace& ws) {
  return d.convw && op_bf16 && !d.conv && d.a_t && d.lda == d.M && !d.c_bf16 && !d.bias && !d.relu && !d.fp8 &&
         d.M == d.convw->Cout && d.N >= 49 && d.N <= 64 && d.ldc == d.N &&
         d.K == d.convw->N * d.convw->Ho * d.convw->Wo && conv_wgrad_stem_ok(*d.convw, d.B, d.A, ws);
}

int gemm(const GemmDesc& d, bool op_bf16, const GemmWorkspace& ws, cudaStream_t s,
         KernelTimer* timer) {
  if (d.M <= 0 || d.N <= 0) return DDPPO_OK;
  if (d.K <= 0) {
    set_error("gemm: K must be positive");
    return DDPPO_E_CONFIG;
  }
  if (d.fp8 && (!op_bf16 || d.c_bf16)) {
    set_error("gemm: E4M3 operands need the tensor-core path and an fp32 output");
    return DDPPO_E_CONFIG;
  }
  if (d.c_bf16 && d.beta != 0.f) {
    set_error("gemm: bf16 output cannot accumulate");
    return DDPPO_E_CONFIG;
  }
  if (d.conv && !d.fp8 && !(op_bf16 && (gemm_conv_supported(*d.conv, d.A) || conv_c1_ok(d)))) {
    set_error("gemm: implicit convolution not supported for this shape");
    return DDPPO_E_CONFIG;
  }
  const bool stem_w = wgrad_stem_ok(d, op_bf16, ws);
  if (d.convw && !stem_w && !(op_bf16 && !d.conv && d.a_t && d.lda == d.M && d.lda % 8 == 0 && !d.c_bf16 && !d.bias && !d.relu &&
                   d.N == d.convw->k * d.convw->k * d.convw->C &&
                   d.K == d.convw->N * d.convw->Ho * d.convw->Wo &&
                   (conv_wgrad_halo_ok(*d.convw, d.B, d.A) ||
                    gemm_convw_supported(*d.convw, d.B, d.A)))) {
    set_error("gemm: implicit weight gradient not supported for this shape");
    return DDPPO_E_CONFIG;
  }
  const bool rec = timer && timer->on && timer->n + 2 <= 2 * 4096;
  if (timer && timer->on) timer->flops_all += 2.0 * d.M * d.N * d.K;
  // inside a stream capture the records are external: they become event nodes of the graph
  unsigned rec_flags = cudaEventRecordDefault;
  if (rec) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusActive)
      rec_flags = cudaEventRecordExternal;
    cudaEventRecordWithFlags(timer->ev[timer->n], s, rec_flags);
  }
  int rc;
  if (d.fp8) {
    rc = gemm_fp8(d, ws, s);
    if (ws.tc && ws.tc->on) {
      ws.tc->launches += 1;
      ws.tc->flops += 2.0 * d.M * d.N * d.K;
    }
  } else if (stem_w) {
    rc = conv_wgrad_stem(*d.convw, d.B, d.A, (float*)d.C, d.ldc, d.beta, ws, s);
    if (ws.tc && ws.tc->on) {
      ws.tc->launches += 1;
      ws.tc->flops += 2.0 * d.M * d.N * d.K;
    }
  } else if (op_bf16 && conv_c1_ok(d) && conv_stem_ok(*d.conv, d.A) && !((uintptr_t)d.C & 15)) {
    rc = conv_stem(*d.conv, d.A, d.B, d.ldb, (float*)d.C, d.beta, ws, s);
    if (ws.tc && ws.tc->on) {
      ws.tc->launches += 1;
      ws.tc->flops += 2.0 * d.M * d.N * d.K;
    }
  } else if (op_bf16 && conv_c1_ok(d)) {
    // a single-channel convolution (the stem): patches gathered in shared memory
    const ConvShape& c = *d.conv;
    ConvC1 a{};
    a.N = c.N; a.H = c.H; a.W = c.W; a.k = c.k; a.s = c.s; a.p = c.p; a.Ho = c.Ho; a.Wo = c.Wo;
    a.Cout = c.Cout; a.ldw = d.ldb;
    a.x = (const __nv_bfloat16*)d.A; a.w = (const __nv_bfloat16*)d.B; a.y = (float*)d.C;
    a.beta = d.beta; a.err = ws.err;
    rc = launch_conv_c1_tc(a, ws.num_sms, s);
    if (ws.tc && ws.tc->on) {
      ws.tc->launches += 1;
      ws.tc->flops += 2.0 * d.M * d.N * d.K;
    }
  } else if (op_bf16 && gemm_small_supported(d)) {
    rc = gemm_small(d, s);  // latency-bound small-M shapes: no tensor-memory pipeline
  } else if (op_bf16 && d.convw && conv_wgrad_halo_ok(*d.convw, d.B, d.A)) {
    rc = conv_wgrad_halo(*d.convw, d.B, d.A, (float*)d.C, d.ldc, d.beta, ws, s);
  } else if (op_bf16 && d.convw && conv_wgrad_rows_ok(*d.convw, d.B, d.A, ws)) {
    rc = conv_wgrad_rows(*d.convw, d.B, d.A, (float*)d.C, d.ldc, d.beta, ws, s);
    if (ws.tc && ws.tc->on) {
      ws.tc->launches += 1;
      ws.tc->flops += 2.0 * d.M * d.N * d.K;
    }
  } else if (op_bf16 && (d.conv || d.convw || gemm_tc_supported(d))) {
    rc = gemm_tc(d, ws, s);
    if (ws.tc && ws.tc->on) {
      ws.tc->launches += 1;
      ws.tc->flops += 2.0 * d.M * d.N * d.K;
    }
  } else {
    rc = gemm_simt(d, op_bf16, ws, s);
  }
  if (rec) {
    cudaEventRecordWithFlags(timer->ev[timer->n + 1], s, rec_flags);
    const double es = d.fp8 ? 1.0 : op_bf16 ? 2.0 : 4.0, cs = d.c_bf16 ? 2.0 : 4.0;
    timer->work[timer->n / 2] = 2.0 * d.M * d.N * d.K;
    // operands read once, result written once (and read when accumulating); an implicit
    // convolution reads its input tensor, not the M x K patch matrix
    const ConvShape* cv = d.conv ? d.conv : d.convw;
    const double in_elems = cv ? (double)cv->N * cv->H * cv->W * cv->C : 0.0;
    const double a_elems = d.conv ? in_elems : (double)d.M * d.K;
    const double b_elems = d.convw ? in_elems : (double)d.N * d.K;
    timer->bytes[timer->n / 2] = (a_elems + b_elems) * es +
                                 (double)d.M * d.N * cs * (d.beta != 0.f ? 2.0 : 1.0);
    timer->n += 2;
    timer->flops += 2.0 * d.M * d.N * d.K;
    timer->launches += 1;
  }
  return rc;
}

}  // namespace ddppo
