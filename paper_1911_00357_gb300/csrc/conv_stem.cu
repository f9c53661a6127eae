// The stem (7x7 / stride 2 / pad 3 on one input channel) and its weight gradient on tcgen05,
// patches built in shared memory from the staged input rows.
//
// A tile is 128 output pixels, whole rows of one image. The input rows it reads are staged
// once (16-byte loads; a 4-pixel zero border each side), so that the seven taps of a filter
// row are halves 1..7 of four consecutive words at the pixel's own word. A thread builds the
// 49 taps of its pixel in (ky, kx) order -- 28 shared words, consecutive over the warp, 25
// byte permutations -- as one 128-byte row in the 128-byte swizzle, zero from tap 49 to 63.
//
//   forward:  y[pixel, co] = patches (K-major, 128 x 64) . w (resident, Cout x 64): the MMAs of
//             the im2col matrix' GEMM, in their order, hence the same bits.
//   gradient: dw[tap, co] = sum over pixels: the same rows read as an MN-major operand
//             (M = taps; the upper 64 accumulator rows take the block one row on and are
//             discarded) and dz (MN-major) as the other; a CTA keeps its sums in tensor
//             memory over all its tiles and a second kernel adds the CTAs in order.
//
// Six CTAs (forward) or six building groups (gradient) an SM hide one another's build, MMA and
// epilogue. Every wait is bounded.
// Bound: building the patches -- the shared-memory data pipe is 77% (forward) and 78% (gradient)
// busy with their words and rows, HBM 51% and 36% (912 images of 128x128 into 32 channels). With
// the patch matrix (1.9 GB for 4096 images) written by one kernel (827 us) and read by the GEMM
// the encoder's pass took 19.5 ms; with this 16.7: 458 us forward, 412 the gradient.
#include <algorithm>

#include "gemm.cuh"
#include "nn_kernels.cuh"
#include "tma.cuh"

namespace ddppo {

namespace {

constexpr int ST_THREADS = 128;

struct StemArgs {
  int N, H, W, Ho, Wo, lwo, lw8, R, tpi, ldw;  // lwo, lw8: log2 of Wo and of W / 8; R: output rows a tile
  const __nv_bfloat16* x;
  const __nv_bfloat16* w;
  float* y;
  float beta;
  const __nv_bfloat16* dz;
  float* part;
  int kchunk;  // gradient: pixels a split
  int32_t* err;
};

__device__ __forceinline__ uint32_t st_sw128(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

// input rows of a tile into shared memory: row r = image row 2 oy0 - 3 + r, word 2 + i its
// pixels 2 i and 2 i + 1 (zero outside the image)
__device__ __forceinline__ void stage_rows(const StemArgs& a, int tile, uint32_t* sx, int tid) {
  const int img = tile / a.tpi, iy0 = 2 * (tile - img * a.tpi) * a.R - 3;
  const int rows = 2 * a.R + 5, pw = a.W / 2 + 4;
  const __nv_bfloat16* xi = a.x + (size_t)img * a.H * a.W;
  for (int i = tid; i < rows << a.lw8; i += ST_THREADS) {
    const int r = i >> a.lw8, c = i & ((1 << a.lw8) - 1), iy = iy0 + r;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (iy >= 0 && iy < a.H) v = __ldg(reinterpret_cast<const uint4*>(xi + (size_t)iy * a.W + 8 * c));
    uint32_t* d = sx + r * pw + 2 + 4 * c;
    *reinterpret_cast<uint2*>(d) = make_uint2(v.x, v.y);
    *reinterpret_cast<uint2*>(d + 2) = make_uint2(v.z, v.w);
  }
}
__device__ __forceinline__ void zero_borders(const StemArgs& a, uint32_t* sx, int tid) {
  const int rows = 2 * a.R + 5, pw = a.W / 2 + 4;
  for (int i = tid; i < rows * 4; i += ST_THREADS) {
    const int r = i >> 2, b = i & 3;
    sx[r * pw + (b < 2 ? b : a.W / 2 + b)] = 0u;
  }
}
// pixel m of the tile: 64 taps into its row of the patch tile
__device__ __forceinline__ void build_patch(const StemArgs& a, const uint32_t* sx, uint8_t* sa, int m) {
  const int pw = a.W / 2 + 4;
  const uint32_t* p = sx + 2 * (m >> a.lwo) * pw + (m & (a.Wo - 1));
  uint32_t w[7][4];
#pragma unroll
  for (int ky = 0; ky < 7; ++ky)
#pragma unroll
    for (int i = 0; i < 4; ++i) w[ky][i] = p[ky * pw + i];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int t = c * 8 + 2 * i;  // taps t and t + 1: halves 1 + kx of their rows
      if (t >= 49) {
        o[i] = 0u;
      } else {
        const int ha = 1 + t % 7, tb = t + 1 < 49 ? t + 1 : t, hb = 1 + tb % 7;
        const uint32_t both = __byte_perm(w[t / 7][ha >> 1], w[tb / 7][hb >> 1],
                                          ((ha & 1) ? 0x32 : 0x10) | (((hb & 1) ? 0x76 : 0x54) << 8));
        o[i] = t + 1 < 49 ? both : both & 0xffffu;
      }
    }
    *reinterpret_cast<uint4*>(sa + st_sw128(m, c)) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

struct StemCtl {
  uint64_t bar;
  uint32_t tmem_base;
  int abort_flag;
};
// `it` batches of MMAs were committed; after an abort the last one has completed (bounded)
// before the accumulator is freed
__device__ __forceinline__ void stem_end(StemCtl& ctl, int warp, uint32_t tmem, uint32_t cols, uint32_t it) {
  __syncthreads();
  if (ctl.abort_flag && threadIdx.x == 0 && it) mbar_drain_wait(&ctl.bar, (it - 1) & 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
  }
}

}  // namespace

template <int COUT>
__global__ void __launch_bounds__(ST_THREADS, 6) conv_stem_kernel(const StemArgs a) {
  extern __shared__ __align__(1024) uint8_t dyn[];
  __shared__ StemCtl ctl;
  uint8_t* base = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
  uint8_t* sA = base;                                  // 128 patch rows; then the epilogue's staging
  uint8_t* sB = base + 128 * 128;                      // COUT weight rows
  uint32_t* sX = (uint32_t*)(sB + COUT * 128);         // input rows
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  volatile int* abort = &ctl.abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&ctl.bar, 1);
    ctl.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&ctl.tmem_base)),
                 "r"(COUT));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  DDPPO_PDL_ENTRY();  // after the barrier set-up and the tensor-memory allocation
  const uint32_t tmem = ctl.tmem_base;
  const int ntiles = a.N * a.tpi;
  // resident weights: row co = its 49 taps, zero up to 64
  for (int i = threadIdx.x; i < COUT * 32; i += ST_THREADS) {
    const int co = i >> 5, t = 2 * (i & 31);
    uint32_t v = 0u;
    if (t < 49) v = __bfloat16_as_ushort(a.w[(size_t)co * a.ldw + t]);
    if (t + 1 < 49) v |= (uint32_t)__bfloat16_as_ushort(a.w[(size_t)co * a.ldw + t + 1]) << 16;
    *reinterpret_cast<uint32_t*>(sB + st_sw128(co, t >> 3) + (t & 7) * 2) = v;
  }
  zero_borders(a, sX, threadIdx.x);
  const uint32_t idesc = f16_idesc(128, COUT, 0, 0);
  bool ok = true;
  uint32_t it = 0;
  if ((int)blockIdx.x < ntiles) stage_rows(a, blockIdx.x, sX, threadIdx.x);
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    if (!__syncthreads_and(ok ? 1 : 0)) break;  // the input rows are staged
    build_patch(a, sX, sA, threadIdx.x);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();  // ... and read; the previous accumulator has been read
    if (warp == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          tc_mma(tmem, sw128_desc(smem_addr(sA) + k * 32), sw128_desc(smem_addr(sB) + k * 32), idesc, k > 0, 0);
        tc_commit(&ctl.bar);
      }
      __syncwarp();
    }
    if (tile + (int)gridDim.x < ntiles) stage_rows(a, tile + gridDim.x, sX, threadIdx.x);
    ok = warp_wait(&ctl.bar, it & 1u, abort, a.err);
    ++it;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) continue;
    // warp w: accumulator rows 32 w .. 32 w + 31, through its part of the patch tile (which the
    // MMAs have read), out as 16-byte stores of whole 128-byte rows
    uint8_t* st = sA + warp * 4096;
    float* y0 = a.y + ((size_t)tile * 128 + warp * 32) * COUT;
#pragma unroll
    for (int c0 = 0; c0 < COUT; c0 += 32) {
      uint32_t r[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
#pragma unroll
      for (int c = 0; c < 8; ++c)
        *reinterpret_cast<uint4*>(st + st_sw128(lane, c)) = make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int row = i * 4 + (lane >> 3), c = lane & 7;
        float4 v = *reinterpret_cast<const float4*>(st + st_sw128(row, c));
        float4* d = reinterpret_cast<float4*>(y0 + (size_t)row * COUT + c0 + c * 4);
        if (a.beta != 0.f) {
          const float4 o = *d;
          v.x = __fmaf_rn(a.beta, o.x, v.x); v.y = __fmaf_rn(a.beta, o.y, v.y);
          v.z = __fmaf_rn(a.beta, o.z, v.z); v.w = __fmaf_rn(a.beta, o.w, v.w);
        }
        *d = v;
      }
      __syncwarp();
    }
  }
  stem_end(ctl, warp, tmem, COUT, it);
}

// Weight gradient: CTA z sums the pixels of split z, in ascending order -- the splits, and the
// order within one, of the GEMM over the patch matrix, hence its bits (the truncating
// accumulation of a chain of a few thousand MMAs depends on its length). Three groups of 128
// threads build tiles in turn, a 13th warp issues their MMAs.
constexpr int SW_GROUPS = 3, SW_THREADS = SW_GROUPS * 128 + 32;

template <int COUT>
__global__ void __launch_bounds__(SW_THREADS, 2) wgrad_stem_kernel(const StemArgs a) {
  extern __shared__ __align__(1024) uint8_t dyn[];
  __shared__ StemCtl ctl;
  __shared__ uint64_t full[SW_GROUPS], empty[SW_GROUPS];
  constexpr int DB = COUT * 2, NCH = DB / 16;          // bytes and 16-byte chunks of a dz row
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  volatile int* abort = &ctl.abort_flag;
  // a group: 128 patch rows, 128 dz rows (what the row after the patches reads, too), input rows
  constexpr uint32_t GB = 128 * 128 + 128 * DB;
  uint8_t* base = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
  const int xwords = (2 * a.R + 5) * (a.W / 2 + 4);
  if (threadIdx.x == 0) {
    mbar_init(&ctl.bar, 1);
    for (int g = 0; g < SW_GROUPS; ++g) {
      mbar_init(&full[g], 128);
      mbar_init(&empty[g], 1);
    }
    ctl.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&ctl.tmem_base)),
                 "r"(COUT));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  DDPPO_PDL_ENTRY();  // after the barrier set-up and the tensor-memory allocation
  const uint32_t tmem = ctl.tmem_base;
  const int K = a.N * a.Ho * a.Wo;
  const int p0 = blockIdx.x * a.kchunk, p1 = min(K, p0 + a.kchunk);  // multiples of 64
  const int t0 = p0 >> 7, t1 = (p1 + 127) >> 7;

  if (warp < 4 * SW_GROUPS) {
    const int g = warp >> 2, m = threadIdx.x & 127;
    uint8_t* sA = base + g * GB;
    uint8_t* sD = sA + 128 * 128;
    uint32_t* sX = (uint32_t*)(base + SW_GROUPS * GB) + g * xwords;
    zero_borders(a, sX, m);
    uint4 d[NCH];
    const auto fetch = [&](int tile) {
      stage_rows(a, tile, sX, m);
      const uint4* p = reinterpret_cast<const uint4*>(a.dz + ((size_t)tile * 128 + m) * COUT);
#pragma unroll
      for (int c = 0; c < NCH; ++c) d[c] = __ldg(p + c);
    };
    if (t0 + g < t1) fetch(t0 + g);
    uint32_t j = 0;
    for (int t = t0 + g; t < t1; t += SW_GROUPS, ++j) {
      // the MMAs have read the group's last tile; its next input rows are staged
      const bool ok = warp_wait(&empty[g], (j & 1u) ^ 1u, abort, a.err);
      uint32_t all;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
          "barrier.cta.red.and.pred q, %2, 128, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
          : "=r"(all)
          : "r"((uint32_t)ok), "r"(1 + g)
          : "memory");
      if (!all) break;
      build_patch(a, sX, sA, m);
#pragma unroll
      for (int c = 0; c < NCH; ++c) {  // the swizzle of 64- or 128-byte rows
        const int sc = COUT == 32 ? c ^ ((m >> 1) & 3) : c ^ (m & 7);
        *reinterpret_cast<uint4*>(sD + m * DB + sc * 16) = d[c];
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&full[g])) : "memory");
      asm volatile("barrier.cta.sync %0, 128;" ::"r"(1 + g) : "memory");  // the input rows are read
      if (t + SW_GROUPS < t1) fetch(t + SW_GROUPS);
    }
  } else {
    const uint32_t idesc = f16_idesc(128, COUT, 1, 1);
    uint32_t ph = 0, acc = 0;
    int g = 0;
    for (int t = t0; t < t1; ++t) {
      if (!warp_wait(&full[g], ph, abort, a.err)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // the tile's part of the split, 16 pixels an MMA
      const int k0 = max(p0 - t * 128, 0) >> 4, k1 = min(p1 - t * 128, 128) >> 4;
      const uint32_t a0 = smem_addr(base + g * GB);
      if (elect_one()) {
        for (int k = k0; k < k1; ++k) {
          const uint32_t d0 = a0 + 128 * 128 + k * 16 * DB;
          uint64_t db = sw128_mn_desc(d0);
          if (COUT == 32)  // 64-byte rows and swizzle, 8-row groups 512 bytes apart
            db = (uint64_t)((d0 >> 4) & 0x3FFF) | (uint64_t)(4096 >> 4) << 16 | (uint64_t)(512 >> 4) << 32 |
                 (uint64_t)1 << 46 | (uint64_t)4 << 61;
          tc_mma(tmem, sw128_mn_desc(a0 + k * 16 * 128, 128u), db, idesc, acc | (uint32_t)(k != k0), 0);
        }
        tc_commit(&empty[g]);
      }
      __syncwarp();
      acc = 1u;
      if (++g == SW_GROUPS) { g = 0; ph ^= 1u; }
    }
    if (elect_one()) tc_commit(&ctl.bar);
    __syncwarp();
    // after an abort the others no longer wait: every MMA of this warp has completed
    if (*abort) mbar_drain_wait(&ctl.bar, 0u);
  }
  __syncwarp();
  if (warp < 2) {  // taps 0 .. 63
    const bool ok = warp_wait(&ctl.bar, 0u, abort, a.err);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    float* dst = a.part + ((size_t)blockIdx.x * 64 + warp * 32 + lane) * COUT;
#pragma unroll
    for (int c0 = 0; c0 < COUT; c0 += 32) {
      uint32_t r[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
#pragma unroll
      for (int j = 0; j < 32; j += 4)
        *reinterpret_cast<uint4*>(dst + c0 + j) = ok ? make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3])
                                                     : make_uint4(0u, 0u, 0u, 0u);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COUT));
  }
}

// dw[co, tap] (+)= the splits' sums, in order; a block takes one tap
__global__ void __launch_bounds__(64) wgrad_stem_reduce_kernel(const float* __restrict__ part, int splits,
                                                               float* __restrict__ dw, int ldw, float beta) {
  DDPPO_PDL_ENTRY();
  const int tap = blockIdx.x, co = threadIdx.x, Cout = blockDim.x;
  const float* p = part + (size_t)tap * Cout + co;
  const size_t step = (size_t)64 * Cout;
  float s = 0.f;
  int i = 0;
  for (; i + 16 <= splits; i += 16, p += 16 * step) {
    float u[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) u[k] = p[k * step];
#pragma unroll
    for (int k = 0; k < 16; ++k) s += u[k];
  }
  for (; i < splits; ++i, p += step) s += *p;
  float* d = dw + (size_t)co * ldw + tap;
  *d = beta != 0.f ? __fmaf_rn(beta, *d, s) : s;
}

// whole rows of one image in a 128-pixel tile, rows of 16-byte groups. Other single-channel
// convolutions gather their patches per tap or through an im2col matrix.
static bool stem_plan(const ConvShape& c, StemArgs* a) {
  if (c.C != 1 || c.k != 7 || c.s != 2 || c.p != 3 || (c.Cout != 32 && c.Cout != 64) || c.N < 1) return false;
  if (c.Wo < 16 || c.Wo > 128 || (c.Wo & (c.Wo - 1)) || c.W != 2 * c.Wo || c.H != 2 * c.Ho) return false;
  const int R = 128 / c.Wo;
  if (c.Ho % R || (int64_t)c.N * c.Ho * c.Wo >= (1ll << 31)) return false;
  if (a) {
    int l = 4;
    while ((1 << l) < c.Wo) ++l;
    a->N = c.N; a->H = c.H; a->W = c.W; a->Ho = c.Ho; a->Wo = c.Wo;
    a->lwo = l; a->lw8 = l - 2; a->R = R; a->tpi = c.Ho / R;
  }
  return true;
}

static size_t stem_smem(const StemArgs& a, int row_bytes) {  // row_bytes: resident rows beside the patches
  return 1024 + 128 * 128 + (size_t)row_bytes + (size_t)(2 * a.R + 5) * (a.W / 2 + 4) * 4;
}

// CTAs an SM: shared memory (227 KiB, 1 KiB reserved a CTA), tensor memory (512 columns) and
// the registers of the launch bounds, at most 8
template <typename K>
static int stem_grid(K kern, size_t smem, int cout, int ntiles, int num_sms, int* grid) {
  cudaFuncAttributes fa{};
  DDPPO_CHECK_CUDA(cudaFuncGetAttributes(&fa, kern));
  const int regs = std::max(8, (fa.numRegs + 7) / 8 * 8) * ST_THREADS;
  const int occ = std::max(1, std::min({8, (int)(232448 / (smem + fa.sharedSizeBytes + 1024)), 512 / cout, 65536 / regs}));
  *grid = std::min(ntiles, num_sms * occ);
  return DDPPO_OK;
}

bool conv_stem_ok(const ConvShape& c, const void* x) {
  return !((uintptr_t)x & 15) && stem_plan(c, nullptr);
}

int conv_stem(const ConvShape& c, const void* x, const void* w, int ldw, float* y, float beta,
              const GemmWorkspace& ws, cudaStream_t s) {
  StemArgs a{};
  if (!stem_plan(c, &a)) {
    set_error("conv_stem: unsupported shape");
    return DDPPO_E_CONFIG;
  }
  a.x = (const __nv_bfloat16*)x; a.w = (const __nv_bfloat16*)w; a.ldw = ldw; a.y = y; a.beta = beta; a.err = ws.err;
  auto kern = c.Cout == 32 ? conv_stem_kernel<32> : conv_stem_kernel<64>;
  const size_t smem = stem_smem(a, c.Cout * 128);
  int grid = 0;
  DDPPO_TRY(stem_grid(kern, smem, c.Cout, a.N * a.tpi, ws.num_sms, &grid));
  ::ddppo::launch_k(kern, grid, ST_THREADS, smem, s, a);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

// the K splits of the GEMM over the patch matrix (two 64-wide CTAs an SM, one tile): pixels
// of one, a multiple of 64
static int stem_wgrad_chunk(const ConvShape& c, int kp, const GemmWorkspace& ws) {
  const int K = c.N * c.Ho * c.Wo;
  int splits = 1;
  if (K >= 8 * 64) {
    splits = std::min(2 * ws.num_sms, K / (4 * 64));
    splits = (int)std::min((size_t)splits, ws.partial_elems / ((size_t)c.Cout * kp));
    if (splits < 2) splits = 1;
  }
  return ((K + splits - 1) / splits + 63) / 64 * 64;
}
bool conv_wgrad_stem_ok(const ConvShape& c, const void* x, const void* dz, const GemmWorkspace& ws) {
  return !((uintptr_t)x & 15) && !((uintptr_t)dz & 15) && stem_plan(c, nullptr) &&
         ws.partial_elems >= (size_t)2 * ws.num_sms * 64 * c.Cout;
}

// dw[co, 0 .. ldw) (+)= the gradient, zero past tap 48 (ldw <= 64)
int conv_wgrad_stem(const ConvShape& c, const void* x, const void* dz, float* dw, int ldw, float beta,
                    const GemmWorkspace& ws, cudaStream_t s) {
  StemArgs a{};
  if (!stem_plan(c, &a) || ldw > 64) {
    set_error("wgrad_stem: unsupported shape");
    return DDPPO_E_CONFIG;
  }
  a.x = (const __nv_bfloat16*)x; a.dz = (const __nv_bfloat16*)dz; a.err = ws.err;
  DDPPO_TRY(ws.sums(s, &a.part));
  a.kchunk = stem_wgrad_chunk(c, ldw, ws);
  const int splits = (c.N * c.Ho * c.Wo + a.kchunk - 1) / a.kchunk;
  auto kern = c.Cout == 32 ? wgrad_stem_kernel<32> : wgrad_stem_kernel<64>;
  const size_t smem = 1024 + SW_GROUPS * (size_t)(128 * 128 + 128 * c.Cout * 2 + (2 * a.R + 5) * (a.W / 2 + 4) * 4);
  DDPPO_CHECK_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ::ddppo::launch_k(kern, splits, SW_THREADS, smem, s, a);
  DDPPO_CHECK_LAUNCH();
  ::ddppo::launch_k(wgrad_stem_reduce_kernel, ldw, c.Cout, 0, s, a.part, splits, dw, ldw, beta);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

}  // namespace ddppo
