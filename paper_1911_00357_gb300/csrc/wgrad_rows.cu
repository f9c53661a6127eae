// Weight gradient of the 3x3 / stride-1 / pad-1 convolutions with 64 or more channels
// (stages 2 to 4 of the encoder, the compression layer; bf16 operands, fp32 accumulation on
// tcgen05):
//   dW[co, (ky, kx, c)] = sum over output pixels a of dz[a, co] x[a + (ky - 1, kx - 1), c].
//
// The reduction runs over pixels, so both operands are MN-major (channels contiguous, one
// 128-byte row of 64 channels per pixel). A unit of work is RB rows of ni images, laid out
// as "anchors" (row, image, column) of pitch Wp = W + 2 whose two extra columns carry
// dz = 0 (the copy engine's zero fill); images sit inside a row so that a vertical tap is
// again a constant shift and small maps fill a unit. A filter tap is then a shift of x by
// whole anchors: every tap reads the same staged box through a shifted descriptor, where
// the gather form copies the box once per tap (9 times, which bound it by L2 traffic).
//
//   all taps (64 -> 64 channels): one box of x with its halo per unit; an MMA (M = 128, N =
//     64, K = 16 anchors) takes two column taps, its two 64-channel atoms one anchor apart
//     (the fourth column tap of a pair is discarded); 6 accumulators of 64 columns;
//   by row tap (C and Cout multiples of 128): a job is a filter row, 128 input and 128
//     output channels; the x box is fetched already shifted by the row, the three column
//     taps are three MMAs (M = N = 128) into 3 accumulators of 128 columns. N = 128 keeps
//     the MMA at its full rate (256 bytes of operands per 4 shared-memory cycles).
//
// Each CTA (one per SM: all of TMEM) accumulates every unit of its split of the job and
// writes its sums once; a second kernel adds the splits in order. Rows past the last shift
// of a box are zeros that no copy overwrites: they meet dz = 0, and stale values there could
// be NaN. Pad anchors meet real pixels too (the last column through the left tap, the next
// row's first through the right one, the last row through the upper one where a unit reaches
// past the image): with dz = 0 that adds nothing unless the pixel is an infinity or a NaN, of
// which 0 x makes a NaN. The second kernel therefore forms a sum that is not finite again, from
// the pixels of its own tap alone.
//
// Measured (4096 images): 16x16, 64 -> 64 channels 97 us against 367 us for the gather form
// (0.73 PFLOP/s; the tensor pipe is taken 77% of the time but computes 51%: MMAs of N = 64 wait
// for their operands' shared-memory reads; x and dz come from memory once, 269 MB); the seven
// convolutions of stages 3, 4 and the compression layer 72 us each on average, reduction
// included. The encoder's ten such gradients: 0.80 ms against 2.9 ms.
#include <algorithm>
#include <cstring>

#include "gemm.cuh"
#include "tma.cuh"

namespace ddppo {

namespace {

constexpr int WR_THREADS = 128, WR_STAGES = 6;
constexpr size_t WR_SMEM_MAX = 222 * 1024;
constexpr uint32_t WR_PAD = 1024;  // zero rows behind a box (8 anchors)

struct WrArgs {
  int by_row;               // 1: jobs by filter row, 0: all taps
  int Wp, ni, RB, nrb;      // anchor pitch, images and rows per unit, row blocks per image
  int nunits, ksteps, cpj;  // units, 16-anchor steps per unit, CTAs per job
  int cb128, stages;        // 128-channel blocks of the input; ring depth
  uint32_t x_bytes, d_bytes, x_stride, d_stride;  // one box delivered / its slot
};

template <int NB>
__global__ void __launch_bounds__(WR_THREADS, 1)
    wgrad_rows_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapD,
                      WrArgs a, float* __restrict__ part, int32_t* err) {
  extern __shared__ __align__(1024) uint8_t dyn[];
  __shared__ uint64_t full[WR_STAGES], empty[WR_STAGES], done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  __shared__ uint32_t n_issued, n_consumed;
  constexpr int NX = NB / 64;             // boxes of 64 channels per operand
  constexpr int NACC = NB == 64 ? 6 : 3;  // accumulators of NB columns
  uint8_t* base = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
  const uint32_t stage_bytes = NX * (a.x_stride + a.d_stride);
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  volatile int* abort = &abort_flag;
  if (threadIdx.x == 0) {
    for (int i = 0; i < a.stages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(&done, 1);
    abort_flag = 0;
    n_issued = 0;
    n_consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&tmem_base)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // the zero rows behind every x box
  for (uint32_t i = threadIdx.x; i < (uint32_t)a.stages * NX * (WR_PAD / 16); i += WR_THREADS) {
    const uint32_t s = i / (NX * (WR_PAD / 16)), r = i - s * (NX * (WR_PAD / 16));
    const uint32_t b = r / (WR_PAD / 16), o = r - b * (WR_PAD / 16);
    *reinterpret_cast<uint4*>(base + s * stage_bytes + b * a.x_stride + a.x_bytes + o * 16) =
        make_uint4(0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  DDPPO_PDL_ENTRY();  // after the barrier set-up and the tensor-memory allocation
  const uint32_t tmem = tmem_base;
  const int job = blockIdx.x / a.cpj, split = blockIdx.x - job * a.cpj;
  const int ky = a.by_row ? job % 3 : 0;
  const int cb = a.by_row ? (job / 3) % a.cb128 : 0, nb = a.by_row ? job / (3 * a.cb128) : 0;
  const bool has_work = split < a.nunits;

  if (warp == 0) {
    uint32_t it = 0, ph = 0;
    int s = 0;
    for (int u = split; u < a.nunits; u += a.cpj, ++it) {
      const int ib = u / a.nrb, y0 = (u - ib * a.nrb) * a.RB, n0 = ib * a.ni;
      if (!warp_wait(&empty[s], ph ^ 1u, abort, err)) break;
      if (elect_one()) {
        uint8_t* sx = base + s * stage_bytes;
        uint8_t* sd = sx + NX * a.x_stride;
        mbar_expect_tx(&full[s], NX * (a.x_bytes + a.d_bytes));
#pragma unroll
        for (int i = 0; i < NX; ++i) {
          tma_load_4d(sx + i * a.x_stride, &mapX, &full[s], cb * 128 + i * 64, -1, n0, y0 - 1 + ky);
          tma_load_4d(sd + i * a.d_stride, &mapD, &full[s], nb * 128 + i * 64, 0, n0, y0);
        }
      }
      __syncwarp();
      if (++s == a.stages) { s = 0; ph ^= 1u; }
    }
    if (lane == 0) n_issued = it;
  } else if (warp == 1) {
    const uint32_t idesc = f16_idesc(128, NB, 1, 1);
    uint32_t it = 0, ph = 0;
    int s = 0;
    for (int u = split; u < a.nunits; u += a.cpj, ++it) {
      if (!warp_wait(&full[s], ph, abort, err)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t x0 = smem_addr(base + s * stage_bytes), d0 = x0 + NX * a.x_stride;
      if (elect_one()) {
        for (int k = 0; k < a.ksteps; ++k) {
          const uint64_t db = sw128_mn_desc(d0 + (uint32_t)k * 16 * 128, a.d_stride);
          const uint32_t acc = (it | k) ? 1u : 0u;
#pragma unroll
          for (int q = 0; q < NACC; ++q) {
            // all taps: accumulator (ky, pair) reads the box from row ky, columns 2 pair and
            // 2 pair + 1; by row: accumulator kx, the second atom is the next 64 channels
            const int shift = NB == 64 ? (q >> 1) * a.ni * a.Wp + 2 * (q & 1) : q;
            const uint64_t da = sw128_mn_desc(x0 + (uint32_t)(shift + k * 16) * 128,
                                              NB == 64 ? 128u : a.x_stride);
            tc_mma(tmem + q * NB, da, db, idesc, acc, 0);
          }
        }
        tc_commit(&empty[s]);
      }
      __syncwarp();
      if (++s == a.stages) { s = 0; ph ^= 1u; }
    }
    if (elect_one()) tc_commit(&done);
    if (lane == 0) n_consumed = it;
    // after an abort the epilogue no longer waits for `done`; this warp does, so that
    // every MMA it issued has completed before the accumulators are freed
    if (*abort) mbar_drain_wait(&done, 0u);
  }
  __syncwarp();
  const bool ok = has_work ? mbar_wait(&done, 0u, abort, err) : true;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
  for (int q = 0; q < NACC; ++q) {
    if (NB == 64 && (q & 1) && warp >= 2) continue;  // the discarded fourth column tap
    float* dst = part + (((size_t)blockIdx.x * NACC + q) * 128 + warp * 32 + lane) * NB;
#pragma unroll 1
    for (int c0 = 0; c0 < NB; c0 += 32) {
      uint32_t r[32];
      tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(q * NB + c0), r);
#pragma unroll
      for (int j = 0; j < 32; j += 4)
        *reinterpret_cast<float4*>(dst + c0 + j) =
            (has_work && ok) ? make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                           __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]))
                             : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (abort_flag) {  // uniform: no thread writes it after the barrier
    if (threadIdx.x == 0) drain_unconsumed(full, n_consumed, n_issued, a.stages, nullptr);
    __syncthreads();
  }
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// One weight's gradient from its own pixels alone, in plain order (zero outside the image).
// Out of line and last in its caller: no stack frame there, 48 registers a thread (32 without
// it), 0.25 us a call (97.1 us at 4096 x 16x16, 64 -> 64).
struct WrPixels {
  const __nv_bfloat16* x;
  const __nv_bfloat16* dz;
  int N, H, W, C, Cout;
};
__device__ __noinline__ void wgrad_plain(const WrPixels& p, int ky, int kx, int ci, int co, float* d,
                                         float beta) {
  double sum = 0.0;
  for (int r = 0; r < p.N * p.H; ++r) {
    const int iy = r % p.H + ky - 1;
    const bool in_row = iy >= 0 && iy < p.H;
    const __nv_bfloat16* dz = p.dz + (size_t)r * p.W * p.Cout + co;
    const __nv_bfloat16* x = p.x + ((size_t)(r + ky - 1) * p.W + kx - 1) * p.C + ci;
    float row = 0.f;
#pragma unroll 4
    for (int c = 0; c < p.W; ++c) {
      const bool in = in_row && c + kx >= 1 && c + kx <= p.W;
      const float v = in ? __bfloat162float(x[(ptrdiff_t)c * p.C]) : 0.f;
      row = fmaf(__bfloat162float(dz[(size_t)c * p.Cout]), v, row);
    }
    sum += row;
    if (isnan(sum)) break;  // and stays so
  }
  const float t = (float)sum;
  *d = beta != 0.f ? beta * *d + t : t;
}

// dw (+)= the splits' sums. A block takes 8 accumulator rows (input channels) x 32 columns
// (output channels) of one accumulator of one job: 64 threads of 16-byte loads by 4 slices
// of the splits, the slices added in order; 8 consecutive input channels are written
// together.
template <int NB>
__global__ void __launch_bounds__(256) wgrad_rows_reduce_kernel(const float* __restrict__ part,
                                                                WrArgs a, const __grid_constant__ WrPixels px,
                                                                float* __restrict__ dw, int ldw, float beta) {
  DDPPO_PDL_ENTRY();
  constexpr int NACC = NB == 64 ? 6 : 3;
  __shared__ float sh[4][8][33];
  const int job = blockIdx.z, q = blockIdx.y;
  const int r0 = (blockIdx.x / (NB / 32)) * 8, c0 = (blockIdx.x % (NB / 32)) * 32;
  if (NB == 64 && (q & 1) && r0 >= 64) return;
  const int slice = threadIdx.x >> 6, i = threadIdx.x & 63, r = i >> 3, c = (i & 7) * 4;
  const float* p = part + (((size_t)job * a.cpj * NACC + q) * 128 + r0 + r) * NB + c0 + c;
  const size_t step = (size_t)NACC * 128 * NB;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
  for (int s = slice; s < a.cpj; s += 4) {
    const float4 t = *reinterpret_cast<const float4*>(p + s * step);
    v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
  }
  sh[slice][r][c] = v.x; sh[slice][r][c + 1] = v.y; sh[slice][r][c + 2] = v.z; sh[slice][r][c + 3] = v.w;
  __syncthreads();
  const int rr = threadIdx.x & 7, n = threadIdx.x >> 3;
  const float t = ((sh[0][rr][n] + sh[1][rr][n]) + sh[2][rr][n]) + sh[3][rr][n];
  const int row = r0 + rr;
  int ky, kx, ci, co;
  if (NB == 64) {
    ky = q >> 1; kx = 2 * (q & 1) + (row >> 6); ci = row & 63; co = c0 + n;
  } else {
    ky = job % 3; kx = q; ci = (job / 3) % a.cb128 * 128 + row; co = job / (3 * a.cb128) * 128 + c0 + n;
  }
  float* d = dw + (size_t)co * ldw + (size_t)(ky * 3 + kx) * px.C + ci;
  if (isfinite(t)) *d = beta != 0.f ? beta * *d + t : t;
  else wgrad_plain(px, ky, kx, ci, co, d, beta);
}

// units, ring and shared memory for a convolution; false when it is not covered
struct WrPlan {
  WrArgs a;
  int jobs, nb, x_rows, d_rows;
  size_t smem;
};
bool wr_plan(const ConvShape& c, WrPlan* o) {
  if (c.k != 3 || c.s != 1 || c.p != 1 || c.Ho != c.H || c.Wo != c.W || c.N < 1) return false;
  const bool all = c.C == 64 && c.Cout == 64;
  if (!all && (c.C % 128 || c.Cout % 128 || !c.C || !c.Cout)) return false;
  WrArgs& a = o->a;
  memset(&a, 0, sizeof(a));
  a.by_row = all ? 0 : 1;
  a.Wp = c.W + 2;
  if (a.Wp > 256) return false;
  o->nb = all ? 64 : 128;
  const int nx = o->nb / 64;
  a.cb128 = all ? 1 : c.C / 128;
  o->jobs = all ? 1 : 3 * a.cb128 * (c.Cout / 128);
  // the unit that wastes the fewest anchors (pad columns, rows and images past the end)
  // among those of 64 to 288 anchors, three ring stages rather than two, few halo rows per
  // row (all taps); taller, then larger, on a tie
  double best = 0.0;
  for (int RB = std::min(c.H, 64); RB >= 1; --RB)
    for (int ni = 1; ni <= 16; ++ni) {
      const int anchors = RB * ni * a.Wp;
      if (anchors % 16 || anchors > 288 || (anchors < 64 && ni < 16 && RB < c.H) || ni * a.Wp > 288) continue;
      const int xr = (all ? RB + 2 : RB) * ni * a.Wp;
      const uint32_t xb = 128u * xr, db = 128u * anchors;
      const uint32_t xs = (xb + WR_PAD + 1023) / 1024 * 1024, dsz = (db + 1023) / 1024 * 1024;
      const size_t stage = (size_t)nx * (xs + dsz);
      const int st = (int)std::min<size_t>(WR_STAGES, (WR_SMEM_MAX - 2048) / stage);
      if (st < 2) continue;
      const int nrb = (c.H + RB - 1) / RB, nblk = (c.N + ni - 1) / ni;
      const double use = (double)c.N * c.H * c.W / ((double)nrb * nblk * anchors) * (st >= 3 ? 1.0 : 0.9) *
                         (all ? 0.8 + 0.2 * RB / (RB + 2) : 1.0) * (1.0 + 1e-4 * anchors);
      if (use <= best) continue;
      best = use;
      a.ni = ni; a.RB = RB; a.nrb = nrb; a.nunits = nrb * nblk; a.ksteps = anchors / 16;
      a.stages = st; a.x_bytes = xb; a.d_bytes = db; a.x_stride = xs; a.d_stride = dsz;
      o->x_rows = all ? RB + 2 : RB; o->d_rows = RB;
      o->smem = st * stage + 1024;
    }
  return best > 0.0;
}

bool wr_map(CUtensorMap* m, const void* p, int C, const ConvShape& c, int Wp, int ni, int rows) {
  // dimensions (channel, column, image, row): a box holds `rows` rows of ni images
  cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)c.W, (cuuint64_t)c.N, (cuuint64_t)c.H};
  cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)c.H * c.W * C * 2, (cuuint64_t)c.W * C * 2};
  cuuint32_t box[4] = {64, (cuuint32_t)Wp, (cuuint32_t)ni, (cuuint32_t)rows};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return encode_fn()(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p), dims, strides, box,
                     estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int NB>
int launch_wr(const WrPlan& p, const CUtensorMap& mx, const CUtensorMap& md, const WrPixels& px,
              float* dw, int ldw, float beta, const GemmWorkspace& ws, cudaStream_t s) {
  static bool attr_done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && !attr_done[dev]) {
    DDPPO_CHECK_CUDA(cudaFuncSetAttribute(wgrad_rows_kernel<NB>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WR_SMEM_MAX));
    attr_done[dev] = true;
  }
  float* part = nullptr;
  DDPPO_TRY(ws.sums(s, &part));
  ::ddppo::launch_k(wgrad_rows_kernel<NB>, p.jobs * p.a.cpj, WR_THREADS, p.smem, s, mx, md, p.a, part, ws.err);
  DDPPO_CHECK_LAUNCH();
  ::ddppo::launch_k(wgrad_rows_reduce_kernel<NB>, dim3(16 * (NB / 32), NB == 64 ? 6 : 3, p.jobs), 256, 0, s,
                    part, p.a, px, dw, ldw, beta);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

// CTAs per job that the SMs, the units and the workspace of partial sums allow (0: none)
int wr_splits(const WrPlan& p, const GemmWorkspace& ws) {
  const size_t per = (size_t)(p.nb == 64 ? 6 : 3) * 128 * p.nb;
  size_t cpj = std::max(1, ws.num_sms / p.jobs);
  cpj = std::min(cpj, ws.partial_elems / (per * p.jobs));
  return (int)std::min<size_t>(cpj, (size_t)p.a.nunits);
}

}  // namespace

bool conv_wgrad_rows_ok(const ConvShape& c, const void* x, const void* dz, const GemmWorkspace& ws) {
  WrPlan p;
  return encode_fn() && !((uintptr_t)x & 15) && !((uintptr_t)dz & 15) && wr_plan(c, &p) &&
         wr_splits(p, ws) >= 1;
}

int conv_wgrad_rows(const ConvShape& c, const void* x, const void* dz, float* dw, int ldw, float beta,
                    const GemmWorkspace& ws, cudaStream_t s) {
  WrPlan p;
  if (!wr_plan(c, &p) || (p.a.cpj = wr_splits(p, ws)) < 1) {
    set_error("wgrad_rows: unsupported shape or workspace too small");
    return DDPPO_E_CONFIG;
  }
  CUtensorMap mx, md;
  if (!wr_map(&mx, x, c.C, c, p.a.Wp, p.a.ni, p.x_rows) ||
      !wr_map(&md, dz, c.Cout, c, p.a.Wp, p.a.ni, p.d_rows)) {
    set_error("wgrad_rows: tensor map encoding failed");
    return DDPPO_E_CUDA;
  }
  const WrPixels px{(const __nv_bfloat16*)x, (const __nv_bfloat16*)dz, c.N, c.H, c.W, c.C, c.Cout};
  if (p.nb == 64) return launch_wr<64>(p, mx, md, px, dw, ldw, beta, ws, s);
  return launch_wr<128>(p, mx, md, px, dw, ldw, beta, ws, s);
}

}  // namespace ddppo
