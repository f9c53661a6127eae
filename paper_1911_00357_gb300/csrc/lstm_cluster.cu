// The LSTM recurrence of a whole segment, one launch per layer and direction, for batches
// of at most 64 envs (App. "Agent Design"; Sec. 4 "Training": back-propagation through the
// rollout). A step is a contraction of a few MFLOP whose result every unit of the next step
// needs, so the chain of steps bounds it, not arithmetic or bandwidth: step by step, the
// recurrent contraction and the cell kernel cost 10.5 us per step and layer.
//
// Here a thread-block cluster of H / 32 CTAs (16 at H = 512) carries at most 8 envs through
// all T steps; clusters share nothing, so they need not be resident together. CTA j owns
// the 32 units [32 j, 32 j + 32). Its rows of W_hh (forward) or W_hh^T (backward), 128 KB of
// bf16 at H = 512, stay in the register file as warp-level MMA fragments (m16n8k16, the
// envs on the 8-wide side) for the whole segment: no weight is read again. What a step
// exchanges is small (the masked state, 8 envs x H bf16; the gate gradients, four times
// that) and goes straight into the shared memory of every CTA of the cluster with st.async,
// whose bytes complete the receiver's mbarrier: no grid barrier and no trip through L2.
// Two buffers alternate: a CTA sends the data of step t + 2 only after it has received all
// of step t + 1, which every CTA sent after it had read step t's buffer.
//
// tcgen05 is not used: with 8 envs the MMA's useful side is 8 columns, and a TMEM round
// trip per step costs more than the 4 k-step chains of the register form (the tcgen05
// kernel in lstm_tc.cu takes 7 us a step).
//
// The sums are formed exactly as the step-by-step path forms them (gemm_small_kernel: K
// split into eight slices, each one chain of MMAs, added in slice order), so results are
// bit-identical with it.
//
// Measured on the 2 x 512 LSTM over 128 steps x 32 envs: one layer's recurrence takes 184 us
// forward (1.4 us a step) and 236 us backward (1.8 us a step) against 1.35 ms each step by
// step; the whole pass, input and weight gradients included, 1.24 ms against 5.52 ms. What
// is left per step is the chain: wait, operand loads and MMAs, cell, block barrier, remote
// stores.
//
// Every wait is bounded: on a run-out the sticky timeout flag is set, the CTA sends and
// stores nothing more, and every CTA meets the cluster barrier at the end; one that gave up
// then waits (bounded) for the blocks still on their way to it before its shared memory is
// released.
#include <algorithm>
#include <atomic>

#include "cluster.cuh"
#include "lstm_cell.cuh"
#include "nn_kernels.cuh"

namespace ddppo {

namespace {

constexpr int LC_THREADS = 256;  // 8 warps
constexpr int LC_UNITS = 32;     // hidden units per CTA
constexpr int LC_ENVS = 8;       // envs per cluster at most (the MMA's N side)
constexpr int LC_BLOCK = 512;    // bytes of one [8 envs][32 units] bf16 block
constexpr int LC_RED_PITCH = 36; // backward partial sums: floats per env row

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t saddr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(saddr)
               : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// byte offset of (env row n, unit u) inside a block: rows of 64 bytes whose 16-byte chunks
// are swizzled so that the 8 rows of an ldmatrix tile fall into distinct banks
__device__ __forceinline__ int blk_off(int n, int u) {
  return n * 64 + (((u >> 3) ^ ((n >> 1) & 3)) << 4) + (u & 7) * 2;
}
// this lane's ldmatrix row address inside a block: four 8 x 8 tiles = 32 units of 8 envs
__device__ __forceinline__ int ldsm_off(int lane) {
  return blk_off(lane & 7, (lane >> 3) * 8);
}
__device__ __forceinline__ uint32_t ld_w2(const __nv_bfloat16* p) {
  return __ldg(reinterpret_cast<const uint32_t*>(p));
}

template <int KS>
__global__ void __launch_bounds__(LC_THREADS, 1) lstm_cl_fwd_kernel(LstmCl a) {
  DDPPO_PDL_ENTRY();
  constexpr int H = KS * 16, CL = H / LC_UNITS;
  constexpr int PER = (KS + 7) / 8, NSL = KS / PER;  // k-steps per slice, slices
  __shared__ __align__(128) uint8_t hs[2][CL * LC_BLOCK];
  __shared__ __align__(16) uint8_t stage[2][LC_BLOCK];
  __shared__ uint64_t full[2];
  __shared__ int sent[kClusterMax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  const int cta = (int)cluster_rank();
  const int e0 = (int)(blockIdx.x / CL) * a.epc, ne = min(a.epc, a.E - e0);
  // this thread's cell: unit u of the CTA, env n of the cluster
  const int hi = lane >> 4, u = warp * 4 + (g & 3), n = 2 * t4 + hi;
  const bool mine = n < ne;
  const int unit = cta * LC_UNITS + u, e = e0 + (mine ? n : 0);

  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (a.T > 1) expect_bytes(&full[1], (uint32_t)(CL * ne * 64));
    if (a.T > 2) expect_bytes(&full[0], (uint32_t)(CL * ne * 64));
  }
  // the masked state entering step 0, and zero rows for the missing envs
  for (int i = threadIdx.x; i < CL * 32; i += LC_THREADS) {
    const int j = i >> 5, row = (i >> 2) & 7, k = j * LC_UNITS + (i & 3) * 8;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (row < ne) {
      const size_t o = (size_t)(e0 + row) * H + k;
      if (a.m[e0 + row]) {
        __nv_bfloat162 p[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) p[q] = __floats2bfloat162_rn(a.h0[o + 2 * q], a.h0[o + 2 * q + 1]);
        v = *reinterpret_cast<uint4*>(p);
      }
      if (j == cta) *reinterpret_cast<uint4*>((__nv_bfloat16*)a.hm + o) = v;
    }
    *reinterpret_cast<uint4*>(&hs[0][j * LC_BLOCK + blk_off(row, (i & 3) * 8)]) = v;
    *reinterpret_cast<uint4*>(&hs[1][j * LC_BLOCK + blk_off(row, (i & 3) * 8)]) = make_uint4(0u, 0u, 0u, 0u);
  }
  // this warp's 16 gate rows: MMA row r is gate r / 4 of unit warp * 4 + r % 4
  uint32_t w[KS][4];
  {
    const __nv_bfloat16* r0 = (const __nv_bfloat16*)a.W + (size_t)((g >> 2) * H + unit) * H + 2 * t4;
    const __nv_bfloat16* r1 = r0 + (size_t)2 * H * H;  // rows 8 .. 15: gates g, o
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      w[ks][0] = ld_w2(r0 + ks * 16);
      w[ks][1] = ld_w2(r1 + ks * 16);
      w[ks][2] = ld_w2(r0 + ks * 16 + 8);
      w[ks][3] = ld_w2(r1 + ks * 16 + 8);
    }
  }
  const size_t EG = (size_t)a.E * 4 * H, EH = (size_t)a.E * H;
  const float* gxp = a.gx + (size_t)e * 4 * H + unit;
  float c = mine ? a.c0[(size_t)e * H + unit] : 0.f;
  bool mk = mine && a.m[e];
  float gx[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) gx[q] = mine ? gxp[q * H] : 0.f;
  __syncthreads();
  cluster_sync();  // every barrier is initialised and every buffer zeroed before a send

  bool ok = true;
  int t = 0;
  for (; t < a.T; ++t) {
    if (t > 0) ok = wait_bytes(&full[step_bar(t)], step_parity(t), a.err) && ok;
    if (threadIdx.x == 0 && ok && t > 0 && t + 2 < a.T)
      expect_bytes(&full[t & 1], (uint32_t)(CL * ne * 64));
    // the next step's input projection and mask, in flight during this step's MMAs
    float gn[4] = {0.f, 0.f, 0.f, 0.f};
    bool mn = false;
    if (mine && t + 1 < a.T) {
      const float* p = gxp + (size_t)(t + 1) * EG;
#pragma unroll
      for (int q = 0; q < 4; ++q) gn[q] = __ldg(p + q * H);
      mn = a.m[(size_t)(t + 1) * a.E + e] != 0;
    }
    float acc[NSL][4];
#pragma unroll
    for (int s = 0; s < NSL; ++s)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[s][q] = 0.f;
    const uint32_t hb = smem_addr(&hs[t & 1][0]) + (uint32_t)ldsm_off(lane);
    if constexpr (PER == 1) {
#pragma unroll
      for (int s = 0; s < NSL; s += 2) {
        uint32_t b[4];
        ldsm4(b, hb + (s / 2) * LC_BLOCK);
        mma16816(acc[s], w[s], b[0], b[1]);
        mma16816(acc[s + 1], w[s + 1], b[2], b[3]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < PER; i += 2) {
        uint32_t b[NSL][4];
#pragma unroll
        for (int s = 0; s < NSL; ++s) ldsm4(b[s], hb + ((s * PER + i) / 2) * LC_BLOCK);
#pragma unroll
        for (int s = 0; s < NSL; ++s) mma16816(acc[s], w[s * PER + i], b[s][0], b[s][1]);
#pragma unroll
        for (int s = 0; s < NSL; ++s) mma16816(acc[s], w[s * PER + i + 1], b[s][2], b[s][3]);
      }
    }
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = 0.f;
#pragma unroll
      for (int s = 0; s < NSL; ++s) v[q] += acc[s][q];
    }
    // lanes 0..15 hold gates i, g of envs 2 t4 and 2 t4 + 1, lanes 16..31 gates f, o of the
    // same units: after the exchange each lane holds all four of its own env
    const float x0 = __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[1], 16);
    const float x1 = __shfl_xor_sync(0xffffffffu, hi ? v[2] : v[3], 16);
    const float ri = hi ? x0 : v[0], rf = hi ? v[1] : x0;
    const float rg = hi ? x1 : v[2], ro = hi ? v[3] : x1;
    float gi, gf, gg, go, h;
    const float cp = mk ? c : 0.f;
    lstm_cell_fwd(gx[0] + ri, gx[1] + rf, gx[2] + rg, gx[3] + ro, cp, gi, gf, gg, go, c, h);
    const __nv_bfloat16 hn = __float2bfloat16_rn(mn ? h : 0.f);
    const bool last = t + 1 == a.T;
    bool stop = last;
    if (!last) {
      if (mine) *reinterpret_cast<__nv_bfloat16*>(&stage[t & 1][blk_off(n, u)]) = hn;
      if (__syncthreads_or(ok ? 0 : 1)) ok = false;
      stop = !ok;
    }
    // the block of new states to every CTA of the cluster (two destinations per warp)
    if (!stop && (lane >> 2) < ne) {
      const uint4 blk = *reinterpret_cast<const uint4*>(&stage[t & 1][lane * 16]);
      const int nb = (t + 1) & 1;
      const uint32_t dst = smem_addr(&hs[nb][cta * LC_BLOCK + lane * 16]), bar = smem_addr(&full[nb]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const uint32_t r = (uint32_t)(warp * 2 + q);
        if (r < (uint32_t)CL) send16(map_rank(dst, r), blk, map_rank(bar, r));
      }
    }
    // the step's results leave while the states travel
    if (mine && ok) {
      const size_t gb = (size_t)t * EG + (size_t)e * 4 * H + unit, ho = (size_t)t * EH + (size_t)e * H + unit;
      a.gates[gb] = gi;
      a.gates[gb + H] = gf;
      a.gates[gb + 2 * H] = gg;
      a.gates[gb + 3 * H] = go;
      a.c[ho] = c;
      a.h[ho] = h;
      ((__nv_bfloat16*)a.y)[ho] = __float2bfloat16_rn(h);
      if (!last) ((__nv_bfloat16*)a.hm)[ho + EH] = hn;
    }
    if (stop) break;
#pragma unroll
    for (int q = 0; q < 4; ++q) gx[q] = gn[q];
    mk = mn;
  }
  cluster_end(full, sent, CL, t, a.T, (uint32_t)(ne * 64), !ok);
}

// back-propagation: CTA j owns units [32 j, 32 j + 32), i.e. rows of W_hh^T [H, 4H]. The
// recurrent gradient of a unit sums over all 4H gate gradients; warp s takes slice s of
// that sum (gate s / 2, unit half s % 2) for the CTA's 32 rows (two MMA row tiles sharing
// the operand fragments), and the eight slices meet in shared memory in slice order.
template <int KS>
__global__ void __launch_bounds__(LC_THREADS, 1) lstm_cl_bwd_kernel(LstmCl a) {
  DDPPO_PDL_ENTRY();
  constexpr int H = KS * 16, CL = H / LC_UNITS, PER = H / 32;  // k-steps per slice
  extern __shared__ __align__(128) uint8_t ds[];  // [2][CL][4 gates][LC_BLOCK]
  __shared__ __align__(16) uint8_t stage[4 * LC_BLOCK];
  __shared__ float red[8][LC_ENVS][LC_RED_PITCH];
  __shared__ uint64_t full[2];
  __shared__ int sent[kClusterMax];
  constexpr int BUF = CL * 4 * LC_BLOCK;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t4 = lane & 3;
  const int cta = (int)cluster_rank();
  const int e0 = (int)(blockIdx.x / CL) * a.epc, ne = min(a.epc, a.E - e0);
  const int n = warp, u = lane;  // this thread's cell
  const bool mine = n < ne;
  const int unit = cta * LC_UNITS + u, e = e0 + (mine ? n : 0);
  const uint32_t bytes = (uint32_t)(CL * 4 * ne * 64);

  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (a.T > 1) expect_bytes(&full[1], bytes);
    if (a.T > 2) expect_bytes(&full[0], bytes);
  }
  for (int i = threadIdx.x; i < 2 * BUF / 16; i += LC_THREADS)
    *reinterpret_cast<uint4*>(ds + i * 16) = make_uint4(0u, 0u, 0u, 0u);
  uint32_t w[2][PER][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    const __nv_bfloat16* r0 = (const __nv_bfloat16*)a.W + (size_t)(cta * LC_UNITS + mt * 16 + g) * 4 * H +
                              (size_t)warp * PER * 16 + 2 * t4;
    const __nv_bfloat16* r1 = r0 + (size_t)8 * 4 * H;
#pragma unroll
    for (int ks = 0; ks < PER; ++ks) {
      w[mt][ks][0] = ld_w2(r0 + ks * 16);
      w[mt][ks][1] = ld_w2(r1 + ks * 16);
      w[mt][ks][2] = ld_w2(r0 + ks * 16 + 8);
      w[mt][ks][3] = ld_w2(r1 + ks * 16 + 8);
    }
  }
  const size_t EG = (size_t)a.E * 4 * H, EH = (size_t)a.E * H;
  const size_t gofs = (size_t)e * 4 * H + unit, hofs = (size_t)e * H + unit;
  float c = mine ? a.c[(size_t)(a.T - 1) * EH + hofs] : 0.f, dcc = 0.f;
  bool mnext = false;
  __syncthreads();
  cluster_sync();

  bool ok = true;
  int it = 0;
  for (; it < a.T; ++it) {
    const int t = a.T - 1 - it;
    // forward values of the step, in flight during the wait and the MMAs
    float gt[4] = {0.f, 0.f, 0.f, 0.f}, cprev = 0.f, dha = 0.f;
    bool mk = false;
    if (mine) {
      const float* gp = a.gates + (size_t)t * EG + gofs;
#pragma unroll
      for (int q = 0; q < 4; ++q) gt[q] = gp[q * H];
      cprev = t == 0 ? a.c0[hofs] : a.c[(size_t)(t - 1) * EH + hofs];
      dha = a.dh_above[(size_t)t * EH + hofs];
      mk = a.m[(size_t)t * a.E + e] != 0;
    }
    float rec = 0.f;
    if (it > 0) {
      ok = wait_bytes(&full[step_bar(it)], step_parity(it), a.err) && ok;
      if (threadIdx.x == 0 && ok && it + 2 < a.T) expect_bytes(&full[it & 1], bytes);
      float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
      // slice = gate warp / 2, units of CTAs (warp % 2) CL / 2 ..
      const uint32_t db = smem_addr(ds + (it & 1) * BUF) + (uint32_t)ldsm_off(lane) +
                          (uint32_t)((warp & 1) * (CL / 2) * 4 + (warp >> 1)) * LC_BLOCK;
#pragma unroll
      for (int ks = 0; ks < PER; ks += 2) {
        uint32_t b[4];
        ldsm4(b, db + (ks / 2) * 4 * LC_BLOCK);
        mma16816(acc[0], w[0][ks], b[0], b[1]);
        mma16816(acc[1], w[1][ks], b[0], b[1]);
        mma16816(acc[0], w[0][ks + 1], b[2], b[3]);
        mma16816(acc[1], w[1][ks + 1], b[2], b[3]);
      }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        red[warp][2 * t4][mt * 16 + g] = acc[mt][0];
        red[warp][2 * t4 + 1][mt * 16 + g] = acc[mt][1];
        red[warp][2 * t4][mt * 16 + g + 8] = acc[mt][2];
        red[warp][2 * t4 + 1][mt * 16 + g + 8] = acc[mt][3];
      }
      if (__syncthreads_or(ok ? 0 : 1)) { ok = false; break; }
#pragma unroll
      for (int s = 0; s < 8; ++s) rec += red[s][n][u];
    }
    const float cp = mk ? cprev : 0.f;
    float dh = dha;
    if (mnext && it > 0) dh += rec;
    float dz[4], dco;
    lstm_cell_bwd(gt[0], gt[1], gt[2], gt[3], c, cp, dh, mnext, dcc, dz[0], dz[1], dz[2], dz[3], dco);
    dcc = dco;
    c = cprev;
    mnext = mk;
    __nv_bfloat16 db16[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) db16[q] = __float2bfloat16_rn(dz[q]);
    if (t > 0) {
      if (mine) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<__nv_bfloat16*>(&stage[q * LC_BLOCK + blk_off(n, u)]) = db16[q];
      }
      __syncthreads();
      if ((lane >> 2) < ne) {
        const int nb = (it + 1) & 1;
        const uint32_t dst = smem_addr(ds + nb * BUF + cta * 4 * LC_BLOCK + lane * 16), bar = smem_addr(&full[nb]);
        uint4 blk[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) blk[q] = *reinterpret_cast<const uint4*>(&stage[q * LC_BLOCK + lane * 16]);
#pragma unroll
        for (int d = 0; d < 2; ++d) {
          const uint32_t r = (uint32_t)(warp * 2 + d);
          if (r >= (uint32_t)CL) break;
          const uint32_t rd = map_rank(dst, r), rb = map_rank(bar, r);
#pragma unroll
          for (int q = 0; q < 4; ++q) send16(rd + q * LC_BLOCK, blk[q], rb);
        }
      }
    }
    // the step's results leave while the gradients travel
    if (mine) {
      const size_t gb = (size_t)t * EG + gofs;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a.dg32[gb + q * H] = dz[q];
        ((__nv_bfloat16*)a.dg_op)[gb + q * H] = db16[q];
      }
    }
  }
  cluster_end(full, sent, CL, it, a.T, (uint32_t)(4 * ne * 64), !ok);
}

// ---- FP32 operands: the same scheme on the CUDA cores ----
// CTA j owns 32 units; its weights (64 KB at H = 128) are registers: warp w holds gate w / 2
// of them over K half w % 2 (forward), or slice w of the 4H gate gradients (backward), lane =
// unit, and multiplies with the envs' rows broadcast from shared memory. The eight partial
// sums of a (unit, env) meet in shared memory; thread (env = warp, unit = lane) updates the
// cell and sends its value to every CTA. Covered to H = 256 (128 weight registers a thread).
template <int K2>
__device__ __forceinline__ void load_row(float (&w)[K2], const float* p) {
#pragma unroll
  for (int k = 0; k < K2; k += 4) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p + k));
    w[k] = v.x; w[k + 1] = v.y; w[k + 2] = v.z; w[k + 3] = v.w;
  }
}
template <int K2>
__device__ __forceinline__ float dot_row(const float (&w)[K2], const float* h) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < K2; k += 4) {
    const float4 v = *reinterpret_cast<const float4*>(h + k);
    s[0] = fmaf(w[k], v.x, s[0]);
    s[1] = fmaf(w[k + 1], v.y, s[1]);
    s[2] = fmaf(w[k + 2], v.z, s[2]);
    s[3] = fmaf(w[k + 3], v.w, s[3]);
  }
  return (s[0] + s[1]) + (s[2] + s[3]);
}

template <int H>
__global__ void __launch_bounds__(LC_THREADS, 1) lstm_cl32_fwd_kernel(LstmCl a) {
  DDPPO_PDL_ENTRY();
  constexpr int CL = H / LC_UNITS, K2 = H / 2;
  __shared__ __align__(16) float hs[2][LC_ENVS][H];
  __shared__ float red[8][LC_ENVS][LC_UNITS];
  __shared__ uint64_t full[2];
  __shared__ int sent[kClusterMax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = (int)cluster_rank();
  const int e0 = (int)(blockIdx.x / CL) * a.epc, ne = min(a.epc, a.E - e0);
  const bool mine = warp < ne;
  const int unit = cta * LC_UNITS + lane, e = e0 + (mine ? warp : 0);
  const uint32_t bytes = (uint32_t)(H * ne * 4);
  float* hm = (float*)a.hm;
  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (a.T > 1) expect_bytes(&full[1], bytes);
    if (a.T > 2) expect_bytes(&full[0], bytes);
  }
  for (int i = threadIdx.x; i < ne * H; i += LC_THREADS) {
    const int row = i / H, k = i - row * H;
    const size_t o = (size_t)(e0 + row) * H + k;
    const float v = a.m[e0 + row] ? a.h0[o] : 0.f;
    hs[0][row][k] = v;
    if (k / LC_UNITS == cta) hm[o] = v;
  }
  float w[K2];
  load_row<K2>(w, (const float*)a.W + (size_t)((warp >> 1) * H + unit) * H + (warp & 1) * K2);
  const size_t EG = (size_t)a.E * 4 * H, EH = (size_t)a.E * H;
  const float* gxp = a.gx + (size_t)e * 4 * H + unit;
  float c = mine ? a.c0[(size_t)e * H + unit] : 0.f;
  bool mk = mine && a.m[e];
  float gx[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) gx[q] = mine ? gxp[q * H] : 0.f;
  __syncthreads();
  cluster_sync();

  bool ok = true;
  int t = 0;
  for (; t < a.T; ++t) {
    if (t > 0) ok = wait_bytes(&full[step_bar(t)], step_parity(t), a.err) && ok;
    if (threadIdx.x == 0 && ok && t > 0 && t + 2 < a.T) expect_bytes(&full[t & 1], bytes);
    const bool last = t + 1 == a.T;
    float gn[4] = {0.f, 0.f, 0.f, 0.f};
    bool mn = false;
    if (mine && !last) {
      const float* p = gxp + (size_t)(t + 1) * EG;
#pragma unroll
      for (int q = 0; q < 4; ++q) gn[q] = __ldg(p + q * H);
      mn = a.m[(size_t)(t + 1) * a.E + e] != 0;
    }
    for (int n = 0; n < ne; ++n) red[warp][n][lane] = dot_row<K2>(w, &hs[t & 1][n][(warp & 1) * K2]);
    // (the buffer of partial sums is free again at the next step: its wait ends only after
    // every cell of this CTA has been read, updated and sent)
    if (__syncthreads_or(ok ? 0 : 1)) { ok = false; break; }
    if (mine) {
      float z[4], gi, gf, gg, go, h;
#pragma unroll
      for (int q = 0; q < 4; ++q) z[q] = gx[q] + (red[2 * q][warp][lane] + red[2 * q + 1][warp][lane]);
      lstm_cell_fwd(z[0], z[1], z[2], z[3], mk ? c : 0.f, gi, gf, gg, go, c, h);
      const float hn = mn ? h : 0.f;
      if (!last) {
        const int nb = (t + 1) & 1;
        const uint32_t dst = smem_addr(&hs[nb][warp][unit]), bar = smem_addr(&full[nb]);
#pragma unroll
        for (int r = 0; r < CL; ++r) send4(map_rank(dst, r), hn, map_rank(bar, r));
      }
      const size_t gb = (size_t)t * EG + (size_t)e * 4 * H + unit, ho = (size_t)t * EH + (size_t)e * H + unit;
      a.gates[gb] = gi;
      a.gates[gb + H] = gf;
      a.gates[gb + 2 * H] = gg;
      a.gates[gb + 3 * H] = go;
      a.c[ho] = c;
      a.h[ho] = h;
      ((float*)a.y)[ho] = h;
      if (!last) hm[ho + EH] = hn;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) gx[q] = gn[q];
    mk = mn;
  }
  cluster_end(full, sent, CL, t, a.T, (uint32_t)(LC_UNITS * ne * 4), !ok);
}

template <int H>
__global__ void __launch_bounds__(LC_THREADS, 1) lstm_cl32_bwd_kernel(LstmCl a) {
  DDPPO_PDL_ENTRY();
  constexpr int CL = H / LC_UNITS, K2 = H / 2, ROW = 4 * H;
  extern __shared__ __align__(128) float dz_in[];  // [2][LC_ENVS][4H]
  __shared__ float red[8][LC_ENVS][LC_UNITS];
  __shared__ uint64_t full[2];
  __shared__ int sent[kClusterMax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = (int)cluster_rank();
  const int e0 = (int)(blockIdx.x / CL) * a.epc, ne = min(a.epc, a.E - e0);
  const bool mine = warp < ne;
  const int unit = cta * LC_UNITS + lane, e = e0 + (mine ? warp : 0);
  const uint32_t bytes = (uint32_t)(ROW * ne * 4);
  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (a.T > 1) expect_bytes(&full[1], bytes);
    if (a.T > 2) expect_bytes(&full[0], bytes);
  }
  float w[K2];
  load_row<K2>(w, (const float*)a.W + (size_t)unit * ROW + warp * K2);
  const size_t EG = (size_t)a.E * ROW, EH = (size_t)a.E * H;
  const size_t gofs = (size_t)e * ROW + unit, hofs = (size_t)e * H + unit;
  float c = mine ? a.c[(size_t)(a.T - 1) * EH + hofs] : 0.f, dcc = 0.f;
  bool mnext = false;
  __syncthreads();
  cluster_sync();

  bool ok = true;
  int it = 0;
  for (; it < a.T; ++it) {
    const int t = a.T - 1 - it;
    float gt[4] = {0.f, 0.f, 0.f, 0.f}, cprev = 0.f, dha = 0.f;
    bool mk = false;
    if (mine) {
      const float* gp = a.gates + (size_t)t * EG + gofs;
#pragma unroll
      for (int q = 0; q < 4; ++q) gt[q] = gp[q * H];
      cprev = t == 0 ? a.c0[hofs] : a.c[(size_t)(t - 1) * EH + hofs];
      dha = a.dh_above[(size_t)t * EH + hofs];
      mk = a.m[(size_t)t * a.E + e] != 0;
    }
    float rec = 0.f;
    if (it > 0) {
      ok = wait_bytes(&full[step_bar(it)], step_parity(it), a.err) && ok;
      if (threadIdx.x == 0 && ok && it + 2 < a.T) expect_bytes(&full[it & 1], bytes);
      const float* in = dz_in + (size_t)(it & 1) * LC_ENVS * ROW + warp * K2;
      for (int n = 0; n < ne; ++n) red[warp][n][lane] = dot_row<K2>(w, in + n * ROW);
      if (__syncthreads_or(ok ? 0 : 1)) { ok = false; break; }
      if (mine) {
#pragma unroll
        for (int s = 0; s < 8; ++s) rec += red[s][warp][lane];
      }
    }
    if (!mine) continue;
    float dh = dha;
    if (mnext && it > 0) dh += rec;
    float dz[4], dco;
    lstm_cell_bwd(gt[0], gt[1], gt[2], gt[3], c, mk ? cprev : 0.f, dh, mnext, dcc, dz[0], dz[1], dz[2],
                  dz[3], dco);
    dcc = dco;
    c = cprev;
    mnext = mk;
    if (t > 0) {
      const int nb = (it + 1) & 1;
      const uint32_t dst = smem_addr(dz_in + ((size_t)nb * LC_ENVS + warp) * ROW + unit), bar = smem_addr(&full[nb]);
#pragma unroll
      for (int r = 0; r < CL; ++r) {
        const uint32_t rd = map_rank(dst, r), rb = map_rank(bar, r);
#pragma unroll
        for (int q = 0; q < 4; ++q) send4(rd + q * H * 4, dz[q], rb);
      }
    }
    const size_t gb = (size_t)t * EG + gofs;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      a.dg32[gb + q * H] = dz[q];
      ((float*)a.dg_op)[gb + q * H] = dz[q];
    }
  }
  cluster_end(full, sent, CL, it, a.T, (uint32_t)(4 * LC_UNITS * ne * 4), !ok);
}

typedef void (*ClKernel)(LstmCl);
struct ClForm {
  ClKernel fwd = nullptr, bwd = nullptr;
  int CL = 0;
  size_t bwd_smem = 0;
};
template <int KS>
ClForm bf16_form() {
  return ClForm{lstm_cl_fwd_kernel<KS>, lstm_cl_bwd_kernel<KS>, KS / 2,
                (size_t)2 * (KS / 2) * 4 * LC_BLOCK};
}
template <int H>
ClForm fp32_form() {
  return ClForm{lstm_cl32_fwd_kernel<H>, lstm_cl32_bwd_kernel<H>, H / LC_UNITS,
                (size_t)2 * LC_ENVS * 4 * H * sizeof(float)};
}
constexpr int LC_SIZES[4] = {64, 128, 256, 512};
// the kernels of hidden size LC_SIZES[i]; fwd null where not covered
ClForm form_of(int i, bool bf) {
  switch (i) {
    case 0: return bf ? bf16_form<4>() : fp32_form<64>();
    case 1: return bf ? bf16_form<8>() : fp32_form<128>();
    case 2: return bf ? bf16_form<16>() : fp32_form<256>();
    case 3: return bf ? bf16_form<32>() : ClForm{};
    default: return ClForm{};
  }
}
int size_index(int H) {
  for (int i = 0; i < 4; ++i)
    if (LC_SIZES[i] == H) return i;
  return -1;
}

cudaLaunchConfig_t cl_config(int clusters, int CL, size_t smem, cudaStream_t s,
                             cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * CL));
  cfg.blockDim = dim3(LC_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  return cfg;
}

// clusters of this hidden size that the current device holds at once (0: none, or the size
// is not covered); asked once per device, size and operand type
int cl_resident(int H, bool bf) {
  static std::atomic<int> cache[64][8];  // 0: not asked yet, else the answer + 1
  const int i = size_index(H);
  int dev = 0;
  if (i < 0 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  const ClForm f = form_of(i, bf);
  if (!f.fwd) return 0;
  std::atomic<int>& slot = cache[dev][2 * i + (bf ? 1 : 0)];
  const int known = slot.load();
  if (known) return known - 1;
  int least = 1 << 20;
  for (int dir = 0; dir < 2; ++dir) {
    const ClKernel k = dir ? f.bwd : f.fwd;
    const size_t smem = dir ? f.bwd_smem : 0;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cl_config(1, f.CL, smem, nullptr, attr);
    cfg.numAttrs = 1;
    int num = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&num, k, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      num = 0;
    }
    least = std::min(num, least);
  }
  slot.store(least + 1);
  return least;
}

int launch_cl(const LstmCl& in, bool bf, bool bwd, cudaStream_t s) {
  const int room = cl_resident(in.H, bf);
  if (room < 1) {
    set_error("lstm: the cluster form does not cover this hidden size or device");
    return DDPPO_E_CONFIG;
  }
  const ClForm f = form_of(size_index(in.H), bf);
  LstmCl a = in;
  // as few envs per cluster as keep all clusters resident at once (fewer bytes to exchange
  // per step), at most 8
  a.epc = std::min(LC_ENVS, (a.E + room - 1) / room);
  const int clusters = (a.E + a.epc - 1) / a.epc;
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = cl_config(clusters, f.CL, bwd ? f.bwd_smem : 0, s, attr);
  DDPPO_CHECK_CUDA(cudaLaunchKernelEx(&cfg, bwd ? f.bwd : f.fwd, a));
  return DDPPO_OK;
}

}  // namespace

// BF16: segments of more than one step and up to 64 envs. Above that the step-by-step
// contraction is the tcgen05 one, which sums in another order, and the recurrence would no
// longer give that path's bits; a single step measured no gain (the act pass: 597 us with
// it, 584 without). 57 to 64 envs at H = 512 take two waves of clusters (7 are resident at
// once), about 3.5 us a step, still a third of the steps'.
// FP32: any segment that fits one wave of clusters (H = 128: 592 envs); the step-by-step
// form costs 12 us a step there against 0.9 us (H = 128, 32 steps x 8 envs: 29 us forward, 27 us
// backward a segment; the 16-env update 6.96 -> 3.54 ms).
bool lstm_cl_supported(int H, int T, int E, bool bf) {
  if (T < 1 || E < 1 || (bf && (T < 2 || E > 64))) return false;
  const int room = cl_resident(H, bf);
  return room >= 1 && (bf || E <= LC_ENVS * room);
}
int launch_lstm_cl_fwd(const LstmCl& a, bool bf, cudaStream_t s) { return launch_cl(a, bf, false, s); }
int launch_lstm_cl_bwd(const LstmCl& a, bool bf, cudaStream_t s) { return launch_cl(a, bf, true, s); }

}  // namespace ddppo
