// The operand copies of the FP32 master weights that the contractions read (GEMM layouts in
// the operand dtype), all layers in one launch.
//
// A weight tensor is rows x (cin x kk): output channels (or gate rows) by input channels by
// filter taps (1 for the LSTM, the pixels of the feature map for the visual FC). Up to three
// copies are formed: wg [rows][tap][cin] (leading dimension ld), wgT [tap][cin][rows] and,
// for the convolutions whose input gradient is a convolution, wgR [cin][tap reversed][rows].
// A block stages a tile of 32 rows x ~144 consecutive source columns in shared memory, so
// that the source is read once, in whole runs, and every copy is written in runs of the
// index that is contiguous in it (64 bytes where the rows are, 32 bytes or more else).
//
// Bound: 4 bytes read and 2 to 6 written per weight, 8.5 M weights in the ResNet agent
// (L2-resident after the optimizer). One launch per tensor and copy took 45 launches of 2-5
// us, 180 us in all; this one takes 24 us.
#include <algorithm>

#include "nn_kernels.cuh"

namespace ddppo {

namespace {

constexpr int WP_ROWS = 32, WP_COLS = 144, WP_THREADS = 256;

template <typename T> __device__ __forceinline__ T wp_cast(float v);
template <> __device__ __forceinline__ float wp_cast<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 wp_cast<__nv_bfloat16>(float v) {
  return __float2bfloat16_rn(v);
}

// input channels per tile (whole taps), or 0: tiles cut the taps too
__host__ __device__ __forceinline__ int wp_ci(int kk) {
  if (kk > WP_COLS) return 0;
  const int c = WP_COLS / kk;
  return c >= 8 ? c / 8 * 8 : c;
}

template <typename T>
__global__ void __launch_bounds__(WP_THREADS) weight_prep_kernel(const WPrep* __restrict__ table,
                                                                 const uint16_t* __restrict__ entry,
                                                                 const float* __restrict__ params) {
  DDPPO_PDL_ENTRY();
  __shared__ float tile[WP_ROWS][WP_COLS + 1];
  const WPrep e = table[entry[blockIdx.x]];
  const int b = (int)blockIdx.x - e.first;
  if (e.kk == 0) {  // element-wise sum of two vectors (the LSTM's biases), kept in fp32
    const int i = b * WP_THREADS + threadIdx.x;
    if (i < e.rows) ((float*)e.wg)[i] = params[e.src + i] + params[e.src2 + i];
    return;
  }
  const int L = e.cin * e.kk, ci = wp_ci(e.kk), step = ci ? ci * e.kk : WP_COLS;
  const int ntc = (L + step - 1) / step;
  const int r0 = (b / ntc) * WP_ROWS, j0 = (b % ntc) * step;
  const int W = min(step, L - j0), R = min(WP_ROWS, e.rows - r0);
  // where the tile's columns go, once per block: column q of wg's order (input channel
  // fastest) reads tile column s_col and goes to row offset s_wg; source column q goes to
  // row s_t of wgT and s_r of wgR
  __shared__ int s_col[WP_COLS], s_wg[WP_COLS], s_t[WP_COLS], s_r[WP_COLS];
  if (threadIdx.x < W) {
    const int q = threadIdx.x, c = (j0 + q) / e.kk, tap = j0 + q - c * e.kk;
    s_t[q] = tap * e.cin + c;
    s_r[q] = c * e.kk + (e.kk - 1 - tap);
    if (ci) {
      const int cn = W / e.kk, t2 = q / cn, c2 = q - t2 * cn;
      s_col[q] = c2 * e.kk + t2;
      s_wg[q] = t2 * e.cin + j0 / e.kk + c2;
    } else {
      s_col[q] = q;
      s_wg[q] = s_t[q];
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NW = WP_THREADS / 32;
  const float* src = params + e.src + (size_t)r0 * L + j0;
#pragma unroll
  for (int r = warp; r < WP_ROWS; r += NW)
#pragma unroll
    for (int c = lane; c < WP_COLS; c += 32)
      if (r < R && c < W) tile[r][c] = src[(size_t)r * L + c];
  __syncthreads();
  T* wg = (T*)e.wg + (size_t)r0 * e.ld;
#pragma unroll
  for (int c = lane; c < WP_COLS; c += 32) {
    if (c >= W) break;
    const int col = s_col[c], o = s_wg[c];
#pragma unroll
    for (int r = warp; r < WP_ROWS; r += NW)
      if (r < R) wg[(size_t)r * e.ld + o] = wp_cast<T>(tile[r][col]);
  }
  T* wgT = (T*)e.wgT;
  T* wgR = (T*)e.wgR;
  if ((!wgT && !wgR) || lane >= R) return;
#pragma unroll 6
  for (int q = warp; q < W; q += NW) {
    const T v = wp_cast<T>(tile[lane][q]);
    if (wgT) wgT[(size_t)s_t[q] * e.rows + r0 + lane] = v;
    if (wgR) wgR[(size_t)s_r[q] * e.rows + r0 + lane] = v;
  }
}

}  // namespace

int weight_prep_blocks(const WPrep& e) {
  if (e.kk == 0) return (e.rows + WP_THREADS - 1) / WP_THREADS;
  const int L = e.cin * e.kk, ci = wp_ci(e.kk), step = ci ? ci * e.kk : WP_COLS;
  return (e.rows + WP_ROWS - 1) / WP_ROWS * ((L + step - 1) / step);
}

int launch_weight_prep(const WPrep* table, const uint16_t* entry, int blocks, const float* params,
                       bool op_bf16, cudaStream_t s) {
  if (!blocks) return DDPPO_OK;
  if (op_bf16)
    ::ddppo::launch_k(weight_prep_kernel<__nv_bfloat16>, blocks, WP_THREADS, 0, s, table, entry, params);
  else
    ::ddppo::launch_k(weight_prep_kernel<float>, blocks, WP_THREADS, 0, s, table, entry, params);
  DDPPO_CHECK_LAUNCH();
  return DDPPO_OK;
}

}  // namespace ddppo
