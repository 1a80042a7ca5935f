// Element-wise tick kernels (loss, activation backward) and the fp32 SIMT grouped GEMMs.
//
// Every kernel is "grouped": blockIdx.z (or .y) selects the stage, the per-tick table says
// whether that stage is active and which ring slots it touches.  Within a tick the stages
// only read what earlier ticks left in their rings and mailboxes, so one launch covers all.
#include <algorithm>

#include "pm_tick.cuh"

namespace pm {

template <typename AT> __device__ __forceinline__ AT* ring_ptr(const TickArgs& t, uint64_t off, int slot, uint64_t slot_elems) {
  return ring_at<AT>(t, off, slot, slot_elems);
}
template <typename AT> __device__ __forceinline__ AT* ws_ptr(const TickArgs& t, uint64_t off) { return ws_at<AT>(t, off); }

// ---- MSE loss at the last stage ------------------------------------------------------------------
// loss = mean over T*out of (y - y*)^2 ;  dy = 2 (y - y*) / (T*out), stored in the activation type.
// Fixed summation order: each block sums a contiguous chunk (strided per-thread partials, fixed tree), the last block to
// finish adds the per-block partials: 32 lanes every 32nd of them, then a tree over the lanes.
constexpr int kLossBlocks = 96, kLossThreads = 256;     // partial sums and the counter share a 512-byte block of the workspace

template <typename AT>
__global__ void __launch_bounds__(kLossThreads) mse_loss_kernel(TickArgs t) {
  pdl_trigger();
  pdl_wait();
  const StageDyn& d = t.dyn[t.P - 1];
  if (d.b_mb < 0) return;
  const StageDev& sl = t.st[t.P - 1];
  const uint64_t n = (uint64_t)t.T * t.n_out_last;
  const int par = (int)((d.tick + 1) & 1);            // written during the previous tick
  const AT* y = ws_ptr<AT>(t, t.yout_off) + (uint64_t)par * n;
  const float* tg = ws_ptr<float>(t, t.tgt_off) + (uint64_t)(d.b_mb % (t.P + 1)) * n;
  AT* dy = gin_read<AT>(t, sl, d);
  float* partial = ws_ptr<float>(t, t.lossred_off);
  unsigned int* counter = reinterpret_cast<unsigned int*>(partial + kLossBlocks);
  const float scale = (float)(2.0 / (double)n * (double)t.loss_scale);
  const LinDev& Ll = sl.lin[sl.n_lin - 1];
  const int act = (Ll.flags & LF_DZ_FUSED) ? Ll.act : PM_ACT_NONE;       // the last Linear receives dz itself
  const AT* z = act != PM_ACT_NONE ? ring_ptr<AT>(t, Ll.z_ring, d.b_slot, n) : nullptr;
  const uint64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const uint64_t lo = (uint64_t)blockIdx.x * chunk, hi = lo + chunk < n ? lo + chunk : n;
  float part = 0.f;
#pragma unroll 4
  for (uint64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    float r = __fsub_rn(to_f<AT>(y[i]), tg[i]);
    part = __fadd_rn(part, __fmul_rn(r, r));
    AT g = from_f<AT>(__fmul_rn(scale, r));
    if (act != PM_ACT_NONE) g = from_f<AT>(__fmul_rn(to_f<AT>(g), act_grad(to_f<AT>(z[i]), act)));
    dy[i] = g;
  }
  __shared__ float red[kLossThreads];
  __shared__ bool last;
  red[threadIdx.x] = part;
  __syncthreads();
  for (int off = kLossThreads / 2; off > 0; off >>= 1) {
    if ((int)threadIdx.x < off) red[threadIdx.x] = __fadd_rn(red[threadIdx.x], red[threadIdx.x + off]);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = red[0];
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x < 32) {                     // lane l adds partials l, l + 32, l + 64, then a fixed tree
    __threadfence();
    float sum = 0.f;
#pragma unroll
    for (int b = 0; b < kLossBlocks / 32; ++b) sum = __fadd_rn(sum, __ldcg(partial + 32 * b + threadIdx.x));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum = __fadd_rn(sum, __shfl_xor_sync(0xffffffffu, sum, off));
    if (threadIdx.x == 0) {
      ws_ptr<float>(t, t.loss_off)[d.b_mb % t.loss_cap] = sum / (float)n;
      *counter = 0;                                   // ready for the next tick
    }
  }
}

cudaError_t launch_ce_loss(const TickArgs& t, int dtype, cudaStream_t stream);   // pm_xfmr.cu

cudaError_t launch_loss(const TickArgs& t, int dtype, cudaStream_t stream) {
  if (t.loss_kind == PM_LOSS_CE) return launch_ce_loss(t, dtype, stream);
  return launch_pdl(dtype == PM_F32 ? mse_loss_kernel<float> : mse_loss_kernel<__nv_bfloat16>, dim3(kLossBlocks), dim3(kLossThreads), 0, stream, t.pdl, t);
}

// ---- activation backward ---------------------------------------------------------------------------
// dz = dy * act'(z), stored in the activation type (the bias gradient, its column sums, comes from the weight-gradient GEMM).
// A block owns 256 columns, or 32 of a microbatch of up to kActSmallRows rows; eight columns per lane, a lane has four rows in
// flight.  Bounded by latency for short microbatches, by HBM for long ones.

// rows r, r + step, ... < r1 of 8 columns: N of them are loaded before the first is used (no branch between the loads: the
// compiler would wait for each)
template <typename AT, int ACT, int N>
__device__ __forceinline__ void actbwd_rows_n(const AT* __restrict__ dy, const AT* __restrict__ z, AT* __restrict__ dz, int n_out, int c, int r, int step) {
  float g[N][8], zz[N][8];
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const uint64_t i = (uint64_t)(r + u * step) * n_out + c;
    load8<AT>(dy + i, g[u]);
    load8<AT>(z + i, zz[u]);
  }
#pragma unroll
  for (int u = 0; u < N; ++u) {
#pragma unroll
    for (int k = 0; k < 8; ++k) g[u][k] = round_as<AT>(__fmul_rn(g[u][k], act_grad(zz[u][k], ACT)));
    store8<AT>(dz + (uint64_t)(r + u * step) * n_out + c, g[u]);
  }
}
template <typename AT, int ACT>
__device__ __forceinline__ void actbwd_rows(const AT* __restrict__ dy, const AT* __restrict__ z, AT* __restrict__ dz, int n_out, int c, int r, int step, int r1) {
  for (; r + 3 * step < r1; r += 4 * step) actbwd_rows_n<AT, ACT, 4>(dy, z, dz, n_out, c, r, step);
  if (r + step < r1) { actbwd_rows_n<AT, ACT, 2>(dy, z, dz, n_out, c, r, step); r += 2 * step; }
  if (r < r1) actbwd_rows_n<AT, ACT, 1>(dy, z, dz, n_out, c, r, step);
}

// rows a block of the launch covers: all of a short microbatch; in a launch of one stage few enough for several blocks per SM; more where
// the grid's second dimension, at most 65535, would not reach the last row
__host__ __device__ inline int act_block_rows(const TickArgs& t) {
  int rows = t.T <= kActSmallRows ? t.T : (t.sel_p >= 0 ? 64 : 256);
  while (((int64_t)t.T + rows - 1) / rows > 65535) rows *= 2;
  return rows;
}

template <typename AT>
__global__ void __launch_bounds__(256) actbwd_kernel(TickArgs t, int lvl) {
  pdl_trigger();
  pdl_wait();
  const int* start = t.act_start + (size_t)lvl * (t.P + 1);
  int lo = 0, hi = t.P - 1;                                 // stage of this column block: largest p with start[p] <= its index
  const int blk = (int)blockIdx.x + t.act_first[lvl];
  if (t.sel_p >= 0) lo = hi = t.sel_p;                     // a launch of one stage: no search
  while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (start[mid] <= blk) lo = mid; else hi = mid - 1; }
  const int p = lo;
  const StageDyn& d = t.dyn[p];
  const StageDev& s = t.st[p];
  if (d.b_mb < 0 || lvl >= s.n_lin) return;
  const LinDev& L = s.lin[lvl];
  if (bwd_act(L) == PM_ACT_NONE) return;                    // without an activation (or with one applied upstream) dz = dy
  const bool small = t.T <= kActSmallRows;
  const int cols = small ? kActSmallCols : kActCols;
  const int c0 = (blk - start[p]) * cols;
  if (c0 >= L.n_out) return;
  const int rows = act_block_rows(t), r0 = (int)blockIdx.y * rows, r1 = r0 + min(t.T - r0, rows);
  const uint64_t n = (uint64_t)t.T * L.n_out;
  const AT* dy = (lvl < s.n_lin - 1) ? ws_ptr<AT>(t, L.dy_off) : (feeds_attention(s.post) ? ws_ptr<AT>(t, s.dy) : gin_read<AT>(t, s, d));
  // the pre-activation stash, or for a ReLU without one the stashed output (same sign pattern)
  const AT* z = !(L.flags & LF_ACT_FROM_Y) ? ring_ptr<AT>(t, L.z_ring, d.b_slot, n)
                : (lvl < s.n_lin - 1 ? ring_ptr<AT>(t, L.h_ring, d.b_slot, n) : ring_ptr<AT>(t, t.st[p + 1].x_ring, d.b_next_xslot, n));
  AT* dz = ws_ptr<AT>(t, L.dz_off);
  if ((L.n_out & 7) == 0) {                                 // vector path needs 8-element alignment of every row
    const int per = cols / 8, c = c0 + 8 * (int)(threadIdx.x % per), r = r0 + (int)(threadIdx.x / per), step = 256 / per;
    if (c >= L.n_out) return;
    if (L.act == PM_ACT_RELU) actbwd_rows<AT, PM_ACT_RELU>(dy, z, dz, L.n_out, c, r, step, r1);
    else actbwd_rows<AT, PM_ACT_GELU>(dy, z, dz, L.n_out, c, r, step, r1);
  } else {                                                  // fp32 only: bf16 Linears have widths that are multiples of 8
    const int c1 = min(L.n_out, c0 + cols), w = c1 - c0;
    for (int o = (int)threadIdx.x; o < w * (r1 - r0); o += 256) {
      const uint64_t i = (uint64_t)(r0 + o / w) * L.n_out + c0 + o % w;
      dz[i] = from_f<AT>(round_as<AT>(__fmul_rn(to_f<AT>(dy[i]), act_grad(to_f<AT>(z[i]), L.act))));
    }
  }
}

cudaError_t launch_actbwd(const TickArgs& t, int dtype, int lvl, cudaStream_t stream) {
  if (t.act_blocks[lvl] == 0) return cudaSuccess;
  const int rows = act_block_rows(t);
  return launch_pdl(dtype == PM_F32 ? actbwd_kernel<float> : actbwd_kernel<__nv_bfloat16>, dim3(t.act_blocks[lvl], (t.T + rows - 1) / rows), dim3(256), 0, stream, t.pdl, t, lvl);
}

// ---- bias gradient of networks with a fused update ------------------------------------------------------
// Their weight-gradient GEMMs, which sum the columns of dz elsewhere, run in the update phase, and the bias gradients belong to the
// backward phase.  The additions and their order are those of the GEMM's summing warps (pm_umma.cu), so that a fused run keeps the bits of
// one that is not: per column eight row groups (rows rho + 8 j of every 64), eight rows pairwise, the 64-row blocks one after the other, the
// groups pairwise.  A block owns 32 columns; its warps form the sums of eight 64-row blocks side by side (8 KB of shared memory,
// two buffers), 256 threads add them to (row group, column).  Bound by the round trip per 512 rows, and in networks of many rows by
// the second pass over dz: a tick of the 6-layer encoder with a fused update takes 1081 us (1007 with the sums in the GEMM, 1385 with
// the column sums before those), an update of the encoder-decoder of 2 + 2 layers of width 1024 4278 (4226, 5367).
constexpr int kBgCols = 32;
__global__ void __launch_bounds__(256) bias_grad_kernel(TickArgs t, int lvl, int per) {
  pdl_trigger();
  pdl_wait();
  const int* start = t.act_start + (size_t)lvl * (t.P + 1);
  const int blk = (int)blockIdx.x / per;                    // entry of the list of column blocks, `per` of these blocks each
  int lo = 0, hi = t.P - 1;
  while (lo < hi) { const int mid = (lo + hi + 1) >> 1; if (start[mid] <= blk) lo = mid; else hi = mid - 1; }
  const StageDyn& d = t.dyn[lo];
  const StageDev& s = t.st[lo];
  if (d.b_mb < 0 || lvl >= s.n_lin) return;
  const LinDev& L = s.lin[lvl];
  const int c0 = ((blk - start[lo]) * per + (int)blockIdx.x % per) * kBgCols;
  if (c0 >= L.n_out) return;
  __shared__ float part[2][8][8][kBgCols];                  // [buffer][64-row block][row group][column]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rho = lane >> 2, c = c0 + 8 * (lane & 3);
  const __nv_bfloat16* dz = dz_src<__nv_bfloat16>(t, s, d, lvl) + (c < L.n_out ? c : 0);   // (widths are multiples of 8)
  const int n_kb = (t.T + 63) / 64;
  const int g = (int)threadIdx.x >> 5, col = (int)threadIdx.x & 31;
  float acc = 0.f;
  for (int kb0 = 0, buf = 0; kb0 < n_kb; kb0 += 8, buf ^= 1) {
    const int row = (kb0 + warp) * 64 + rho;
    float v[8][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) load8<__nv_bfloat16>(dz + (uint64_t)min(row + 8 * j, t.T - 1) * L.n_out, v[j]);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (row + 8 * j >= t.T)
#pragma unroll
        for (int e = 0; e < 8; ++e) v[j][e] = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      part[buf][warp][rho][8 * (lane & 3) + e] = __fadd_rn(__fadd_rn(__fadd_rn(v[0][e], v[1][e]), __fadd_rn(v[2][e], v[3][e])),
                                                           __fadd_rn(__fadd_rn(v[4][e], v[5][e]), __fadd_rn(v[6][e], v[7][e])));
    __syncthreads();                                        // (the other buffer is written next: one barrier per step is enough)
#pragma unroll
    for (int k = 0; k < 8; ++k) if (kb0 + k < n_kb) acc = __fadd_rn(acc, part[buf][k][g][col]);
  }
  __shared__ float fin[8][kBgCols];
  fin[g][col] = acc;
  __syncthreads();
  if (g == 0 && c0 + col < L.n_out) {
    auto two = [&](int a, int b) { return __fadd_rn(fin[a][col], fin[b][col]); };
    const float sum = __fadd_rn(__fadd_rn(two(0, 4), two(1, 5)), __fadd_rn(two(2, 6), two(3, 7)));
    t.a.grad[L.b_off + c0 + col] = d.accum ? __fadd_rn(t.a.grad[L.b_off + c0 + col], sum) : sum;
  }
}

cudaError_t launch_bias_grad(const TickArgs& t, int lvl, cudaStream_t stream) {
  const int per = act_cols((uint64_t)t.T) / kBgCols;
  return launch_pdl(bias_grad_kernel, dim3((unsigned)(t.act_blocks[lvl] * per)), dim3(256), 0, stream, t.pdl, t, lvl, per);
}

// ---- fp32 SIMT grouped GEMM ------------------------------------------------------------------------
// C[M,N] = sum_k A(m,k) B(k,n) with fused multiply-adds in fp32.
//   mode 0 forward:  A = x [T,in],        B(k,n) = W[n,k]            -> z = C + b, y = act(z)
//   mode 1 dgrad:    A = dz [T,out],      B(k,n) = W[k,n]-gap*delta  -> dx = C, times act'(z) of the Linear that receives it
//   mode 2 wgrad:    A(m,k) = dz[k,m],    B(k,n) = x[k,n]            -> dW = C; db = the row sums of A (the bias gradient
//                    without a launch of its own)
// What bounds it: latency.  The fp32 workloads have a few hundred rows and columns and a reduction of as many, so a
// launch is a handful of loads deep; a k loop that loads, synchronises and multiplies in turn paid one L2 round trip
// per 16 k.  Here the eight warps of a block split the reduction: warp w owns the 16-deep k chunks w, w + 8, ..., brings
// them into its own part of shared memory with asynchronous copies (kF32Buf chunks ahead, so a reduction of up to
// 16 * 8 * kF32Buf is in flight at once) and multiplies without any block-wide barrier; the eight partial tiles are added
// pairwise at the end.  Warp tile (4 TM) x (8 TN), TM x TN outputs per lane.  Measured against a 64 x 64 tile with a
// serial k loop: a tick of the 4-stage 256-wide MLP at 32 rows 87.6 -> 44.4 us, an update of the 6-stage 200-wide MLP (two
// Linears per stage, two microbatches of 50 rows, microbatch-major order) 1483 -> 562 us.
constexpr int kF32KC = 16;

template <int TM, int TN, int NBUF, int MODE> struct F32Cfg {
  static constexpr int BM = 4 * TM, BN = 8 * TN;
  // k-contiguous operands keep rows of 16 k (stride 20: the eight rows a quarter-warp reads fall into distinct banks),
  // the others rows of BM / BN columns
  static constexpr int kA = MODE == 2 ? kF32KC * (BM + 4) : BM * (kF32KC + 4);
  static constexpr int kB = MODE == 0 ? BN * (kF32KC + 4) : kF32KC * (BN + 4);
  static constexpr int kBuf = kA + kB * (MODE == 1 ? 2 : 1);                     // mode 1: w and delta
  static constexpr int kPanels = 8 * NBUF * kBuf;
  static constexpr int kRed = 8 * BM * (BN + 4) + (MODE == 2 ? 8 * BM : 0);      // partial tiles; mode 2: partial row sums of A
  static constexpr int kBytes = 4 * (kPanels > kRed ? kPanels : kRed);
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" :: "r"(dst), "l"(src), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" :: "r"(dst), "l"(src), "r"(on ? 4 : 0) : "memory");
}

// R rows (r0 .. of n_rows) x 16 k (k0 .. of K) of a matrix with k contiguous -> dst[r][k], stride 20; zeros outside
template <int R>
__device__ __forceinline__ void f32_load_kc(float* dst, const float* __restrict__ src, int ld, int r0, int n_rows, int k0, int K, bool vec, int lane) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if (vec) {
#pragma unroll
    for (int f = lane; f < R * 4; f += 32) {
      const int r = f >> 2, q = (f & 3) * 4;
      const bool on = r0 + r < n_rows && k0 + q < K;
      cp_async16(d + 4u * (uint32_t)(r * (kF32KC + 4) + q), on ? src + (uint64_t)(r0 + r) * ld + k0 + q : src, on);
    }
  } else {
    for (int f = lane; f < R * kF32KC; f += 32) {
      const int r = f >> 4, k = f & 15;
      const bool on = r0 + r < n_rows && k0 + k < K;
      cp_async4(d + 4u * (uint32_t)(r * (kF32KC + 4) + k), on ? src + (uint64_t)(r0 + r) * ld + k0 + k : src, on);
    }
  }
}
// 16 k (k0 .. of K) x R columns (c0 .. of n_cols) of a matrix with columns contiguous -> dst[k][c], stride R + 4
template <int R>
__device__ __forceinline__ void f32_load_nc(float* dst, const float* __restrict__ src, int ld, int c0, int n_cols, int k0, int K, bool vec, int lane) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if (vec) {
#pragma unroll
    for (int f = lane; f < kF32KC * (R / 4); f += 32) {
      const int k = f / (R / 4), c = (f % (R / 4)) * 4;
      const bool on = c0 + c < n_cols && k0 + k < K;
      cp_async16(d + 4u * (uint32_t)(k * (R + 4) + c), on ? src + (uint64_t)(k0 + k) * ld + c0 + c : src, on);
    }
  } else {
    for (int f = lane; f < kF32KC * R; f += 32) {
      const int k = f / R, c = f % R;
      const bool on = c0 + c < n_cols && k0 + k < K;
      cp_async4(d + 4u * (uint32_t)(k * (R + 4) + c), on ? src + (uint64_t)(k0 + k) * ld + c0 + c : src, on);
    }
  }
}

// the eight warps' partial sums, pairwise: three roundings per term instead of seven
__device__ __forceinline__ float f32_sum8(const float* p, int stride) {
  const float a = __fadd_rn(__fadd_rn(p[0], p[stride]), __fadd_rn(p[2 * stride], p[3 * stride]));
  const float b = __fadd_rn(__fadd_rn(p[4 * stride], p[5 * stride]), __fadd_rn(p[6 * stride], p[7 * stride]));
  return __fadd_rn(a, b);
}

template <int TM, int TN, int NBUF, int MODE>
__global__ void __launch_bounds__(256, 2) f32_gemm_kernel(TickArgs t, int lvl) {
  using C = F32Cfg<TM, TN, NBUF, MODE>;
  constexpr int BM = C::BM, BN = C::BN, KC = kF32KC;
  pdl_trigger();
  const int p = stage_of_block(t, blockIdx.y);
  const StageDyn& d = t.dyn[p];
  const StageDev& s = t.st[p];
  const LinDev& L = s.lin[lvl < s.n_lin ? lvl : 0];
  const int T = t.T;
  const int M = MODE == 2 ? L.n_out : T, N = MODE == 0 ? L.n_out : L.n_in, K = MODE == 0 ? L.n_in : (MODE == 1 ? L.n_out : T);
  const unsigned tiles_n = (unsigned)(N + BN - 1) / BN;      // the grid holds the tiles of the launch's largest Linear
  const int m0 = (int)(blockIdx.x / tiles_n) * BM, n0 = (int)(blockIdx.x % tiles_n) * BN;
  if (lvl >= s.n_lin || (MODE == 0 ? d.f_mb < 0 : d.b_mb < 0) || m0 >= M || n0 >= N ||
      (MODE == 1 && p == 0 && lvl == 0 && s.pre != PRE_EMBED)) {          // raw network inputs need no gradient
    pdl_wait();
    return;
  }

  // operand sources
  const float* asrc = MODE == 0 ? lin_input<float>(t, s, d, lvl, true) : dz_src<float>(t, s, d, lvl);
  const float* wf = fwd_weights<float>(t, s, d, L.w_off);  // forward operand: the weights of the version the forward reads
  // dgrad: w - gap * delta formed here, or (weight stashing, written-out corrected weights) the queued version as it is
  const bool corr = MODE == 1 && !t.stash && d.use_delta != 0;
  const float* bsrc = MODE == 0 ? wf : (MODE == 1 ? (t.stash ? wf : t.a.w + L.w_off) : lin_input<float>(t, s, d, lvl, false));
  const float* dl = t.a.delta + L.w_off;
  const int lda = MODE == 0 ? L.n_in : L.n_out, ldb = L.n_in;
  const bool va = (lda & 3) == 0, vb = (ldb & 3) == 0;     // 16-byte copies need rows that start on 16 bytes
  const float gapf = (float)s.gap;

  extern __shared__ __align__(16) float f32_sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, tx = lane & 7, ty = lane >> 3;
  float* mine = f32_sm + warp * NBUF * C::kBuf;
  const int chunks = (K + KC - 1) / KC;
  auto load_b = [&](int c, float* buf) {
    if (c >= chunks) return;
    if (MODE == 0) f32_load_kc<BN>(buf + C::kA, bsrc, ldb, n0, N, c * KC, K, vb, lane);
    else f32_load_nc<BN>(buf + C::kA, bsrc, ldb, n0, N, c * KC, K, vb, lane);
    if (corr) f32_load_nc<BN>(buf + C::kA + C::kB, dl, ldb, n0, N, c * KC, K, vb, lane);
  };
  auto load_a = [&](int c, float* buf) {                   // closes the chunk's group of copies
    if (c < chunks) {
      if (MODE == 2) f32_load_nc<BM>(buf, asrc, lda, m0, M, c * KC, K, va, lane);
      else f32_load_kc<BM>(buf, asrc, lda, m0, M, c * KC, K, va, lane);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;
  float rows[TM];                                          // mode 2, first column of tiles: row sums of A over this warp's k
#pragma unroll
  for (int i = 0; i < TM; ++i) rows[i] = 0.f;
  const bool bias_tile = MODE == 2 && n0 == 0;

  // weights and delta are written by no launch of this phase: their copies start before the predecessor has ended
  if (MODE == 2) pdl_wait();
#pragma unroll
  for (int b = 0; b < NBUF; ++b) load_b(warp + 8 * b, mine + b * C::kBuf);
  if (MODE != 2) pdl_wait();
#pragma unroll
  for (int b = 0; b < NBUF; ++b) load_a(warp + 8 * b, mine + b * C::kBuf);
  int slot = 0;
  for (int c = warp; c < chunks; c += 8) {
    asm volatile("cp.async.wait_group %0;" :: "n"(NBUF - 1) : "memory");
    __syncwarp();
    float* buf = mine + slot * C::kBuf;
    float* pb = buf + C::kA;
    if (corr) {                                            // T2: w - (tau_fwd - tau_bkwd) * delta
#pragma unroll
      for (int f = lane; f < KC * (BN / 4); f += 32) {
        const int o = (f / (BN / 4)) * (BN + 4) + (f % (BN / 4)) * 4;
        float4 w4 = *reinterpret_cast<float4*>(pb + o);
        const float4 d4 = *reinterpret_cast<const float4*>(pb + C::kB + o);
        w4.x = __fsub_rn(w4.x, __fmul_rn(gapf, d4.x)); w4.y = __fsub_rn(w4.y, __fmul_rn(gapf, d4.y));
        w4.z = __fsub_rn(w4.z, __fmul_rn(gapf, d4.z)); w4.w = __fsub_rn(w4.w, __fmul_rn(gapf, d4.w));
        *reinterpret_cast<float4*>(pb + o) = w4;
      }
      __syncwarp();
    }
#pragma unroll
    for (int k = 0; k < KC; k += 4) {
      float av[TM][4], bv[TN][4];                          // [row or column of this lane][k]
      if (MODE == 2) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int i = 0; i < TM; i += 4) {
            const float4 v = *reinterpret_cast<const float4*>(buf + (k + kk) * (BM + 4) + ty * TM + i);
            av[i][kk] = v.x; av[i + 1][kk] = v.y; av[i + 2][kk] = v.z; av[i + 3][kk] = v.w;
          }
      } else {
#pragma unroll
        for (int i = 0; i < TM; ++i) *reinterpret_cast<float4*>(av[i]) = *reinterpret_cast<const float4*>(buf + (ty + 4 * i) * (KC + 4) + k);
      }
      if (MODE == 0) {
#pragma unroll
        for (int j = 0; j < TN; ++j) *reinterpret_cast<float4*>(bv[j]) = *reinterpret_cast<const float4*>(pb + (tx + 8 * j) * (KC + 4) + k);
      } else {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int j = 0; j < TN; j += 2) {
            const float2 v = *reinterpret_cast<const float2*>(pb + (k + kk) * (BN + 4) + tx * TN + j);
            bv[j][kk] = v.x; bv[j + 1][kk] = v.y;
          }
      }
      if (bias_tile) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int i = 0; i < TM; ++i) rows[i] = __fadd_rn(rows[i], av[i][kk]);
      }
      // four products first, then one addition to the running sum: a quarter as many roundings at the size of the sum
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j)
          acc[i][j] = __fadd_rn(acc[i][j], fmaf(av[i][3], bv[j][3], fmaf(av[i][2], bv[j][2], fmaf(av[i][1], bv[j][1], __fmul_rn(av[i][0], bv[j][0])))));
    }
    __syncwarp();
    load_b(c + 8 * NBUF, buf);
    load_a(c + 8 * NBUF, buf);
    if (++slot == NBUF) slot = 0;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();                                         // the panels become the partial tiles
  {
    float* red = f32_sm + warp * BM * (BN + 4);
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int m = MODE == 2 ? ty * TM + i : ty + 4 * i, n = MODE == 0 ? tx + 8 * j : tx * TN + j;
        red[m * (BN + 4) + n] = acc[i][j];
      }
    if (bias_tile && tx == 0)
#pragma unroll
      for (int i = 0; i < TM; ++i) f32_sm[8 * BM * (BN + 4) + warp * BM + ty * TM + i] = rows[i];
  }
  __syncthreads();
  if (bias_tile && tid < BM && m0 + tid < M) {
    const float v = f32_sum8(f32_sm + 8 * BM * (BN + 4) + tid, BM);
    float* db = t.a.grad + L.b_off + m0 + tid;
    *db = d.accum ? __fadd_rn(*db, v) : v;
  }

  // epilogue: consecutive threads take consecutive columns of a row
  const uint64_t n_xout = (uint64_t)T * L.n_out;
  float* zout = MODE == 0 && (L.flags & LF_WRITE_Z) ? ring_ptr<float>(t, L.z_ring, d.f_slot, n_xout) : nullptr;
  float* yout = MODE == 0 ? y_dest<float>(t, p, s, d, lvl) : nullptr;
  float* lout = MODE == 0 && (L.flags & LF_OUT_F32) ? ws_ptr<float>(t, t.yout_off) + (uint64_t)(d.tick & 1) * n_xout : nullptr;
  const float* bias = fwd_small<float>(t, s, d, L.b_off, L.b_soff);
  float* dx = MODE == 1 ? dx_dest<float>(t, p, s, d, lvl) : nullptr;
  const float* z = nullptr;
  const int dact = MODE == 1 ? dx_fused_act<float>(t, p, s, d, lvl, &z) : PM_ACT_NONE;
  float* dW = t.a.grad + L.w_off;
#pragma unroll
  for (int o = tid; o < BM * BN; o += 256) {
    const int r = o / BN, c = o % BN, m = m0 + r, n = n0 + c;
    float v = f32_sum8(f32_sm + r * (BN + 4) + c, BM * (BN + 4));
    if (m >= M || n >= N) continue;
    const uint64_t i = (uint64_t)m * N + n;
    if (MODE == 0) {
      v = __fadd_rn(v, bias[n]);
      if (lout) lout[i] = v;
      if (zout) zout[i] = v;
      if (yout) yout[i] = act_fwd(v, L.act);
    } else if (MODE == 1) dx[i] = dact != PM_ACT_NONE ? __fmul_rn(v, act_grad(z[i], dact)) : v;
    else dW[i] = d.accum ? __fadd_rn(dW[i], v) : v;
  }
}

template <int TM, int TN, int NBUF, int MODE>
static cudaError_t launch_f32_t(const TickArgs& t, int lvl, uint64_t tiles, cudaStream_t stream) {
  using C = F32Cfg<TM, TN, NBUF, MODE>;
  return launch_pdl(f32_gemm_kernel<TM, TN, NBUF, MODE>, dim3((unsigned)tiles, t.sel_p >= 0 ? 1 : t.P), dim3(256), C::kBytes, stream, t.pdl, t, lvl);
}

// The instances: small tiles with one chunk per warp in flight, two, or the most that leave two blocks on an SM; large tiles with one or two.
#define PM_F32_INSTANCES(X) X(4, 2, 1, 0) X(4, 2, 2, 0) X(4, 2, 4, 0) X(4, 2, 1, 1) X(4, 2, 2, 1) X(4, 2, 3, 1) X(4, 2, 1, 2) X(4, 2, 2, 2) X(4, 2, 4, 2) \
                            X(8, 4, 1, 0) X(8, 4, 2, 0) X(8, 4, 1, 1) X(8, 4, 2, 1) X(8, 4, 1, 2) X(8, 4, 2, 2)

// opt-in shared-memory sizes, on the current device
cudaError_t simt_gemm_set_limits() {
  cudaError_t e = cudaSuccess;
#define PM_F32_LIMIT(TM, TN, NB, MODE) if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)f32_gemm_kernel<TM, TN, NB, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, F32Cfg<TM, TN, NB, MODE>::kBytes);
  PM_F32_INSTANCES(PM_F32_LIMIT)
#undef PM_F32_LIMIT
  return e;
}

// 16 x 16 tiles while the 32 x 32 ones of all stages of the launch would number no more than the SMs: a smaller tile has a
// quarter of the multiplies on its critical path and the chip is not full anyway.
// Tiles are counted over the launch's own Linears.  (Sized by the widest Linear of the network, the launches of a network with a
// large vocabulary were mostly blocks without a tile: a tick of a 6-layer encoder of width 64, 64 rows and a vocabulary of
// 8000 took 2368 us and takes 211, of a 2-layer one of width 64, 384 rows and a vocabulary of 1000 165 and 152.)
// A warp has at most as many chunks of the reduction in flight as it owns (one in eight): a panel it never fills is shared memory
// that the blocks of the launches beside it could use.  (A tick of the 4-stage MLP, whose forward, input and weight gradients run side
// by side, 33.0 -> 31.9 us.)
cudaError_t launch_simt_gemm(const TickArgs& t, const std::vector<StageDev>& st, int mode, int lvl, cudaStream_t stream) {
  uint64_t all32 = 0, most32 = 1, most16 = 1;
  int chunks = 1;                                          // of the deepest reduction, per warp
  for (int p = t.sel_p >= 0 ? t.sel_p : 0; p < (t.sel_p >= 0 ? t.sel_p + 1 : t.P); ++p) {
    if (lvl >= st[p].n_lin || (mode == 1 && p == 0 && lvl == 0 && st[p].pre != PRE_EMBED)) continue;
    const LinDev& L = st[p].lin[lvl];
    const uint64_t M = mode == 2 ? L.n_out : t.T, N = mode == 0 ? L.n_out : L.n_in;
    const int K = mode == 2 ? t.T : (mode == 0 ? L.n_in : L.n_out);
    const uint64_t n32 = ((M + 31) / 32) * ((N + 31) / 32);
    all32 += n32;
    most32 = std::max(most32, n32);
    most16 = std::max(most16, ((M + 15) / 16) * ((N + 15) / 16));
    chunks = std::max(chunks, (K + 8 * kF32KC - 1) / (8 * kF32KC));
  }
  const bool small = all32 <= kSms;
  const int tm = small ? 4 : 8, nb = chunks <= 2 ? chunks : (small ? (mode == 1 ? 3 : 4) : 2);
#define PM_F32_LAUNCH(TM, TN, NB, MODE) if (tm == TM && nb == NB && mode == MODE) return launch_f32_t<TM, TN, NB, MODE>(t, lvl, small ? most16 : most32, stream);
  PM_F32_INSTANCES(PM_F32_LAUNCH)
#undef PM_F32_LAUNCH
  return cudaErrorInvalidValue;
}

}  // namespace pm
