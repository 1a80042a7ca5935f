// bf16 grouped GEMMs of the pipeline on the 5th-generation tensor cores.
//
// One launch covers every stage that is active in this tick.  The kernel is persistent: one CTA per SM
// walks a flattened list of 128x128 output tiles (stage, row tile, column tile).  Operands are staged in
// shared memory in the 128-byte-swizzled canonical layouts, the accumulators live in tensor memory
// (two buffers of 128 lanes x 128 fp32 columns, so the epilogue of one tile overlaps the main loop of
// the next), one elected thread issues tcgen05.mma, and eight warps drain the accumulators with
// tcgen05.ld.
//
//   mode 0 forward  D[T,out]  = x[T,in] * W[out,in]^T      A K-major (TMA), B K-major (TMA, bf16 shadow)
//                   z = bf16(D + b) -> ring,  y = bf16(act(z)) -> next consumer
//   mode 1 dgrad    D[T,in]   = dz[T,out] * Wc[out,in]     A K-major (TMA), B MN-major (TMA): a queued version of the weights, or
//                   the T2-corrected weights bf16(w - gap*delta) (Section 3.2).  Where a launch has fewer than 256 rows or columns,
//                   umma_dgrad_kernel forms those itself from the fp32 master weights and the accumulator delta
//   mode 2 wgrad    D[out,in] = dz[T,out]^T * x[T,in]      A MN-major (TMA), B MN-major (TMA), fp32 out
//
// Warp roles: warp 0 = TMA producer, warp 1 = MMA issuer + TMEM owner, (mode 2: warps 2..5 = column sums,) last eight warps =
// epilogue (two per TMEM lane group, each taking 64 of the 128 columns).
// Every wait on an mbarrier is bounded; on expiry the CTA records a code in a status word, stops
// issuing work, waits (bounded) for its copies in flight, frees its tensor memory and returns.
#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "pm_copy_parity.cuh"
#include "pm_ptx.cuh"
#include "pm_umma.cuh"
#include "pm_update_math.cuh"

namespace pm {

constexpr int TILE_M = 128, TILE_N = 128, TILE_K = 64;     // bf16: 64 elements = one 128-byte swizzle row
constexpr int A_BYTES = TILE_M * TILE_K * 2;               // 16 KB
constexpr int B_BYTES = TILE_N * TILE_K * 2;               // 16 KB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int STG_HALF_BYTES = TILE_K * TILE_N * 4;        // one fp32 [64 x 128] tile: 32 KB
constexpr int STG_BYTES = 2 * STG_HALF_BYTES;              // w tile + delta tile
constexpr int ACC_COLS = 128, TMEM_COLS = 2 * ACC_COLS;
constexpr int N_EPI_WARPS = 8;

// MODE 0 forward, 2 wgrad, 1 dgrad against a plain bf16 operand: a queued weight version (weight stashing, corrected weights that the update
// wrote out) or, on CTA pairs, the corrected weights in scratch.  Elsewhere umma_dgrad_kernel forms the corrected operand.  MODE 2: four warps sum the columns of dz, the bias gradient, from the A tiles in shared
// memory.  FUSE (MODE 2): the update is applied in the epilogue; the bias gradients belong to the backward phase (bias_grad_kernel).
template <int MODE, bool FUSE> struct Cfg {
  static constexpr int kStages = 4;                        // operand ring depth
  static constexpr int kSumWarps = MODE == 2 && !FUSE ? 4 : 0;
  static constexpr int kThreads = 32 * (2 + kSumWarps + N_EPI_WARPS);
  static constexpr int kOutWarpBytes = 8192;               // per epilogue warp: two boxes of 32 rows x 128 B
  static constexpr int kOutBytes = N_EPI_WARPS * kOutWarpBytes;
  static constexpr int kTileBytes = kStages * STAGE_BYTES + kOutBytes;
  static constexpr int kSmemBytes = kTileBytes + 1024 /*alignment slack*/ + 512 /*barriers*/;
};

enum { MAP_ACT_K = 0, MAP_W_K = 1, MAP_DZ_K = 2, MAP_DZ_MN = 3, MAP_ACT_MN = 4, MAP_W_F32 = 5, MAP_D_F32 = 6,
       MAP_Z_OUT = 7, MAP_Y_OUT = 8, MAP_DX_OUT = 9, MAP_DW_OUT = 10, MAP_W_MN = 11, MAP_W_K32 = 12, MAP_SKIP = 13, MAPS_PER_LINEAR = 14 };
}  // namespace pm
#include "pm_umma_row.cuh"     // the kernel of launches with few tiles; uses the tensor maps above
namespace pm {

// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = 128, operand majors as given.
__device__ __forceinline__ uint32_t make_idesc(int a_mn_major, int b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn_major << 15) | ((uint32_t)b_mn_major << 16) |
         ((uint32_t)(TILE_N >> 3) << 17) | ((uint32_t)(TILE_M >> 4) << 24);
}

// One epilogue warp's staging buffer: SLOTS boxes of 4 KB (32 rows of one 128-byte swizzle row), each its own TMA store.
template <int SLOTS>
struct EpiStage {
  uint8_t* buf; uint32_t buf_s; int lane;
  uint32_t bar;               // counts the skip tensor's copies into the box
  uint32_t off = 0;           // the box written next
  CopyParity copy{};          // of those copies
  bool stored = false;
  // the box's earlier store has finished reading it
  __device__ __forceinline__ uint8_t* begin() {
    if (lane == 0 && stored) { if (SLOTS == 1) tma_store_wait_read(); else tma_store_wait_read_1(); }
    __syncwarp();
    return buf + off;
  }
  template <class Store> __device__ __forceinline__ void end(Store store) {
    fence_async_smem();                                           // staging writes -> visible to the TMA engine
    __syncwarp();
    if (lane == 0) { store(buf_s + off); tma_store_commit(); }
    stored = true;
    if (SLOTS == 2) off ^= 4096u;
  }
  // a residual stage's unit: its block of the skip tensor comes into the box in the layout the sum leaves it in
  __device__ __forceinline__ void fetch(const CUtensorMap* map, int n, int m, int slot) {
    begin();
    if (lane == 0) { mbar_arrive_expect_tx(bar, 4096); tma_load_3d(buf_s + off, map, bar, n, m, slot); }
  }
  __device__ __forceinline__ bool fetched(volatile int* abort_flag, int* status) {
    return copy.await([&](uint32_t parity) { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status, 11)) != 0; });
  }
  // a CTA that gives up: the copy still lands here (bounded wait)
  __device__ __forceinline__ void drain() {
    const long long t0 = clock64();
    copy.drain([&](uint32_t parity) { return mbar_try_wait(bar, parity); }, [&] { return clock64() - t0 < WAIT_LIMIT_CYCLES; });
  }
};

// The PipeMare update of one 32-row x 32-column block of a Linear matrix, applied to the weight gradient while it is
// still on chip (r: the block's accumulators, lane = row).  The block goes through the warp's staging buffer
// once, in the layout the dW store uses, and comes back with a lane owning four consecutive columns of a row, so
// that every access to the master weights, the moments and delta is a full 128-byte line per eight lanes.  Per
// element the arithmetic is upd_one's, i.e. exactly what the stand-alone update kernel does with a stored gradient.
template <int OPT>
__device__ __forceinline__ void epi_update_block(const TickArgs& t, const StageDyn& d, const LinDev& L, int M, int N, int mrow, int nb,
                                                 const uint32_t (&r)[32], uint8_t* obuf, int lane) {
  const uint32_t row_off = (uint32_t)lane * 128, sw = (uint32_t)(lane & 7);
  __syncwarp();                                                   // the previous block's reads of the buffer are done
#pragma unroll
  for (int g = 0; g < 8; ++g)                                     // 16-byte chunks swizzled by row
    *reinterpret_cast<uint4*>(obuf + row_off + (((uint32_t)g ^ sw) << 4)) = make_uint4(r[g * 4], r[g * 4 + 1], r[g * 4 + 2], r[g * 4 + 3]);
  __syncwarp();
  UpdScalars sc;
  sc.alpha = d.alpha; sc.gamma = d.gamma; sc.omg = d.one_minus_gamma; sc.bc1 = d.bc1; sc.bc2 = d.bc2; sc.use_delta = d.use_delta;
  sc.lp_shift = d.lp_shift; sc.rc_shift = d.rc_uslot >= 0 ? d.rc_shift : -1; sc.rc_gap = d.rc_gap;
  const bool need_dl = sc.use_delta || sc.rc_shift >= 0;
  const float beta1 = t.upd_beta1, beta2 = t.upd_beta2, eps = t.upd_eps;
  const float omb1 = __fsub_rn(1.0f, beta1), omb2 = __fsub_rn(1.0f, beta2);
  const int rr0 = lane >> 3, ch = lane & 7;                       // row within a group of four, 16-byte chunk of the 32 columns
  constexpr int NB = 2;                                           // row groups whose loads are in flight together
#pragma unroll 1
  for (int it0 = 0; it0 < 8; it0 += NB) {                         // eight groups of four rows
    float4 g4[NB], w4[NB], m4[NB], s4[NB], d4[NB];
    uint64_t e[NB];
    bool on[NB];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      const int rr = (it0 + u) * 4 + rr0;
      const int row = mrow + rr, col = nb + ch * 4;
      on[u] = row < M && col < N;
      e[u] = L.w_off + (uint64_t)row * (uint64_t)N + (uint64_t)col;
      g4[u] = *reinterpret_cast<const float4*>(obuf + rr * 128 + (((uint32_t)ch ^ (uint32_t)(rr & 7)) << 4));
      if (on[u]) {
        w4[u] = __ldcs(reinterpret_cast<const float4*>(t.a.w + e[u]));
        m4[u] = __ldcs(reinterpret_cast<const float4*>(t.a.m + e[u]));
        if (need_dl) d4[u] = __ldcs(reinterpret_cast<const float4*>(t.a.delta + e[u]));
        if (OPT == PM_ADAM) s4[u] = __ldcs(reinterpret_cast<const float4*>(t.a.s + e[u]));
      }
    }
#pragma unroll
    for (int u = 0; u < NB; ++u) {
      if (!on[u]) continue;
      float4 wn;
      wn.x = upd_one<OPT>(g4[u].x, w4[u].x, m4[u].x, s4[u].x, d4[u].x, sc, beta1, beta2, omb1, omb2, eps);
      wn.y = upd_one<OPT>(g4[u].y, w4[u].y, m4[u].y, s4[u].y, d4[u].y, sc, beta1, beta2, omb1, omb2, eps);
      wn.z = upd_one<OPT>(g4[u].z, w4[u].z, m4[u].z, s4[u].z, d4[u].z, sc, beta1, beta2, omb1, omb2, eps);
      wn.w = upd_one<OPT>(g4[u].w, w4[u].w, m4[u].w, s4[u].w, d4[u].w, sc, beta1, beta2, omb1, omb2, eps);
      __stcs(reinterpret_cast<float4*>(t.a.w + e[u]), wn);
      __stcs(reinterpret_cast<float4*>(t.a.m + e[u]), m4[u]);
      if (OPT == PM_ADAM) __stcs(reinterpret_cast<float4*>(t.a.s + e[u]), s4[u]);
      if (sc.use_delta) __stcs(reinterpret_cast<float4*>(t.a.delta + e[u]), d4[u]);
      {
        __nv_bfloat162 lo2 = __floats2bfloat162_rn(wn.x, wn.y), hi2 = __floats2bfloat162_rn(wn.z, wn.w);
        uint2 pk; pk.x = *reinterpret_cast<uint32_t*>(&lo2); pk.y = *reinterpret_cast<uint32_t*>(&hi2);
        *reinterpret_cast<uint2*>(t.upd_lp + (sc.lp_shift + (int64_t)e[u])) = pk;              // re-read by a later forward: default caching
      }
      if (sc.rc_shift >= 0) {                                     // corrected recompute weights of the new version (T2 for recompute)
        const float gp = sc.rc_gap;
        __nv_bfloat162 lo2 = __floats2bfloat162_rn(__fsub_rn(wn.x, __fmul_rn(gp, d4[u].x)), __fsub_rn(wn.y, __fmul_rn(gp, d4[u].y)));
        __nv_bfloat162 hi2 = __floats2bfloat162_rn(__fsub_rn(wn.z, __fmul_rn(gp, d4[u].z)), __fsub_rn(wn.w, __fmul_rn(gp, d4[u].w)));
        uint2 pk; pk.x = *reinterpret_cast<uint32_t*>(&lo2); pk.y = *reinterpret_cast<uint32_t*>(&hi2);
        *reinterpret_cast<uint2*>(t.upd_lp + (sc.rc_shift + (int64_t)e[u])) = pk;
      }
    }
  }
}

// What an epilogue warp needs to know of a tile's Linear, read before the accumulator is awaited: behind it every asm with a
// memory clobber would make the compiler read the tables again.
struct EpiTile {
  int flags, act;             // MODE 0: LF_* and PM_ACT_* of the Linear
  bool resid;                 // MODE 0: the stage adds its skip tensor to z here, from slot skip_slot of its buffer
  int skip_slot;
  int slot;                   // ring slot of z (MODE 0) or dx (MODE 1); MODE 2: gradients add to the arena
  int yslot;                  // MODE 0: ring slot of y, or of the fp32 logits
  const float* bias;          // MODE 0
  uint2* mask;                // the mask bits a ReLU writes (MODE 0) or the gradient of its output reads (MODE 1); null: none
};

// this lane's eight bytes of the mask bits of a block of 32 rows x 64 columns (row0 a multiple of 32, n a multiple of 64)
__device__ __forceinline__ uint2* mask_at(const TickArgs& t, uint64_t ring_off, int slot, int N, int row0, int n, int lane) {
  const uint64_t cb = (uint64_t)(N + 63) / 64, rb = (uint64_t)(t.T + 31) / 32;
  return reinterpret_cast<uint2*>(t.ring + ring_off) + (((uint64_t)slot * rb + row0 / 32) * cb + n / 64) * 32 + lane;
}

template <int MODE>
__device__ __forceinline__ EpiTile epi_tile(const TickArgs& t, const StageDev& s, const StageDyn& d, const LinDev& L, int p, int lvl, int mrow, int nb, int lane) {
  EpiTile e{};
  if (MODE == 0) {
    e.flags = L.flags; e.act = L.act;
    e.resid = s.post == POST_RESIDUAL && !((L.flags & LF_WRITE_Z) && (L.flags & LF_WRITE_Y));
    e.skip_slot = d.skip_rslot;
    e.slot = d.f_slot;
    e.yslot = lvl < s.n_lin - 1 ? d.f_slot : (s.emit_memory ? (int)(d.f_mb % t.mem_depth) : (p < t.P - 1 ? d.f_next_xslot : (int)(d.tick & 1)));
    e.bias = fwd_small<__nv_bfloat16>(t, s, d, L.b_off, L.b_soff);
    if (L.mask_out) e.mask = mask_at(t, L.mask_out, e.yslot, L.n_out, mrow, nb, lane);
  } else if (MODE == 1) {
    e.slot = (lvl == 0 && s.pre == PRE_NONE) ? d.prev_wslot : 0;
    if (L.mask_in) e.mask = mask_at(t, L.mask_in, (lvl == 0 && s.pre == PRE_NONE) ? d.b_xslot : d.b_slot, L.n_in, mrow, nb, lane);
  } else {
    e.slot = d.accum;
  }
  return e;
}

// One epilogue unit: 32 rows x 64 columns of the accumulator at tensor-memory address `taddr`, read 32 columns at a time
// and passed through this warp's swizzled staging boxes to TMA stores (full 128-byte rows; rows and columns beyond the
// tensor are clipped).  Called by a whole warp; lane = row within the block.  `release` is called once the accumulator has
// been read.  A residual stage's skip values wait in the box (EpiStage::fetch).
// What bounds it is the number of instructions: a tile of 128 x 256 per CTA is sixteen units on four schedulers, and the tensor core
// takes 4096 cycles for it at a reduction of 512.  Hence two columns per instruction everywhere (a bf16 sum of two bf16 values
// rounded once is what the fp32 sum rounds to: at most 16 binary digits apart the fp32 sum is exact, further apart neither
// reaches a tie), and one branch per half on what the Linear does.
// bias: that of columns 2 l and 2 l + 1 in lane l.  mask: this row's mask bits where a ReLU's backward is applied (MODE 1).  (With one column per instruction the
// forward of the 6-layer encoder's tick took 194 us, 164 now; reading the skip values row by row into registers 172.)
template <int MODE, bool FUSE, int SLOTS, class Release>
__device__ __forceinline__ void epi_unit(const TickArgs& t, const CUtensorMap* lm, const StageDev& s, const StageDyn& d, const LinDev& L, const EpiTile& et,
                                         int M, int N, int mrow, int nb, uint32_t taddr, EpiStage<SLOTS>& es,
                                         const float2 bias, const uint2 mask, Release release) {
  const int lane = es.lane;
  const uint32_t row_off = (uint32_t)lane * 128, sw = (uint32_t)(lane & 7);
  uint32_t r[32];
  auto load_half = [&](int h) {
    tmem_ld32(taddr + 32 * h, r);
    tmem_ld_wait();
    if (h == 1) release();
  };
  if (mrow >= M || nb >= N) { release(); return; }                // nothing of this unit lies in the tensor
  auto bias4 = [&](int h, int g) {
    const int src = 16 * h + 2 * g;
    return make_float4(__shfl_sync(0xffffffffu, bias.x, src), __shfl_sync(0xffffffffu, bias.y, src),
                       __shfl_sync(0xffffffffu, bias.x, src + 1), __shfl_sync(0xffffffffu, bias.y, src + 1));
  };
  auto pair = [&](int i, float bx, float by) {                    // two columns of the half in r, with the bias
    const float2 v = make_float2(__uint_as_float(r[i]), __uint_as_float(r[i + 1]));
    return MODE == 0 ? add_f32x2(v, make_float2(bx, by)) : v;
  };
  if (MODE == 2 || (MODE == 0 && (et.flags & LF_OUT_F32))) {      // two boxes of 32 fp32 columns
#pragma unroll (FUSE ? 2 : 1)
    for (int h = 0; h < 2; ++h) {
      load_half(h);
      if (MODE == 2 && FUSE) {                                    // the update is applied here; nothing is stored to the grad arena
        if (t.upd_opt == PM_SGDM) epi_update_block<PM_SGDM>(t, d, L, M, N, mrow, nb + 32 * h, r, es.buf, lane);
        else epi_update_block<PM_ADAM>(t, d, L, M, N, mrow, nb + 32 * h, r, es.buf, lane);
        continue;
      }
      uint8_t* box = es.begin();
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        const float4 b = MODE == 0 ? bias4(h, g) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float2 v0 = pair(4 * g, b.x, b.y), v1 = pair(4 * g + 2, b.z, b.w);
        *reinterpret_cast<float4*>(box + row_off + (((uint32_t)g ^ sw) << 4)) = make_float4(v0.x, v0.y, v1.x, v1.y);
      }
      es.end([&](uint32_t src) {
        if (nb + 32 * h >= N) return;
        if (MODE == 0) tma_store_3d(lm + MAP_Y_OUT, src, nb + 32 * h, mrow, et.yslot);
        else if (et.slot) tma_reduce_add_2d(lm + MAP_DW_OUT, src, nb + 32 * h, mrow);   // a later microbatch of the minibatch: dW adds to the arena
        else tma_store_2d(lm + MAP_DW_OUT, src, nb + 32 * h, mrow);
      });
    }
    return;
  }
  const bool both = MODE == 0 && (et.flags & LF_WRITE_Z) && (et.flags & LF_WRITE_Y);   // z, then y = act(z) from the staged z
  // A stage that ends in a residual add writes the sum itself: out = bf16(skip + bf16(acc + b)), straight into the
  // next stage's input (or the memory ring); the skip tensor was sent by the emitting stage skip_depth - 1 ticks ago.
  enum { PLAIN, RELU, RESIDUAL, MASKED };
  uint2 bits = make_uint2(0u, 0u);                                // the mask bits a ReLU leaves
  uint8_t* box = nullptr;
  auto half = [&](int h, auto kind) {
    constexpr int KIND = decltype(kind)::value;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const float4 b0 = MODE == 0 ? bias4(h, 2 * g) : make_float4(0.f, 0.f, 0.f, 0.f), b1 = MODE == 0 ? bias4(h, 2 * g + 1) : b0;
      const float2 v0 = pair(8 * g, b0.x, b0.y), v1 = pair(8 * g + 2, b0.z, b0.w), v2 = pair(8 * g + 4, b1.x, b1.y), v3 = pair(8 * g + 6, b1.z, b1.w);
      uint4 o = make_uint4(pack_bf16(v0.x, v0.y), pack_bf16(v1.x, v1.y), pack_bf16(v2.x, v2.y), pack_bf16(v3.x, v3.y));
      if (KIND == RELU) o = make_uint4(relu_bf16x2(o.x), relu_bf16x2(o.y), relu_bf16x2(o.z), relu_bf16x2(o.w));   // bf16(max(x, 0)) = max(bf16(x), 0)
      if (KIND == RELU) {
        const uint32_t w[4] = {o.x, o.y, o.z, o.w};
        uint32_t m = 0u;
#pragma unroll
        for (int e = 0; e < 4; ++e) m |= positive_bf16x2(w[e]) & (0x00010001u << (4 * g + e));
        if (h == 0) bits.x |= m; else bits.y |= m;
      }
      if (KIND == MASKED) {                                         // dz = bf16(dx) * (1 or 0)
        const uint32_t m = h == 0 ? mask.x : mask.y;
        o = make_uint4(mask_bf16x2(o.x, m << (15 - 4 * g)), mask_bf16x2(o.y, m << (14 - 4 * g)), mask_bf16x2(o.z, m << (13 - 4 * g)), mask_bf16x2(o.w, m << (12 - 4 * g)));
      }
      if (KIND == RESIDUAL) {
        const uint4 k = *reinterpret_cast<const uint4*>(box + row_off + (((uint32_t)(4 * h + g) ^ sw) << 4));
        o = make_uint4(add_bf16x2(k.x, o.x), add_bf16x2(k.y, o.y), add_bf16x2(k.z, o.z), add_bf16x2(k.w, o.w));
      }
      *reinterpret_cast<uint4*>(box + row_off + (((uint32_t)(4 * h + g) ^ sw) << 4)) = o;
    }
  };
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    load_half(h);
    if (h == 0) box = MODE == 0 && et.resid ? es.buf + es.off : es.begin();
    if (MODE == 0 && et.resid) half(h, std::integral_constant<int, RESIDUAL>());
    else if (MODE == 0 && et.act == PM_ACT_RELU && !both) half(h, std::integral_constant<int, RELU>());
    else if (MODE == 1 && et.mask) half(h, std::integral_constant<int, MASKED>());
    else half(h, std::integral_constant<int, PLAIN>());
  }
  if (MODE == 0 && et.mask) *et.mask = bits;
  es.end([&](uint32_t src) {
    // dx: to the previous stage's gradient mailbox, or this stage's own scratch when a pre-op stands before the Linear
    if (MODE == 1) tma_store_3d(lm + MAP_DX_OUT, src, nb, mrow, et.slot);
    else if (et.flags & LF_WRITE_Z) tma_store_3d(lm + MAP_Z_OUT, src, nb, mrow, et.slot);
    else if (et.flags & LF_WRITE_Y) tma_store_3d(lm + MAP_Y_OUT, src, nb, mrow, et.yslot);
  });
  if (!both) return;
  // With an activation in front of a residual add the skip tensor joins y: out = bf16(skip + y).  (Read plainly, a row per lane: the
  // box holds z, and none of the networks this library's configurations describe has such a stage.)
  const __nv_bfloat16* skip = s.post == POST_RESIDUAL && mrow + lane < M ? ws_at<__nv_bfloat16>(t, s.skip_in) + ((uint64_t)et.skip_slot * M + mrow + lane) * N + nb : nullptr;
  uint8_t* ybox = es.begin();                                     // one slot: z's own box, which its store has read by now
  auto write_y = [&](auto a) {
    constexpr int ACT = decltype(a)::value;
#pragma unroll 1
    for (int g = 0; g < 8; ++g) {
      const uint32_t off = row_off + (((uint32_t)g ^ sw) << 4);
      const uint4 z = *reinterpret_cast<const uint4*>(box + off);
      uint32_t o[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&o[e]));
        if (ACT != PM_ACT_NONE) o[e] = pack_bf16(act_fwd(f.x, ACT), act_fwd(f.y, ACT));
      }
      if (skip && nb + 8 * g < N) {                                 // widths are multiples of 8
        const uint4 k = ld_chain16(skip + 8 * g);
        o[0] = add_bf16x2(k.x, o[0]); o[1] = add_bf16x2(k.y, o[1]); o[2] = add_bf16x2(k.z, o[2]); o[3] = add_bf16x2(k.w, o[3]);
      }
      *reinterpret_cast<uint4*>(ybox + off) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  };
  if (et.act == PM_ACT_GELU) write_y(std::integral_constant<int, PM_ACT_GELU>());
  else if (et.act == PM_ACT_RELU) write_y(std::integral_constant<int, PM_ACT_RELU>());
  else write_y(std::integral_constant<int, PM_ACT_NONE>());
  es.end([&](uint32_t src) { tma_store_3d(lm + MAP_Y_OUT, src, nb, mrow, et.yslot); });
}

// ---- tile walk ---------------------------------------------------------------------------------------
// tile_start[p] .. tile_start[p+1] are the flattened tile ids of stage p for this (mode, level).
// the tile a CTA's slot holds: from the launch's order list, or, in a launch of one stage (its tiles in ascending
// order), from the launch arguments alone, so that no role starts with a chain of dependent global loads
__device__ __forceinline__ int tile_at(const TickArgs& t, const int* __restrict__ order, int slot) {
  return t.sel_p >= 0 ? t.sel_tile0 + slot : order[slot];
}

// A tile as one lane decodes it.  sa, sb: ring slots of the operands.
struct Tile { int p, m0, n0, n_kb, sa, sb; };                         // p < 0: the slot holds no tile, or one of an idle stage

// TS: rows and columns of a tile
template <int MODE, int TS>
__device__ __forceinline__ Tile decode_tile(const TickArgs& t, const int* __restrict__ tile_start, const int* __restrict__ order, int n_slots, int lvl, int slot) {
  Tile r{-1, 0, 0, 0, 0, 0};
  if (slot >= n_slots) return r;
  const int tile = tile_at(t, order, slot);
  if (tile < 0) return r;
  const int p = t.sel_p >= 0 ? t.sel_p : tile_start[t.P + 1 + tile];                            // the stage of this tile: table behind the P + 1 starts
  const StageDyn& d = t.dyn[p];
  const StageDev& s = t.st[p];
  if (lvl >= s.n_lin || (MODE == 0 ? d.f_mb < 0 : d.b_mb < 0) || (MODE == 1 && p == 0 && lvl == 0 && s.pre != PRE_EMBED)) return r;
  const LinDev& L = s.lin[lvl];
  const int N = MODE == 0 ? L.n_out : L.n_in, K = MODE == 0 ? L.n_in : (MODE == 1 ? L.n_out : t.T);
  const int tiles_n = (N + TS - 1) / TS, local = tile - (t.sel_p >= 0 ? t.sel_tile0 : tile_start[p]);
  r.p = p;
  r.m0 = local / tiles_n * TS;
  r.n0 = local % tiles_n * TS;
  r.n_kb = (K + TILE_K - 1) / TILE_K;
  const bool own_input = lvl == 0 && s.pre == PRE_NONE;
  // dz operand: the dz scratch, or (no activation) the incoming gradient itself, which for the last Linear of a stage without
  // attention is the rotating mailbox slot written during the previous tick
  if (MODE != 0) r.sa = (bwd_act(L) == PM_ACT_NONE && lvl == s.n_lin - 1 && !feeds_attention(s.post)) ? dz_mailbox_slot(t, s, d) : 0;
  else r.sa = own_input ? d.f_xslot : d.f_slot;
  // wgrad: the input's slot; else the weight version, or the corrected weights
  r.sb = MODE == 2 ? (own_input ? d.b_xslot : d.b_slot) : (MODE == 1 && L.wc_off ? 0 : d.f_vslot);
  return r;
}

// A role's walk over its CTA's tiles.  The tables that say what a tile is are four dependent loads deep, several microseconds of
// an idle tensor core when every role reads them between two tiles (a tick's forward of the 6-layer encoder, eight k-blocks per
// tile: 205 us, 194 with this walk).  So the lanes of a warp decode 32 tiles at a time, each its own, and hand them round.
// `body` runs warp-wide and returns (the same in all lanes) whether to go on.  `mine`: the first 32, decoded before the launch
// waited for its predecessor.
template <class Decode, class Body>
__device__ __forceinline__ void walk_tiles(Tile mine, int first, int step, int n_slots, int lane, Decode decode, Body body) {
  for (int s0 = first;;) {
    uint32_t todo = __ballot_sync(0xffffffffu, mine.p >= 0);
    while (todo) {
      const int j = __ffs(todo) - 1;
      todo &= todo - 1;
      Tile tl;
      tl.p = __shfl_sync(0xffffffffu, mine.p, j); tl.m0 = __shfl_sync(0xffffffffu, mine.m0, j); tl.n0 = __shfl_sync(0xffffffffu, mine.n0, j);
      tl.n_kb = __shfl_sync(0xffffffffu, mine.n_kb, j); tl.sa = __shfl_sync(0xffffffffu, mine.sa, j); tl.sb = __shfl_sync(0xffffffffu, mine.sb, j);
      if (!body(tl)) return;
    }
    s0 += 32 * step;
    if (s0 >= n_slots) return;
    mine = decode(s0 + lane * step);
  }
}

struct Ring {                       // position in a ring of mbarrier-guarded slots
  int idx; uint32_t phase;
  __device__ __forceinline__ void advance(int n) { if (++idx == n) { idx = 0; phase ^= 1u; } }
};

// ---- bias gradient: column sums of dz in the weight-gradient kernels -----------------------------------
// The A operand of the weight gradient is dz itself, so db needs no pass of its own: in the tiles of the first column the
// tensor core's release of an operand slot goes to four summing warps first, which take the slot's 64 rows of dz to registers,
// hand it to the producer and add.  Warp w owns the columns 32 w .. 32 w + 31 of the CTA's 128: lane = (16-byte chunk of eight
// columns, row group); the two row groups of a quarter-warp differ in bit 2, which the swizzle turns into distinct banks.  Eight
// rows are added pairwise, then to the running sum of their row group, the eight row groups pairwise at the end.
// What it replaced: launches that read dz again, 92 + 15 us of a tick of the 6-layer encoder (57 now, for the activations alone), 121 us of
// an update of the encoder-decoder of 2 + 2 layers of width 1024; the weight gradients themselves 148 -> 146 and 532 -> 493 us, the
// sums costing them less than the elected-lane loops gave.  (Releasing the slot only after the additions: 166 us.)
__device__ __forceinline__ void colsum_add8(const uint4 (&q)[8], float (&acc)[8]) {
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    float lo[8], hi[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t x = w == 0 ? q[j].x : w == 1 ? q[j].y : w == 2 ? q[j].z : q[j].w;
      lo[j] = __uint_as_float(x << 16); hi[j] = __uint_as_float(x & 0xFFFF0000u);
    }
    auto sum8 = [](const float (&v)[8]) {
      return __fadd_rn(__fadd_rn(__fadd_rn(v[0], v[1]), __fadd_rn(v[2], v[3])), __fadd_rn(__fadd_rn(v[4], v[5]), __fadd_rn(v[6], v[7])));
    };
    acc[2 * w] = __fadd_rn(acc[2 * w], sum8(lo));
    acc[2 * w + 1] = __fadd_rn(acc[2 * w + 1], sum8(hi));
  }
}
// the lanes of a column chunk meet; lanes 0..3 write eight columns each
__device__ __forceinline__ void colsum_store(const TickArgs& t, const StageDyn& d, const LinDev& L, int m, int lane, float (&acc)[8]) {
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    acc[e] = __fadd_rn(acc[e], __shfl_xor_sync(0xffffffffu, acc[e], 4));
    acc[e] = __fadd_rn(acc[e], __shfl_xor_sync(0xffffffffu, acc[e], 8));
    acc[e] = __fadd_rn(acc[e], __shfl_xor_sync(0xffffffffu, acc[e], 16));
  }
  if (lane < 4 && m < L.n_out) {                                  // widths are multiples of 8
    float* db = t.a.grad + L.b_off + m;
    if (d.accum) { float o[8]; load8<float>(db, o);
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] = __fadd_rn(o[e], acc[e]); }
    store8<float>(db, acc);
  }
}
// One summing warp's part of a tile.  `done` completes when the MMAs have read a slot of a summed tile (phases: the parity of
// each slot's next completion), the arrival on `empty` hands the slot back.
template <int NS>
__device__ __forceinline__ void colsum_tile(const TickArgs& t, int lvl, const Tile& tl, int row0, int sw, int lane, int& idx, uint32_t& phases, bool& ok,
                                            const uint8_t* tiles_ptr, uint32_t bar_done, uint32_t bar_empty, volatile int* abort_flag, int* status) {
  if (tl.n0 != 0) { idx = (idx + tl.n_kb) % NS; return; }
  const int r = lane >> 2, chunk = 4 * sw + (lane & 3), row = ((r & 1) << 2) | (r >> 1);
  const uint32_t off = (uint32_t)(chunk >> 3) * (A_BYTES / 2) + (uint32_t)row * 128 + (uint32_t)(((chunk & 7) ^ row) << 4);   // rows row + 8 j: the same swizzle
  float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int kb = 0; kb < tl.n_kb; ++kb) {
    const bool ready = mbar_wait(bar_done + 8 * idx, (phases >> idx) & 1u, abort_flag, status, 9);
    ok = __all_sync(0xffffffffu, ready) && ok;                    // a CTA that gives up: the warps still meet at every k-block
    phases ^= 1u << idx;
    uint4 q[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) q[j] = *reinterpret_cast<const uint4*>(tiles_ptr + idx * STAGE_BYTES + off + j * 1024);
    asm volatile("bar.sync 1, 128;" ::: "memory");                // the four summing warps have read the slot
    if (ok && sw == 0 && lane == 0) mbar_arrive(bar_empty + 8 * idx);
    colsum_add8(q, acc);
    if (++idx == NS) idx = 0;
  }
  if (ok) colsum_store(t, t.dyn[tl.p], t.st[tl.p].lin[lvl], tl.m0 + row0 + 8 * chunk, lane, acc);
}

// ---- the kernel --------------------------------------------------------------------------------------
template <int MODE, bool FUSE>
__global__ void __launch_bounds__(Cfg<MODE, FUSE>::kThreads, 1)
umma_gemm_kernel(TickArgs t, const CUtensorMap* __restrict__ maps, const int* __restrict__ tile_start, const int* __restrict__ order, int n_slots, int lvl, int* status) {
  using C = Cfg<MODE, FUSE>;
  constexpr int NS = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;                      // swizzled tiles need 1024-byte alignment
  uint8_t* tiles_ptr = smem_raw + (tiles - raw);
  const uint32_t outs = tiles + NS * STAGE_BYTES;                     // epilogue staging for TMA stores
  uint8_t* outs_ptr = tiles_ptr + NS * STAGE_BYTES;
  const uint32_t bars = tiles + C::kTileBytes;
  // barrier block: full[NS] empty[NS] done[NS] tfull[2] tempty[2] skip[one per epilogue warp], then tmem base word and abort flag
  const uint32_t bar_full = bars, bar_empty = bar_full + 8 * NS, bar_done = bar_empty + 8 * NS, bar_tfull = bar_done + 8 * NS, bar_tempty = bar_tfull + 16, bar_skip = bar_tempty + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tiles_ptr + C::kTileBytes + 8 * (3 * NS + 4 + N_EPI_WARPS));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 1); mbar_init(bar_done + 8 * i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar_tfull + 8 * i, 1); mbar_init(bar_tempty + 8 * i, N_EPI_WARPS); }
    for (int i = 0; i < N_EPI_WARPS; ++i) mbar_init(bar_skip + 8 * i, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    __syncwarp();
    tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
    tmem_relinquish();
  }
  const int first = (int)blockIdx.x, step = (int)gridDim.x;
  auto decode = [&](int slot) { return decode_tile<MODE, TILE_N>(t, tile_start, order, n_slots, lvl, slot); };
  const Tile mine = decode(first + lane * step);                      // tables no launch of the phase writes
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_trigger();                                                      // behind the tensor-memory allocation: a successor's must not come first
  pdl_wait();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    Ring op{0, 0};
    int issued_op = 0;
    walk_tiles(mine, first, step, n_slots, lane, decode, [&](const Tile& tl) {
      const CUtensorMap* lm = maps + ((size_t)tl.p * PM_MAX_LINEARS + lvl) * MAPS_PER_LINEAR;
      for (int kb = 0; kb < tl.n_kb; ++kb) {
        const int k0 = kb * TILE_K;
        if (!__all_sync(0xffffffffu, mbar_wait(bar_empty + 8 * op.idx, op.phase ^ 1, abort_flag, status, 1))) return false;
        const uint32_t sa = tiles + op.idx * STAGE_BYTES, sb = sa + A_BYTES, fb = bar_full + 8 * op.idx;
        if (elect_one()) {
          mbar_arrive_expect_tx(fb, A_BYTES + B_BYTES);
          if (MODE == 0) {
            tma_load_3d(sa, lm + MAP_ACT_K, fb, k0, tl.m0, tl.sa);
            tma_load_3d(sb, lm + MAP_W_K, fb, k0, tl.n0, tl.sb);
          } else if (MODE == 1) {
            // dx = dz W: dz K-major, the weights as the MN-major operand, two 64-column runs
            tma_load_3d(sa, lm + MAP_DZ_K, fb, k0, tl.m0, tl.sa);
            tma_load_3d(sb, lm + MAP_W_MN, fb, tl.n0, k0, tl.sb);
            tma_load_3d(sb + B_BYTES / 2, lm + MAP_W_MN, fb, tl.n0 + 64, k0, tl.sb);
          } else {
            tma_load_3d(sa, lm + MAP_DZ_MN, fb, tl.m0, k0, tl.sa);
            tma_load_3d(sa + A_BYTES / 2, lm + MAP_DZ_MN, fb, tl.m0 + 64, k0, tl.sa);
            tma_load_3d(sb, lm + MAP_ACT_MN, fb, tl.n0, k0, tl.sb);
            tma_load_3d(sb + B_BYTES / 2, lm + MAP_ACT_MN, fb, tl.n0 + 64, k0, tl.sb);
          }
        }
        __syncwarp();
        op.advance(NS); ++issued_op;
      }
      return true;
    });
    if (lane == 0 && *abort_flag) {
      // copies already issued still land in this CTA's shared memory: wait for them (bounded) before leaving
      for (int back = 1; back <= NS && back <= issued_op; ++back) {
        const int it = issued_op - back;
        const long long t0 = clock64();
        while (!mbar_try_wait(bar_full + 8 * (it % NS), (uint32_t)(it / NS) & 1u) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t idesc = make_idesc(MODE == 2, MODE != 0);
    // K-major: 16 elements = 32 bytes along the swizzled row.  MN-major: 16 k-rows of 128 bytes.
    const uint64_t dba = MODE == 2 ? desc_base(A_BYTES / 2, 1024) : desc_base(16, 1024);
    const uint64_t dbb = MODE == 0 ? desc_base(16, 1024) : desc_base(B_BYTES / 2, 1024);
    const uint32_t ka = MODE == 2 ? 2048 : 32, kb_ = MODE == 0 ? 32 : 2048;
    Ring op{0, 0}, acc{0, 0};
    walk_tiles(mine, first, step, n_slots, lane, decode, [&](const Tile& tl) {
      if (!__all_sync(0xffffffffu, mbar_wait(bar_tempty + 8 * acc.idx, acc.phase ^ 1, abort_flag, status, 6))) return false;
      tc_fence_after();
      const uint32_t tmem_acc = tmem_base + (uint32_t)(acc.idx * ACC_COLS);
      // a slot is free once these MMAs have read it (first column of a weight gradient: by way of the summing warps)
      const uint32_t release = C::kSumWarps && tl.n0 == 0 ? bar_done : bar_empty;
      for (int kb = 0; kb < tl.n_kb; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(bar_full + 8 * op.idx, op.phase, abort_flag, status, 2))) return false;
        tc_fence_after();
        const uint32_t sa = tiles + op.idx * STAGE_BYTES, sb = sa + A_BYTES;
        if (elect_one()) {
#pragma unroll
          for (int k16 = 0; k16 < TILE_K / 16; ++k16)
            tc_mma_bf16(tmem_acc, desc_at(dba, sa + k16 * ka), desc_at(dbb, sb + k16 * kb_), idesc, (kb > 0 || k16 > 0) ? 1u : 0u);
          tc_commit(release + 8 * op.idx);
          if (kb == tl.n_kb - 1) tc_commit(bar_tfull + 8 * acc.idx);   // accumulator complete
        }
        __syncwarp();
        op.advance(NS);
      }
      acc.advance(2);
      return true;
    });
  } else if (warp < 2 + C::kSumWarps) {
    // ---------------- bias gradient: column sums of dz ----------------
    int idx = 0;
    uint32_t phases = 0;
    bool ok = true;
    walk_tiles(mine, first, step, n_slots, lane, decode, [&](const Tile& tl) {
      colsum_tile<NS>(t, lvl, tl, 0, warp - 2, lane, idx, phases, ok, tiles_ptr, bar_done, bar_empty, abort_flag, status);
      return true;
    });
  } else {
    // ---------------- epilogue: 8 warps, warp%4 = TMEM lane group, two warps per group split the columns ----------------
    const int q = warp & 3;
    const int ew = warp - 2 - C::kSumWarps;                           // 0..7
    const int half = ew >> 2;                                         // 0: columns 0..63, 1: columns 64..127
    EpiStage<2> es{outs_ptr + ew * C::kOutWarpBytes, outs + ew * C::kOutWarpBytes, lane, bar_skip + 8 * ew};
    Ring acc{0, 0};
    walk_tiles(mine, first, step, n_slots, lane, decode, [&](const Tile& tl) {
      const StageDyn& d = t.dyn[tl.p];
      const StageDev& s = t.st[tl.p];
      const LinDev& L = s.lin[lvl];
      const CUtensorMap* lm = maps + ((size_t)tl.p * PM_MAX_LINEARS + lvl) * MAPS_PER_LINEAR;
      const int M = MODE == 2 ? L.n_out : t.T, N = MODE == 0 ? L.n_out : L.n_in;
      const int mrow = tl.m0 + q * 32, nb = tl.n0 + half * 64;        // this warp's block
      const EpiTile et = epi_tile<MODE>(t, s, d, L, tl.p, lvl, mrow, nb, lane);
      // (written by the forward phase, which this launch's predecessors ended: read behind the wait)
      const uint2 mask = MODE == 1 && et.mask && mrow < M && nb < N ? *et.mask : make_uint2(0u, 0u);
      const float* bias = et.bias;
      const float2 bias2 = MODE == 0 && nb + 2 * lane < N ? __ldg(reinterpret_cast<const float2*>(bias + nb + 2 * lane)) : make_float2(0.f, 0.f);
      const bool fetch = MODE == 0 && et.resid && mrow < M && nb < N;
      if (fetch) es.fetch(lm + MAP_SKIP, nb, mrow, et.skip_slot);
      const bool ready = mbar_wait(bar_tfull + 8 * acc.idx, acc.phase, abort_flag, status, 4);
      bool go = __all_sync(0xffffffffu, ready);                       // tcgen05.ld needs the whole warp
      if (fetch && go) go = es.fetched(abort_flag, status);
      if (!go) { if (fetch) es.drain(); return false; }
      tc_fence_after();
      epi_unit<MODE, FUSE, 2>(t, lm, s, d, L, et, M, N, mrow, nb, tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc.idx * ACC_COLS + half * 64), es, bias2, mask, [&] {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tempty + 8 * acc.idx);         // the accumulator buffer may be overwritten now
      });
      acc.advance(2);
      return true;
    });
    if (lane == 0 && es.stored) tma_store_wait_all();                    // global writes complete before the CTA retires
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// ---- CTA-pair GEMM: 256 x 256 output tiles ---------------------------------------------------------------
// The same products on tiles of 256 x 256 computed by two CTAs of a cluster with one
// tcgen05.mma.cta_group::2 per 16 k-columns.  Each CTA loads its 128 rows of A and its 128 of the 256
// columns of B, so a CTA ingests 32 KB per 128x256x64 product: half the shared-memory fill per FLOP of the
// single-CTA kernel, whose tensor pipe waits on that fill.  Roles per CTA: warp 0 = TMA producer (loads
// land in its own shared memory and are counted on the leader's `full` barrier), warp 1 = TMEM owner and,
// in the leader (cluster rank 0), MMA issuer; sixteen epilogue warps drain the CTA's own 128 accumulator
// rows (four warps per lane group, 64 columns each).  tcgen05.commit arrives on the
// `empty` / `tfull` barriers of both CTAs; the epilogue warps of both arrive on the leader's `tempty`.
// Used when every GEMM of the launch has at least 256 rows and columns; smaller shapes keep the kernel above.
constexpr int P2_TILE = 256;
constexpr int P2_STAGES = 5;
constexpr int P2_ACC_COLS = 256;                                      // two accumulators fill the 512 TMEM columns
constexpr int P2_TILE_BYTES = P2_STAGES * STAGE_BYTES + 16 * 4096;
constexpr int P2_SMEM_BYTES = P2_TILE_BYTES + 1024 + 512;
template <int MODE, bool FUSE> struct P2Cfg {
  static constexpr int kSumWarps = Cfg<MODE, FUSE>::kSumWarps;
  static constexpr int kEpiWarps = FUSE ? 8 : 16;        // those with more registers per thread
  static constexpr int kUnits = 16 / kEpiWarps;                       // 32 x 64 blocks of the CTA's accumulator per warp
  static constexpr int kThreads = 32 * (2 + kSumWarps + kEpiWarps);
};

template <int MODE, bool FUSE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(P2Cfg<MODE, FUSE>::kThreads, 1)
umma_pair_gemm_kernel(TickArgs t, const CUtensorMap* __restrict__ maps, const int* __restrict__ tile_start, const int* __restrict__ order, int n_slots, int lvl, int* status) {
  constexpr int NS = P2_STAGES, SUM = P2Cfg<MODE, FUSE>::kSumWarps, UNITS = P2Cfg<MODE, FUSE>::kUnits;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;                      // same offset in both CTAs of the pair
  uint8_t* tiles_ptr = smem_raw + (tiles - raw);
  const uint32_t outs = tiles + NS * STAGE_BYTES;
  uint8_t* outs_ptr = tiles_ptr + NS * STAGE_BYTES;
  const uint32_t bars = tiles + P2_TILE_BYTES;
  // barrier block: full[NS] (used in the leader) empty[NS] done[NS] tfull[2] tempty[2] (leader) skip[one per epilogue warp], tmem base word, abort flag
  const uint32_t bar_full = bars, bar_empty = bar_full + 8 * NS, bar_done = bar_empty + 8 * NS, bar_tfull = bar_done + 8 * NS, bar_tempty = bar_tfull + 16, bar_skip = bar_tempty + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tiles_ptr + P2_TILE_BYTES + 8 * (3 * NS + 4 + 16));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();                            // 0 = leader
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 1); mbar_init(bar_done + 8 * i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar_tfull + 8 * i, 1); mbar_init(bar_tempty + 8 * i, 2 * P2Cfg<MODE, FUSE>::kEpiWarps); }
    for (int i = 0; i < P2Cfg<MODE, FUSE>::kEpiWarps; ++i) mbar_init(bar_skip + 8 * i, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    __syncwarp();
    tmem_alloc_pair(smem_u32(tmem_slot), 2 * P2_ACC_COLS);
    tmem_relinquish_pair();
  }
  auto decode = [&](int slot) { return decode_tile<MODE, P2_TILE>(t, tile_start, order, n_slots, lvl, slot); };
  const Tile mine = decode(pair + lane * n_pairs);                    // tables no launch of the phase writes
  tc_fence_before();
  cluster_sync_all();                                                 // barriers of both CTAs are initialised
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_trigger();                                                      // behind the tensor-memory allocation: a successor's must not come first
  pdl_wait();

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs) ----------------
    Ring op{0, 0};
    int issued_op = 0;
    const uint32_t leader_full = mapa_shared(bar_full, 0);
    walk_tiles(mine, pair, n_pairs, n_slots, lane, decode, [&](const Tile& tl) {
      const CUtensorMap* lm = maps + ((size_t)tl.p * PM_MAX_LINEARS + lvl) * MAPS_PER_LINEAR;
      const int ma = tl.m0 + rank * TILE_M, nbh = tl.n0 + rank * TILE_N;   // this CTA's rows of A and of B
      for (int kb = 0; kb < tl.n_kb; ++kb) {
        const int k0 = kb * TILE_K;
        if (!__all_sync(0xffffffffu, mbar_wait(bar_empty + 8 * op.idx, op.phase ^ 1, abort_flag, status, 31))) return false;
        const uint32_t sa = tiles + op.idx * STAGE_BYTES, sb = sa + A_BYTES;
        const uint32_t fb = leader_full + 8 * op.idx;
        if (elect_one()) {
          if (rank == 0) mbar_arrive_expect_tx(bar_full + 8 * op.idx, 2 * (A_BYTES + B_BYTES));   // the bytes of both CTAs
          if (MODE == 0) {
            tma_load_3d_pair(sa, lm + MAP_ACT_K, fb, k0, ma, tl.sa);
            tma_load_3d_pair(sb, lm + MAP_W_K, fb, k0, nbh, tl.sb);
          } else if (MODE == 1) {
            tma_load_3d_pair(sa, lm + MAP_DZ_K, fb, k0, ma, tl.sa);
            tma_load_3d_pair(sb, lm + MAP_W_MN, fb, nbh, k0, tl.sb);
            tma_load_3d_pair(sb + B_BYTES / 2, lm + MAP_W_MN, fb, nbh + 64, k0, tl.sb);
          } else {
            tma_load_3d_pair(sa, lm + MAP_DZ_MN, fb, ma, k0, tl.sa);
            tma_load_3d_pair(sa + A_BYTES / 2, lm + MAP_DZ_MN, fb, ma + 64, k0, tl.sa);
            tma_load_3d_pair(sb, lm + MAP_ACT_MN, fb, nbh, k0, tl.sb);
            tma_load_3d_pair(sb + B_BYTES / 2, lm + MAP_ACT_MN, fb, nbh + 64, k0, tl.sb);
          }
        }
        __syncwarp();
        op.advance(NS); ++issued_op;
      }
      return true;
    });
    // Copies already issued still land here: give them time (bounded) before leaving.  Rank 1's copies are counted on the same
    // barriers of the leader (the expected bytes are those of both CTAs), and no CTA of the pair leaves before the cluster
    // barrier at the end of the kernel, which the leader reaches only after these waits: rank 1 needs no wait of its own.
    if (lane == 0 && *abort_flag && rank == 0)
      for (int back = 1; back <= NS && back <= issued_op; ++back) {
        const int it = issued_op - back;
        const long long t0 = clock64();
        while (!mbar_try_wait(bar_full + 8 * (it % NS), (uint32_t)(it / NS) & 1u) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
      }
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA only) ----------------
    const uint32_t idesc = make_idesc_mn(P2_TILE, P2_TILE, MODE == 2, MODE != 0);
    const uint64_t dba = MODE == 2 ? desc_base(A_BYTES / 2, 1024) : desc_base(16, 1024);
    const uint64_t dbb = MODE == 0 ? desc_base(16, 1024) : desc_base(B_BYTES / 2, 1024);
    const uint32_t ka = MODE == 2 ? 2048 : 32, kb_ = MODE == 0 ? 32 : 2048;
    Ring op{0, 0}, acc{0, 0};
    if (rank == 0) walk_tiles(mine, pair, n_pairs, n_slots, lane, decode, [&](const Tile& tl) {
      if (!__all_sync(0xffffffffu, mbar_wait(bar_tempty + 8 * acc.idx, acc.phase ^ 1, abort_flag, status, 36))) return false;
      tc_fence_after();
      const uint32_t tmem_acc = tmem_base + (uint32_t)(acc.idx * P2_ACC_COLS);
      // a slot is free in both CTAs once these MMAs have read it (first column of a weight gradient: by way of the summing warps)
      const uint32_t release = SUM && tl.n0 == 0 ? bar_done : bar_empty;
      for (int kb = 0; kb < tl.n_kb; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait(bar_full + 8 * op.idx, op.phase, abort_flag, status, 32))) return false;
        tc_fence_after();
        const uint32_t sa = tiles + op.idx * STAGE_BYTES, sb = sa + A_BYTES;
        if (elect_one()) {
#pragma unroll
          for (int k16 = 0; k16 < TILE_K / 16; ++k16)
            tc_mma_bf16_pair(tmem_acc, desc_at(dba, sa + k16 * ka), desc_at(dbb, sb + k16 * kb_), idesc, (kb > 0 || k16 > 0) ? 1u : 0u);
          tc_commit_pair(release + 8 * op.idx, 3);
          if (kb == tl.n_kb - 1) tc_commit_pair(bar_tfull + 8 * acc.idx, 3);   // accumulator complete, both CTAs
        }
        __syncwarp();
        op.advance(NS);
      }
      acc.advance(2);
      return true;
    });
  } else if (warp < 2 + SUM) {
    // ---------------- bias gradient: column sums of this CTA's rows of the A tile ----------------
    int idx = 0;
    uint32_t phases = 0;
    bool ok = true;
    walk_tiles(mine, pair, n_pairs, n_slots, lane, decode, [&](const Tile& tl) {
      colsum_tile<NS>(t, lvl, tl, rank * TILE_M, warp - 2, lane, idx, phases, ok, tiles_ptr, bar_done, bar_empty, abort_flag, status);
      return true;
    });
  } else {
    // ---------------- epilogue: 16 warps per CTA (fused update: 8), warp%4 = TMEM lane group, the warps of a group split the 256 columns ----------------
    const int q = warp & 3;
    const int ew = warp - 2 - SUM;
    const int part = (ew >> 2) * UNITS;                               // first of this warp's blocks of 64 columns
    const uint32_t leader_tempty = mapa_shared(bar_tempty, 0);
    EpiStage<1> es{outs_ptr + ew * 4096, outs + ew * 4096, lane, bar_skip + 8 * ew};
    Ring acc{0, 0};
    walk_tiles(mine, pair, n_pairs, n_slots, lane, decode, [&](const Tile& tl) {
      const StageDyn& d = t.dyn[tl.p];
      const StageDev& s = t.st[tl.p];
      const LinDev& L = s.lin[lvl];
      const CUtensorMap* lm = maps + ((size_t)tl.p * PM_MAX_LINEARS + lvl) * MAPS_PER_LINEAR;
      const int M = MODE == 2 ? L.n_out : t.T, N = MODE == 0 ? L.n_out : L.n_in;
      const int mrow = tl.m0 + rank * TILE_M + q * 32, nb = tl.n0 + part * 64;   // this warp's (first) block
      const EpiTile et = epi_tile<MODE>(t, s, d, L, tl.p, lvl, mrow, nb, lane);
      // (written by the forward phase, which this launch's predecessors ended: read behind the wait)
      const uint2 mask = MODE == 1 && et.mask && mrow < M && nb < N ? *et.mask : make_uint2(0u, 0u);
      const float* bias = et.bias;
      const float2 bias2 = MODE == 0 && nb + 2 * lane < N ? __ldg(reinterpret_cast<const float2*>(bias + nb + 2 * lane)) : make_float2(0.f, 0.f);
      const bool fetch = MODE == 0 && et.resid && mrow < M && nb < N;
      if (fetch) es.fetch(lm + MAP_SKIP, nb, mrow, et.skip_slot);
      const bool ready = mbar_wait(bar_tfull + 8 * acc.idx, acc.phase, abort_flag, status, 34);
      bool go = __all_sync(0xffffffffu, ready);                       // tcgen05.ld needs the whole warp
      if (fetch && go) go = es.fetched(abort_flag, status);
      if (!go) { if (fetch) es.drain(); return false; }
      tc_fence_after();
#pragma unroll 1
      for (int u = 0; u < UNITS; ++u) {                               // (MODE 0: one)
        epi_unit<MODE, FUSE, 1>(t, lm, s, d, L, et, M, N, mrow, nb + 64 * u, tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc.idx * P2_ACC_COLS + (part + u) * 64), es, bias2, mask, [&] {
          if (u != UNITS - 1) return;
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(leader_tempty + 8 * acc.idx);   // this warp has read its part of the accumulator
        });
      }
      acc.advance(2);
      return true;
    });
    if (lane == 0 && es.stored) tma_store_wait_all();                    // global writes complete before the CTA retires
  }
  tc_fence_before();
  cluster_sync_all();                                                 // no barrier or shared memory of a CTA is touched after this
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 2 * P2_ACC_COLS);
  }
}

// ---- dgrad with reuse of the corrected operand -----------------------------------------------------------
// D[T,in] = dz[T,out] * Wc[out,in], launches of fewer than 256 rows or columns (the others: corr_weights_kernel below).  The fp32 w and
// delta tiles (64 KB per k-block) and their conversion would be repeated for every 128-row tile; here one CTA computes up to
// four 128-row tiles against the SAME converted tile: per k-block the staging ring receives w and delta once, the transform warps
// write bf16(w - gap*delta) once, and the MMA warp issues one product per row tile into its own accumulator
// (4 x 128 TMEM columns).  Traffic per 128x128x64 product drops from 80 KB to 32 KB.
constexpr int DG_MG = 4;                                   // row tiles per B tile
constexpr int DG_NA = 3, DG_NB = 2, DG_NG = 2;             // A ring, B (converted) ring, fp32 staging ring
constexpr int DG_EPI_WARPS = 4;
constexpr int DG_XF_WARPS = 8;                             // transform warps: 32 of the 64 k-rows per half
constexpr int DG_THREADS = 32 * (2 + DG_XF_WARPS + DG_EPI_WARPS);
constexpr int DG_TILE_BYTES = DG_NG * STG_BYTES + DG_NB * B_BYTES + DG_NA * A_BYTES + DG_EPI_WARPS * 4096;
constexpr int DG_SMEM_BYTES = DG_TILE_BYTES + 1024 + 512;

struct DgTile { int p, m0, n0, n_m, M, N, K, n_kb; bool valid; };

__device__ __forceinline__ DgTile decode_dgrad(const TickArgs& t, const int* __restrict__ tile_start, int lvl, int tile) {
  DgTile r;
  const int lo = t.sel_p >= 0 ? t.sel_p : tile_start[t.P + 1 + tile];                           // the stage of this tile: table behind the P + 1 starts
  r.p = lo;
  const StageDyn& d = t.dyn[lo];
  const StageDev& s = t.st[lo];
  r.valid = lvl < s.n_lin && d.b_mb >= 0 && !(lo == 0 && lvl == 0 && s.pre != PRE_EMBED);
  const LinDev& L = s.lin[lvl < s.n_lin ? lvl : 0];
  r.M = t.T; r.N = L.n_in; r.K = L.n_out;
  const int tiles_n = (r.N + TILE_N - 1) / TILE_N;
  const int tiles_m = (r.M + TILE_M - 1) / TILE_M;
  const int local = tile - (t.sel_p >= 0 ? t.sel_tile0 : tile_start[lo]);
  const int mg = local / tiles_n;
  r.m0 = mg * DG_MG * TILE_M;
  r.n0 = (local % tiles_n) * TILE_N;
  r.n_m = min(DG_MG, tiles_m - mg * DG_MG);
  r.n_kb = (r.K + TILE_K - 1) / TILE_K;
  return r;
}

__global__ void __launch_bounds__(DG_THREADS, 1)
umma_dgrad_kernel(TickArgs t, const CUtensorMap* __restrict__ maps, const int* __restrict__ tile_start, const int* __restrict__ order, int n_slots, int lvl, int* status) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  const uint32_t stg = base;                                          // [DG_NG][w 32 KB | delta 32 KB]
  const uint32_t sB = stg + DG_NG * STG_BYTES;                        // [DG_NB][16 KB] converted operand
  const uint32_t sA = sB + DG_NB * B_BYTES;                           // [DG_NA][16 KB] dz tiles
  const uint32_t sO = sA + DG_NA * A_BYTES;                           // [4][4 KB] epilogue staging
  uint8_t* stg_ptr = base_ptr;
  uint8_t* sB_ptr = base_ptr + DG_NG * STG_BYTES;
  uint8_t* sO_ptr = sB_ptr + DG_NB * B_BYTES + DG_NA * A_BYTES;
  const uint32_t bars = base + DG_TILE_BYTES;
  const uint32_t bar_sfull = bars, bar_sempty = bar_sfull + 8 * DG_NG, bar_bfull = bar_sempty + 8 * DG_NG,
                 bar_bempty = bar_bfull + 8 * DG_NB, bar_afull = bar_bempty + 8 * DG_NB, bar_aempty = bar_afull + 8 * DG_NA,
                 bar_tfull = bar_aempty + 8 * DG_NA, bar_tempty = bar_tfull + 8;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + DG_TILE_BYTES + 8 * (2 * DG_NG + 2 * DG_NB + 2 * DG_NA + 2));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < DG_NG; ++i) { mbar_init(bar_sfull + 8 * i, 1); mbar_init(bar_sempty + 8 * i, DG_XF_WARPS); }
    for (int i = 0; i < DG_NB; ++i) { mbar_init(bar_bfull + 8 * i, DG_XF_WARPS); mbar_init(bar_bempty + 8 * i, 1); }
    for (int i = 0; i < DG_NA; ++i) { mbar_init(bar_afull + 8 * i, 1); mbar_init(bar_aempty + 8 * i, 1); }
    mbar_init(bar_tfull, 1);
    mbar_init(bar_tempty, DG_EPI_WARPS);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    __syncwarp();
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_trigger();                                                      // behind the tensor-memory allocation: a successor's must not come first
  pdl_wait();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    // Two cursors walk the same (tile, k-block) sequence: the fp32 staging loads run one k-block ahead of the dz
    // loads, so that the load + conversion of the next weight tile overlaps the products of the current one.
    if (lane == 0) {
      struct Cursor { int tile, kb; DgTile tl; bool done; };
      auto seek = [&](Cursor& c) {                                    // move to the next valid tile at or after c.tile
        for (; c.tile < n_slots; c.tile += gridDim.x) {              // c.tile walks the slots of the order array
          const int tile = tile_at(t, order, c.tile);
          if (tile < 0) continue;
          c.tl = decode_dgrad(t, tile_start, lvl, tile);
          if (c.tl.valid) { c.kb = 0; c.done = false; return; }
        }
        c.done = true;
      };
      auto step = [&](Cursor& c) { if (++c.kb >= c.tl.n_kb) { c.tile += gridDim.x; seek(c); } };
      Cursor cs{(int)blockIdx.x, 0, DgTile{}, false}, ca{(int)blockIdx.x, 0, DgTile{}, false};
      seek(cs); seek(ca);
      Ring sg{0, 0}, ar{0, 0};
      int issued_sg = 0, issued_a = 0;
      bool ok = true;
      auto issue_staging = [&](const Cursor& c) {
        const StageDyn& d = t.dyn[c.tl.p];
        const CUtensorMap* lm = maps + ((size_t)c.tl.p * PM_MAX_LINEARS + lvl) * MAPS_PER_LINEAR;
        if (!mbar_wait(bar_sempty + 8 * sg.idx, sg.phase ^ 1, abort_flag, status, 21)) { ok = false; return; }
        const uint32_t sw = stg + sg.idx * STG_BYTES, fb = bar_sfull + 8 * sg.idx;
        const bool corr = d.use_delta != 0;
        mbar_arrive_expect_tx(fb, corr ? STG_BYTES : STG_HALF_BYTES);
        tma_load_2d(sw, lm + MAP_W_F32, fb, c.tl.n0, c.kb * TILE_K);
        if (corr) tma_load_2d(sw + STG_HALF_BYTES, lm + MAP_D_F32, fb, c.tl.n0, c.kb * TILE_K);
        sg.advance(DG_NG); ++issued_sg;
      };
      if (!cs.done) { issue_staging(cs); step(cs); }
      while (!ca.done && ok) {
        if (!cs.done) { issue_staging(cs); step(cs); if (!ok) break; }
        const StageDyn& d = t.dyn[ca.tl.p];
        const StageDev& sd_ = t.st[ca.tl.p];
        const CUtensorMap* lm = maps + ((size_t)ca.tl.p * PM_MAX_LINEARS + lvl) * MAPS_PER_LINEAR;
        const int dz_slot = (bwd_act(sd_.lin[lvl]) == PM_ACT_NONE && lvl == sd_.n_lin - 1 && !feeds_attention(sd_.post)) ? dz_mailbox_slot(t, sd_, d) : 0;
        for (int mi = 0; mi < ca.tl.n_m; ++mi) {
          if (!mbar_wait(bar_aempty + 8 * ar.idx, ar.phase ^ 1, abort_flag, status, 22)) { ok = false; break; }
          const uint32_t fa = bar_afull + 8 * ar.idx;
          mbar_arrive_expect_tx(fa, A_BYTES);
          tma_load_3d(sA + ar.idx * A_BYTES, lm + MAP_DZ_K, fa, ca.kb * TILE_K, ca.tl.m0 + mi * TILE_M, dz_slot);
          ar.advance(DG_NA); ++issued_a;
        }
        step(ca);
      }
      if (*abort_flag) {
        for (int back = 1; back <= DG_NG && back <= issued_sg; ++back) {
          const int it = issued_sg - back;
          const long long t0 = clock64();
          while (!mbar_try_wait(bar_sfull + 8 * (it % DG_NG), (uint32_t)(it / DG_NG) & 1u) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
        }
        for (int back = 1; back <= DG_NA && back <= issued_a; ++back) {
          const int it = issued_a - back;
          const long long t0 = clock64();
          while (!mbar_try_wait(bar_afull + 8 * (it % DG_NA), (uint32_t)(it / DG_NA) & 1u) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      const uint32_t idesc = make_idesc(0, 1);
      const uint64_t dba = desc_base(16, 1024), dbb = desc_base(B_BYTES / 2, 1024);
      Ring br{0, 0}, ar{0, 0};
      uint32_t tphase = 0;
      bool ok = true;
      for (int slot = blockIdx.x; slot < n_slots && ok; slot += gridDim.x) {
        const int tile = tile_at(t, order, slot);
        if (tile < 0) continue;
        const DgTile tl = decode_dgrad(t, tile_start, lvl, tile);
        if (!tl.valid) continue;
        if (!mbar_wait(bar_tempty, tphase ^ 1, abort_flag, status, 23)) { ok = false; break; }
        tc_fence_after();
        for (int kb = 0; kb < tl.n_kb && ok; ++kb) {
          if (!mbar_wait(bar_bfull + 8 * br.idx, br.phase, abort_flag, status, 24)) { ok = false; break; }
          const uint32_t sb = sB + br.idx * B_BYTES;
          for (int mi = 0; mi < tl.n_m; ++mi) {
            if (!mbar_wait(bar_afull + 8 * ar.idx, ar.phase, abort_flag, status, 25)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sa = sA + ar.idx * A_BYTES;
#pragma unroll
            for (int k16 = 0; k16 < TILE_K / 16; ++k16)
              tc_mma_bf16(tmem_base + (uint32_t)(mi * ACC_COLS), desc_at(dba, sa + k16 * 32), desc_at(dbb, sb + k16 * 2048),
                          idesc, (kb > 0 || k16 > 0) ? 1u : 0u);
            tc_commit(bar_aempty + 8 * ar.idx);
            ar.advance(DG_NA);
          }
          if (ok) tc_commit(bar_bempty + 8 * br.idx);
          br.advance(DG_NB);
        }
        if (ok) tc_commit(bar_tfull);
        tphase ^= 1;
      }
    }
  } else if (warp < 2 + DG_XF_WARPS) {
    // ---------------- operand transform: fp32 w, delta in staging -> bf16(w - gap*delta), MN-major ----------------
    const int tt = (threadIdx.x - 64) & 127;                          // position within a group of four warps
    const int hsel = (threadIdx.x - 64) >> 7;                         // which half of the 64 k-rows this group converts
    const int c = tt & 15, rb = tt >> 4;
    const uint32_t dst_in_tile = (uint32_t)(c >> 3) * (B_BYTES / 2) + (uint32_t)rb * 128 + (uint32_t)(((c & 7) ^ rb) << 4);
    const uint32_t src_in_tile = (uint32_t)rb * (TILE_N * 4) + (uint32_t)c * 32;
    Ring br{0, 0}, sg{0, 0};
    bool ok = true;
    for (int slot = blockIdx.x; slot < n_slots && ok; slot += gridDim.x) {
      const int tile = tile_at(t, order, slot);
      if (tile < 0) continue;
      const DgTile tl = decode_dgrad(t, tile_start, lvl, tile);
      if (!tl.valid) continue;
      const float gapf = (float)t.st[tl.p].gap;
      const bool corr = t.dyn[tl.p].use_delta != 0;
      for (int kb = 0; kb < tl.n_kb; ++kb) {
        bool go = mbar_wait(bar_sfull + 8 * sg.idx, sg.phase, abort_flag, status, 26);
        go = go && mbar_wait(bar_bempty + 8 * br.idx, br.phase ^ 1, abort_flag, status, 27);
        go = __all_sync(0xffffffffu, go);
        if (!go) { ok = false; break; }
        const uint8_t* src = stg_ptr + sg.idx * STG_BYTES + src_in_tile;
        uint8_t* dst = sB_ptr + br.idx * B_BYTES + dst_in_tile;
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const int j = hsel * 4 + jj;
          const float4 w0 = *reinterpret_cast<const float4*>(src + j * 8 * TILE_N * 4);
          const float4 w1 = *reinterpret_cast<const float4*>(src + j * 8 * TILE_N * 4 + 16);
          float v[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
          if (corr) {
            const float4 d0 = *reinterpret_cast<const float4*>(src + STG_HALF_BYTES + j * 8 * TILE_N * 4);
            const float4 d1 = *reinterpret_cast<const float4*>(src + STG_HALF_BYTES + j * 8 * TILE_N * 4 + 16);
            const float dd[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = __fsub_rn(v[e], __fmul_rn(gapf, dd[e]));   // w - (tau_fwd - tau_bkwd) * delta
          }
          *reinterpret_cast<uint4*>(dst + j * 1024) =
              make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) { mbar_arrive(bar_bfull + 8 * br.idx); mbar_arrive(bar_sempty + 8 * sg.idx); }
        br.advance(DG_NB); sg.advance(DG_NG);
      }
    }
  } else {
    // ---------------- epilogue: one warp per TMEM lane group, 64 columns at a time through a swizzled staging buffer ----------------
    const int q = warp & 3;
    const int ew = warp - 2 - DG_XF_WARPS;
    uint8_t* obuf = sO_ptr + ew * 4096;
    const uint32_t obuf_s = sO + ew * 4096;
    const uint32_t row_off = (uint32_t)lane * 128, sw = (uint32_t)(lane & 7);
    uint32_t tphase = 0;
    bool ok = true, stored = false;
    for (int slot = blockIdx.x; slot < n_slots && ok; slot += gridDim.x) {
      const int tile = tile_at(t, order, slot);
      if (tile < 0) continue;
      const DgTile tl = decode_dgrad(t, tile_start, lvl, tile);
      if (!tl.valid) continue;
      const StageDyn& d = t.dyn[tl.p];
      const StageDev& s = t.st[tl.p];
      const CUtensorMap* lm = maps + ((size_t)tl.p * PM_MAX_LINEARS + lvl) * MAPS_PER_LINEAR;
      bool ready = mbar_wait(bar_tfull, tphase, abort_flag, status, 28);
      ready = __all_sync(0xffffffffu, ready);
      if (!ready) { ok = false; break; }
      tc_fence_after();
      const int dslot = (lvl == 0 && s.pre == PRE_NONE) ? d.prev_wslot : 0;
      for (int mi = 0; mi < tl.n_m; ++mi) {
        const int mrow = tl.m0 + mi * TILE_M + q * 32;
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          const int nb = tl.n0 + half * 64;
          uint32_t r0[32], r1[32];
          const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(mi * ACC_COLS + half * 64);
          tmem_ld32(taddr, r0);
          tmem_ld32(taddr + 32, r1);
          tmem_ld_wait();
          if (mrow >= tl.M || nb >= tl.N) continue;
          if (lane == 0 && stored) tma_store_wait_read();
          __syncwarp();
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            float f[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(g < 4 ? r0[(g & 3) * 8 + e] : r1[(g & 3) * 8 + e]);
            *reinterpret_cast<uint4*>(obuf + row_off + (((uint32_t)g ^ sw) << 4)) =
                make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), pack_bf16(f[6], f[7]));
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) { tma_store_3d(lm + MAP_DX_OUT, obuf_s, nb, mrow, dslot); tma_store_commit(); }
          stored = true;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_tempty);                         // all four accumulators have been read
      tphase ^= 1;
    }
    if (lane == 0 && stored) tma_store_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// ---- the corrected weights as an operand ------------------------------------------------------------------
// Launches of many rows (CTA pairs) read the T2-corrected weights bf16(w - gap*delta) from a scratch copy that this kernel forms at
// the start of the backward phase, so that their dgrad is the plain GEMM above.  Forming them inside the GEMM costs every group of
// row tiles the fp32 stream (8 B per weight through L2 and shared memory) and the conversion again, and their staging left room
// for 1.5 k-blocks of latency: an update of the encoder-decoder of 4 + 4 layers of width 1024 spent 1700 us in such a dgrad, and spends
// 222 here (6.9 TB/s) and 1005 in the plain one; a tick of the 6-layer encoder 215, and 35 + 142.  With fewer rows the stream is read
// once either way and umma_dgrad_kernel stays.
// One block per entry of the list: up to 8192 consecutive weights of one Linear.  Bound by HBM (10 B per weight).
struct CorrBlock { uint32_t src64, dst64, n64; int32_t stage; };      // in groups of 64 elements; dst64 from the workspace's start
constexpr int CORR_THREADS = 256, CORR_GROUPS = 4;                    // groups of eight elements per thread
constexpr uint32_t CORR_N64 = CORR_THREADS * CORR_GROUPS * 8 / 64;

__global__ void __launch_bounds__(CORR_THREADS) corr_weights_kernel(TickArgs t, const CorrBlock* list) {
  pdl_trigger();
  pdl_wait();
  const CorrBlock b = list[blockIdx.x];
  const StageDyn& d = t.dyn[b.stage];
  if (d.b_mb < 0) return;
  const bool corr = d.use_delta != 0;
  const float gapf = (float)t.st[b.stage].gap;
  const float* w = t.a.w + (uint64_t)b.src64 * 64;
  const float* dl = t.a.delta + (uint64_t)b.src64 * 64;
  __nv_bfloat16* out = ws_at<__nv_bfloat16>(t, (uint64_t)b.dst64 * 128);
  const uint32_t n8 = b.n64 * 8;
  float4 w0[CORR_GROUPS], w1[CORR_GROUPS], d0[CORR_GROUPS], d1[CORR_GROUPS];
#pragma unroll
  for (int u = 0; u < CORR_GROUPS; ++u) {
    const uint32_t i = min(threadIdx.x + u * CORR_THREADS, n8 - 1);     // (beyond the end: the last group again, not stored)
    w0[u] = __ldcs(reinterpret_cast<const float4*>(w) + 2 * i); w1[u] = __ldcs(reinterpret_cast<const float4*>(w) + 2 * i + 1);
    if (corr) { d0[u] = __ldcs(reinterpret_cast<const float4*>(dl) + 2 * i); d1[u] = __ldcs(reinterpret_cast<const float4*>(dl) + 2 * i + 1); }
  }
#pragma unroll
  for (int u = 0; u < CORR_GROUPS; ++u) {
    const uint32_t i = threadIdx.x + u * CORR_THREADS;
    if (i >= n8) break;
    float v[8] = {w0[u].x, w0[u].y, w0[u].z, w0[u].w, w1[u].x, w1[u].y, w1[u].z, w1[u].w};
    if (corr) {
      const float dd[8] = {d0[u].x, d0[u].y, d0[u].z, d0[u].w, d1[u].x, d1[u].y, d1[u].z, d1[u].w};
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = __fsub_rn(v[e], __fmul_rn(gapf, dd[e]));   // w - (tau_fwd - tau_bkwd) * delta
    }
    store8<__nv_bfloat16>(out + (uint64_t)i * 8, v);
  }
}

// ---- host side -----------------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct UmmaPlan {
  const CUtensorMap* d_maps = nullptr;
  const int* d_tile_start = nullptr;     // per (mode, level) at ts_off: [P+1] starts, then the stage of each tile
  size_t ts_off[4][PM_MAX_LINEARS] = {};
  const int* d_orders = nullptr;         // concatenated order arrays
  int* d_status = nullptr;
  int n_slots[4][PM_MAX_LINEARS] = {};
  int grid[4][PM_MAX_LINEARS] = {};
  bool pair[4][PM_MAX_LINEARS] = {};     // launch uses the CTA-pair kernel (256 x 256 tiles)
  size_t order_off[4][PM_MAX_LINEARS] = {};
  int P = 0;
  // launches of one stage (microbatch-major order): the stage's tiles in ascending order are a slice of the identity list
  std::vector<int> h_tile_start;         // host copy of the tile starts
  RowShape row[2][PM_MAX_LINEARS];       // launches over all stages (forward, dgrad) with few tiles: pm_umma_row.cuh
  int row_n[2][PM_MAX_LINEARS] = {};
  std::vector<StageDev> st;              // host copy of the stages (launches of one stage with few tiles)
  const int* d_identity = nullptr;       // 0, 1, 2, ...
  const CorrBlock* d_corr = nullptr;     // blocks of the corrected weights, and each stage's first
  std::vector<uint32_t> corr_first;
  int max_ctas = kSms;
};

// Tile tables of every (mode, level): the flattened tile ids per stage, and the order in which the persistent
// CTAs walk them.  CTA b takes order[b], order[b + G], ...: the lists are a longest-processing-time-first
// assignment (weight = k-blocks x row tiles + a constant per tile), so that one very deep GEMM (a vocabulary
// projection next to d_model-sized layers) does not leave most SMs idle.  Unused slots hold -1.
struct TileTables {
  std::vector<int> tile_start;           // per (mode, level): [P+1] starts, then the stage of each tile
  size_t ts_off[4][PM_MAX_LINEARS] = {};
  std::vector<int> orders;
  int n_slots[4][PM_MAX_LINEARS] = {};
  int grid[4][PM_MAX_LINEARS] = {};
  bool pair[4][PM_MAX_LINEARS] = {};
  size_t order_off[4][PM_MAX_LINEARS] = {};
  int max_tiles = 0;                     // most tiles of any (mode, level)
};

static int device_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
    cudaGetLastError();
    return kSms;
  }
  return sms;
}

// PM_UMMA_PAIR=0 in the environment keeps every launch on the single-CTA kernels (for comparisons).
static bool pair_kernels_allowed() {
  const char* v = getenv("PM_UMMA_PAIR");
  return !(v && v[0] == '0');
}

// Launches of a level whose GEMMs all have at least 256 rows and columns run on CTA pairs.
static bool level_on_pairs(int T, const std::vector<StageDev>& st, int mode, int l) {
  int n = 0;
  for (size_t p = 0; p < st.size(); ++p)
    if (l < st[p].n_lin) {
      const LinDev& L = st[p].lin[l];
      if ((mode == 2 ? L.n_out : T) < P2_TILE || (mode == 0 ? L.n_out : L.n_in) < P2_TILE) return false;
      if ((mode == 0 || mode == 2) || p > 0 || l > 0 || st[p].pre == PRE_EMBED) ++n;   // the first Linear of the network has no input gradient
    }
  return n > 0 && pair_kernels_allowed();
}

// Does the dgrad of Linear l of stage p read the corrected weights from scratch?  one_stage: in launches of its stage alone; grouped: in
// launches over all stages.
bool umma_corr_weights(int T, const std::vector<StageDev>& st, int p, int l, bool one_stage, bool grouped) {
  if (l >= st[p].n_lin || (p == 0 && l == 0 && st[p].pre != PRE_EMBED) || device_sms() < 2 || !level_on_pairs(T, st, 3, l)) return false;
  int n;
  return (one_stage && row_dgrad_shape(T, st[p].lin[l].n_in, st[p].lin[l].n_out).bn == 0) || (grouped && row_grouped_shape(T, st, 1, l, &n).bn == 0);
}

// Do the forward of Linear l of stage p / its dgrad run on the kernels above in every launch the context makes (queued: against a
// queued version of the weights)?
bool umma_fwd_plain(int T, const std::vector<StageDev>& st, int p, int l, bool one_stage, bool grouped) {
  int n;
  return (!one_stage || row_shape(T, st[p].lin[l].n_out, st[p].lin[l].n_in).bn == 0) && (!grouped || row_grouped_shape(T, st, 0, l, &n).bn == 0);
}
bool umma_dgrad_plain(int T, const std::vector<StageDev>& st, int p, int l, bool one_stage, bool grouped, bool queued) {
  if (!queued && (device_sms() < 2 || !level_on_pairs(T, st, 3, l))) return false;
  int n;
  return (!one_stage || row_dgrad_shape(T, st[p].lin[l].n_in, st[p].lin[l].n_out).bn == 0) && (!grouped || row_grouped_shape(T, st, 1, l, &n).bn == 0);
}

static TileTables build_tile_tables(int T, const std::vector<StageDev>& st, int sms) {
  const int P = (int)st.size();
  TileTables tt;
  auto cdiv = [](int a, int b) { return (a + b - 1) / b; };
  for (int mode = 0; mode < 4; ++mode)                      // 1: dgrad on the kernel that forms the corrected operand; 3: as a plain GEMM
    for (int l = 0; l < PM_MAX_LINEARS; ++l) {
      // block of this (mode, level): P + 1 tile starts, then the stage of every tile (one load instead of a search)
      tt.ts_off[mode][l] = tt.tile_start.size();
      std::vector<int> ts_block((size_t)P + 1, 0);
      int* ts = ts_block.data();
      std::vector<std::pair<long long, int>> work;          // (weight, tile id)
      const bool pair = mode != 1 && sms >= 2 && level_on_pairs(T, st, mode, l);
      tt.pair[mode][l] = pair;
      const bool dg = mode == 1;
      const int tile_m = pair ? P2_TILE : TILE_M, tile_n = tile_m;
      const int mg_rows = DG_MG;                            // mode 1: row tiles sharing one converted weight tile
      int acc = 0;
      for (int p = 0; p < P; ++p) {
        ts[p] = acc;
        if (l < st[p].n_lin) {
          const LinDev& L = st[p].lin[l];
          const int M = mode == 2 ? L.n_out : T, N = mode == 0 ? L.n_out : L.n_in, K = mode == 0 ? L.n_in : (mode == 2 ? T : L.n_out);
          const int tm = cdiv(M, tile_m), tn = cdiv(N, tile_n), n_kb = cdiv(K, TILE_K);
          const int groups = dg ? cdiv(tm, mg_rows) : tm;
          for (int g = 0; g < groups; ++g) {
            const int n_m = dg ? std::min(mg_rows, tm - g * mg_rows) : 1;
            for (int n = 0; n < tn; ++n) work.push_back({(long long)n_kb * n_m + 3 * n_m, acc + g * tn + n});
          }
          acc += groups * tn;
        }
      }
      ts[P] = acc;
      tt.max_tiles = std::max(tt.max_tiles, acc);
      tt.tile_start.insert(tt.tile_start.end(), ts_block.begin(), ts_block.end());
      for (int p = 0; p < P; ++p) tt.tile_start.insert(tt.tile_start.end(), (size_t)(ts_block[p + 1] - ts_block[p]), p);
      const int G = std::max(1, std::min(acc, pair ? sms / 2 : sms));     // persistent CTAs, or CTA pairs
      tt.grid[mode][l] = pair ? 2 * G : G;
      tt.order_off[mode][l] = tt.orders.size();
      if (acc == 0) { tt.n_slots[mode][l] = 0; continue; }
      std::stable_sort(work.begin(), work.end(), [](const std::pair<long long, int>& a, const std::pair<long long, int>& b) { return a.first > b.first; });
      std::vector<std::vector<int>> lists(G);
      std::vector<long long> load(G, 0);
      for (const auto& w : work) {
        int best = 0;
        for (int b = 1; b < G; ++b) if (load[b] < load[best]) best = b;
        lists[best].push_back(w.second);
        load[best] += w.first;
      }
      size_t max_len = 0;
      for (const auto& li : lists) max_len = std::max(max_len, li.size());
      tt.n_slots[mode][l] = (int)(max_len * G);
      tt.orders.resize(tt.orders.size() + max_len * G, -1);
      int* ord = tt.orders.data() + tt.order_off[mode][l];
      for (int b = 0; b < G; ++b)
        for (size_t k = 0; k < lists[b].size(); ++k) ord[k * G + b] = lists[b][k];
    }
  return tt;
}

// the blocks of corr_weights_kernel, stage by stage; first: per stage its first block, and the total
static std::vector<CorrBlock> corr_list(const std::vector<StageDev>& st, std::vector<uint32_t>* first) {
  std::vector<CorrBlock> out;
  for (size_t p = 0; p < st.size(); ++p) {
    if (first) first->push_back((uint32_t)out.size());
    for (int l = 0; l < st[p].n_lin; ++l) {
      const LinDev& L = st[p].lin[l];
      if (!L.wc_off) continue;
      const uint32_t n64 = (uint32_t)((uint64_t)L.n_in * L.n_out / 64);          // dimensions are multiples of 8
      for (uint32_t o = 0; o < n64; o += CORR_N64)
        out.push_back(CorrBlock{(uint32_t)(L.w_off / 64) + o, (uint32_t)(L.wc_off / 128) + o, std::min(CORR_N64, n64 - o), (int32_t)p});
    }
  }
  if (first) first->push_back((uint32_t)out.size());
  return out;
}

static uint64_t maps_bytes(int P) { return (uint64_t)P * PM_MAX_LINEARS * MAPS_PER_LINEAR * sizeof(CUtensorMap); }
static uint64_t ints_bytes(size_t n) { return ((uint64_t)n * sizeof(int) + 255) / 256 * 256; }

uint64_t umma_workspace_bytes(int T, const std::vector<StageDev>& st) {
  const TileTables tt = build_tile_tables(T, st, device_sms());
  return 256 + maps_bytes((int)st.size()) + ints_bytes(tt.tile_start.size()) + ints_bytes(tt.orders.size()) + ints_bytes((size_t)tt.max_tiles) +
         corr_list(st, nullptr).size() * sizeof(CorrBlock);
}

static bool encode(EncodeTiledFn fn, CUtensorMap* m, int kind, void* base, int rank, const uint64_t* dims,
                   const uint64_t* strides_bytes, const uint32_t* box, std::string& err) {
  cuuint64_t gd[3]; cuuint64_t gs[2]; cuuint32_t bx[3]; cuuint32_t es[3] = {1, 1, 1};
  for (int i = 0; i < rank; ++i) { gd[i] = dims[i]; bx[i] = box[i]; }
  for (int i = 0; i + 1 < rank; ++i) gs[i] = strides_bytes[i];
  CUresult r = fn(m, kind >= 2 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, base, gd, gs, bx, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, kind == 3 ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) { err = "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r); return false; }
  return true;
}

pm_status umma_plan_create(UmmaPlan** out, const TickArgs& t, const std::vector<StageDev>& st, void* ws_region, cudaStream_t stream, std::string& err) {
  *out = nullptr;
  void* fnp = nullptr;
  cudaDriverEntryPointQueryResult qres;
  cudaError_t ce = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fnp, cudaEnableDefault, &qres);
  if (ce != cudaSuccess || qres != cudaDriverEntryPointSuccess || !fnp) { err = "cuTensorMapEncodeTiled is not available from this driver"; return PM_ERR_CUDA; }
  EncodeTiledFn fn = (EncodeTiledFn)fnp;
  const int P = t.P;
  std::vector<CUtensorMap> maps((size_t)P * PM_MAX_LINEARS * MAPS_PER_LINEAR);
  memset(maps.data(), 0, maps.size() * sizeof(CUtensorMap));
  UmmaPlan* plan = new UmmaPlan();
  plan->P = P;
  const uint64_t T = (uint64_t)t.T;
  for (int p = 0; p < P; ++p) {
    const StageDev& s = st[p];
    for (int l = 0; l < s.n_lin; ++l) {
      const LinDev& L = s.lin[l];
      CUtensorMap* m = maps.data() + ((size_t)p * PM_MAX_LINEARS + l) * MAPS_PER_LINEAR;
      // input activation of this Linear: ring [slots][T][n_in]
      const bool in_is_x = l == 0 && s.pre == PRE_NONE;
      char* act_base = t.ring + (l > 0 ? s.lin[l - 1].h_ring : (in_is_x ? s.x_ring : s.u_ring));
      const uint64_t slots = in_is_x ? (uint64_t)s.xdepth : (uint64_t)s.depth;
      const uint64_t n_in = (uint64_t)L.n_in, n_out = (uint64_t)L.n_out;
      bool okm = true;
      {
        uint64_t dims[3] = {n_in, T, slots}, strides[2] = {n_in * 2, T * n_in * 2};
        uint32_t box_k[3] = {TILE_K, TILE_M, 1}, box_mn[3] = {64, TILE_K, 1};
        okm = okm && encode(fn, m + MAP_ACT_K, 0, act_base, 3, dims, strides, box_k, err);
        okm = okm && encode(fn, m + MAP_ACT_MN, 0, act_base, 3, dims, strides, box_mn, err);
      }
      {
        uint64_t dims[2] = {n_in, n_out}, strides[1] = {n_in * 2}, strides4[1] = {n_in * 4};
        uint32_t box[2] = {TILE_K, TILE_N}, box4[2] = {TILE_N, TILE_K};
        {
          // forward operand: the bf16 copy of w; in microbatch-major order one copy per version the forward can reach
          uint64_t dims3[3] = {n_in, n_out, 1}, strides3[2] = {n_in * 2, n_in * n_out * 2};
          uint32_t box3[3] = {TILE_K, TILE_N, 1};
          void* wbase = (void*)(t.a.w_lp + L.w_off);
          if (t.mb_major) {
            dims3[2] = (uint64_t)(s.vdepth + s.rdepth); strides3[1] = (s.end - s.begin) * 2;
            wbase = (void*)(reinterpret_cast<__nv_bfloat16*>(t.ring + s.v_ring) + (L.w_off - s.begin));
          }
          okm = okm && encode(fn, m + MAP_W_K, 0, wbase, 3, dims3, strides3, box3, err);
          uint32_t box32[3] = {TILE_K, 32, 1};                          // 32 columns of an output tile (launches with few tiles)
          okm = okm && encode(fn, m + MAP_W_K32, 0, wbase, 3, dims3, strides3, box32, err);
          uint32_t box3mn[3] = {64, TILE_K, 1};                         // the same copies as an MN-major operand (dgrad against a queued version),
          if (L.wc_off) { wbase = (void*)(t.ws + L.wc_off); dims3[2] = 1; strides3[1] = n_in * n_out * 2; }   // or the corrected weights
          okm = okm && encode(fn, m + MAP_W_MN, 0, wbase, 3, dims3, strides3, box3mn, err);
        }
        okm = okm && encode(fn, m + MAP_W_F32, 3, (void*)(t.a.w + L.w_off), 2, dims, strides4, box4, err);
        okm = okm && encode(fn, m + MAP_D_F32, 3, (void*)(t.a.delta + L.w_off), 2, dims, strides4, box4, err);
      }
      {
        // dz operand (same rule as dz_src): dz scratch | gradient inside the stage | attention's dy | rotating incoming-gradient mailbox
        char* dzb; uint64_t dz_slots = 1;
        if (bwd_act(L) != PM_ACT_NONE) dzb = t.ws + L.dz_off;
        else if (l < s.n_lin - 1) dzb = t.ws + L.dy_off;
        else if (feeds_attention(s.post)) dzb = t.ws + s.dy;
        else if (s.emit_memory) { dzb = t.ws + t.gmem_off; dz_slots = (uint64_t)t.gmem_depth; }
        else { dzb = t.ws + s.gin; dz_slots = (uint64_t)s.gin_depth; }
        uint64_t dims[3] = {n_out, T, dz_slots}, strides[2] = {n_out * 2, T * n_out * 2};
        uint32_t box_k[3] = {TILE_K, TILE_M, 1}, box_mn[3] = {64, TILE_K, 1};
        okm = okm && encode(fn, m + MAP_DZ_K, 0, dzb, 3, dims, strides, box_k, err);
        okm = okm && encode(fn, m + MAP_DZ_MN, 0, dzb, 3, dims, strides, box_mn, err);
      }
      {
        // outputs: 32-row boxes of one 128-byte swizzle row (64 bf16 or 32 fp32 columns)
        uint32_t box_bf[3] = {64, 32, 1}, box_f32[2] = {32, 32};
        uint64_t zd[3] = {n_out, T, (uint64_t)s.depth}, zs[2] = {n_out * 2, T * n_out * 2};
        if (L.flags & LF_WRITE_Z) okm = okm && encode(fn, m + MAP_Z_OUT, 1, t.ring + L.z_ring, 3, zd, zs, box_bf, err);
        if (L.flags & LF_OUT_F32) {
          uint64_t ld[3] = {n_out, T, 2}, ls[2] = {n_out * 4, T * n_out * 4};
          uint32_t box3[3] = {32, 32, 1};
          okm = okm && encode(fn, m + MAP_Y_OUT, 2, t.ws + t.yout_off, 3, ld, ls, box3, err);
        } else if (L.flags & LF_WRITE_Y) {
          char* ybase; uint64_t yslots;
          if (l < s.n_lin - 1) { ybase = t.ring + L.h_ring; yslots = (uint64_t)s.depth; }
          else if (s.emit_memory) { ybase = t.ring + t.mem_ring; yslots = (uint64_t)t.mem_depth; }   // the residual sum is the memory
          else if (p < P - 1) { ybase = t.ring + st[p + 1].x_ring; yslots = (uint64_t)st[p + 1].xdepth; }
          else { ybase = t.ws + t.yout_off; yslots = 2; }
          uint64_t yd[3] = {n_out, T, yslots};
          okm = okm && encode(fn, m + MAP_Y_OUT, 1, ybase, 3, yd, zs, box_bf, err);
        }
        if (s.post == POST_RESIDUAL && l == s.n_lin - 1) {
          uint64_t sd[3] = {n_out, T, (uint64_t)s.skip_depth};
          okm = okm && encode(fn, m + MAP_SKIP, 1, t.ws + s.skip_in, 3, sd, zs, box_bf, err);
        }
        if (!(p == 0 && l == 0 && s.pre != PRE_EMBED)) {
          const bool to_prev = l == 0 && s.pre == PRE_NONE;
          char* xbase = to_prev ? t.ws + st[p - 1].gin : t.ws + (l > 0 ? s.lin[l - 1].dy_off : s.dh);
          uint64_t xd[3] = {n_in, T, (uint64_t)(to_prev ? st[p - 1].gin_depth : 1)}, xs[2] = {n_in * 2, T * n_in * 2};
          okm = okm && encode(fn, m + MAP_DX_OUT, 1, xbase, 3, xd, xs, box_bf, err);
        }
        uint64_t wd[2] = {n_in, n_out}, wst[1] = {n_in * 4};
        okm = okm && encode(fn, m + MAP_DW_OUT, 2, (void*)(t.a.grad + L.w_off), 2, wd, wst, box_f32, err);
      }
      if (!okm) { delete plan; return PM_ERR_CUDA; }
    }
  }
  const TileTables tt = build_tile_tables(t.T, st, device_sms());
  for (int mode = 0; mode < 4; ++mode)
    for (int l = 0; l < PM_MAX_LINEARS; ++l) {
      plan->n_slots[mode][l] = tt.n_slots[mode][l];
      plan->grid[mode][l] = tt.grid[mode][l];
      plan->pair[mode][l] = tt.pair[mode][l];
      plan->order_off[mode][l] = tt.order_off[mode][l];
      plan->ts_off[mode][l] = tt.ts_off[mode][l];
    }
  char* region = (char*)ws_region;
  cudaError_t e = cudaMemcpyAsync(region + 256, maps.data(), maps_bytes(P), cudaMemcpyHostToDevice, stream);
  char* ts_dev = region + 256 + maps_bytes(P);
  char* ord_dev = ts_dev + ints_bytes(tt.tile_start.size());
  if (e == cudaSuccess) e = cudaMemcpyAsync(ts_dev, tt.tile_start.data(), tt.tile_start.size() * sizeof(int), cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess && !tt.orders.empty()) e = cudaMemcpyAsync(ord_dev, tt.orders.data(), tt.orders.size() * sizeof(int), cudaMemcpyHostToDevice, stream);
  char* id_dev = ord_dev + ints_bytes(tt.orders.size());
  std::vector<int> identity((size_t)tt.max_tiles);
  for (int i = 0; i < tt.max_tiles; ++i) identity[(size_t)i] = i;
  if (e == cudaSuccess && tt.max_tiles > 0) e = cudaMemcpyAsync(id_dev, identity.data(), identity.size() * sizeof(int), cudaMemcpyHostToDevice, stream);
  char* corr_dev = id_dev + ints_bytes(identity.size());
  const std::vector<CorrBlock> corr = corr_list(st, &plan->corr_first);
  if (e == cudaSuccess && !corr.empty()) e = cudaMemcpyAsync(corr_dev, corr.data(), corr.size() * sizeof(CorrBlock), cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(region, 0, 256, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) { err = std::string("tensor map upload: ") + cudaGetErrorString(e); delete plan; return PM_ERR_CUDA; }
  e = cudaFuncSetAttribute((const void*)umma_gemm_kernel<0, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<0, false>::kSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_dgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DG_SMEM_BYTES);
  if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_gemm_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<2, false>::kSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_gemm_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<2, true>::kSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_pair_gemm_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, P2_SMEM_BYTES);
  if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_gemm_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<1, false>::kSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_pair_gemm_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, P2_SMEM_BYTES);
  if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_pair_gemm_kernel<0, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, P2_SMEM_BYTES);
  if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_pair_gemm_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, P2_SMEM_BYTES);
  if (e == cudaSuccess) e = row_set_limits<0>();
  if (e == cudaSuccess) e = row_set_limits<1>();
  if (e == cudaSuccess) e = row_set_limits<2>();
  if (e != cudaSuccess) { err = std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e); delete plan; return PM_ERR_CUDA; }
  plan->d_status = (int*)region;
  plan->d_maps = (const CUtensorMap*)(region + 256);
  plan->d_tile_start = (const int*)ts_dev;
  plan->d_orders = (const int*)ord_dev;
  plan->d_identity = (const int*)id_dev;
  plan->d_corr = (const CorrBlock*)corr_dev;
  plan->h_tile_start = tt.tile_start;
  plan->max_ctas = device_sms();
  plan->st = st;
  for (int mode = 0; mode < 2; ++mode)
    for (int l = 0; l < PM_MAX_LINEARS; ++l) plan->row[mode][l] = row_grouped_shape(t.T, st, mode, l, &plan->row_n[mode][l]);
  *out = plan;
  return PM_OK;
}

void umma_plan_destroy(UmmaPlan* plan) { delete plan; }

// ---- self-test of the bounded wait ---------------------------------------------------------------------------
// One CTA, one thread: waits on an mbarrier on which nothing ever arrives, through the same bounded wait the GEMM
// kernels use, with the cycle limit given as an argument.  No tensor memory is allocated and no copy is in flight, so
// giving up is safe: the wait returns false, the abort flag and the status word are set, the kernel ends.
__global__ void wait_timeout_probe_kernel(int* status, long long limit_cycles, int* returned) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  const uint32_t b = smem_u32(&bar);
  mbar_init(b, 1);
  abort_flag = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  const bool ok = mbar_try_wait(b, 0) || mbar_wait_slow(b, 0, &abort_flag, status, 99, limit_cycles);
  *returned = ok ? 1 : (abort_flag ? 2 : 3);         // 2: gave up and raised the abort flag
}

cudaError_t umma_wait_timeout_probe(UmmaPlan* plan, long long limit_cycles, int* d_returned, cudaStream_t stream) {
  wait_timeout_probe_kernel<<<1, 1, 0, stream>>>(plan->d_status, limit_cycles, d_returned);
  return cudaGetLastError();
}
cudaError_t umma_clear_status(UmmaPlan* plan, cudaStream_t stream) { return cudaMemsetAsync(plan->d_status, 0, sizeof(int), stream); }

int* umma_status_word(UmmaPlan* plan) { return plan ? plan->d_status : nullptr; }

bool umma_row_dgrad(int T, const LinDev& L) { return row_dgrad_shape(T, L.n_in, L.n_out).bn != 0; }

int umma_corr_blocks(const UmmaPlan* plan, int p) { return (int)(p >= 0 ? plan->corr_first[p + 1] - plan->corr_first[p] : plan->corr_first.back()); }

cudaError_t umma_corr_launch(UmmaPlan* plan, const TickArgs& t, cudaStream_t stream) {
  const int n = umma_corr_blocks(plan, t.sel_p);
  if (n == 0) return cudaSuccess;
  return launch_pdl(corr_weights_kernel, dim3((unsigned)n), dim3(CORR_THREADS), 0, stream, t.pdl, t, plan->d_corr + (t.sel_p >= 0 ? plan->corr_first[t.sel_p] : 0));
}

cudaError_t umma_launch(UmmaPlan* plan, const TickArgs& t, int mode, int lvl, cudaStream_t stream) {
  const bool queued = mode == 1 && t.stash;                           // dgrad against a queued version of the weights
  if (t.sel_p >= 0 && mode != 2) {
    const LinDev& L = plan->st[t.sel_p].lin[lvl];
    const int N = mode == 0 ? L.n_out : L.n_in;
    const RowShape r = mode == 0 ? row_shape(t.T, N, L.n_in) : row_dgrad_shape(t.T, N, L.n_out);
    if (r.bn != 0)
      return mode == 0 ? row_launch<0>(t, r, plan->d_maps, lvl, N, 1, plan->d_status, stream)
             : !queued ? row_launch<1>(t, r, plan->d_maps, lvl, N, 1, plan->d_status, stream)
                       : row_launch<2>(t, r, plan->d_maps, lvl, N, 1, plan->d_status, stream);
  }
  if (t.sel_p < 0 && mode < 2 && !queued && plan->row[mode][lvl].bn != 0)
    return mode == 0 ? row_launch<0>(t, plan->row[0][lvl], plan->d_maps, lvl, plan->row_n[0][lvl], t.P, plan->d_status, stream)
                     : row_launch<1>(t, plan->row[1][lvl], plan->d_maps, lvl, plan->row_n[1][lvl], t.P, plan->d_status, stream);
  if (mode == 1 && (queued || plan->pair[3][lvl])) mode = 3;          // a plain GEMM: a queued version, or the corrected weights in scratch
  int n_slots = plan->n_slots[mode][lvl];
  if (n_slots == 0) return cudaSuccess;
  int grid = plan->grid[mode][lvl];                                   // one persistent CTA per SM
  const int* ts = plan->d_tile_start + plan->ts_off[mode][lvl];
  const int* ord = plan->d_orders + plan->order_off[mode][lvl];
  const bool pair = plan->pair[mode][lvl];
  int tile0 = 0;
  if (t.sel_p >= 0) {                                                 // the tiles of one stage, in ascending order
    const int* hts = plan->h_tile_start.data() + plan->ts_off[mode][lvl];
    const int first = hts[t.sel_p];
    n_slots = hts[t.sel_p + 1] - first;
    if (n_slots == 0) return cudaSuccess;
    ord = plan->d_identity + first;
    tile0 = first;
    const int G = std::max(1, std::min(n_slots, pair ? plan->max_ctas / 2 : plan->max_ctas));
    grid = pair ? 2 * G : G;
  }
  TickArgs ta = t;
  ta.sel_tile0 = tile0;
  auto go = [&](auto kernel, int threads, int smem) {
    return launch_pdl(kernel, dim3(grid), dim3(threads), smem, stream, t.pdl, ta, plan->d_maps, ts, ord, n_slots, lvl, plan->d_status);
  };
  if (pair) {
    if (mode == 0) return go(umma_pair_gemm_kernel<0, false>, P2Cfg<0, false>::kThreads, P2_SMEM_BYTES);
    if (mode == 3) return go(umma_pair_gemm_kernel<1, false>, P2Cfg<1, false>::kThreads, P2_SMEM_BYTES);
    if (t.fuse_upd) return go(umma_pair_gemm_kernel<2, true>, P2Cfg<2, true>::kThreads, P2_SMEM_BYTES);
    return go(umma_pair_gemm_kernel<2, false>, P2Cfg<2, false>::kThreads, P2_SMEM_BYTES);
  }
  if (mode == 0) return go(umma_gemm_kernel<0, false>, Cfg<0, false>::kThreads, Cfg<0, false>::kSmemBytes);
  if (mode == 1) return go(umma_dgrad_kernel, DG_THREADS, DG_SMEM_BYTES);
  if (mode == 3) return go(umma_gemm_kernel<1, false>, Cfg<1, false>::kThreads, Cfg<1, false>::kSmemBytes);
  if (t.fuse_upd) return go(umma_gemm_kernel<2, true>, Cfg<2, true>::kThreads, Cfg<2, true>::kSmemBytes);
  return go(umma_gemm_kernel<2, false>, Cfg<2, false>::kThreads, Cfg<2, false>::kSmemBytes);
}

}  // namespace pm
