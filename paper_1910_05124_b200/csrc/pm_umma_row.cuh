// bf16 GEMMs of launches with few output tiles: one stage of a microbatch-major network, or all stages of a small one.
//
// What bounds such a launch is its own length, not a pipe: a 128 x 1024 x 1024 product is 0.3 GFLOP and 2 MB of weights, but
// on 128-column tiles it is eight CTAs, each walking sixteen k-blocks behind a ring, and the launches of a microbatch
// follow one another because every Linear needs the one before.  So here
//   - a tile is 128 rows x BN = 32 or 64 columns, and the S CTAs of a cluster split its reduction (S up to 4): the operands
//     of a CTA are a few k-blocks, requested at once;
//   - the partial accumulators meet in the CTA that owns a quarter (half, all) of the rows, through distributed shared
//     memory, and are added there in rank order;
//   - the weights are operands no other launch of the chain writes, so their loads (dgrad: the loads, the T2 correction
//     w - gap*delta and its rounding) are issued before the launch waits for its predecessor (programmatic dependent
//     launch); a CTA keeps half an SM's shared memory, so that the next launch's CTAs fit beside it;
//   - the dgrad epilogue applies the receiving Linear's act'(z) (LF_DZ_FUSED), so no activation-backward launch stands
//     between two dgrads.
// B is K-major in all modes: the forward's rows of W arrive by TMA, the dgrad's columns of W are read by a warp, 32
// columns x 8 k at a time, and stored as 16-byte chunks of k.
// MODE: 0 forward, 1 dgrad with the corrected weights, 2 dgrad against a queued bf16 version as it is.
#pragma once
#include "pm_ptx.cuh"
#include "pm_umma.cuh"

namespace pm {

constexpr int ROW_M = 128, ROW_K = 64, ROW_THREADS = 320;      // warp 0 TMA, warp 1 MMA + TMEM, warps 2..9 operand transform and epilogue
template <int BN, int S> struct RowCfg {
  static constexpr int kStages = BN == 32 ? 4 : 3;
  static constexpr int kA = ROW_M * ROW_K * 2, kB = BN * ROW_K * 2;
  static constexpr int kRows = ROW_M / S;                      // rows a CTA of the cluster finishes
  static constexpr int kRedLd = BN + 4;                        // floats; rows of a quarter-warp start in distinct banks
  static constexpr int kTiles = kStages * (kA + kB);
  static constexpr int kRed = ROW_M * kRedLd * 4;              // [rank of the sender][own row][BN]
  static constexpr int kBytes = kTiles + kRed + 1024 /*alignment*/ + 256 /*barriers*/;
  static_assert(2 * (kBytes + 1024) <= 227 * 1024, "two CTAs per SM");
  static constexpr int kGroups = kRows * BN / 4 / 256;         // groups of four columns per epilogue thread
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ float4 unpack4(uint2 q) {
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&q.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float bf16_rn(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

template <int MODE, int BN, int S>
__global__ void __launch_bounds__(ROW_THREADS, 2) umma_row_kernel(TickArgs t, const CUtensorMap* __restrict__ maps, int lvl, int tiles_n, int* status) {
  using C = RowCfg<BN, S>;
  constexpr int NS = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;
  uint8_t* tiles_ptr = smem_raw + (tiles - raw);
  const uint32_t sB = tiles + NS * C::kA;
  uint8_t* sB_ptr = tiles_ptr + NS * C::kA;
  const uint32_t sRed = tiles + C::kTiles;
  const float* red = reinterpret_cast<const float*>(tiles_ptr + C::kTiles);
  const uint32_t bar_full = sRed + C::kRed, bar_empty = bar_full + 8 * NS, bar_acc = bar_empty + 8 * NS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tiles_ptr + C::kTiles + C::kRed + 8 * (2 * NS + 1));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  const int p = stage_of_block(t, blockIdx.y);
  const StageDyn& d = t.dyn[p];
  const StageDev& s = t.st[p];
  const LinDev& L = s.lin[lvl < s.n_lin ? lvl : 0];
  const int M = t.T, N = MODE == 0 ? L.n_out : L.n_in, K = MODE == 0 ? L.n_in : L.n_out;
  const int rank = S > 1 ? (int)(blockIdx.x % S) : 0;
  const int tile = (int)(blockIdx.x / S), m0 = tile / tiles_n * ROW_M, n0 = tile % tiles_n * BN;
  // the same for every CTA of a cluster
  if (lvl >= s.n_lin || (MODE == 0 ? d.f_mb < 0 : d.b_mb < 0) || (MODE != 0 && p == 0 && lvl == 0 && s.pre != PRE_EMBED) || m0 >= M || n0 >= N) {
    pdl_wait();                                                // a launch must not end before the one it depends on
    return;
  }
  const int kb_all = (K + ROW_K - 1) / ROW_K;
  const int kb0 = kb_all * rank / S, n_kb = kb_all * (rank + 1) / S - kb0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) { mbar_init(bar_full + 8 * i, MODE == 0 ? 1 : 9); mbar_init(bar_empty + 8 * i, 1); }
    mbar_init(bar_acc, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    __syncwarp();
    tmem_alloc(smem_u32(tmem_slot), BN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();                                               // behind the tensor-memory allocation: a successor's must not come first
  if (S > 1) cluster_arrive();                                 // "this CTA runs": awaited before anything is written into it
  const uint32_t tmem = *tmem_slot;
  const CUtensorMap* lm = maps + ((size_t)p * PM_MAX_LINEARS + lvl) * MAPS_PER_LINEAR;

  // What the epilogue will need (256 threads, groups of four columns of the rows this CTA owns): addresses come from the
  // stage tables by dependent loads, so they are formed, and the operands fetched, before the accumulators are awaited.
  using bf16 = __nv_bfloat16;
  const int tid = (int)threadIdx.x - 64;
  const int c4 = tid % (BN / 4) * 4, n = n0 + c4;
  const uint64_t nx = (uint64_t)M * N;
  const bf16* aux = nullptr;                                   // skip tensor (forward, residual) or act' stash (dgrad)
  bf16 *out = nullptr, *zout = nullptr;
  float* lout = nullptr;
  int act = PM_ACT_NONE;
  bool resid = false;
  float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
  uint2 ax[C::kGroups];

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      const CUtensorMap* am = lm + (MODE == 0 ? MAP_ACT_K : MAP_DZ_K);
      const int aslot = MODE == 0 ? ((lvl == 0 && s.pre == PRE_NONE) ? d.f_xslot : d.f_slot)
                        : ((bwd_act(L) == PM_ACT_NONE && lvl == s.n_lin - 1 && !feeds_attention(s.post)) ? dz_mailbox_slot(t, s, d) : 0);
      auto load_b = [&](int i) {
        const int st = i % NS;
#pragma unroll
        for (int h = 0; h < BN / 32; ++h)
          tma_load_3d(sB + st * C::kB + h * 4096, lm + MAP_W_K32, bar_full + 8 * st, (kb0 + i) * ROW_K, n0 + 32 * h, d.f_vslot);
      };
      const int first = n_kb < NS ? n_kb : NS;
      tma_prefetch_desc(am);
      for (int i = 0; i < first; ++i) {
        mbar_arrive_expect_tx(bar_full + 8 * i, MODE == 0 ? C::kA + C::kB : C::kA);
        if (MODE == 0) load_b(i);
      }
      pdl_wait();
      int issued = 0;
      bool ok = true;
      for (int i = 0; i < n_kb; ++i) {
        const int st = i % NS;
        if (i >= NS) {
          if (!mbar_wait(bar_empty + 8 * st, (uint32_t)(i / NS - 1) & 1u, abort_flag, status, 61)) { ok = false; break; }
          mbar_arrive_expect_tx(bar_full + 8 * st, MODE == 0 ? C::kA + C::kB : C::kA);
          if (MODE == 0) load_b(i);
        }
        tma_load_3d(tiles + st * C::kA, am, bar_full + 8 * st, (kb0 + i) * ROW_K, m0, aslot);
        ++issued;
      }
      if (!ok || *abort_flag) {
        // copies already issued still land in this CTA's shared memory: wait for them (bounded) before leaving
        for (int i = issued > NS ? issued - NS : 0; i < issued; ++i) {
          const long long t0 = clock64();
          while (!mbar_try_wait(bar_full + 8 * (i % NS), (uint32_t)(i / NS) & 1u) && clock64() - t0 < WAIT_LIMIT_CYCLES) {}
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t idesc = make_idesc_mn(ROW_M, BN, 0, 0);
    const uint64_t base = desc_base(16, 1024);
    for (int i = 0; i < n_kb; ++i) {
      const int st = i % NS;
      if (!__all_sync(0xffffffffu, mbar_wait(bar_full + 8 * st, (uint32_t)(i / NS) & 1u, abort_flag, status, 62))) break;
      tc_fence_after();
      if (elect_one()) {
#pragma unroll
        for (int k16 = 0; k16 < ROW_K / 16; ++k16)
          tc_mma_bf16(tmem, desc_at(base, tiles + st * C::kA + k16 * 32), desc_at(base, sB + st * C::kB + k16 * 32), idesc, (i > 0 || k16 > 0) ? 1u : 0u);
        tc_commit(bar_empty + 8 * st);
        if (i == n_kb - 1) tc_commit(bar_acc);
      }
      __syncwarp();
    }
    if (n_kb == 0 && lane == 0) tc_commit(bar_acc);
  } else {
    const int w = warp - 2;
    if (MODE != 0) {
      // ---------------- operand transform: w - gap*delta (or a queued version) -> K-major bf16 ----------------
      // warp w owns the k rows 8 w .. 8 w + 7 of every k-block, lane = column; four (k-block, 32 columns) items are requested together
      const float gapf = (float)s.gap;
      const bool corr = MODE == 1 && d.use_delta != 0;
      const float* wm = t.a.w + L.w_off;
      const float* dl = t.a.delta + L.w_off;
      const __nv_bfloat16* wq = fwd_weights<__nv_bfloat16>(t, s, d, L.w_off);
      constexpr int H = BN / 32, U = 4;
      bool ok = true;
      for (int i0 = 0; i0 < n_kb * H && ok; i0 += U) {
        float v[U][8], dv[U][8];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int it = i0 + u, k = (kb0 + it / H) * ROW_K + 8 * w, n = n0 + 32 * (it % H) + lane;
          const bool on = it < n_kb * H && n < N;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const bool onk = on && k + j < K;
            const uint64_t e = (uint64_t)(k + j) * N + n;
            if (MODE == 2) v[u][j] = onk ? __bfloat162float(wq[e]) : 0.f;
            else {
              v[u][j] = onk ? wm[e] : 0.f;
              if (corr) dv[u][j] = onk ? dl[e] : 0.f;
            }
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int it = i0 + u, i = it / H, st = i % NS;
          if (it >= n_kb * H) break;
          if (corr) {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[u][j] = __fsub_rn(v[u][j], __fmul_rn(gapf, dv[u][j]));   // w - (tau_fwd - tau_bkwd) * delta
          }
          if (i >= NS && it % H == 0) {
            bool go = mbar_wait(bar_empty + 8 * st, (uint32_t)(i / NS - 1) & 1u, abort_flag, status, 63);
            if (!__all_sync(0xffffffffu, go)) { ok = false; break; }
          }
          const int nl = 32 * (it % H) + lane;
          *reinterpret_cast<uint4*>(sB_ptr + st * C::kB + (nl >> 3) * 1024 + (nl & 7) * 128 + ((w ^ (nl & 7)) << 4)) =
              make_uint4(pack_bf16(v[u][0], v[u][1]), pack_bf16(v[u][2], v[u][3]), pack_bf16(v[u][4], v[u][5]), pack_bf16(v[u][6], v[u][7]));
          if (it % H == H - 1) {
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_full + 8 * st);
          }
        }
      }
    }
    // ---------------- partial accumulators -> the CTA that finishes their rows ----------------
    if (MODE == 0) {
      act = L.act;
      resid = s.post == POST_RESIDUAL && lvl == s.n_lin - 1;
      if (n < N) b4 = *reinterpret_cast<const float4*>(fwd_small<bf16>(t, s, d, L.b_off, L.b_soff) + n);
      if (L.flags & LF_OUT_F32) lout = ws_at<float>(t, t.yout_off) + (uint64_t)(d.tick & 1) * nx;
      if (L.flags & LF_WRITE_Z) zout = ring_at<bf16>(t, L.z_ring, d.f_slot, nx);
      if (L.flags & LF_WRITE_Y) {
        if (!resid) out = y_dest<bf16>(t, p, s, d, lvl);
        else if (s.emit_memory) out = mem_at<bf16>(t, d.f_mb);
        else if (p < t.P - 1) out = ring_at<bf16>(t, t.st[p + 1].x_ring, d.f_next_xslot, nx);
        else out = ws_at<bf16>(t, t.yout_off) + (uint64_t)(d.tick & 1) * nx;
      }
      if (resid) aux = ws_at<bf16>(t, s.skip_in) + (uint64_t)d.skip_rslot * nx;
    } else {
      out = dx_dest<bf16>(t, p, s, d, lvl);
      act = dx_fused_act<bf16>(t, p, s, d, lvl, &aux);
    }
    pdl_wait();
#pragma unroll
    for (int g = 0; g < C::kGroups; ++g) {
      const int m = m0 + rank * C::kRows + (tid + 256 * g) / (BN / 4);
      ax[g] = (aux && m < M && n < N) ? *reinterpret_cast<const uint2*>(aux + (uint64_t)m * N + n) : make_uint2(0u, 0u);
    }
    const int q = warp & 3, half = w >> 2;                     // TMEM lane group (32 rows), half of the columns
    bool ready = mbar_wait(bar_acc, 0, abort_flag, status, 64);
    ready = __all_sync(0xffffffffu, ready);
    uint32_t r[BN / 2];
#pragma unroll
    for (int c = 0; c < BN / 2; ++c) r[c] = 0u;
    if (ready && n_kb > 0) {
      tc_fence_after();
      const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * (BN / 2));
      if constexpr (BN == 32) tmem_ld16(ta, r); else tmem_ld32(ta, r);
      tmem_ld_wait();
      tc_fence_before();
    }
    __syncwarp();
    if (S > 1) cluster_wait();
    {
      const int row = q * 32 + lane;
      const uint32_t own = sRed + (uint32_t)((rank * C::kRows + row % C::kRows) * C::kRedLd + half * (BN / 2)) * 4u;
      const uint32_t dst = S > 1 ? mapa_shared(own, (uint32_t)(row / C::kRows)) : own;
#pragma unroll
      for (int c = 0; c < BN / 2; c += 4) {
        const float4 v = make_float4(__uint_as_float(r[c]), __uint_as_float(r[c + 1]), __uint_as_float(r[c + 2]), __uint_as_float(r[c + 3]));
        if (S > 1) st_cluster4(dst + 4 * c, v);
        else *reinterpret_cast<float4*>(tiles_ptr + (dst - tiles) + 4 * c) = v;
      }
    }
  }
  __syncwarp();
  if (S > 1) {
    if (warp < 2) cluster_wait();                              // (the other warps awaited the first phase above)
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, BN);
  }
  if (warp < 2) return;

  // ---------------- epilogue ----------------
  if (n >= N) return;                                          // widths are multiples of 8
#pragma unroll
  for (int g = 0; g < C::kGroups; ++g) {
    const int rl = (tid + 256 * g) / (BN / 4), m = m0 + rank * C::kRows + rl;
    if (m >= M) break;
    float4 v = *reinterpret_cast<const float4*>(red + rl * C::kRedLd + c4);
#pragma unroll
    for (int k = 1; k < S; ++k) {
      const float4 o = *reinterpret_cast<const float4*>(red + (k * C::kRows + rl) * C::kRedLd + c4);
      v.x = __fadd_rn(v.x, o.x); v.y = __fadd_rn(v.y, o.y); v.z = __fadd_rn(v.z, o.z); v.w = __fadd_rn(v.w, o.w);
    }
    const uint64_t e = (uint64_t)m * N + n;
    const float4 a = unpack4(ax[g]);
    if (MODE == 0) {
      v.x = __fadd_rn(v.x, b4.x); v.y = __fadd_rn(v.y, b4.y); v.z = __fadd_rn(v.z, b4.z); v.w = __fadd_rn(v.w, b4.w);
      if (lout) { *reinterpret_cast<float4*>(lout + e) = v; continue; }   // logits stay fp32
      v = make_float4(bf16_rn(v.x), bf16_rn(v.y), bf16_rn(v.z), bf16_rn(v.w));
      if (!out && act == PM_ACT_RELU) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));   // z alone: what attention reads
      if (zout) *reinterpret_cast<uint2*>(zout + e) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
      v = make_float4(act_fwd(v.x, act), act_fwd(v.y, act), act_fwd(v.z, act), act_fwd(v.w, act));
      if (resid) {                                             // skip + bf16(y)
        v.x = __fadd_rn(a.x, bf16_rn(v.x)); v.y = __fadd_rn(a.y, bf16_rn(v.y)); v.z = __fadd_rn(a.z, bf16_rn(v.z)); v.w = __fadd_rn(a.w, bf16_rn(v.w));
      }
    } else if (act != PM_ACT_NONE) {                           // dz = bf16(bf16(dx) * act'(z))
      v.x = __fmul_rn(bf16_rn(v.x), act_grad(a.x, act)); v.y = __fmul_rn(bf16_rn(v.y), act_grad(a.y, act));
      v.z = __fmul_rn(bf16_rn(v.z), act_grad(a.z, act)); v.w = __fmul_rn(bf16_rn(v.w), act_grad(a.w, act));
    }
    if (out) *reinterpret_cast<uint2*>(out + e) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
  }
}

// ---- host: tile width and split of the reduction -------------------------------------------------------------------
// Up to two CTAs of 64-column tiles per SM (296 tiles): beyond that the chip is full and the larger tiles of pm_umma.cu read less.
// Columns of 32 while those number one per SM; the reduction is split while the CTAs still fit (a 128 x 1024 x 1024 launch takes
// 1.3 us less with four parts than with two) and a part keeps two k-blocks.
struct RowShape { int bn = 0, split = 1; };                    // bn = 0: the launch has enough tiles for the kernels of pm_umma.cu

inline RowShape row_shape_of(long long t32, long long t64, int kb) {      // tiles of 32 and 64 columns, k-blocks
  RowShape r;
  if (t64 > 2 * kSms) return r;
  r.bn = t32 <= kSms ? 32 : 64;
  const long long base = r.bn == 32 ? t32 : t64;
  r.split = (base <= 40 && kb >= 8) ? 4 : ((base <= kSms && kb >= 4) ? 2 : 1);   // CTAs: about one per SM in four parts, two in two
  return r;
}
inline RowShape row_shape(int T, int N, int K) {
  const int tm = (T + ROW_M - 1) / ROW_M;
  return row_shape_of((long long)tm * ((N + 31) / 32), (long long)tm * ((N + 63) / 64), (K + ROW_K - 1) / ROW_K);
}

template <int MODE, int BN, int S>
static cudaError_t row_launch_t(const TickArgs& t, const CUtensorMap* maps, int lvl, int T, int N, int stages, int* status, cudaStream_t stream) {
  using C = RowCfg<BN, S>;
  const int tiles_n = (N + BN - 1) / BN, tiles_m = (T + ROW_M - 1) / ROW_M;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(S * tiles_m * tiles_n), (unsigned)stages);
  cfg.blockDim = dim3(ROW_THREADS);
  cfg.dynamicSmemBytes = C::kBytes;
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = S; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = t.pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, umma_row_kernel<MODE, BN, S>, t, maps, lvl, tiles_n, status);
}

// dgrad: every row tile forms its operand again, four 64 x 32 pieces per round trip of its loads, so many row tiles of a deep
// reduction belong to the CTA-pair kernels where those apply (256 rows and columns).  An update of a 3-layer encoder at width
// 512 takes 1202 us with this kernel everywhere and 1022 without it at 4096 rows (K = 512 to 2048, 32 row tiles); at 1024
// rows 680 with it and 702 without.
inline RowShape row_dgrad_shape(int T, int N, int K) {
  RowShape r = row_shape(T, N, K);
  const int items = ((K + ROW_K - 1) / ROW_K + r.split - 1) / r.split * (r.bn / 32);
  if (T >= 256 && N >= 256 && items * ((T + ROW_M - 1) / ROW_M) > 200) r.bn = 0;
  return r;
}

// A launch over all stages (tick-major order): by the tiles of all of them and the shallowest reduction; `n` is the widest output.
// (Ticks against the persistent 128-column kernels: 4 stages of width 1024 and 100 rows 94.9 -> 83.3 us, 12 x 2 Linears of 256 and
// 200 rows 116.1 -> 109.1, 16 x 2 of 96 and 40 rows 77.8 -> 64.0, 6 stages of 512 and 512 rows 102.4 -> 94.3.)
inline RowShape row_grouped_shape(int T, const std::vector<StageDev>& st, int mode, int lvl, int* n) {
  const int tm = (T + ROW_M - 1) / ROW_M;
  long long t32 = 0, t64 = 0;
  int kb = 1 << 30;
  *n = 0;
  for (size_t p = 0; p < st.size(); ++p) {
    if (lvl >= st[p].n_lin || (mode != 0 && p == 0 && lvl == 0 && st[p].pre != PRE_EMBED)) continue;
    const LinDev& L = st[p].lin[lvl];
    const int N = mode == 0 ? L.n_out : L.n_in, K = mode == 0 ? L.n_in : L.n_out;
    t32 += (long long)tm * ((N + 31) / 32); t64 += (long long)tm * ((N + 63) / 64);
    kb = std::min(kb, (K + ROW_K - 1) / ROW_K);
    *n = std::max(*n, N);
    if (mode != 0 && row_dgrad_shape(T, N, K).bn == 0) return RowShape{};
  }
  return *n > 0 ? row_shape_of(t32, t64, kb) : RowShape{};
}

template <int MODE>
static cudaError_t row_set_limits() {
  cudaError_t e = cudaSuccess;
#define PM_ROW_LIMIT(BN, S) if (e == cudaSuccess) e = cudaFuncSetAttribute((const void*)umma_row_kernel<MODE, BN, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, RowCfg<BN, S>::kBytes)
  PM_ROW_LIMIT(32, 1); PM_ROW_LIMIT(32, 2); PM_ROW_LIMIT(32, 4); PM_ROW_LIMIT(64, 1); PM_ROW_LIMIT(64, 2);
#undef PM_ROW_LIMIT
  return e;
}

template <int MODE>
static cudaError_t row_launch(const TickArgs& t, const RowShape& r, const CUtensorMap* maps, int lvl, int N, int stages, int* status, cudaStream_t stream) {
  if (r.bn == 32) {
    if (r.split == 4) return row_launch_t<MODE, 32, 4>(t, maps, lvl, t.T, N, stages, status, stream);
    if (r.split == 2) return row_launch_t<MODE, 32, 2>(t, maps, lvl, t.T, N, stages, status, stream);
    return row_launch_t<MODE, 32, 1>(t, maps, lvl, t.T, N, stages, status, stream);
  }
  if (r.split == 2) return row_launch_t<MODE, 64, 2>(t, maps, lvl, t.T, N, stages, status, stream);
  return row_launch_t<MODE, 64, 1>(t, maps, lvl, t.T, N, stages, status, stream);
}

}  // namespace pm
