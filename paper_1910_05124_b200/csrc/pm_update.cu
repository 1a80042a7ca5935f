// Tick scheduler and the fused multi-tensor PipeMare update.
//
// The update is a pure HBM stream: per parameter it reads g, w, m, delta (and s for
// Adam) and writes w, m, delta (and s) in fp32 plus a bfloat16 copy of w: 30 bytes per
// parameter for momentum SGD, 38 for Adam.  One launch covers every stage; a block finds
// the stage of its first 64-element group in the table of stage bounds (by an even split's
// guess, else by binary search), and that stage's scalars (T1 step size, T2 decay, Adam
// bias corrections) come from the table the scheduler wrote for this tick.
//
// Arithmetic order (each operation rounded once in fp32, no fused multiply-add, so that
// results can be reproduced bit for bit by any IEEE implementation):
//   SGD-m (Appendix B.3):  v' = beta*v - alpha*g ;  w' = w + v'
//   Adam:  m' = b1*m + (1-b1)*g ;  s' = b2*s + (1-b2)*(g*g) ;
//          w' = w - (alpha*(m'/bc1)) / (sqrt(s'/bc2) + eps)
//   T2 (Section 3.2):      delta' = gamma*delta + (1-gamma)*(w' - w)
#include "pm_update.cuh"
#include "pm_tick.cuh"
#include "pm_update_math.cuh"

namespace pm {

// ---- scheduler -------------------------------------------------------------------------------
//
// Tick s, stage i (1-based): forward of the microbatch that entered at tick s-(i-1); backward and update of
// the one that entered at tick s-(2P-i) (microbatch = entry tick, except during a synchronous warm-up).  T1 (Eq. 2): alpha_i = alpha_base(k) / tau_i^p, p = 1 - min(k/K, 1).
// T2: gamma_i = D^(1/(tau_fwd,i - tau_bkwd,i)).  Scalars are evaluated in double and rounded to
// float once.
// non-negative a modulo d, without the 64-bit division while a fits 32 bits
__device__ __forceinline__ int32_t slot_of(int64_t a, int32_t d) {
  return ((uint64_t)a >> 32) == 0 ? (int32_t)((uint32_t)a % (uint32_t)d) : (int32_t)(a % d);
}

// The launch is as long as one thread's chain of double-precision powers, so four neighbouring lanes share a stage: lane r of
// the quad evaluates scalar r (step size, T2 decay, Adam's two bias corrections) of update index kk, and all four are
// handed round.  Every lane of the warp must come here.
struct DynScalars { float alpha, gamma, bc1, bc2; };
__device__ __forceinline__ DynScalars quad_scalars(const StageSched& s, const HyperDev& hp, int64_t kk) {
  const int lane = threadIdx.x & 31, r = lane & 3;
  // warm-up microbatches (Section 4) are synchronous: standard step size, no correction, delta left alone; the T1
  // annealing counts from the first PipeMare step
  const bool sync = kk < hp.warm;
  float v = r == 0 ? 0.f : (r == 1 ? 0.f : 1.f);
  if (kk >= 0) {
    // v = scale * base^expo (alpha: base step / tau^p), 1 - base^expo (bias corrections) or base^expo (gamma): one call of pow
    double base = 1.0, expo = 0.0, step = hp.alpha_const;
    if (r == 0) {
      if (hp.alpha_tab != nullptr) step = hp.alpha_tab[kk < hp.alpha_len ? kk : hp.alpha_len - 1];
      if (hp.t1 && !sync) {
        const double q = (double)(kk - hp.warm) / (double)hp.K;
        base = (double)(s.tau_f > 1 ? s.tau_f : 1);
        expo = 1.0 - (q < 1.0 ? q : 1.0);
      }
    } else if (r == 1) {
      if (hp.t2 && s.gap > 0 && !sync) { base = hp.D; expo = 1.0 / (double)s.gap; }
    } else {
      base = r == 2 ? (double)hp.beta1 : (double)hp.beta2;
      expo = (double)(kk + 1);
    }
    const double pw = pow(base, expo);
    if (r == 0) v = (float)((hp.t1 && !sync) ? step / pw : step);
    else if (r == 1) v = (hp.t2 && s.gap > 0 && !sync) ? (float)pw : 0.f;
    else v = hp.optimizer == PM_ADAM ? (float)(1.0 - pw) : 1.f;
  }
  DynScalars o;
  o.alpha = __shfl_sync(0xffffffffu, v, lane & ~3);
  o.gamma = __shfl_sync(0xffffffffu, v, (lane & ~3) + 1);
  o.bc1 = __shfl_sync(0xffffffffu, v, (lane & ~3) + 2);
  o.bc2 = __shfl_sync(0xffffffffu, v, (lane & ~3) + 3);
  return o;
}

// Per-stage state of one tick: forward microbatch a and backward microbatch b (-1: idle), `ver` updates applied to the
// stage so far, the version `fver` its forward reads; k >= 0 activates the update with that index.
// kb: the update index the microbatch in backward belongs to (one microbatch per update: itself).
__device__ StageDyn make_dyn(const StageSched& s, const HyperDev& hp, int64_t tick, int64_t a, int64_t b, int64_t k,
                             int64_t ver, int64_t fver, bool slots, int64_t kb) {
  StageDyn d;
  d.tick = tick;
  d.accum = 0; d._pad2 = 0;
  d.rc_uslot = -1; d.rc_shift = 0; d.r_ver = fver; d.rc_gap = 0.f; d.g_shift = 0;
  const bool fa = a >= 0, ba = b >= 0;
  d.f_mb = a; d.b_mb = b; d.k = k;
  d.f_slot = (fa && slots) ? slot_of(a, s.depth) : 0;
  d.f_xslot = (fa && slots) ? slot_of(a, s.xdepth) : 0;
  d.f_next_xslot = (fa && slots && s.next_xdepth > 0) ? slot_of(a, s.next_xdepth) : 0;
  d.b_slot = (ba && slots) ? slot_of(b, s.depth) : 0;
  d.b_xslot = (ba && slots) ? slot_of(b, s.xdepth) : 0;
  d.gin_rslot = s.gin_depth > 0 ? slot_of(tick + s.gin_depth - 1, s.gin_depth) : 0;
  d.prev_wslot = s.prev_gin_depth > 0 ? slot_of(tick, s.prev_gin_depth) : 0;
  d.gmem_slot = (s.gmem_depth > 0 && ba) ? slot_of(b, s.gmem_depth) : 0;
  d.skip_wslot = s.skip_dst_depth > 0 ? slot_of(tick, s.skip_dst_depth) : 0;
  d.skip_rslot = s.skip_depth > 0 ? slot_of(tick + 1, s.skip_depth) : 0;
  d.b_next_xslot = (ba && slots && s.next_xdepth > 0) ? slot_of(b, s.next_xdepth) : 0;
  d.f_ver = fver;
  d.b_ver = ver;
  // version rings (microbatch-major order): version v sits in slot v % vdepth
  d.f_vslot = s.vdepth > 1 ? slot_of(fver, s.vdepth) : 0;
  d.u_vslot = s.vdepth > 1 ? slot_of(ver + 1, s.vdepth) : 0;
  d.lp_shift = hp.mb_major ? (int64_t)(s.v_ring / (uint64_t)hp.lp_elem) + (int64_t)d.u_vslot * (int64_t)s.count - (int64_t)s.begin : 0;
  if (hp.mb_major && s.rdepth > 0) {
    // corrected recompute weights of version ver + 1: slot vdepth + (ver + 1) % rdepth of the same rings
    d.rc_uslot = s.vdepth + slot_of(ver + 1, s.rdepth);
    d.rc_shift = (int64_t)(s.v_ring / (uint64_t)hp.lp_elem) + (int64_t)d.rc_uslot * (int64_t)s.count - (int64_t)s.begin;
    d.rc_gap = (float)(s.tau_f - s.tau_r);
  }
  d.active_update = k >= 0 ? 1 : 0;
  const int64_t kk = k >= 0 ? k : kb;                 // the update index of the microbatch in backward
  const DynScalars sc = quad_scalars(s, hp, kk);
  d.use_delta = (kk >= 0 && hp.t2 && s.gap > 0 && !(kk < hp.warm)) ? 1 : 0;
  d.alpha = kk >= 0 ? sc.alpha : 0.f;
  d.gamma = d.use_delta ? sc.gamma : 0.f;
  d.one_minus_gamma = d.use_delta ? 1.0f - sc.gamma : 1.f;
  d.bc1 = sc.bc1; d.bc2 = sc.bc2;
  return d;
}

// one quad of lanes per stage; every lane of the block must come here
__device__ __forceinline__ void schedule_tick(const StageSched* __restrict__ sched, const int64_t* __restrict__ nupd,
                                              StageDyn* __restrict__ dyn, const HyperDev& hp, int64_t tick, int64_t n_fed, int block) {
  const int quad = (block * (int)blockDim.x + (int)threadIdx.x) >> 2;
  const int P = hp.n_stages, i = quad < P ? quad : P - 1;
  const StageSched s = sched[i];
  const int64_t ver = nupd[i];
  int64_t a = mb_at_tick(tick - i, hp.warm, hp.period, hp.entry_period);
  int64_t b = mb_at_tick(tick - (2 * (int64_t)P - (i + 1)), hp.warm, hp.period, hp.entry_period);
  if (!(a >= 0 && a < n_fed)) a = -1;
  if (!(b >= 0 && b < n_fed)) b = -1;
  // One microbatch per tick: the weights a stage holds ARE version max(0, a - tau).  With a microbatch only every E
  // ticks more updates have landed by the time a forward runs, and the forward takes the version Table 1's delay
  // names from the stage's queue.
  int64_t fver = ver;
  if (hp.entry_period > 1 && a >= 0) { fver = a - s.tau_f; if (fver < 0) fver = 0; }
  const StageDyn d = make_dyn(s, hp, tick, a, b, b, ver, fver, true, b);
  if (quad < P && (threadIdx.x & 3) == 0) dyn[i] = d;
}

// Microbatch-major order (the paper's own statement of the method, Section 2.1: a queue of weight versions per
// stage).  Microbatch t runs alone: stage i's forward in sub-tick i, its backward in sub-tick 2P-1-i, on the same
// mailbox-slot arithmetic as a pipeline tick (virtual tick = 2P t + sub-tick).  The forward reads version
// max(0, t - tau_fwd,i) from the stage's version ring (during a synchronous warm-up version t, afterwards nothing
// older than the end of the warm-up), the backward the live weights (version t).  Table v in 0..2P-1 serves the
// launches of sub-tick v; table 2P marks every stage in backward with its own backward sub-tick's slots and an
// active update: it serves the grouped weight-gradient launch and the fused update.
__device__ __forceinline__ void schedule_mb(const StageSched* __restrict__ sched, StageDyn* __restrict__ tables, const HyperDev& hp, int64_t t,
                                            const int32_t* __restrict__ delays, const int64_t* __restrict__ nupd, int block, int v) {
  const int P = hp.n_stages;
  const int quad = (block * (int)blockDim.x + (int)threadIdx.x) >> 2, i = quad < P ? quad : P - 1;
  const bool store = quad < P && (threadIdx.x & 3) == 0;
  const StageSched s = sched[i];
  const int64_t base = 2 * (int64_t)P * t;
  // N microbatches per update (Section 2.1): versions, delays and step indices count updates; microbatch t belongs to
  // update u = t / N, every microbatch of a minibatch reads the same versions, the update follows the N-th
  const int64_t N = hp.n_micro > 1 ? hp.n_micro : 1;
  const int64_t u = t / N;
  int64_t fver = u - s.tau_f;
  if (u < hp.warm) fver = u; else if (fver < hp.warm) fver = hp.warm;
  if (fver < 0) fver = 0;
  StageDyn d;
  if (hp.stochastic > 0) {
    // Stage-wise stochastic delays (Appendix E): forward and backward of microbatch t on the stage's current weights
    // (version = updates it has applied); the update table activates the stage when the gradient of microbatch
    // t - delay exists, points it at that microbatch's slot of the gradient ring and indexes its step-size schedule,
    // T1 annealing and bias corrections by the stage's own update count
    const int64_t ver = nupd[i];
    const int64_t src = t - (int64_t)delays[i];
    if (v < 2 * P) d = make_dyn(s, hp, base + v, v == i ? t : -1, v == 2 * P - 1 - i ? t : -1, -1, ver, ver, true, ver);
    else {
      d = make_dyn(s, hp, base + 2 * P - 1 - i, -1, t, src >= 0 ? ver : -1, ver, ver, true, ver);
      d.g_shift = src >= 0 ? (src % hp.stochastic) * (int64_t)hp.total : 0;
    }
    d.r_ver = src >= 0 ? src : -1;
    if (store) tables[(size_t)v * P + i] = d;
    return;
  }
  // PipeMare Recompute (Appendix A.2, Appendix D): the version the recomputation reads, clamped like the forward's
  int64_t rver = u - s.tau_r;
  if (u < hp.warm) rver = u; else if (rver < hp.warm) rver = hp.warm;
  if (rver < 0) rver = 0;
  const int seg = hp.segment > 0 ? i / hp.segment : 0;
  if (v < 2 * P) d = make_dyn(s, hp, base + v, v == i ? t : -1, v == 2 * P - 1 - i ? t : -1, -1, u, fver, true, u);
  else if (v == 2 * P) d = make_dyn(s, hp, base + 2 * P - 1 - i, -1, t, (t % N == N - 1) ? u : -1, u, fver, true, u);
  else if (v == 2 * P + 1) {
    // the stage's forward entry again (same virtual tick, so the same mailbox and skip slots), reading the recompute
    // weights: the corrected queue behind the version slots when the stage keeps one, else the plain version
    d = make_dyn(s, hp, base + i, t, -1, -1, u, fver, true, u);
    d.f_vslot = s.rdepth > 0 ? s.vdepth + (int32_t)(rver % s.rdepth) : (s.vdepth > 1 ? (int32_t)(rver % s.vdepth) : 0);
  } else {
    // backward entries of one segment alone: the grouped weight-gradient launch that follows the segment's backward
    const bool mine = seg == v - (2 * P + 2);
    d = make_dyn(s, hp, base + 2 * P - 1 - i, -1, mine ? t : -1, -1, u, fver, true, u);
  }
  d.r_ver = rver;
  if (hp.materialize && (v >= 2 * P || v == 2 * P - 1 - i)) {
    // a backward entry: its version slot is the one the update filled with w - tau delta of the live version (stages that
    // keep none -- no gap, or T2 off -- read the live version itself)
    d.f_vslot = s.rdepth > 0 ? s.vdepth : (s.vdepth > 1 ? (int32_t)(u % s.vdepth) : 0);
  }
  d.accum = (t % N != 0) ? 1 : 0;
  if (store) tables[(size_t)v * P + i] = d;
}

// ---- start of a tick ------------------------------------------------------------------------------
// One launch writes the schedule table(s) and copies the microbatch in, which depend on nothing of each other: the first
// `sched_blocks` blocks schedule, the rest copy.
// MLP: inputs [T, n_in] (activation type) -> stage 1's input ring slot; targets [T, n_out] float -> target ring.
// Encoder: token ids [T] int32 per stream -> the id ring slots of the embedding stages; target ids [T] int32 -> target ring.
template <typename E>
__device__ __forceinline__ void copy_in(E* __restrict__ dst, const E* __restrict__ src, uint64_t n, uint64_t gid, uint64_t stride) {
  constexpr uint64_t V = 16 / sizeof(E);
  uint64_t done = 0;
  if ((((uintptr_t)dst | (uintptr_t)src) & 15) == 0) {      // the caller's pointer and an odd-sized slot may start anywhere
    done = n / V * V;
    for (uint64_t i = gid; i < n / V; i += stride) reinterpret_cast<uint4*>(dst)[i] = reinterpret_cast<const uint4*>(src)[i];
  }
  for (uint64_t i = done + gid; i < n; i += stride) dst[i] = src[i];
}

constexpr int kBeginThreads = 128;

template <typename AT, bool MB>
__global__ void __launch_bounds__(kBeginThreads) begin_kernel(const StageSched* __restrict__ sched, StageDyn* __restrict__ dyn, HyperDev hp, int64_t tick, int64_t n_fed,
                                                              const int32_t* __restrict__ delays, const int64_t* __restrict__ nupd, int sched_blocks, int per_table,
                                                              TickArgs t, const void* __restrict__ inputs, const void* __restrict__ targets, int64_t mb) {
  if ((int)blockIdx.x < sched_blocks) {
    if (MB) schedule_mb(sched, dyn, hp, mb, delays, nupd, (int)blockIdx.x % per_table, (int)blockIdx.x / per_table);
    else schedule_tick(sched, nupd, dyn, hp, tick, n_fed, (int)blockIdx.x);
    return;
  }
  const StageDev& s0 = t.st[0];
  const uint64_t gid = (uint64_t)(blockIdx.x - sched_blocks) * blockDim.x + threadIdx.x, stride = (uint64_t)(gridDim.x - sched_blocks) * blockDim.x;
  const uint64_t T = (uint64_t)t.T;
  if (s0.pre == PRE_EMBED) {
    const int32_t* ids = reinterpret_cast<const int32_t*>(inputs);
    copy_in<int32_t>(ring_at<int32_t>(t, s0.ids_ring, (int)(mb % s0.ids_depth), T), ids, T, gid, stride);
    if (t.n_streams > 1) {                                    // second token stream -> the stage that embeds it
      const StageDev& s1 = t.st[t.second_embed_stage];
      copy_in<int32_t>(ring_at<int32_t>(t, s1.ids_ring, (int)(mb % s1.ids_depth), T), ids + T, T, gid, stride);
    }
  } else {
    const uint64_t n = T * t.n_in_first;
    copy_in<AT>(ring_at<AT>(t, s0.x_ring, (int)(mb % s0.xdepth), n), reinterpret_cast<const AT*>(inputs), n, gid, stride);
  }
  if (t.loss_kind == PM_LOSS_CE) {
    copy_in<int32_t>(ws_at<int32_t>(t, t.tgt_off) + (uint64_t)(mb % (t.P + 1)) * T, reinterpret_cast<const int32_t*>(targets), T, gid, stride);
  } else {
    const uint64_t n = T * t.n_out_last;
    copy_in<float>(ws_at<float>(t, t.tgt_off) + (uint64_t)(mb % (t.P + 1)) * n, reinterpret_cast<const float*>(targets), n, gid, stride);
  }
}

cudaError_t launch_begin(const StageSched* sched, StageDyn* dyn, HyperDev hp, int64_t tick, int64_t n_fed, bool mb_order, const int32_t* delays,
                         const int64_t* nupd, const TickArgs& t, int dtype, const void* inputs, const void* targets, int64_t mb, cudaStream_t stream) {
  const int per_table = (4 * hp.n_stages + kBeginThreads - 1) / kBeginThreads;
  const int sched_blocks = per_table * (mb_order ? mb_table_count(hp.n_stages, hp.segment) : 1);
  int copy_blocks = 0;
  if (inputs) {
    // 16 bytes per thread and array; the larger of the arrays decides, capped at a chip-full of blocks
    const uint64_t x = t.n_in_first > 0 ? (uint64_t)t.T * t.n_in_first * (dtype == PM_F32 ? 4 : 2) : (uint64_t)t.T * 4;
    const uint64_t y = t.loss_kind == PM_LOSS_CE ? (uint64_t)t.T * 4 : (uint64_t)t.T * t.n_out_last * 4;
    const uint64_t need = ((x > y ? x : y) / 16 + kBeginThreads) / kBeginThreads;
    copy_blocks = (int)(need < 1184 ? need : 1184);
  }
#define PM_BEGIN(AT, MB) begin_kernel<AT, MB><<<sched_blocks + copy_blocks, kBeginThreads, 0, stream>>>(sched, dyn, hp, tick, n_fed, delays, nupd, sched_blocks, per_table, t, inputs, targets, mb)
  if (dtype == PM_F32) { if (mb_order) PM_BEGIN(float, true); else PM_BEGIN(float, false); }
  else { if (mb_order) PM_BEGIN(__nv_bfloat16, true); else PM_BEGIN(__nv_bfloat16, false); }
#undef PM_BEGIN
  return cudaGetLastError();
}

// ---- read-back ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) report_kernel(const float* log, int64_t first, int n, int64_t cap, const int* status0, const int* status1, float* host, int words) {
  for (int i = (int)threadIdx.x; i < n; i += 128) host[i] = log[(first + i) % cap];
  if (threadIdx.x < 2) {
    const int* w = threadIdx.x == 0 ? status0 : status1;
    reinterpret_cast<int*>(host)[words + threadIdx.x] = w ? *w : 0;
  }
  __threadfence_system();
}

cudaError_t launch_report(const float* log, int64_t first, int n, int64_t cap, const int* status0, const int* status1, float* host, int words, cudaStream_t stream) {
  report_kernel<<<1, 128, 0, stream>>>(log, first, n, cap, status0, status1, host, words);
  return cudaGetLastError();
}

// ---- stand-alone update: stage tables ------------------------------------------------------------------------
// The caller's stage split comes as a kernel argument (no copy from pageable host memory in front of the launch); the kernel
// writes the bounds, the scalars of update index k and zeroed counters into the workspace.
template <int N>
__global__ void __launch_bounds__(128) flat_table_kernel(__grid_constant__ const FlatTable<N> tab, HyperDev hp, int64_t k, uint32_t* __restrict__ begin64,
                                                         uint32_t* __restrict__ end64, StageDyn* __restrict__ dyn, int64_t* __restrict__ nupd) {
  pdl_trigger();
  const int quad = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 2;
  const int P = hp.n_stages, i = quad < P ? quad : P - 1;
  StageSched s{};
  s.tau_f = tab.tau_f[i]; s.gap = tab.gap[i]; s.depth = 1; s.xdepth = 1;
  const StageDyn d = make_dyn(s, hp, 0, -1, -1, k, 0, 0, false, -1);
  if (quad < P && (threadIdx.x & 3) == 0) { dyn[i] = d; nupd[i] = 0; begin64[i] = tab.begin64[i]; end64[i] = tab.end64[i]; }
}

template <int N>
static cudaError_t flat_table_t(const FlatStage* st, HyperDev hp, int64_t k, uint32_t* begin64, uint32_t* end64, StageDyn* dyn, int64_t* nupd, cudaStream_t stream) {
  FlatTable<N> tab;
  for (int i = 0; i < hp.n_stages; ++i) { tab.begin64[i] = st[i].begin64; tab.end64[i] = st[i].end64; tab.tau_f[i] = st[i].tau_f; tab.gap[i] = st[i].gap; }
  flat_table_kernel<N><<<(4 * hp.n_stages + 127) / 128, 128, 0, stream>>>(tab, hp, k, begin64, end64, dyn, nupd);
  return cudaGetLastError();
}

cudaError_t launch_flat_table(const FlatStage* st, HyperDev hp, int64_t k, uint32_t* begin64, uint32_t* end64, StageDyn* dyn, int64_t* nupd, cudaStream_t stream) {
  // argument sizes of 1, 4 and 16 KB: a launch copies all of them
  if (hp.n_stages <= 64) return flat_table_t<64>(st, hp, k, begin64, end64, dyn, nupd, stream);
  if (hp.n_stages <= 256) return flat_table_t<256>(st, hp, k, begin64, end64, dyn, nupd, stream);
  return flat_table_t<PM_MAX_STAGES>(st, hp, k, begin64, end64, dyn, nupd, stream);
}

// ---- fused update ------------------------------------------------------------------------------

__device__ __forceinline__ float4 ld_stream(const float* p) { return __ldcs(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ void st_stream(float* p, float4 v) { __stcs(reinterpret_cast<float4*>(p), v); }

constexpr int kUpdThreads = 128;

// What bounds the kernel: HBM.  One block per 1024 elements, in ascending order, and not a persistent grid: resident blocks then
// work on one moving window of the arenas, where grid-stride blocks drift apart and the nine streams lose their DRAM pages.
// 100 M parameters, Adam, 64 stages: 674 us with eight persistent blocks of 256 threads per SM, 633 with a block of 256 threads
// per chunk, 615 when the look-up tries the stage an even split would give before it searches, 598 with blocks of 128 threads
// (6.36 TB/s).  U: float4 groups per thread and array.  Two while there are many waves of blocks (one: 602 us); one for small
// networks, where a launch is as long as a thread's chain of divisions (a tick of the 4-stage MLP 36.9 -> 34.8 us).

// The stage tables and gradients come from launches that may still be running when this one starts, so they are read by plain
// loads behind the wait: a read-only (non-coherent) load is defined for memory that nobody writes during the kernel's
// lifetime, and the compiler may move it across the wait.
// LP: operand-type copy of the new weights: 0 none, 1 bfloat16, 2 float (a version-ring slot of fp32 operands);
// element e of the arenas goes to lp_base[lp_shift + e], lp_shift from the stage's table entry (0: the w_lp arena)
// PARTS: only the parts of the stages that the weight-gradient GEMM's epilogue has not updated, a block per chunk of one part.
// (Blocks over the whole arenas find nothing to do for most of a large network: beside the fused weight gradients of an
// encoder-decoder of 4 + 4 layers of width 1024 the kernels of the update took 557 us, these 403; of the 6-layer encoder 60 and 38.)
template <int OPT, int LP, int U, bool PARTS>
__global__ void __launch_bounds__(kUpdThreads, 6)
update_kernel(ArenasDev a, void* lp_base, const uint32_t* begin64, const uint32_t* end64,
              const StageDyn* dyn, int64_t* nupd, int n_stages, uint64_t total_vec4,
              float beta1, float beta2, float eps, uint64_t first_vec4, const UpdPart* parts, int n_parts,
              const float* gsrc, float stages_per_group) {
  pdl_trigger();
  pdl_wait();
  const float omb1 = __fsub_rn(1.0f, beta1), omb2 = __fsub_rn(1.0f, beta2);
  uint64_t base = first_vec4 + (uint64_t)blockIdx.x * kUpdThreads * U, counter = ~0ull;   // PARTS: the element group whose thread keeps the stage's counter
  int lo0 = 0;
  if (PARTS) {
    int pi = 0, hi = n_parts - 1;                                           // the part of this chunk: the last that starts at or before it
    while (pi < hi) { const int mid = (pi + hi + 1) >> 1; if (parts[mid].first_chunk <= blockIdx.x) pi = mid; else hi = mid - 1; }
    const UpdPart q = parts[pi];
    lo0 = q.stage;
    base = (uint64_t)q.begin64 * 16 + (uint64_t)(blockIdx.x - q.first_chunk) * kUpdThreads * U;
    total_vec4 = (uint64_t)q.end64 * 16;
    if (q.counts) counter = (uint64_t)q.begin64 * 16;
  } else {
    // the stage of the block's first group: the largest i with begin64[i] <= g0 (every thread searches, on the same addresses)
    const uint32_t g0 = (uint32_t)(base >> 4);
    int hi = n_stages - 1;
    const int q = min(hi, (int)((float)g0 * stages_per_group));            // where it is if all stages have the same size
    if (begin64[q] <= g0 && (q == hi || g0 < begin64[q + 1])) lo0 = hi = q;
    while (lo0 < hi) { const int mid = (lo0 + hi + 1) >> 1; if (begin64[mid] <= g0) lo0 = mid; else hi = mid - 1; }
  }
  uint64_t v[U];
  int stage[U];
  UpdScalars sc[U];
  float4 g[U], w[U], m[U], dl[U], s[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    v[u] = base + (uint64_t)u * kUpdThreads + threadIdx.x;
    stage[u] = -1;
    if (v[u] < total_vec4) {
      const uint32_t e64 = (uint32_t)(v[u] >> 4);
      int lo = lo0;
      if (!PARTS) while (lo + 1 < n_stages && begin64[lo + 1] <= e64) ++lo;      // a block spans 8 or 16 groups: rarely more than one stage on
      if ((PARTS || (begin64[lo] <= e64 && e64 < end64[lo])) && dyn[lo].active_update) stage[u] = lo;
    }
    if (stage[u] >= 0) {
      const uint64_t e = v[u] * 4;
      const StageDyn& d = dyn[stage[u]];
      g[u] = ld_stream(gsrc + (d.g_shift + (int64_t)e));
      w[u] = ld_stream(a.w + e);
      m[u] = ld_stream(a.m + e);
      sc[u].alpha = d.alpha; sc[u].gamma = d.gamma; sc[u].omg = d.one_minus_gamma;
      sc[u].bc1 = d.bc1; sc[u].bc2 = d.bc2; sc[u].use_delta = d.use_delta;
      if (LP != 0) { sc[u].lp_shift = d.lp_shift; sc[u].rc_shift = d.rc_uslot >= 0 ? d.rc_shift : -1; sc[u].rc_gap = d.rc_gap; }
      if (sc[u].use_delta || (LP != 0 && sc[u].rc_shift >= 0)) dl[u] = ld_stream(a.delta + e);
      if (OPT == PM_ADAM) s[u] = ld_stream(a.s + e);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (stage[u] < 0) continue;
    const uint64_t e = v[u] * 4;
    float4 wn;
    wn.x = upd_one<OPT>(g[u].x, w[u].x, m[u].x, s[u].x, dl[u].x, sc[u], beta1, beta2, omb1, omb2, eps);
    wn.y = upd_one<OPT>(g[u].y, w[u].y, m[u].y, s[u].y, dl[u].y, sc[u], beta1, beta2, omb1, omb2, eps);
    wn.z = upd_one<OPT>(g[u].z, w[u].z, m[u].z, s[u].z, dl[u].z, sc[u], beta1, beta2, omb1, omb2, eps);
    wn.w = upd_one<OPT>(g[u].w, w[u].w, m[u].w, s[u].w, dl[u].w, sc[u], beta1, beta2, omb1, omb2, eps);
    st_stream(a.w + e, wn);
    st_stream(a.m + e, m[u]);
    if (OPT == PM_ADAM) st_stream(a.s + e, s[u]);
    if (sc[u].use_delta) st_stream(a.delta + e, dl[u]);
    if (LP == 1) {
      __nv_bfloat162 lo2 = __floats2bfloat162_rn(wn.x, wn.y);
      __nv_bfloat162 hi2 = __floats2bfloat162_rn(wn.z, wn.w);
      uint2 packed;
      packed.x = *reinterpret_cast<uint32_t*>(&lo2);
      packed.y = *reinterpret_cast<uint32_t*>(&hi2);
      *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(lp_base) + (sc[u].lp_shift + (int64_t)e)) = packed;   // re-read by a later forward: default caching
    } else if (LP == 2) {
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(lp_base) + (sc[u].lp_shift + (int64_t)e)) = wn;
    }
    if (LP != 0 && sc[u].rc_shift >= 0) {
      // T2 for recompute (Appendix D): the weights a recomputation tau_recomp updates from now reads, corrected with the
      // accumulator as it stands with this version: w' - (tau_fwd - tau_recomp) * delta'
      const float gp = sc[u].rc_gap;
      float4 r;
      r.x = __fsub_rn(wn.x, __fmul_rn(gp, dl[u].x)); r.y = __fsub_rn(wn.y, __fmul_rn(gp, dl[u].y));
      r.z = __fsub_rn(wn.z, __fmul_rn(gp, dl[u].z)); r.w = __fsub_rn(wn.w, __fmul_rn(gp, dl[u].w));
      if (LP == 1) {
        __nv_bfloat162 lo2 = __floats2bfloat162_rn(r.x, r.y);
        __nv_bfloat162 hi2 = __floats2bfloat162_rn(r.z, r.w);
        uint2 packed;
        packed.x = *reinterpret_cast<uint32_t*>(&lo2);
        packed.y = *reinterpret_cast<uint32_t*>(&hi2);
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(lp_base) + (sc[u].rc_shift + (int64_t)e)) = packed;
      } else {
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(lp_base) + (sc[u].rc_shift + (int64_t)e)) = r;
      }
    }
    if (PARTS ? v[u] == counter : (v[u] >> 4) == begin64[stage[u]] && (v[u] & 15) == 0) nupd[stage[u]] += 1;
  }
}

// up to four waves of blocks at one float4 group per thread and array
static bool few_chunks(uint64_t vec4) { return vec4 <= 4ull * kSms * 8 * kUpdThreads; }

UpdParts update_parts(const uint32_t* begin64, const uint32_t* end64, const uint32_t* skip_b64, const uint32_t* skip_e64, int n_stages) {
  UpdParts p;
  uint64_t groups = 0;
  for (int i = 0; i < n_stages; ++i) groups += (skip_b64[i] - begin64[i]) + (end64[i] - skip_e64[i]);
  p.unroll = few_chunks(groups * 16) ? 1 : 2;
  const uint32_t per = (uint32_t)(kUpdThreads * p.unroll / 16);              // groups of a chunk
  auto add = [&](int stage, uint32_t b, uint32_t e, int counts) {
    if (b < e) { p.list.push_back(UpdPart{p.chunks, b, e, stage, counts}); p.chunks += (e - b + per - 1) / per; }
  };
  for (int i = 0; i < n_stages; ++i) {
    add(i, begin64[i], skip_b64[i], 0);
    add(i, skip_e64[i], end64[i], 1);                                        // never empty: the Linear's bias follows its matrix
  }
  return p;
}

bool update_is_short(uint64_t groups64) { return few_chunks(groups64 * 16); }

cudaError_t launch_update(ArenasDev a, const uint32_t* begin64, const uint32_t* end64, const StageDyn* dyn,
                          int64_t* nupd, int n_stages, uint64_t total64, int optimizer, float beta1, float beta2,
                          float eps, cudaStream_t stream, void* lp_base, int lp_elem, uint64_t first64, const float* gsrc, bool pdl) {
  if (total64 == 0 || n_stages == 0 || first64 >= total64) return cudaSuccess;
  uint64_t total_vec4 = total64 * 16;
  const uint64_t first_vec4 = first64 * 16;
  const bool small = few_chunks(total_vec4 - first_vec4);
  const uint64_t per_block = (uint64_t)kUpdThreads * (small ? 1 : 2);
  const unsigned blocks = (unsigned)((total_vec4 - first_vec4 + per_block - 1) / per_block);   // 1024 elements per block: 2^31 blocks are 2e12 elements
  // the operand-type copy: the w_lp arena (bfloat16) unless the caller names a version ring and its element size
  if (lp_base == nullptr) { lp_base = a.w_lp; lp_elem = 2; }
  if (gsrc == nullptr) gsrc = a.grad;
  const int lp = lp_base == nullptr ? 0 : (lp_elem == 4 ? 2 : 1);
  const float per_group = (float)n_stages / (float)total64;
#define PM_UPD(OPT, LP) launch_pdl(small ? update_kernel<OPT, LP, 1, false> : update_kernel<OPT, LP, 2, false>, dim3(blocks), dim3(kUpdThreads), 0, stream, pdl, a, lp_base, begin64, end64, dyn, nupd, n_stages, total_vec4, beta1, beta2, eps, first_vec4, nullptr, 0, gsrc, per_group)
  if (optimizer == PM_SGDM) return lp == 0 ? PM_UPD(PM_SGDM, 0) : (lp == 1 ? PM_UPD(PM_SGDM, 1) : PM_UPD(PM_SGDM, 2));
  return lp == 0 ? PM_UPD(PM_ADAM, 0) : (lp == 1 ? PM_UPD(PM_ADAM, 1) : PM_UPD(PM_ADAM, 2));
#undef PM_UPD
}

cudaError_t launch_update_parts(ArenasDev a, const UpdParts& p, const UpdPart* d_parts, const StageDyn* dyn, int64_t* nupd, int optimizer,
                                float beta1, float beta2, float eps, cudaStream_t stream, void* lp_base, bool pdl) {
  if (p.chunks == 0) return cudaSuccess;
  if (lp_base == nullptr) lp_base = a.w_lp;
#define PM_UPD(OPT) launch_pdl(p.unroll == 1 ? update_kernel<OPT, 1, 1, true> : update_kernel<OPT, 1, 2, true>, dim3(p.chunks), dim3(kUpdThreads), 0, stream, pdl, a, lp_base, nullptr, nullptr, dyn, nupd, 0, 0, beta1, beta2, eps, 0, d_parts, (int)p.list.size(), a.grad, 0.f)
  return optimizer == PM_SGDM ? PM_UPD(PM_SGDM) : PM_UPD(PM_ADAM);
#undef PM_UPD
}

// ---- fp32 copies of the small forward-read tensors into the version rings -------------------------------------
// With bfloat16 operands the forward pass still reads biases and LayerNorm parameters in fp32; in microbatch-major
// order their versions sit in a ring of their own, filled here from the master weights after every update.
__global__ void __launch_bounds__(128) push_small_kernel(const float* w, const float* delta, char* ring, const SmallSeg* __restrict__ segs, int n_segs,
                                                         const StageDyn* dyn, int slot_override) {
  pdl_trigger();
  pdl_wait();
  for (int sg = blockIdx.x; sg < n_segs; sg += gridDim.x) {
    const SmallSeg g = segs[sg];
    if (slot_override < 0 && !dyn[g.stage].active_update) continue;          // the stage was not updated this tick
    const int slot = slot_override >= 0 ? slot_override : dyn[g.stage].u_vslot;
    float* base = reinterpret_cast<float*>(ring + g.ring_off);
    float* dst = base + (uint64_t)slot * g.slot_stride;
    const float* src = w + g.arena_off;
    // corrected recompute weights of the same version (T2 for recompute, Appendix D): w - (tau_fwd - tau_recomp) * delta
    const int rslot = g.rc_base < 0 ? -1 : (slot_override >= 0 ? g.rc_base + slot_override : dyn[g.stage].rc_uslot);
    float* rdst = rslot >= 0 ? base + (uint64_t)rslot * g.slot_stride : nullptr;
    const float gap = (rslot >= 0 && slot_override < 0) ? dyn[g.stage].rc_gap : 0.f;
    const float* dl = delta + g.arena_off;
    for (uint32_t i = threadIdx.x * 4; i < g.count; i += blockDim.x * 4) {
      const float4 v = *reinterpret_cast<const float4*>(src + i);
      *reinterpret_cast<float4*>(dst + i) = v;
      if (rdst) {
        float4 r = v;
        if (slot_override < 0) {
          const float4 d4 = *reinterpret_cast<const float4*>(dl + i);
          r.x = __fsub_rn(v.x, __fmul_rn(gap, d4.x)); r.y = __fsub_rn(v.y, __fmul_rn(gap, d4.y));
          r.z = __fsub_rn(v.z, __fmul_rn(gap, d4.z)); r.w = __fsub_rn(v.w, __fmul_rn(gap, d4.w));
        }
        *reinterpret_cast<float4*>(rdst + i) = r;
      }
    }
  }
}

cudaError_t launch_push_small(const float* w, const float* delta, char* ring, const SmallSeg* segs, int n_segs, const StageDyn* dyn,
                              int slot_override, cudaStream_t stream, bool pdl) {
  if (n_segs == 0) return cudaSuccess;
  return launch_pdl(push_small_kernel, dim3(n_segs < 1184 ? n_segs : 1184), dim3(128), 0, stream, pdl, w, delta, ring, segs, n_segs, dyn, slot_override);
}

}  // namespace pm
