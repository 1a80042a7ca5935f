// Tick scheduler and the fused multi-tensor PipeMare update (declarations).
#pragma once
#include <vector>

#include "pm_common.cuh"

namespace pm {

// What the scheduler needs to know about a stage (device table, constant over the run).
struct StageSched {
  int32_t tau_f, gap, depth, xdepth, next_xdepth, gin_depth, prev_gin_depth, gmem_depth;
  int32_t skip_dst_depth, skip_depth;   // slots of the skip buffer this stage writes into / reads from (0: none)
  // version rings (microbatch-major order; vdepth <= 1: none): slots, the stage's element range in the arenas and the
  // byte offset of its operand-type ring in the ring arena
  int32_t vdepth, _pad;
  uint64_t begin, count, v_ring;
  int32_t tau_r, rdepth;                // PipeMare Recompute: delay of the recomputation's weights, slots of their corrected queue
};

struct TickArgs;
// Starts a tick: fills the schedule table(s) and, with inputs, copies the microbatch `mb` into the rings.
// Tick-major order: the table of pipeline tick `tick` with `n_fed` microbatches fed so far.
// Microbatch-major order (mb_order): the tables of microbatch mb ([n_tables][P] entries): table v < 2P for the launches of
// sub-tick v (stage i forward at v = i, backward at v = 2P - 1 - i), table 2P for the grouped weight-gradient launch
// and the update.  With PipeMare Recompute (hp.segment > 0) table 2P + 1 holds every stage's recomputation (its forward
// entry with the recompute weights' slot) and table 2P + 2 + k the backward entries of segment k alone (the grouped
// weight-gradient launch of that segment).
// delays (stochastic delay model only, else null): the step's per-stage delays.  nupd: the stages' update counters.
cudaError_t launch_begin(const StageSched* sched, StageDyn* dyn, HyperDev hp, int64_t tick, int64_t n_fed, bool mb_order, const int32_t* delays,
                         const int64_t* nupd, const TickArgs& t, int dtype, const void* inputs, const void* targets, int64_t mb, cudaStream_t stream);
// Is the update of that many groups of 64 elements a few waves of blocks?
bool update_is_short(uint64_t groups64);
// Losses of microbatches first .. first + n - 1 from the log (a ring of `cap`) and up to two status words (null: 0) into host memory the
// device can write: host[0 .. n) and host[words], host[words + 1].
cudaError_t launch_report(const float* log, int64_t first, int n, int64_t cap, const int* status0, const int* status1, float* host, int words, cudaStream_t stream);
// Stand-alone update: bounds, scalars of update index k and zeroed counters of hp.n_stages stages into device tables.
struct FlatStage { uint32_t begin64, end64; int32_t tau_f, gap; };
template <int N> struct FlatTable { uint32_t begin64[N], end64[N]; int32_t tau_f[N], gap[N]; };
cudaError_t launch_flat_table(const FlatStage* st, HyperDev hp, int64_t k, uint32_t* begin64, uint32_t* end64, StageDyn* dyn, int64_t* nupd, cudaStream_t stream);
inline int mb_table_count(int P, int segment) { return 2 * P + 1 + (segment > 0 ? 1 + (P + segment - 1) / segment : 0); }

// Launches the fused update over all stages whose dyn[i].active_update is set.
// begin64/end64: stage bounds in units of 64 elements, ascending; total64 = end64[P-1].
cudaError_t launch_update(ArenasDev a, const uint32_t* begin64, const uint32_t* end64, const StageDyn* dyn,
                          int64_t* nupd, int n_stages, uint64_t total64, int optimizer, float beta1, float beta2,
                          float eps, cudaStream_t stream, void* lp_base = nullptr, int lp_elem = 0, uint64_t first64 = 0,
                          const float* gsrc = nullptr, bool pdl = false);
// pdl: launched as a programmatic dependent of the launch before it.
// gsrc: where the gradients are read (element e of stage i at gsrc[dyn[i].g_shift + e]); null: the grad arena.
// first64: the walk over the arenas starts at this 64-element group (a launch for one stage starts at that stage's slice).
// lp_base / lp_elem: where the operand-type copy of the new weights goes: by default the bfloat16 arena a.w_lp
// (if there is one); microbatch-major order passes the ring arena and the operand size (2 or 4 bytes), and the
// stages' table entries give the slot (StageDyn::lp_shift).

// When the weight-gradient GEMM has updated the Linear matrices in its epilogue, the parts of the stages it has left: elements in
// groups of 64, in chunks of one block each.  The part that counts keeps the stage's update counter.
struct UpdPart { uint32_t first_chunk, begin64, end64; int32_t stage, counts; };
struct UpdParts { std::vector<UpdPart> list; uint32_t chunks = 0; int32_t unroll = 1; };
// [begin64, skip_b64) and [skip_e64, end64) of every stage (host arrays)
UpdParts update_parts(const uint32_t* begin64, const uint32_t* end64, const uint32_t* skip_b64, const uint32_t* skip_e64, int n_stages);
// d_parts: the list on the device.  bf16 networks: lp_base is the ring arena or null (the w_lp arena).
cudaError_t launch_update_parts(ArenasDev a, const UpdParts& p, const UpdPart* d_parts, const StageDyn* dyn, int64_t* nupd, int optimizer,
                                float beta1, float beta2, float eps, cudaStream_t stream, void* lp_base, bool pdl);

// One fp32 tensor the forward pass reads (a bias, a LayerNorm gain or bias): `count` elements (a multiple of 64,
// padding included) at arena_off of the master weights; its versions sit at ring_off (bytes, slot 0) of the ring
// arena, slot_stride floats apart.
// rc_base: first slot of the stage's corrected recompute weights (= its vdepth), -1 when it keeps none.
struct SmallSeg { uint64_t arena_off, ring_off; uint32_t count, slot_stride; int32_t stage, rc_base; };
// Copies every segment from the master weights into slot dyn[stage].u_vslot of its ring and, for a stage with a queue of
// corrected recompute weights, w - dyn[stage].rc_gap * delta into slot dyn[stage].rc_uslot.  slot_override >= 0 (the
// initial fill, delta = 0): plain copies into that slot and into rc_base + slot_override.
cudaError_t launch_push_small(const float* w, const float* delta, char* ring, const SmallSeg* segs, int n_segs, const StageDyn* dyn,
                              int slot_override, cudaStream_t stream, bool pdl = false);

}  // namespace pm
