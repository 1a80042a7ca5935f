// bf16 tensor-core grouped GEMMs of the pipeline (tcgen05 + TMEM + TMA): interface to the host code.
#pragma once
#include <string>
#include <vector>
#include "pm_tick.cuh"

namespace pm {

struct UmmaPlan;   // tensor maps and launch geometry, built once per context

// Bytes of caller workspace the plan needs (status word, tensor maps, tile tables).
uint64_t umma_workspace_bytes(int T, const std::vector<StageDev>& st);
// ws_region: device memory of at least umma_workspace_bytes(T, stages), 256-byte aligned.  Synchronises `stream`.
pm_status umma_plan_create(UmmaPlan** out, const TickArgs& t, const std::vector<StageDev>& st, void* ws_region,
                           cudaStream_t stream, std::string& err);
void umma_plan_destroy(UmmaPlan* plan);
// Device word that a CTA sets when one of its bounded waits expired (0 = none).
int* umma_status_word(UmmaPlan* plan);
// Self-test: launches a one-thread kernel whose bounded wait (limit in SM cycles) must expire; it sets the plan's status
// word like a real expiry would and writes 2 to *d_returned.  umma_clear_status resets the status word.
cudaError_t umma_wait_timeout_probe(UmmaPlan* plan, long long limit_cycles, int* d_returned, cudaStream_t stream);
cudaError_t umma_clear_status(UmmaPlan* plan, cudaStream_t stream);
// does the dgrad of this Linear, launched for its stage alone, run on the kernel for few tiles (pm_umma_row.cuh)?
bool umma_row_dgrad(int T, const LinDev& L);
// Does the dgrad of Linear l of stage p read the corrected weights from scratch (LinDev::wc_off)?  one_stage / grouped: the context
// launches it for its stage alone / for all stages together.
bool umma_corr_weights(int T, const std::vector<StageDev>& st, int p, int l, bool one_stage, bool grouped);
// Forms them, for the stages in backward (t.sel_p >= 0: that one); umma_corr_blocks: blocks of that launch (p < 0: all stages).
int umma_corr_blocks(const UmmaPlan* plan, int p);
cudaError_t umma_corr_launch(UmmaPlan* plan, const TickArgs& t, cudaStream_t stream);
// Does the forward / the dgrad of Linear l of stage p run on the kernels for many tiles, whose epilogues write and apply ReLU mask bits
// (LinDev::mask_out), in every launch?  queued: the dgrad reads a queued version of the weights.
bool umma_fwd_plain(int T, const std::vector<StageDev>& st, int p, int l, bool one_stage, bool grouped);
bool umma_dgrad_plain(int T, const std::vector<StageDev>& st, int p, int l, bool one_stage, bool grouped, bool queued);
// mode: 0 forward, 1 dgrad (corrected weights, or with t.stash the queued version), 2 wgrad.
cudaError_t umma_launch(UmmaPlan* plan, const TickArgs& t, int mode, int lvl, cudaStream_t stream);

}  // namespace pm
