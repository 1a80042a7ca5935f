"""What pm_query_bytes asks for as workspace: buffers that a network's kernels read, at the sizes they read."""
import ctypes as C

import pytest

import pm_inputs as I
from test_abi_symbols import _describe, built_lib


def workspace(wl, order):
    from paper_1910_05124_b200 import binding as B
    cfg, sd, keep = _describe(wl)
    cfg.loop_order = B.PM_MB_MAJOR if order == "mb_major" else B.PM_TICK_MAJOR
    sb, rb, wb = C.c_uint64(), C.c_uint64(), C.c_uint64()
    assert B.lib().pm_query_bytes(C.byref(cfg), sd, C.byref(sb), C.byref(rb), C.byref(wb)) == 0
    return wb.value


# A layer more costs the same whatever the vocabulary: only the embedding and the projection are as wide as it, and the cross-entropy's
# targets are a word per token.  (Tile tables differ by a few KB.)
@pytest.mark.parametrize("compute,seq", [("f32", 16), ("bf16", 128)])
@pytest.mark.parametrize("order", ["tick_major", "mb_major"])
def test_a_layer_costs_no_vocabulary(built_lib, order, compute, seq):
    need = {}
    for layers in (1, 2):
        for vocab in (264, 8264):
            wl = I.encoder_workload("ws", layers, 512, 8, 2048, seq, 4096 // seq, vocab, compute=compute, optimizer="adam", alpha=1e-3, K=4, D=0.1, steps=1, seed=1)
            need[layers, vocab] = workspace(wl, order)
    wide, narrow = need[2, 8264] - need[1, 8264], need[2, 264] - need[1, 264]
    assert abs(wide - narrow) < 1 << 18, (wide, narrow)


# A bf16 residual stage's GEMM adds the skip tensor itself: nothing waits for a launch that does.  What a layer keeps, in tensors of
# T x d bf16: attention stage 3 (gradient of q, k, v) + 3 mailbox slots + 1 (gradient of the LayerNorm's output); projection 3 mailbox slots +
# 2 of the skip tensor; hidden stage, 4 d wide, 4 x 3 mailbox slots + 4 (dz) + 1; output stage 3 + 2.  Tables and partial sums are less than one.
def test_residual_stages_keep_no_sum_waiting(built_lib):
    T, d, need = 4096, 64, {}
    for layers in (1, 2):
        wl = I.encoder_workload("ws", layers, d, 1, 4 * d, 128, 32, 264, compute="bf16", optimizer="adam", alpha=1e-3, K=4, D=0.1, steps=1, seed=1)
        need[layers] = workspace(wl, "tick_major")
    assert 34 <= (need[2] - need[1]) / (T * d * 2) < 35
