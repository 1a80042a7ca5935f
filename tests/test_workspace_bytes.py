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

