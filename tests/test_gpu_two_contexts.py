"""Contexts of one process do not disturb each other: shared-memory limits belong to a kernel, not to a context."""
import threading

import numpy as np
import pytest

import pm_inputs as I

pytestmark = pytest.mark.gpu


def _pipe(wl, **kw):
    import paper_1910_05124_b200 as pm
    return pm.Pipeline(wl, I.init_encoder_params(wl), loop_order="mb_major", **kw)


def _tokens(wl, t=0):
    import torch
    return tuple(torch.from_numpy(a.astype(np.int32)).cuda() for a in I.token_batch(wl, t))


# the larger network is made first; both of its attention kernels need more than the smaller one's
@pytest.mark.parametrize("compute", ["f32", "bf16"])
def test_smaller_context_made_later(cuda_device, compute):
    kw = dict(compute=compute, optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=1, seed=3)
    large = I.encoder_workload("large", 1, 64, 2, 64, 100, 2, 64, **kw)
    small = I.encoder_workload("small", 1, 32, 1, 64, 8, 2, 64, **kw)
    alone = _pipe(large)
    alone.pm_step(*_tokens(large))
    a, b = _pipe(large), _pipe(small)
    b.pm_step(*_tokens(small))
    a.pm_step(*_tokens(large))
    assert a.pm_get_losses(0, 1)[0] == alone.pm_get_losses(0, 1)[0]


# rows of logits in shared memory (one kernel for both): 131 KB and 33 KB, stepped by two threads on streams of their own, without graphs
def test_two_threads(cuda_device, monkeypatch):
    import torch
    monkeypatch.setenv("PM_CUDA_GRAPHS", "0")
    kw = dict(compute="bf16", optimizer="sgdm", alpha=0.01, K=4, D=0.5, steps=1, seed=3)
    wls = [I.encoder_workload("wide", 1, 64, 1, 64, 8, 1, v, **kw) for v in (32768, 8200)]
    pipes = [_pipe(wl, stream=torch.cuda.Stream()) for wl in wls]
    toks = [_tokens(wl) for wl in wls]
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            for _ in range(4000):
                pipes[i].pm_step(*toks[i])
        except Exception as e:                               # noqa: BLE001
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for p in pipes:
        assert np.isfinite(p.pm_get_losses(3999, 1)).all()
