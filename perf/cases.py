"""The work this framework is timed on: training steps of every network kind, loop order and operand type it builds, and
the fused update on its own.

One pass of a network case is one weight update as a training program makes it: `pm_step` for every microbatch of the
update (one, unless `n_micro` says more) and, where the program logs, the loss it reads back.  A network is a run in
progress: weights from the usual initialisation, optimiser moments and discrepancy accumulator as a resumed run has them,
the pipeline filled (tick-major order) or a few updates old (microbatch-major order).  Microbatches rotate through a small
set that is already on the GPU.  One pass of an update case is one `pm_update_flat`.

Outputs are the whole state an update leaves behind: master weights, moments, discrepancy accumulator, the bf16 weights
where the update writes them to an arena, the gradient of fp32 networks, and the loss where it is read.  The gradient of
a bf16 network is seen through the first moment: at this depth the roundings of one microbatch (six per stage, 2^-9
each) put two correct implementations 3 to 13 % apart in a single gradient, whatever their order of summation, and the
moment averages that.
"""
import math

import torch

import paper_1910_05124_b200 as pm
import pm_inputs

ADAM_S = 3e-4      # a resumed run's second moments are around the square of this (a typical gradient entry)
N_BATCHES = 32
ALPHA = 0.1        # of the configurations' peak step size: a run whose schedule has come down


# ---- the cases -----------------------------------------------------------------------------------------------------

def _update(n, stages, optimizer):
    return dict(kind="update", n=n, stages=stages, optimizer=optimizer)


def _mlp(stages, width, linears, act, rows, compute, optimizer, order, n_micro=1, log=False):
    return dict(kind="mlp", stages=stages, width=width, linears=linears, act=act, rows=rows, compute=compute,
                optimizer=optimizer, order=order, n_micro=n_micro, option="none", log=log)


def _encoder(layers, heads, d_head, d_ff, seq, batch, vocab, compute, order, log=False):
    return dict(kind="encoder", layers=layers, heads=heads, d_head=d_head, d_ff=d_ff, seq=seq, batch=batch, vocab=vocab,
                compute=compute, optimizer="adam", order=order, n_micro=1, option="none", log=log)


def _encdec(enc, dec, heads, d_head, d_ff, seq, batch, vocab, compute, order, option="none", log=False):
    return dict(kind="encdec", enc=enc, dec=dec, heads=heads, d_head=d_head, d_ff=d_ff, seq=seq, batch=batch, vocab=vocab,
                compute=compute, optimizer="adam", order=order, n_micro=1, option=option, log=log)


def listed():
    named = [
        # the smallest training run: a 4-stage fp32 MLP at 32 rows; every kernel is short, launches decide
        ("mlp4_f32", _mlp(4, 256, 1, "relu", 32, "f32", "sgdm", "tick")),
        # fp32 study of a small network in the paper's loop form, two microbatches per update, widths that no tile divides;
        # prints its loss after every update
        ("mlp6_f32_ragged", _mlp(6, 200, 2, "gelu", 50, "f32", "adam", "mb", n_micro=2, log=True)),
        # the convolution-net-like configuration: 32 stages, 67 M parameters, few rows; bound by weight traffic
        ("mlp32_bf16", _mlp(32, 1024, 2, "gelu", 128, "bf16", "sgdm", "tick")),
        # the same network with four microbatches per update, which only microbatch-major order offers
        ("mlp32_bf16_micro4", _mlp(32, 1024, 2, "gelu", 128, "bf16", "sgdm", "mb", n_micro=4)),
        # a mid-sized bf16 network whose width and rows leave remainders in every tile
        ("mlp8_bf16_ragged", _mlp(8, 328, 1, "relu", 72, "bf16", "adam", "tick")),
        # the translation-size encoder: 6 layers, 25 stages, 32 x 128 tokens
        ("encoder6_bf16", _encoder(6, 8, 64, 2048, 128, 32, 8192, "bf16", "tick")),
        # short sequences that are no power of two, an odd batch, in microbatch-major order; prints its loss
        ("encoder2_bf16_ragged", _encoder(2, 3, 64, 520, 96, 7, 1000, "bf16", "mb", log=True)),
        # a small fp32 encoder-decoder, the size people debug with
        ("encdec1_f32_small", _encdec(1, 1, 2, 32, 128, 16, 3, 96, "f32", "tick")),
        # the large encoder-decoder's widths and tokens at 4 + 4 layers (45 stages), microbatch-major order
        ("encdec4_bf16", _encdec(4, 4, 16, 64, 4096, 256, 16, 32000, "bf16", "mb")),
        # the same widths at 2 + 2 layers with the corrected backward weights written out by the update
        ("encdec2_bf16_written", _encdec(2, 2, 16, 64, 4096, 256, 16, 32000, "bf16", "mb", option="written")),
        # the update alone, as a program with its own forward and backward calls it: the smallest and a large model
        ("update_1M_sgdm", _update(1_000_000, 8, "sgdm")),
        ("update_100M_adam", _update(100_000_003, 64, "adam")),
    ]
    return [dict(case, name=name) for name, case in named]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["update", "mlp", "mlp", "mlp", "encoder", "encoder", "encdec", "encdec"])
    if kind == "update":
        return _update(_log_int(rng, 1_000_000, 100_000_000), _log_int(rng, 8, 512), rng.choice(["sgdm", "adam"]))
    order, log = rng.choice(["tick", "mb"]), rng.random() < 0.25
    compute = rng.choice(["f32", "bf16", "bf16"])
    if kind == "mlp":
        optimizer, act = rng.choice(["sgdm", "adam"]), rng.choice(["relu", "gelu"])
        n_micro = rng.choice([1, 2, 4]) if order == "mb" else 1
        if compute == "f32":
            return _mlp(rng.randint(2, 8), _log_int(rng, 64, 384), rng.randint(1, 2), act, _log_int(rng, 16, 128), "f32",
                        optimizer, order, n_micro, log)
        return _mlp(_log_int(rng, 3, 32), 8 * _log_int(rng, 8, 128), rng.randint(1, 2), act, _log_int(rng, 16, 512), "bf16",
                    optimizer, order, n_micro, log)
    if kind == "encoder":
        if compute == "f32":
            heads, d_head, seq = rng.randint(1, 4), rng.choice([16, 32]), _log_int(rng, 8, 48)
            return _encoder(rng.randint(1, 2), heads, d_head, _log_int(rng, 64, 400), seq, rng.randint(2, 8),
                            _log_int(rng, 50, 1000), "f32", order, log)
        heads = rng.randint(2, 8)
        seq = 128 if rng.random() < 0.6 else _log_int(rng, 16, 127)
        return _encoder(rng.randint(1, 4), heads, 64, 8 * _log_int(rng, 32, 256), seq, _log_int(rng, 3, 32),
                        8 * _log_int(rng, 32, 1024), "bf16", order, log)
    if compute == "f32":
        heads, d_head, seq = rng.randint(1, 4), rng.choice([16, 32]), _log_int(rng, 8, 32)
        return _encdec(1, rng.randint(1, 2), heads, d_head, _log_int(rng, 64, 256), seq, rng.randint(2, 6),
                       _log_int(rng, 50, 500), "f32", order, "none", log)
    heads = rng.choice([4, 8, 12, 16])
    option = rng.choice(["none", "none", "written", "recompute"]) if order == "mb" else "none"
    return _encdec(rng.randint(1, 3), rng.randint(1, 3), heads, 64, 256 * heads, rng.choice([128, 256, 256]), rng.randint(3, 16),
                   8 * _log_int(rng, 100, 4000), "bf16", order, option, log)


# ---- preparation -----------------------------------------------------------------------------------------------------

def _workload(case):
    """The workload description of the case, with the hyper-parameters of the repository's configurations."""
    adam = case["optimizer"] == "adam"
    kw = dict(compute=case["compute"], optimizer=case["optimizer"], beta1=0.9, beta2=0.98, eps=1e-8, K=100, D=0.1 if adam else 0.5)
    if case["kind"] == "mlp":
        wl = pm_inputs.mlp_workload("mlp", case["stages"], case["width"], case["linears"], case["act"], case["rows"],
                                    alpha=ALPHA * (5e-4 if adam else 0.01), **kw)
    elif case["kind"] == "encoder":
        wl = pm_inputs.encoder_workload("encoder", case["layers"], case["heads"] * case["d_head"], case["heads"], case["d_ff"],
                                        case["seq"], case["batch"], case["vocab"], alpha=ALPHA * 5e-4, **kw)
    else:
        wl = pm_inputs.encdec_workload("encdec", case["enc"], case["dec"], case["heads"] * case["d_head"], case["heads"],
                                       case["d_ff"], case["seq"], case["batch"], case["vocab"], alpha=ALPHA * 7e-4, **kw)
    wl.tau_fwd, wl.tau_bkwd = pm_inputs.pipemare_delays(wl.n_stages, case["n_micro"])
    return wl


def _act(z, act):
    return torch.relu(z) if act == "relu" else torch.nn.functional.gelu(z)


def _mlp_params(case, normal):
    """Linears N(0, 1/fan_in), rescaled layer by layer so that every pre-activation has unit rms on a calibration batch."""
    w = case["width"]
    h, out = normal(256, w), []
    for _ in range(case["stages"]):
        stage = []
        for _ in range(case["linears"]):
            weight = normal(w, w) / math.sqrt(w)
            z = h @ weight.T
            scale = z.square().mean().rsqrt()
            h = _act(z * scale, case["act"])
            stage.append((weight * scale, torch.zeros(w, device="cuda")))
        out.append(stage)
    return out


def _transformer_params(wl, normal):
    """W ~ N(0, 1/fan_in), tables N(0, 1/d), biases 0, LayerNorm gain 1 and bias 0."""
    out = []
    for sp in wl.stage_specs:
        tensors = []
        if sp.pre in ("embed", "embed_dec"):
            tensors.append(normal(wl.vocab, wl.d_model) / math.sqrt(wl.d_model))
        elif sp.pre == "ln":
            tensors += [torch.ones(sp.n_in, device="cuda"), torch.zeros(sp.n_in, device="cuda")]
        tensors += [normal(sp.n_out, sp.n_in) / math.sqrt(sp.n_in), torch.zeros(sp.n_out, device="cuda")]
        out.append(tensors)
    return out


def _batches(case, wl, gen, normal):
    """Microbatches as a loader hands them over, on the GPU."""
    if case["kind"] == "mlp":
        x = normal(N_BATCHES, case["rows"], case["width"])
        x = x.to(torch.bfloat16) if case["compute"] == "bf16" else x
        y = x.float()
        for stage in _mlp_params(case, normal):
            for weight, bias in stage:
                y = _act(y @ weight.T + bias, case["act"])
        return list(zip(x, y))
    out = []
    shape, vocab = (case["batch"], case["seq"]), case["vocab"]
    if case["kind"] == "encoder":          # uniform ids, the target is the sequence reversed
        for _ in range(N_BATCHES):
            ids = torch.randint(0, vocab, shape, generator=gen, device="cuda", dtype=torch.int32)
            out.append((ids.reshape(-1), ids.flip(1).reshape(-1).contiguous()))
        return out
    # Zipf(1.1) source ids; the target is a fixed permutation of the source, the decoder reads it shifted right
    cdf = torch.arange(1, vocab + 1, dtype=torch.float64).pow(-1.1).cumsum(0)
    cdf = (cdf / cdf[-1]).to(torch.float32).cuda()
    order = torch.randperm(vocab, generator=gen, device="cuda")
    for _ in range(N_BATCHES):
        src = torch.searchsorted(cdf, torch.rand(shape, generator=gen, device="cuda")).clamp_(max=vocab - 1)
        tgt = order[src]
        dec = torch.cat([torch.zeros_like(tgt[:, :1]), tgt[:, :-1]], dim=1)
        out.append((torch.stack([src, dec]).to(torch.int32).reshape(-1), tgt.to(torch.int32).reshape(-1)))
    return out


def _prepare_update(case, gen, normal):
    P, n = case["stages"], case["n"]
    base, rem = divmod(n, P)
    counts = [base + (1 if i < rem else 0) for i in range(P)]
    offsets, total = [], 0
    for c in counts:
        offsets.append(total)
        total += -(-c // 64) * 64
    live = torch.zeros(total, device="cuda")       # 1 where a slice has an element, 0 in its padding
    for o, c in zip(offsets, counts):
        live[o:o + c] = 1
    fwd, bkwd = pm_inputs.pipemare_delays(P)
    adam = case["optimizer"] == "adam"
    update = pm.FlatUpdate(offsets, counts, fwd, bkwd, optimizer=case["optimizer"], alpha=5e-4 if adam else 0.01, K=64, D=0.5)
    w = normal(total).mul_(live)
    return dict(update=update, w=w, m=normal(total).mul_(1e-3).mul_(live), delta=normal(total).mul_(1e-4).mul_(live),
                s=normal(total).mul_(1e-3).square_().mul_(live) if adam else None, grad=normal(total).mul_(1e-3).mul_(live),
                w_lp=w.to(torch.bfloat16), k=10)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    if case["kind"] == "update":
        return _prepare_update(case, gen, normal)
    wl = _workload(case)
    params = _mlp_params(case, normal) if case["kind"] == "mlp" else _transformer_params(wl, normal)
    host = [[tuple(t.cpu().numpy() for t in pair) for pair in stage] if case["kind"] == "mlp" else [t.cpu().numpy() for t in stage]
            for stage in params]
    del params
    P, mb = wl.n_stages, case["order"] == "mb"
    pipe = pm.Pipeline(wl, host, loop_order="mb_major" if mb else "tick_major", n_micro=case["n_micro"],
                       recompute_segment=max(2, int(math.sqrt(P))) if case["option"] == "recompute" else 0,
                       materialize_backward=int(case["option"] == "written"))
    # what a checkpoint restores besides the weights
    pipe.m.copy_(normal(pipe.total)).mul_(3e-5 if case["optimizer"] == "adam" else 1e-5)
    pipe.delta.copy_(normal(pipe.total)).mul_(1e-5)
    if pipe.s is not None:
        pipe.s.copy_(torch.rand(pipe.total, generator=gen, device="cuda")).add_(0.5).mul_(ADAM_S).square_()
    state = dict(pipe=pipe, batches=_batches(case, wl, gen, normal), fed=0, mb=mb, stages=P, n_micro=case["n_micro"],
                 f32=case["compute"] == "f32", log=case["log"])
    for _ in range(4 * case["n_micro"] if mb else 2 * P + 2):
        _feed(state)
    return state


# ---- the pass --------------------------------------------------------------------------------------------------------

def _feed(state):
    x, y = state["batches"][state["fed"] % N_BATCHES]
    state["pipe"].pm_step(x, y)
    state["fed"] += 1


def run(state):
    if "update" in state:
        state["update"].pm_update_flat(state["w"], state["m"], state["s"], state["delta"], state["grad"], state["w_lp"], state["k"])
        state["k"] += 1
        return {key: state[key] for key in ("w", "m", "s", "delta", "w_lp")}
    pipe = state["pipe"]
    for _ in range(state["n_micro"]):
        _feed(state)
    out = dict(w=pipe.w, m=pipe.m, s=pipe.s, delta=pipe.delta, w_lp=None if state["mb"] else pipe.w_lp,
               grad=pipe.grad if state["f32"] else None)
    if state["log"]:       # the losses of the microbatches that have left the pipeline with this update
        done = state["fed"] if state["mb"] else state["fed"] - state["stages"]
        out["loss"] = pipe.pm_get_losses(done - state["n_micro"], state["n_micro"])
    return out


# ---- what a pass cannot do without, and how exact it is ---------------------------------------------------------------

def _linears(case):
    if case["kind"] == "mlp":
        return [(case["width"], case["width"])] * (case["stages"] * case["linears"])
    return [(sp.n_in, sp.n_out) for sp in _workload(case).stage_specs]


def work(case):
    """Bytes: state and weights read and written once per update, every Linear's input written by the forward and read by
    the backward pass.  FLOPs: the three products of every Linear and the attention products, forward and backward."""
    adam = case["optimizer"] == "adam"
    if case["kind"] == "update":
        return {"bytes": (38 if adam else 30) * case["n"], "flops": 0}
    lin = _linears(case)
    d = case["heads"] * case["d_head"] if case["kind"] != "mlp" else 0
    rows = case["rows"] if case["kind"] == "mlp" else case["batch"] * case["seq"]
    params = sum(a * b + b for a, b in lin) + (case["vocab"] * d * (2 if case["kind"] == "encdec" else 1) if d else 0)
    element = 2 if case["compute"] == "bf16" else 4
    micro = case["n_micro"]
    state = (40 if adam else 32) - (2 if element == 4 and case["order"] == "tick" else 0)
    flops = 6.0 * rows * sum(a * b for a, b in lin)
    if d:
        attentions = case["layers"] if case["kind"] == "encoder" else case["enc"] + 2 * case["dec"]
        flops += 12.0 * rows * case["seq"] * d * attentions
    return {"bytes": state * params + micro * 2 * rows * element * sum(a for a, _ in lin), "flops": flops * micro}


def tolerance(case):
    """Measured by permuting hidden units and head columns, which changes the order of every sum and nothing else."""
    if case["kind"] == "update":
        return "exact"                          # elementwise, every operation rounded once in a stated order
    if case["compute"] == "f32":
        if case["kind"] == "mlp" and case["act"] == "gelu":
            return {"rel": 4e-5, "max": 6e-3}   # seen: 1.2e-5 (delta: differences of rounded weights), 1.5e-3 (single entries of it)
        return {"rel": 1e-3, "max": 0.09}       # seen: 2.7e-4, 2.1e-2 where a pre-activation at zero falls on the other side of the ReLU
    return {"rel": 0.03, "max": 0.99}           # seen: up to 1.7e-2 (first moment of 25 stages), 0.46 (single entries)
