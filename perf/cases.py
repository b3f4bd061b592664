"""The work whose speed this repository watches: linear layers of transformer training, forward and
backward, through the calls that a training or evaluation program makes.

`listed()` names the cases, `draw()` gives further ones of the same ranges, `prepare()` makes what a
program holds before a pass (seeded inputs, weights, buffers, a captured graph where such a program
would replay one), `run()` is one pass and returns everything it computed, `work()` counts the bytes
and flops that a pass cannot do without, `tolerance()` says how far a correct result may lie from
another one.
"""
from __future__ import annotations

import math

import torch

from paper_2609_28568_b200 import binding as nb
from paper_2609_28568_b200 import shapes, synth
from paper_2609_28568_b200.stack import LinearStack, LoraStack

DEV = "cuda"
ACTS = {"none": nb.ACT_NONE, "gelu": nb.ACT_GELU, "swiglu": nb.ACT_SWIGLU}
# elements of all parameters of GPT-2 124M: what is cast once per optimizer step
GPT2_PARAMS = shapes.gpt2_param_count()[0]


def listed():
    return [
        # The smallest workload: one MLP fc layer with its GELU, forward and backward, 128 rows
        # (B=2, T=64). A handful of short launches: latency and host time are what counts.
        {"name": "fc_gelu_128", "kind": "layer", "rows": 128, "C": 768, "OC": 3072, "act": "gelu",
         "bias": True, "fused": False, "frozen": False, "micro": 1},
        # A layer of no round size on a batch of no round size, behind a GELU layer whose derivative
        # its backward applies; gradients accumulated over two micro-steps.
        {"name": "layer_odd_1003", "kind": "layer", "rows": 1003, "C": 776, "OC": 1416, "act": "none",
         "bias": True, "fused": True, "frozen": False, "micro": 2},
        # The model's linears on eight rows, as when eight sequences are continued by one token
        # each: every weight is read once for a few rows. Such a loop replays a captured graph.
        {"name": "generate_8", "kind": "forward", "rows": 8, "graph": True},
        # The model's linears, forward only, on one sequence of the full context length: evaluation,
        # or the prompt of a generation.
        {"name": "evaluate_1024", "kind": "forward", "rows": 1024, "graph": False},
        # One transformer block's four linears, forward and backward, B=4, T=1024.
        {"name": "block_4096", "kind": "stack", "model": "gpt2_block", "rows": 4096, "micro": 1,
         "wgrad": True},
        # A training step of the whole model on a small, ragged batch, two micro-steps.
        {"name": "stack_2021x2", "kind": "stack", "model": "gpt2", "rows": 2021, "micro": 2,
         "wgrad": True},
        # The training step the benchmark times by default: B=16, T=1024, four micro-steps.
        {"name": "stack_16384x4", "kind": "stack", "model": "gpt2", "rows": 16384, "micro": 4,
         "wgrad": True},
        # The tied head with its loss at the production batch: logits and softmax statistics, the
        # logits' gradient in place, then both products of the head's backward.
        {"name": "head_loss_16384", "kind": "head", "rows": 16384, "C": 768, "Vp": 50304, "V": 50257},
        # The SwiGLU model's linears, forward and backward with weight gradients, two sequences of 2048.
        {"name": "swiglu_4096", "kind": "stack", "model": "qwen3", "rows": 4096, "micro": 1,
         "wgrad": True},
        # Adapter training, frozen weights, at the adapter stage's batch (B=8, T=2048), four of its
        # 28 layers; the projections of a group as one layer, as the benchmark has them.
        {"name": "adapter_16384", "kind": "lora", "rows": 16384, "layers": 4, "rank": 16, "micro": 1,
         "form": "fused"},
        # Adapter training on one short example of no round length, one set of calls per projection.
        {"name": "adapter_519", "kind": "lora", "rows": 519, "layers": 2, "rank": 8, "micro": 1,
         "form": "plain"},
        # The fp32 master weights cast to the bf16 copies, all parameters of the model.
        {"name": "cast_weights", "kind": "cast", "n": GPT2_PARAMS},
    ]


def _log(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "forward", "stack", "stack", "head", "lora", "lora", "cast"])
    if kind == "layer":
        act = rng.choice(["none", "none", "gelu", "swiglu"])
        return {"kind": kind, "rows": _log(rng, 1, 16384), "C": _log(rng, 64, 4096, 8),
                "OC": _log(rng, 64, 8192, 16), "act": act, "bias": rng.random() < 0.7,
                "fused": act == "none" and rng.random() < 0.4, "frozen": rng.random() < 0.25,
                "micro": rng.choice([1, 1, 2])}
    if kind == "forward":
        rows = _log(rng, 1, 4096)
        return {"kind": kind, "rows": rows, "graph": rows <= 256}
    if kind == "stack":
        model = rng.choice(["gpt2", "gpt2_block", "qwen3"])
        rows = _log(rng, 256, 4096 if model == "qwen3" else 16384)
        micro = rng.choice([1, 1, 2, 4]) if rows <= 4096 else 1
        return {"kind": kind, "model": model, "rows": rows, "micro": micro,
                "wgrad": model != "qwen3" or rng.random() < 0.6}
    if kind == "head":
        Vp = rng.choice([shapes.VOCAB_PADDED, _log(rng, 4096, 50304, 8)])
        return {"kind": kind, "rows": _log(rng, 128, 16384), "C": rng.choice([768, _log(rng, 256, 2048, 8)]),
                "Vp": Vp, "V": Vp - rng.choice([47, 0, 13])}
    if kind == "lora":
        form = rng.choice(["fused", "fused", "stacked", "plain"])
        return {"kind": kind, "rows": _log(rng, 128, 16384), "layers": rng.choice([1, 2]),
                "rank": rng.choice([8, 16]), "micro": rng.choice([1, 2]), "form": form}
    return {"kind": kind, "n": _log(rng, 100_000, GPT2_PARAMS)}


# ---------------------------------------------------------------------------------------- states
class _State:
    pass


def _one_buffer(layers, name):
    """The layers' tensors called `name` laid out one after the other in a single buffer (each on a
    256-byte boundary), as a program that manages its own memory has them. Returns the buffer."""
    have = [L for L in layers if getattr(L, name) is not None]
    if not have:
        return None
    starts, pos = [], 0
    for L in have:
        starts.append(pos)
        pos += (getattr(L, name).numel() + 127) // 128 * 128
    flat = torch.zeros(pos, dtype=getattr(have[0], name).dtype, device=DEV)
    for L, p in zip(have, starts):
        t = getattr(L, name)
        setattr(L, name, flat[p:p + t.numel()].view(t.shape))
    return flat


def prepare(case, seed):
    s = _State()
    s.case = case
    kind = case["kind"]
    if kind == "layer":
        BT, C, OC = case["rows"], case["C"], case["OC"]
        act = ACTS[case["act"]]
        ocols = OC // 2 if case["act"] == "swiglu" else OC
        base = 64 * seed
        s.weight = synth.normal(base + 1, (OC, C), 0.02, DEV)
        s.bias = synth.normal(base + 2, (OC,), 0.02, DEV) if case["bias"] else None
        s.inp = [synth.normal(base + 10 + m, (BT, C), 1.0, DEV) for m in range(case["micro"])]
        s.dout = [synth.normal(base + 20 + m, (BT, ocols), 1e-3, DEV) for m in range(case["micro"])]
        s.inp_pre = [synth.normal(base + 30 + m, (BT, C), 1.0, DEV) if case["fused"] else None
                     for m in range(case["micro"])]
        s.act = act
    elif kind == "forward":
        s.stack = LinearStack("gpt2", case["rows"], 1, seed_offset=seed, wgrad=False)
        s.outputs = [_one_buffer(s.stack.layers, "out"), _one_buffer(s.stack.layers, "pre")]
        s.graph = None
        if case["graph"]:
            s.stack.forward(0)
            torch.cuda.synchronize()
            s.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s.graph):
                s.stack.forward(0)
    elif kind == "stack":
        s.stack = LinearStack(case["model"], case["rows"], case["micro"], seed_offset=seed, wgrad=case["wgrad"],
                              generate=False)
        s.outputs = [_one_buffer(s.stack.layers, n) for n in ("out", "pre", "dinp")]
        if case["wgrad"]:
            s.outputs.append(s.stack.attach_gradient_buckets().flat)
        s.stack.generate_inputs()
    elif kind == "head":
        BT, C, Vp, V = case["rows"], case["C"], case["Vp"], case["V"]
        base = 64 * seed
        s.weight = synth.normal(base + 1, (Vp, C), 0.02, DEV)
        s.weight[V:].zero_()
        s.inp = synth.normal(base + 2, (BT, C), 1.0, DEV)
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        s.targets = torch.randint(0, V, (BT,), dtype=torch.int32, device=DEV, generator=g)
        s.logits = torch.empty((BT, Vp), dtype=torch.bfloat16, device=DEV)
        s.loss = torch.empty(BT, dtype=torch.float32, device=DEV)
        s.lse = torch.empty(BT, dtype=torch.float32, device=DEV)
        s.dinp = torch.empty((BT, C), dtype=torch.bfloat16, device=DEV)
        s.dweight = torch.empty((Vp, C), dtype=torch.float32, device=DEV)
    elif kind == "lora":
        s.stack = LoraStack(case["rows"], case["micro"], r=case["rank"], layers=case["layers"],
                            seed_offset=seed, stacked=case["form"] == "stacked", fused=case["form"] == "fused")
        s.outputs = ([L.out for L in s.stack.layers] + [L.dinp for L in s.stack.layers] +
                     s.stack.gradient_tensors())
    else:
        g = torch.Generator(device=DEV)
        g.manual_seed(seed)
        s.src = torch.randn(case["n"], dtype=torch.float32, device=DEV, generator=g).mul_(0.02)
        s.dst = torch.empty(case["n"], dtype=torch.bfloat16, device=DEV)
    return s


# ---------------------------------------------------------------------------------------- a pass
def _run_layer(s):
    case, got = s.case, []
    dw = db = None
    for m in range(case["micro"]):
        out, pre = nb.linear_forward(s.inp[m], s.weight, s.bias, s.act)
        dinp, dw, db = nb.linear_backward(s.dout[m], s.inp[m], s.weight, pre_act=pre, inp_pre_act=s.inp_pre[m],
                                          act=s.act, dweight=dw, dbias=db, accumulate=m > 0,
                                          need_dweight=not case["frozen"],
                                          need_dbias=case["bias"] and not case["frozen"])
        got += [out, pre, dinp]
    return got + [dw, db]


def _run_head(s):
    c = s.case
    BT, C, Vp, V = c["rows"], c["C"], c["Vp"], c["V"]
    nb.nb_lm_head_ce_forward(s.logits, s.loss, s.lse, s.inp, s.weight, s.targets, BT, C, Vp, V)
    nb.nb_ce_backward(s.logits, s.logits, s.lse, s.targets, 1.0 / BT, BT, Vp, V)
    nb.nb_linear_backward_ex(s.dinp, s.dweight, None, s.logits, s.inp, s.weight, None, None, BT, C, Vp,
                             nb.ACT_NONE, 0)
    return [s.loss, s.lse, s.logits, s.dinp, s.dweight]


def run(s):
    kind = s.case["kind"]
    if kind == "layer":
        return _run_layer(s)
    if kind == "head":
        return _run_head(s)
    if kind == "cast":
        nb.nb_cast_f32_to_bf16(s.dst, s.src, s.case["n"])
        return s.dst
    if kind == "forward":
        if s.graph is not None:
            s.graph.replay()
        else:
            s.stack.forward(0)
    else:
        s.stack.step()
    return s.outputs


# ---------------------------------------------------------------------------------------- accounting
def _linear(BT, C, OC, ocols, micro, backward, wgrad, bias, act, read_dout=True, read_inp=True, extra=0):
    """(bytes, flops) of one layer over all micro-steps: weights once, gradients written once."""
    b = 2 * OC * C + (2 * OC if bias else 0)
    b += micro * 2 * BT * ((C if read_inp else 0) + ocols + (OC if act else 0) + extra)
    f = 2 * BT * C * OC * micro
    if backward:
        b += micro * 2 * BT * ((ocols if read_dout else 0) + C)
        f *= 3 if wgrad else 2
        if wgrad:
            b += 4 * OC * C + (4 * OC if bias else 0)
    return b, f


def work(case):
    kind = case["kind"]
    if kind == "layer":
        OC = case["OC"]
        b, f = _linear(case["rows"], case["C"], OC, OC // 2 if case["act"] == "swiglu" else OC, case["micro"], True,
                       not case["frozen"], case["bias"], case["act"] != "none",
                       extra=case["C"] if case["fused"] else 0)
    elif kind in ("forward", "stack"):
        model = case.get("model", "gpt2")
        if model == "qwen3":
            specs = shapes.qwen3_block() * shapes.QWEN3_LAYERS
        else:
            specs = shapes.gpt2_block() * (shapes.GPT2_LAYERS if model == "gpt2" else 1)
            if model == "gpt2":
                specs = specs + [shapes.gpt2_lm_head()]
        b = f = 0
        for L in specs:
            # a layer behind a GELU layer reads what that one wrote, and writes its dz: both are
            # counted once, where they are written
            behind = L.fused_gelu_bwd
            lb, lf = _linear(case["rows"], L.C, L.OC, L.out_cols, case.get("micro", 1), kind == "stack",
                             case.get("wgrad", False), L.bias, L.act != shapes.ACT_NONE,
                             read_dout=L.act != shapes.ACT_GELU, read_inp=not behind)
            b, f = b + lb, f + lf
    elif kind == "head":
        BT, C, Vp = case["rows"], case["C"], case["Vp"]
        # the logits' gradient stands where the logits were: one result of that size
        b = 2 * BT * C + 2 * Vp * C + 2 * BT * Vp + 12 * BT + 2 * BT * C + 4 * Vp * C
        f = 6 * BT * C * Vp
    elif kind == "lora":
        BT, r, m = case["rows"], case["rank"], case["micro"]
        b = f = 0
        groups = {n: g[0] for g in LoraStack.GROUPS for n in g}
        for L in shapes.qwen3_lora_projections():
            b += 2 * L.C * L.OC + 2 * r * (L.C + L.OC) + 4 * r * (L.C + L.OC)
            b += m * 2 * BT * (2 * L.OC)
            if groups[L.name] == L.name or case["form"] != "fused":
                b += m * 2 * BT * L.C            # input gradients: one per layer of the stack
            if groups[L.name] == L.name:
                b += m * 2 * BT * L.C            # the input, shared by the group
            f += m * (4 * BT * L.C * L.OC + 6 * BT * r * (L.C + L.OC))
        b, f = b * case["layers"], f * case["layers"]
    else:
        b, f = 6 * case["n"], 0
    return {"bytes": b, "flops": f}


def tolerance(case):
    # Results are bf16, rounded once (2^-9 at most, 1.7e-3 in the 2-norm); the gradients of a layer
    # with an activation come from a derivative rounded to bf16 in the same way, and the adapters'
    # from two such intermediates. Against products in 64 bits the results measure 1.6e-3 to 3.0e-3
    # (fp32 gradients without such an intermediate: 4e-7).
    if case["kind"] == "cast":
        return "exact"
    return {"rel": 1e-2}
