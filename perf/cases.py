"""Performance cases of the ERASE training step: whole training steps through the public API.

A case is one training run a user of the library has in hand: a model spec, a schedule and a way of
feeding it.  ``prepare`` builds the model in a caller-owned arena and sets its parameters; ``run`` is
one training step.  The updated parameters and the gradients are returned as views of the arena (they
are the model's own buffers: nothing is copied out of the step); their place in it is found by
content, not by any knowledge of the library's layout.

Keys of a case
  model   "mlp"  w, hidden, blocks, batch, act, dtype          chain of detached MLP blocks, BCE heads, SGD
          "lm"   d, heads, ff, blocks, seq, batch, vocab       pre-LN transformer blocks, softmax heads, AdamW
          "ctr"  batch, rows, tower (three widths as a text), main
                                                               six parallel subarchitectures, BCE heads, Adam;
                                                               main: the undetached main network and trained tables
  sched   "serial"  forward-then-backward order on one stream
          "paper"   B_b released behind F_b and its loss (the paper's placement)
          "wide"    head, optimizer and parameter gradients off the forward's stream (the fastest placement)
  graph   replay the step as one CUDA graph, or enqueue its kernels on every call
  fed     every step copies a pinned host batch in and reads the losses back; otherwise the batch is resident
  update  False: gradients only (gradient accumulation, an optimizer or an exchange of the caller's own)
"""
import math

import numpy as np
import torch

from paper_2608_18469_b200 import binding, synth

_FED_POOL = 4            # host batches a fed loop cycles through


def listed():
    mlp = {"model": "mlp", "act": "gelu", "dtype": "bf16", "blocks": 8, "graph": True, "fed": False, "update": True}
    lm = {"model": "lm", "graph": True, "fed": False, "update": True}
    return [
        # the smallest step there is: fp32, 84 MFLOP, all latency and launches
        dict(mlp, name="mlp_tiny_f32", w=64, hidden=256, blocks=2, batch=256, act="relu", dtype="f32", sched="wide"),
        # narrow end of the width sweep: a chain of small kernels
        dict(mlp, name="mlp_w128_b512", w=128, hidden=512, batch=512, sched="wide"),
        # middle of the sweep through the plain call: one stream, no graph, no flags
        dict(mlp, name="mlp_w512_b4096_plain", w=512, hidden=2048, batch=4096, sched="serial", graph=False),
        # a user's own ragged widths and batch (ReLU)
        dict(mlp, name="mlp_ragged_relu", w=680, hidden=2136, blocks=5, batch=3001, act="relu", sched="wide"),
        # wide end: elementwise passes and GEMMs over large batches
        dict(mlp, name="mlp_w1024_b32768", w=1024, hidden=4096, batch=32768, sched="wide"),
        # the small LM proxy trained in a loop that feeds batches and logs losses
        dict(lm, name="lm_small_fed", d=256, heads=4, ff=1024, blocks=4, seq=256, batch=16, vocab=8192, sched="wide", fed=True),
        # the same model through the paper's placement without graph replay
        dict(lm, name="lm_small_paper", d=256, heads=4, ff=1024, blocks=4, seq=256, batch=16, vocab=8192, sched="paper",
             graph=False),
        # ragged LM: odd sequence length, batch and vocabulary, five heads
        dict(lm, name="lm_ragged", d=320, heads=5, ff=1280, blocks=3, seq=201, batch=7, vocab=5003, sched="wide"),
        # gradients only, serial order: gradient accumulation or a caller's own optimizer
        dict(lm, name="lm_mid_grads", d=512, heads=8, ff=2048, blocks=4, seq=512, batch=8, vocab=16384, sched="serial",
             update=False),
        # the larger LM proxy (the benchmark's headline workload)
        dict(lm, name="lm_large", d=768, heads=12, ff=3072, blocks=12, seq=1024, batch=8, vocab=32768, sched="wide"),
        # the CTR ranking model, fed
        {"name": "ctr_fed", "model": "ctr", "batch": 4096, "rows": 100000, "tower": "1024,512,256", "main": False,
         "sched": "wide", "graph": True, "fed": True, "update": True},
        # CTR with the main network, trained embedding tables and an odd batch
        {"name": "ctr_main", "model": "ctr", "batch": 3001, "rows": 20000, "tower": "512,256,128", "main": True,
         "sched": "wide", "graph": True, "fed": False, "update": True},
    ]


def _logint(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, int(v / step + 0.5) * step)


def draw(rng):
    """One more case of the same ranges; never more work than the largest listed one."""
    while True:
        c = {"sched": rng.choice(["serial", "paper", "wide", "wide"]), "graph": rng.random() < 0.75,
             "fed": rng.random() < 0.3, "update": rng.random() < 0.85}
        kind = rng.choice(["mlp", "mlp", "mlp_f32", "lm", "lm", "ctr"])
        if kind == "mlp_f32":
            w = _logint(rng, 32, 160, 4)
            c.update(model="mlp", dtype="f32", w=w, hidden=w * rng.choice([2, 4]), blocks=rng.randint(2, 6),
                     batch=_logint(rng, 64, 1024), act=rng.choice(["relu", "gelu"]))
        elif kind == "mlp":
            w = _logint(rng, 128, 2048, 8)
            c.update(model="mlp", dtype="bf16", w=w, hidden=w * 4 if rng.random() < 0.6 else _logint(rng, 256, 6144, 8),
                     blocks=rng.randint(2, 8), batch=_logint(rng, 512, 32768), act=rng.choice(["relu", "gelu", "gelu"]))
        elif kind == "lm":
            h = rng.randint(2, 14)
            c.update(model="lm", d=64 * h, heads=h, ff=64 * h * 4 if rng.random() < 0.7 else 64 * h * 3,
                     blocks=rng.randint(2, 12), seq=_logint(rng, 64, 1024), batch=rng.randint(2, 24),
                     vocab=_logint(rng, 2000, 32768, rng.choice([1, 8, 8, 64])))
        else:
            t = rng.choice(["1024,512,256", "512,256,128", "768,384,192"])
            c.update(model="ctr", batch=_logint(rng, 512, 8192), rows=_logint(rng, 1000, 100000), tower=t,
                     main=rng.random() < 0.4)
        most = 3e11 if c["model"] == "lm" and c["vocab"] % 8 else 1.9e13
        if 6e7 <= synth.step_flops(_spec(c)) <= most and _activation_bytes(c) <= 12e9:
            return c


def _spec(case):
    if case["model"] == "mlp":
        return synth.mlp_spec(case["w"], case["hidden"], case["blocks"], case["batch"], case["act"], case["dtype"])
    if case["model"] == "lm":
        return synth.lm_spec(case["blocks"], case["d"], case["heads"], case["ff"], case["seq"], case["batch"], case["vocab"])
    spec = synth.ctr_spec(batch=case["batch"], table_rows=case["rows"], tower=tuple(int(v) for v in case["tower"].split(",")))
    return synth.with_main(spec) if case["main"] else spec


def _activation_bytes(case):
    """A rough bound of what the step keeps on the device besides parameters (bf16 stash and scratch)."""
    if case["model"] == "mlp":
        return case["blocks"] * case["batch"] * (3 * case["hidden"] + 3 * case["w"]) * 2.0
    if case["model"] == "lm":
        return case["blocks"] * case["batch"] * case["seq"] * (case["vocab"] + 16 * case["d"] + 3 * case["ff"]) * 2.0
    return 0.0


def _schedule(case):
    """(n_streams, flags) of the case's schedule."""
    b = len(_spec(case)["blocks"])
    flags = (binding.GRAPH if case["graph"] else 0) | (0 if case["update"] else binding.NO_OPT)
    if case["sched"] == "serial":
        return 1, flags
    if case["sched"] == "wide":
        flags |= binding.EARLY_HEAD | binding.BLOCK_OPT
        flags |= binding.PAR_FWD if case["model"] == "ctr" else binding.SPLIT_BWD
    return b + 1, flags


# ---- inputs, drawn on the GPU from the seed alone --------------------------------------------------

def _bound(spec, block, name, shape, fan_in):
    """Half-width of the uniform initial distribution of one Linear weight or bias."""
    if len(shape) == 1:
        return 1.0 / math.sqrt(fan_in)
    blk = spec["blocks"][block]
    feeds_act = {"mlp": name[1:].isdigit() and int(name[1:]) < len(blk["dims"]) - 2,
                 "transformer": name == "W1"}.get(blk["kind"], name[1:].isdigit() and blk["kind"] != "cross")
    return math.sqrt((6.0 if feeds_act and blk["act"] != "none" else 3.0) / shape[1])


def _parameters(spec, gen):
    """Initial values of every tensor of the model (host fp32), distributed as synth.init_params draws them."""
    flat, fan_in = [], 1
    for block, name, shape, _ in synth.tensor_list(spec):
        if name.startswith("ln"):
            v = torch.full(shape, 1.0 if name.endswith("_g") else 0.0)
        elif block < 0:
            std = {"tok_emb": 1.0, "pos_emb": 0.1}.get(name, 0.125)
            v = torch.randn(shape, generator=gen, device="cuda").mul_(std)
        else:
            fan_in = shape[1] if len(shape) == 2 else fan_in
            v = torch.rand(shape, generator=gen, device="cuda").sub_(0.5).mul_(2.0 * _bound(spec, block, name, shape, fan_in))
        flat.append(v.cpu().numpy())
    return flat


def _batch(spec, gen):
    """One batch on the GPU: features N(0, 1) with balanced labels, uniform tokens, or Zipf(1.1) ids with rare clicks."""
    n = spec["batch"]
    rand = lambda *s: torch.rand(*s, generator=gen, device="cuda")  # noqa: E731
    if spec["input"] == "tokens":
        return {"ids": torch.randint(0, spec["vocab"], (n, spec["seq"] + 1), generator=gen, device="cuda", dtype=torch.int32)}
    if spec["input"] == "dense":
        x = torch.randn(n, spec["width"], generator=gen, device="cuda")
        return {"x": x.bfloat16() if spec["dtype"] == "bf16" else x, "y": (rand(n) < 0.5).float()}
    rows = spec["table_rows"]
    cdf = torch.arange(1, rows + 1, device="cuda", dtype=torch.float64).pow_(-1.1).cumsum_(0)
    rank = torch.searchsorted(cdf / cdf[-1], torch.rand(n, spec["n_sparse"], generator=gen, device="cuda", dtype=torch.float64))
    place = torch.Generator(device="cuda").manual_seed(7)           # which row a rank means: fixed per table
    perm = torch.stack([torch.randperm(rows, generator=place, device="cuda") for _ in range(spec["n_sparse"])], 1)
    ids = perm.gather(0, rank.clamp_(max=rows - 1)).int()
    dense = torch.randn(n, spec["n_dense"], generator=gen, device="cuda").exp_().log1p_()
    return {"x": dense, "ids": ids, "y": (rand(n) < 0.03).float()}


# ---- where the arena keeps what -------------------------------------------------------------------

def _locate(arena, values):
    """Element offset of the host array `values` in the float32 view of the arena."""
    v = torch.from_numpy(np.ascontiguousarray(values, np.float32).reshape(-1)).cuda()
    at = int(v.abs().argmax())
    for beg in range(0, arena.numel(), 1 << 28):
        for hit in (arena[beg:beg + (1 << 28)] == v[at]).nonzero().flatten().tolist():
            off = beg + hit - at
            if off >= 0 and torch.equal(arena[off:off + v.numel()], v):
                return off
    raise RuntimeError("the arena does not hold these values")


def _mark(model, idx, base):
    """Fills tensor idx with values nothing else holds and returns them."""
    n = int(np.prod(model.tensor_info(idx)[2]))
    v = (base + np.arange(n) % 65536).astype(np.float32)
    model.set_params(idx, v.reshape(model.tensor_info(idx)[2]))
    return v


def prepare(case, seed):
    spec = _spec(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    tensors = synth.tensor_list(spec)
    flat = _parameters(spec, gen)
    bytes_ = binding.arena_bytes(spec)
    arena = torch.zeros(bytes_ + 256, dtype=torch.uint8, device="cuda")
    skip = -arena.data_ptr() % 256
    arena = arena[skip:skip + bytes_ // 4 * 4].view(torch.float32)
    torch.cuda.synchronize()
    model = binding.Model(spec, arena.data_ptr(), bytes_)
    model.arena = arena                      # lives as long as the model does
    own = [i for i, t in enumerate(tensors) if t[0] >= 0]
    first, last = own[0], own[-1]
    anchor = next(i for i in own if len(tensors[i][2]) == 2)
    begin = _locate(arena, _mark(model, first, 3.0e6))
    end = _locate(arena, _mark(model, last, 5.0e6)) + flat[last].size
    model.set_all(flat)
    anchor_at = _locate(arena, flat[anchor])
    batches = [_batch(spec, gen) for _ in range(_FED_POOL if case["fed"] else 1)]
    torch.cuda.synchronize()
    dev = {k: v.clone() for k, v in batches[0].items()}
    n_streams, flags = _schedule(case)
    torch.cuda.synchronize()
    model.step(n_streams=1, flags=binding.NO_OPT, **{k: v.data_ptr() for k, v in dev.items()})
    grads = _locate(arena, model.grads(anchor)) - (anchor_at - begin)
    out = {"params": arena[begin:end], "grads": arena[grads:grads + end - begin]}
    if spec.get("train_input"):
        out["tables"] = arena[_locate(arena, flat[0]):_locate(arena, flat[first - 1]) + flat[first - 1].size]
    host = [{k: v.cpu().pin_memory() for k, v in b.items()} for b in batches] if case["fed"] else None
    stream = torch.cuda.ExternalStream(model.main_stream())
    torch.cuda.synchronize()
    # (pinned memory is given back through the stream that read it, which is the model's: it has to go first)
    return {"host": host, "stream": stream, "batch": dev, "ptr": {k: v.data_ptr() for k, v in dev.items()},
            "n_streams": n_streams, "flags": flags, "out": out, "step": 0, "model": model}


def run(state):
    """One step, in order with the caller's stream: it may have written the batch, and reads the results next."""
    model, stream, host = state["model"], state["stream"], state["host"]
    stream.wait_stream(torch.cuda.current_stream())
    if host is not None:
        with torch.cuda.stream(stream):
            for k, v in state["batch"].items():
                v.copy_(host[state["step"] % len(host)][k], non_blocking=True)
        state["step"] += 1
    model.step(n_streams=state["n_streams"], flags=state["flags"], **state["ptr"])
    torch.cuda.current_stream().wait_stream(stream)
    return state["out"] if host is None else dict(state["out"], losses=model.losses())


def work(case):
    """Algorithmic FLOPs of the step; bytes: parameters, moments and gradients once each way, the batch once."""
    spec = _spec(case)
    n = sum(int(np.prod(t[2])) for t in synth.tensor_list(spec) if t[0] >= 0)
    per = 8.0 if not case["update"] else (12.0 if spec["opt"]["kind"] == "sgd" else 28.0)
    rows = spec["batch"] * spec.get("seq", 1)
    bytes_ = n * per
    if spec["input"] == "dense":
        bytes_ += rows * (spec["width"] * (2.0 if spec["dtype"] == "bf16" else 4.0) + 4.0)
    elif spec["input"] == "tokens":
        bytes_ += rows * (4.0 + 8.0 * spec["width"])
    else:
        bytes_ += rows * (4.0 * spec["n_sparse"] * (1 + spec["emb_dim"]) + 4.0 * spec["n_dense"] + 4.0)
    return {"bytes": bytes_, "flops": float(synth.step_flops(spec))}


def tolerance(case):
    """What two correct implementations at the same precision may differ by after one or two steps.

    bf16: measured between the tile shapes, split counts, attention kernels and softmax heads that the library
    has for the same step: gradients and parameters of the LM cases differ by up to 1e-2 (largest single
    element: half of the rms) once an AdamW step -- whose first update is the sign of the gradient -- lies between
    them, by 2e-3 to 5e-3 before; against a float64 step the MLP and CTR cases show 4e-3 to 7e-3.
    fp32: sums of a few thousand terms in another order."""
    if case["model"] == "mlp" and case["dtype"] == "f32":
        return {"rel": 2e-5, "max": 1e-3}
    return {"rel": 3e-2 if case["model"] == "lm" else 2e-2, "max": 0.9}
