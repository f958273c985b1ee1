"""The work a user of this library has it do, as measurable cases: whole calls through the public entry points.

Three kinds of call:
  decode   a job of a serving process: `prefill` of every sequence, then `decode` (pipelined, Algorithm 1) or
           `vanilla_decode` (all recurrences of a token before the next), then the logits of the last target readout;
  prefill  the prompt alone, up to the logits the first token is drawn from (time to first token);
  linear   one stand-alone linear map on a few token rows (`linear`, `linear_tc`, `linear_static`).

Shapes are those of `workloads/configs.py`; prompts are uniform random ids, as in the workloads there.  Decode jobs use an
out-projection scale at which random weights draft as well as trained ones do (the benchmark's acceptance-calibrated
variant: ~90 % of the first proposals are accepted on the large shapes); prefill jobs use the scale of the configuration.
"""
import math

import numpy as np
import torch

import paper_2609_17184_b200 as ls
import workloads as W

CALIBRATED = 1e-4  # the benchmark's out-projection scale of trained-like acceptance


def listed():
    return [
        # one attention output projection of the 1.4B shape on the rows of a decode pass: the smallest call there is
        dict(name="linear_o_proj", kind="linear", op="linear", dtype="bf16", M=4, N=2048, K=2048),
        # gate/up projection of the 1.4B shape on a ragged batch of rows, weights read in place
        dict(name="linear_tc_gate_up", kind="linear", op="linear_tc", dtype="bf16", M=33, N=11264, K=2048),
        # the smallest model: fp32 weights, single proposal, everything is launches and latency
        decode("tiny_greedy", "tiny", prompt=16, tokens=64, d1=1, d2=0, out_scale=0.02),
        # a mid-size model at the paper's sampling setting (T = 1, top-p 0.7); widths that are no multiple of the tiles
        decode("small_top_p", "small_bf16", prompt=130, tokens=48, d1=1, d2=2, T=1.0, top_p=0.7, out_scale=0.01),
        # time to first token: the headline prompt, and a long ragged one that is then decoded with long-context attention
        dict(name="ouro_prefill_512", kind="prefill", model="ouro_1p4b", prompt=512, out_scale=0.3),
        decode("ouro_long_context", "ouro_1p4b", prompt=3001, tokens=48, d1=1, d2=2, T=0.7),
        # the headline job: greedy, two proposals, batch 1
        decode("ouro_greedy", "ouro_1p4b", prompt=512, tokens=192, d1=1, d2=2),
        # the paper's baseline from the same kernels: four passes of one row per token, short chat-like prompt
        decode("ouro_vanilla", "ouro_1p4b", prompt=77, tokens=40, d1=1, d2=2, mode="vanilla"),
        # the paper's sampling setting on the headline shape
        decode("ouro_top_p", "ouro_1p4b", prompt=300, tokens=128, d1=1, d2=2, T=1.0, top_p=0.7),
        # 48 layers, rejection sampling at T = 1, the depths its closed form picks
        decode("ouro_2p6b_sampled", "ouro_2p6b", prompt=256, tokens=64, d1=1, d2=3, T=1.0),
        # prelude / recurrent / coda model: 16 recurrences, grouped-query attention, passes of up to 18 rows
        decode("raven_greedy", "raven", prompt=256, tokens=64, d1=2, d2=8),
        # serving: eight sequences of ragged lengths in one context, T = 0.7, per-sequence rollback
        decode("serve_batch8", "ouro_1p4b", prompt=400, tokens=64, d1=1, d2=2, T=0.7, batch=8),
    ]


def decode(name, model, prompt, tokens, d1, d2, T=0.0, top_k=0, top_p=1.0, gate=True, mode="loopspec", batch=1,
           out_scale=CALIBRATED):
    c = dict(kind="decode", model=model, mode=mode, prompt=prompt, tokens=tokens, batch=batch, d1=d1, d2=d2, gate=gate, T=T,
             top_k=top_k, top_p=top_p, out_scale=out_scale)
    if name:
        c["name"] = name
    return c


def draw(rng):
    """One more case of the ranges above."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["linear", "linear", "prefill", "decode", "decode", "decode", "decode", "serve"])
    if what == "linear":
        op = rng.choice(["linear", "linear_tc", "linear_static"])
        k_unit = 64 if op == "linear_tc" else 8
        c = dict(kind="linear", op=op, dtype=rng.choice(["bf16", "bf16", "fp32"]) if op != "linear_tc" else "bf16", M=log_int(1, 64))
        n_max = 2048 if op == "linear_static" else 12288
        c["N"] = 16 * log_int(16, n_max // 16)
        c["K"] = k_unit * log_int(512 // k_unit, (2048 if op == "linear_static" else 5632) // k_unit)
        return c
    if what == "prefill":
        model = rng.choice(["ouro_1p4b", "ouro_1p4b", "raven", "small_bf16"])
        return dict(kind="prefill", model=model, prompt=log_int(24, 2000 if model != "raven" else 700), out_scale=0.3)
    if what == "serve":
        batch = rng.randint(2, 8)
        return decode(None, "ouro_1p4b", prompt=log_int(40, 3000 // batch), tokens=log_int(12, 48), d1=1, d2=rng.choice([0, 2, 3]),
                      T=rng.choice([0.0, 0.7, 1.0]), batch=batch)
    model = rng.choice(["tiny", "small_bf16", "ouro_1p4b", "ouro_1p4b", "ouro_1p4b", "ouro_2p6b", "raven"])
    T = rng.choice([0.0, 0.0, 0.7, 1.0])
    top_k, top_p = rng.choice([(0, 1.0), (0, 1.0), (0, 0.7), (40, 0.9)]) if T > 0 else (0, 1.0)
    if model == "raven":
        d1, d2 = rng.choice([(2, 8), (4, 8), (2, 4)])
        prompt, tokens = log_int(24, 500), log_int(8, 48)
    else:
        d1, d2 = rng.choice([(1, 2), (1, 2), (1, 3), (1, 0), (2, 0)])
        prompt = log_int(16, {"tiny": 200, "small_bf16": 600, "ouro_1p4b": 2600, "ouro_2p6b": 900}[model])
        tokens = log_int(12, 160 if model != "ouro_2p6b" else 48)
    return decode(None, model, prompt=prompt, tokens=tokens, d1=d1, d2=d2, T=T, top_k=top_k, top_p=top_p,
                  gate=rng.random() < 0.75, mode=rng.choice(["loopspec", "loopspec", "loopspec", "vanilla"]),
                  out_scale={"tiny": 0.02, "small_bf16": 0.01}.get(model, CALIBRATED))


def _weights(shape, out_scale, seed):
    """Random weights of `shape`, drawn on the device: N(0, std), out-projections scaled, norm gains one."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.bfloat16 if shape.weight_dtype == "bf16" else torch.float32
    w = {}
    for name, shp in W.weight_order(shape):
        if len(shp) == 1:
            w[name] = torch.ones(shp, dtype=torch.float32, device="cuda")
            continue
        std = shape.std * (out_scale if name.endswith((".wo", ".wdown")) else 1.0)
        w[name] = torch.randn(shp, generator=g, dtype=torch.float32, device="cuda").mul_(std).to(dt)
    return w


def _lengths(case):
    """Prompt lengths of a job's sequences: ragged around `prompt`, as requests are."""
    return [case["prompt"] + (29 * s) % 64 - (32 if case["batch"] > 1 and case["prompt"] > 64 else 0) for s in range(case["batch"])]


def prepare(case, seed):
    if case["kind"] == "linear":
        g = torch.Generator(device="cuda").manual_seed(seed)
        M, N, K = case["M"], case["N"], case["K"]
        w = torch.randn((N, K), generator=g, device="cuda").mul_(0.02)
        if case["dtype"] == "bf16":
            w = w.to(torch.bfloat16)
        x = torch.randn((M, K), generator=g, device="cuda")
        scratch = None  # the caller keeps its scratch between calls
        if case["op"] == "linear":
            scratch = torch.zeros(ls.linear_scratch_bytes(M, N, K), dtype=torch.uint8, device="cuda")
        elif case["op"] == "linear_tc":
            scratch = torch.zeros(ls.lib.loopspec_linear_tc_scratch_bytes(M, N, K) + 256, dtype=torch.uint8, device="cuda")
        return dict(op=case["op"], w=w, x=x, scratch=scratch)
    shape = W.CONFIGS[case["model"]]
    w = _weights(shape, case["out_scale"], seed)
    rng = np.random.default_rng(seed)
    if case["kind"] == "prefill":
        ctx = ls.LoopSpec(shape, w, d1=2 if shape.R > 4 else 1, d2=8 if shape.R > 4 else 2, max_ctx=case["prompt"] + 32)
        return dict(kind="prefill", ctx=ctx, prompts=[rng.integers(0, shape.vocab, case["prompt"], dtype=np.int32)])
    lengths = _lengths(case)
    ctx = ls.LoopSpec(shape, w, d1=case["d1"], d2=case["d2"], temperature=case["T"], seed=seed, gate=case["gate"],
                      top_k=case["top_k"], top_p=case["top_p"], max_seqs=case["batch"],
                      max_ctx=max(lengths) + case["tokens"] + shape.R // case["d1"] + 16)
    return dict(kind="decode", ctx=ctx, prompts=[rng.integers(0, shape.vocab, n, dtype=np.int32) for n in lengths],
                tokens=case["tokens"], mode=case["mode"])


def run(state):
    if "op" in state:
        if state["op"] == "linear":
            return ls.linear(state["w"], state["x"], state["scratch"])
        if state["op"] == "linear_tc":
            return ls.linear_tc(state["w"], state["x"], state["scratch"], check=False)
        return ls.linear_static(state["w"], state["x"])
    ctx = state["ctx"]
    for s, prompt in enumerate(state["prompts"]):
        ctx.prefill(prompt, seq=s)
    if state["kind"] == "prefill":
        return ctx.debug_logits(0, 0)
    ids = ctx.vanilla_decode(state["tokens"]) if state["mode"] == "vanilla" else ctx.decode(state["tokens"])
    return {"ids": ids, "logits": [ctx.debug_logits(s, 0) for s in range(len(state["prompts"]))]}


def _block_params(shape):
    d = shape.head_dim
    return shape.hidden * d * (2 * shape.n_q_heads + 2 * shape.n_kv_heads) + 3 * shape.hidden * shape.ffn


def work(case):
    if case["kind"] == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": N * K * (2 if case["dtype"] == "bf16" else 4) + 4 * M * (N + K), "flops": 2 * M * N * K}
    shape = W.CONFIGS[case["model"]]
    wb = 2 if shape.weight_dtype == "bf16" else 4
    block, head = _block_params(shape), shape.vocab * shape.hidden
    raven = shape.n_prelude + shape.n_coda > 0
    recurrent = shape.n_recurrent * block + (2 * shape.hidden * shape.hidden if raven else 0)
    kv_row = 4 * shape.n_kv_heads * shape.head_dim  # bytes of a position's keys and values in one plane of one block
    attn = 4 * shape.n_q_heads * shape.head_dim     # flops of one (query, key) pair over the heads of a block
    lengths = [case["prompt"]] if case["kind"] == "prefill" else _lengths(case)
    classes = 3  # readout depths with a cache of their own in the post-layers
    once = shape.n_prelude + classes * shape.n_coda
    # prompt: every weight once per recurrence, keys and values written once and read once
    planes = shape.R * shape.n_recurrent + once
    nbytes = len(lengths) * wb * (shape.R * recurrent + once * block + head)
    nbytes += sum(2 * planes * kv_row * n for n in lengths)
    flops = sum(2 * n * (shape.R * recurrent + once * block) + 2 * head + planes * attn * n * (n + 1) // 2 for n in lengths)
    if case["kind"] == "decode":
        n, R = case["tokens"], shape.R
        # passes: R per token, or - pipelined, every draft accepted - R for the first token and d1 for each later one
        passes = n * R if case["mode"] == "vanilla" else R + (n - 1) * case["d1"]
        readouts = n if case["mode"] == "vanilla" else -(-passes // case["d1"])
        nbytes += wb * (passes * recurrent + readouts * ((shape.n_prelude + shape.n_coda) * block + head))
        nbytes += sum(n * planes * kv_row * (p + n // 2) for p in lengths)  # a token reads its context once per plane
        flops += len(lengths) * n * (2 * (R * recurrent + once * block) + 2 * head) + sum(n * planes * attn * (p + n // 2) for p in lengths)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times what the path differs by when its sums are taken in another order (the skinny kernels for the prompt, the
    wide ones for the decode passes).  The prompt's logits move most: a key or value that lands on the other side of a bf16
    boundary.  In decode jobs the out-projection scale shrinks that to the rounding of the fp32 readout sums; tokens agree."""
    if case["kind"] == "linear":
        return {"rel": 3e-6}
    small = case["model"] == "small_bf16"
    if case["kind"] == "prefill":
        return {"rel": 3e-4 if small else 6e-3}
    return {"rel": 4e-5 if small else 4e-6, "differ": 0.0}
