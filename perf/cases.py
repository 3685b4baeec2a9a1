"""The work a serving loop has this library do, as cases that can be timed and compared.

One case is one call (or the fixed group of calls) of the public entry points on one batch of logits:

    step     speckv_step: signals, controller and verification of one speculation step (the main call)
    signals  speckv_signals + speckv_select_gamma: what a loop runs when the target has not scored yet
    verify   speckv_verify alone: loops that keep gamma fixed
    sample   speckv_sample_draft: the draft side, one token per drafted position
    shard    one rank's four calls of the vocabulary-sharded step (the exchanges between the ranks are
             replaced by the copy of this rank's own part)

Sizes: vocabularies of 32,000 to 151,936 and batches of 1 to 1,024 rows as in
``paper_2605_02888_b200.synth.WORKLOADS`` and in the benchmark, 50,257 as in the tests (an odd vocabulary: the
rows of a contiguous tensor are then not 16-byte aligned).  Logits, draft tokens, uniforms and per-row gamma and
temperature come from the same generator that the benchmark uses.
"""
from __future__ import annotations

import math

import torch

import paper_2605_02888_b200 as speckv
from paper_2605_02888_b200 import synth, vocab_shard

MAX_LOGIT_BYTES = 512 * 17 * 151936 * 4  # storage of the largest listed case
MAX_COST = 512 * 11 * 151936 * 4         # logit bytes it reads


def _case(name, op, B, G, V, dtype, gamma="choices", T="0.8", shards=1):
    return dict(name=name, op=op, B=B, G=G, V=V, dtype=dtype, gamma=gamma, T=T, shards=shards)


def listed():
    return [
        # one interactive stream: a handful of short rows, nothing but latency and launches
        _case("step_b1_fp32_v32k", "step", 1, 4, 32000, "fp32", gamma="full", T="1.0"),
        # a small server: 16 streams of a large-vocabulary model
        _case("step_b16_bf16_v128k", "step", 16, 8, 128256, "bf16"),
        # a medium batch of a small-vocabulary model
        _case("step_b64_bf16_v32k", "step", 64, 8, 32000, "bf16", T="1.0"),
        # odd batch, gamma and vocabulary: rows that are not 16-byte aligned, ragged gamma
        _case("step_b37_bf16_v50257", "step", 37, 5, 50257, "bf16", gamma="ragged", T="mixed"),
        # the batch on which the throughput figure is quoted
        _case("step_b256_bf16_v128k", "step", 256, 8, 128256, "bf16"),
        # the largest: fp32 logits, a quarter of the rows greedy, mixed temperatures
        _case("step_b512_fp32_v152k", "step", 512, 8, 151936, "fp32", T="mixed"),
        # many rows at one short gamma (half of the stored positions are not used)
        _case("step_b1024_bf16_v128k", "step", 1024, 8, 128256, "bf16", gamma="half", T="1.0"),
        # the draft side of the large batch, and of a small one in fp32
        _case("sample_b256_bf16_v128k", "sample", 256, 8, 128256, "bf16"),
        _case("sample_b24_fp32_v32k", "sample", 24, 4, 32000, "fp32", gamma="full", T="1.0"),
        # gamma chosen before the target runs: draft signals and the controller
        _case("signals_b128_bf16_v128k", "signals", 128, 8, 128256, "bf16"),
        # greedy decoding with a fixed gamma
        _case("verify_b96_fp32_greedy", "verify", 96, 4, 151936, "fp32", gamma="full", T="0.0"),
        # tensor-parallel output projection: one of eight ranks
        _case("shard_b256_bf16_8ranks", "shard", 256, 8, 128256, "bf16", shards=8),
    ]


def _cost(c):
    """Logit bytes one pass reads."""
    es = 2 if c["dtype"] == "bf16" else 4
    g = _mean_gamma(c)
    rows = {"step": 2 * g + 1, "verify": 2 * g + 1, "shard": 2 * g + 1, "signals": g, "sample": g}[c["op"]]
    return c["B"] * rows * c["V"] * es / c["shards"]


def draw(rng):
    """Another case of the same ranges: 1 to 1,024 rows, vocabularies of 1,000 to 151,936 (any integer, half of
    them multiples of 64 as model vocabularies are), gamma up to 8, both types, every way gamma and temperature are given."""
    op = rng.choice(["step", "step", "step", "step", "sample", "signals", "verify", "shard"])
    G = rng.randint(1, 8)
    V = int(round(math.exp(rng.uniform(math.log(1000), math.log(151936)))))
    if op == "shard":
        V = int(round(math.exp(rng.uniform(math.log(16000), math.log(151936)))))
    if rng.random() < 0.5:
        V = max(1024, V // 64 * 64)
    c = dict(op=op, B=int(round(math.exp(rng.uniform(0.0, math.log(1024))))), G=G, V=V, dtype=rng.choice(["bf16", "bf16", "fp32"]),
             gamma=rng.choice(["choices", "full", "ragged"]), T=rng.choice(["0.8", "1.0", "mixed", "0.0"]),
             shards=rng.choice([2, 4, 8]) if op == "shard" else 1)
    if G < 2 and c["gamma"] == "choices":
        c["gamma"] = "full"
    es = 2 if c["dtype"] == "bf16" else 4
    while c["B"] * (2 * G + 1) * V * es > MAX_LOGIT_BYTES or _cost(c) > MAX_COST:
        c["B"] = max(1, c["B"] * 3 // 4)
    return c


def _mean_gamma(c):
    if c["gamma"] == "full":
        return c["G"]
    if c["gamma"] == "half":
        return c["G"] // 2
    if c["gamma"] == "ragged":
        return (c["G"] + 1) / 2
    ch = [g for g in synth.GAMMA_CHOICES if g <= c["G"]] or [c["G"]]
    return sum(ch) / len(ch)


def _workload(c, seed):
    kw = dict(gamma_mode="choices") if c["gamma"] == "choices" else dict(gamma_mode="ragged") if c["gamma"] == "ragged" \
        else dict(gamma_mode="fixed", gamma_fixed=c["G"] if c["gamma"] == "full" else c["G"] // 2)
    if c["T"] == "mixed":
        kw.update(temperature_mode="mixed", frac_onehot=0.05)
    else:
        kw.update(temperature=float(c["T"]))
    return synth.Workload("case", B=c["B"], gamma_max=c["G"], V=c["V"], dtype=c["dtype"], sigma_t=2.0,
                          sigma_d=synth.SIGMA_LEVELS, frac_identical=0.1 if c["B"] > 8 else 0.0, seed=int(seed), **kw)


def prepare(case, seed):
    """Inputs, controller weights, output buffers and workspace of one batch, as a loop holds them between steps."""
    dev = torch.device("cuda", torch.cuda.current_device())
    w = _workload(case, seed)
    s = synth.make_step(w, 0, dev)
    st = dict(op=case["op"], comp=s["comp"])
    if case["op"] != "sample":
        mw = synth.make_mlp(w, dev)
        st["mlp"] = speckv.Mlp(mw["W1"], mw["b1"], mw["W2"], mw["b2"])
    if case["op"] in ("sample", "signals"):
        batch = speckv.Batch(draft_logits=s["draft"], gamma=s["gamma"], temperature=s["temperature"])
    else:
        batch = speckv.Batch(draft_logits=s["draft"], target_logits=s["target"], draft_tokens=s["draft_tokens"],
                             gamma=s["gamma"], temperature=s["temperature"], uniforms=s["uniforms"])
    if case["op"] == "sample":
        st["uniforms"] = s["uniforms"][:, :case["G"], 0].contiguous()
    elif case["op"] == "shard":
        _prepare_shard(case, batch, st)
        return st
    else:
        st["out"] = speckv.StepOutputs.allocate(batch, st["mlp"].n_out)
    st["batch"] = batch
    return st


def _prepare_shard(case, full, st):
    """This rank's slice, contiguous, and what the other ranks would have sent."""
    n = case["shards"]
    width, bounds = vocab_shard.shard_bounds(case["V"], n)
    rank = 1
    a, e = bounds[rank]
    local = speckv.Batch(draft_logits=full.draft_logits[:, :, a:e].contiguous(),
                         target_logits=full.target_logits[:, :, a:e].contiguous(), draft_tokens=full.draft_tokens,
                         gamma=full.gamma, temperature=full.temperature, uniforms=full.uniforms)
    buf = vocab_shard.ShardBuffers.allocate(local, n, st["mlp"].n_out)
    parts = [vocab_shard.slice_batch(full, x, y) for x, y in bounds]
    others = [vocab_shard.ShardBuffers.allocate(p, n, st["mlp"].n_out) for p in parts]
    for r, (p, o) in enumerate(zip(parts, others)):
        speckv.speckv_shard_sweep(p, bounds[r][0], o.state, o.tokl, o.workspace)
        buf.all_state[r].copy_(o.state)
        buf.all_tokl[r].copy_(o.tokl)
    speckv.speckv_shard_finish(local, n, width, case["V"], buf.all_state, buf.all_tokl, st["comp"], st["mlp"], buf.out, buf.row_info)
    for r, (p, o) in enumerate(zip(parts, others)):
        speckv.speckv_shard_draw_sums(p, buf.row_info, o.weight, o.workspace)
        buf.all_weight[r].copy_(o.weight)
    st.update(local=local, buf=buf, n=n, width=width, V=case["V"], rank=rank, v_begin=a)


def run(st):
    """One pass; the outputs are the state's own buffers, except for the drafted tokens."""
    op = st["op"]
    if op == "step":
        return speckv.speckv_step(st["batch"], st["comp"], st["mlp"], out=st["out"])
    if op == "verify":
        return speckv.speckv_verify(st["batch"], out=st["out"])
    if op == "sample":
        return speckv.speckv_sample_draft(st["batch"], st["uniforms"])
    if op == "signals":
        o = st["out"]
        r = speckv.speckv_signals(st["batch"], out=o)
        g = speckv.speckv_select_gamma(r["feat"], st["comp"], st["mlp"], scores=o.scores, gamma_next=o.gamma_next)
        return dict(r, **g)
    buf, local = st["buf"], st["local"]
    speckv.speckv_shard_sweep(local, st["v_begin"], buf.state, buf.tokl, buf.workspace)
    buf.all_state[st["rank"]].copy_(buf.state)
    buf.all_tokl[st["rank"]].copy_(buf.tokl)
    speckv.speckv_shard_finish(local, st["n"], st["width"], st["V"], buf.all_state, buf.all_tokl, st["comp"], st["mlp"],
                               buf.out, buf.row_info)
    speckv.speckv_shard_draw_sums(local, buf.row_info, buf.weight, buf.workspace)
    buf.all_weight[st["rank"]].copy_(buf.weight)
    speckv.speckv_shard_draw_pick(local, st["v_begin"], st["rank"], st["n"], buf.row_info, buf.all_weight,
                                  buf.out.out_tokens, buf.workspace)
    return dict(buf.out.as_dict(), weight=buf.weight)  # the exchanged states are opaque: any reference may stand in them


def work(case):
    """Every logit of a position <= gamma read once (at the mean of the case's gamma rule; target rows behind a
    rejection are counted although a step may leave them out), the small outputs written once; per logit one
    exponential and about five more operations."""
    b = _cost(case)
    es = 2 if case["dtype"] == "bf16" else 4
    small = case["B"] * (case["G"] * 4 * 6 + 64)
    return {"bytes": b + small, "flops": 6.0 * b / es}


def tolerance(case):
    """Sums of 1e3 to 1e5 fp32 terms: against the same statistics in fp64 the entropies are off by up to 1.2e-7 (2-norm)
    and 4e-7 (largest), the residual masses (differences of two such sums, a tenth of them) by ten times that.  A drawn token (or, more rarely, a choice of gamma) may differ where the
    threshold falls within rounding of a boundary; at least one such value is allowed where the batch has a hundred."""
    n_tokens = case["B"] * (case["G"] + (0 if case["op"] == "sample" else 1))
    differ = 2e-3 if n_tokens < 100 else max(2e-3, 1.01 / n_tokens)
    return {"rel": 5e-6, "max": 5e-5, "differ": differ}
