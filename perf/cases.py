"""Workloads that stand for what a user of this library runs, with their inputs, their outputs and the work they
cannot do without.  A case is a plain dict; `listed()` names the fixed ones and `draw(rng)` gives more of the same
ranges:

  forward    one forward pass of the MoE branch (scoring, evaluation): 32 .. 32768 tokens, bf16 experts or the
             e4m3 experts, even or Zipf-skewed routing
  step       one training step of the MoE branch: forward, inverse that keeps its intermediates, gradient pass that
             reuses them; gradients written, or the optimiser step (SGD, Adam) fused into the gradient pass;
             256 .. 32768 tokens
  attention  one training step of the attention branch: forward, one-iteration inverse, gradient pass that takes the
             key/value side from the inverse; 256 .. 16384 tokens in sequences of any length, full or grouped
             key/value heads
  stack      one training step of a stack of whole blocks, second stage of the schedule (router frozen): forward
             sweep, then the reversible backward sweep with the expert sets of every layer given (a block's router
             reads a stream that carries the rounding of the attention branch before it, so near ties would
             otherwise fall differently from one correct implementation to the next)

Shapes: "large" is the block of the benchmark (d = 2048, 60 experts of 1408, top-4, shared expert of 5632, 16 heads
of 128); "small" is the d = 512 block of the parity tests, where a pass is a few microseconds of work per launch."""
from __future__ import annotations

import math

import torch

import paper_2512_20920_b200 as rv
from workloads import zipf_router_bias

SHAPES = {
    "large": dict(d_model=2048, n_experts=60, top_k=4, d_expert=1408, d_shared=5632, n_heads=16),
    "small": dict(d_model=512, n_experts=8, top_k=3, d_expert=256, d_shared=384, n_heads=4),
}
UPDATED = ("w_up", "w_down", "w_gate", "w_upx", "w_downx", "ws_gate", "ws_up", "ws_down")


# --------------------------------------------------------------------------- #
# Cases
# --------------------------------------------------------------------------- #
def _forward(tokens, fp8=False, zipf=False):
    return dict(kind="forward", tokens=tokens, fp8=fp8, zipf=zipf)


def _step(tokens, update="none", zipf=False):
    return dict(kind="step", tokens=tokens, update=update, zipf=zipf)


def _attention(batch, seq, kv_heads=16):
    return dict(kind="attention", batch=batch, seq=seq, kv_heads=kv_heads)


def _stack(shape, layers, batch, seq, kv_heads):
    return dict(kind="stack", shape=shape, layers=layers, batch=batch, seq=seq, kv_heads=kv_heads)


def listed():
    return [
        # a handful of tokens to score: every expert's weights are streamed for two or three rows each
        dict(_forward(64), name="forward_64"),
        # evaluation of the benchmark's token batch with the quantised experts
        dict(_forward(8192, fp8=True), name="forward_fp8_8192"),
        # smallest training batch of the token sweep: weights and launches bound it
        dict(_step(512), name="step_512"),
        # an odd token count, as a packed batch of texts has it
        dict(_step(2741), name="step_2741"),
        # the benchmark step (batch 4 x 2048)
        dict(_step(8192), name="step_8192"),
        # skewed expert load with two empty experts
        dict(_step(16384, zipf=True), name="step_zipf_16384"),
        # the large batch of the sweep, where the matrix products alone decide
        dict(_step(32768), name="step_32768"),
        # training with the optimiser step inside the gradient pass: Adam on fp32 master weights
        dict(_step(8192, update="adam"), name="step_adam_8192"),
        # attention branch on the benchmark's token batch
        dict(_attention(4, 2048), name="attention_4x2048"),
        # shorter sequences of an odd length, grouped key/value heads
        dict(_attention(7, 613, kv_heads=4), name="attention_7x613"),
        # a small model: some 400 launches of a few microseconds each
        dict(_stack("small", 4, 2, 192, 2), name="stack_small"),
        # whole blocks at the benchmark shape, as full fine-tuning runs them
        dict(_stack("large", 3, 4, 2048, 16), name="stack_large"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("forward", "forward", "step", "step", "step", "attention", "attention", "stack"))
    if kind == "forward":
        return _forward(_log_int(rng, 32, 32768), fp8=rng.random() < 0.3, zipf=rng.random() < 0.25)
    if kind == "step":
        update = rng.choice(("none", "none", "none", "sgd", "adam"))
        top = 32768 if update == "none" else 16384
        return _step(_log_int(rng, 256, top), update=update, zipf=rng.random() < 0.25)
    if kind == "attention":
        tokens, seq = _log_int(rng, 256, 16384), _log_int(rng, 64, 8192)
        seq = min(seq, tokens)
        return _attention(max(1, tokens // seq), seq, rng.choice((16, 16, 8, 4)))
    if rng.random() < 0.5:
        return _stack("small", rng.randint(2, 8), rng.randint(1, 8), _log_int(rng, 64, 1024), rng.choice((4, 2)))
    tokens, seq = _log_int(rng, 512, 8192), _log_int(rng, 128, 4096)
    seq = min(seq, tokens)
    return _stack("large", rng.randint(1, 2), max(1, tokens // seq), seq, rng.choice((16, 4)))


# --------------------------------------------------------------------------- #
# Inputs
# --------------------------------------------------------------------------- #
def _normal(gen, shape, std=0.02, mean=0.0, dtype=torch.bfloat16):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(mean, std, generator=gen)


def _moe_weights(gen, s, zipf_seed=None):
    d, h, E, I, Is = s["d_model"], s["d_model"] // 2, s["n_experts"], s["d_expert"], s["d_shared"]
    shapes = dict(w_up=(d, h), w_down=(h, d), w_router=(E, d), w_gate=(E, I, d), w_upx=(E, I, d), w_downx=(E, d, I),
                  ws_gate=(Is, d), ws_up=(Is, d), ws_down=(d, Is), ws_sgate=(d,))
    w = {n: _normal(gen, shape) for n, shape in shapes.items()}
    w["norm_gamma"] = _normal(gen, (h,), mean=1.0, dtype=torch.float32)
    if zipf_seed is not None:      # router bias that skews the load towards rank^-1.2; two experts stay empty
        w["b_router"] = torch.from_numpy(zipf_router_bias(E, 1.2, zipf_seed)).cuda()
    return w


def _attn_weights(gen, s, kv_heads):
    d, h = s["d_model"], s["d_model"] // 2
    dkv = kv_heads * (d // s["n_heads"])
    shapes = dict(w_up=(d, h), w_down=(h, d), w_q=(d, d), w_k=(dkv, d), w_v=(dkv, d), w_o=(d, d))
    w = {n: _normal(gen, shape) for n, shape in shapes.items()}
    w["norm_gamma"] = _normal(gen, (h,), mean=1.0, dtype=torch.float32)
    for n, m in (("b_q", d), ("b_k", dkv), ("b_v", dkv)):
        w[n] = _normal(gen, (m,), dtype=torch.float32)
    return w


def _streams(gen, tokens, h, n):
    return [_normal(gen, (tokens, h), 1.0, dtype=torch.float32) for _ in range(n)]


def _like(weights, names, layers=None):
    """fp32 gradient buffers of the named weights; with `layers`, one buffer per name for all layers."""
    lead = () if layers is None else (layers,)
    return {n: torch.empty(lead + tuple(weights[n].shape), dtype=torch.float32, device="cuda") for n in names}


def _moe_shape_args(s):
    return {n: s[n] for n in ("d_model", "n_experts", "top_k", "d_expert", "d_shared")}


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return _PREPARE[case["kind"]](case, gen, int(seed))


def _prepare_forward(case, gen, seed):
    s, T = SHAPES["large"], case["tokens"]
    blk = rv.Block(tokens=T, weight_dtype=rv.BF16, weights=_moe_weights(gen, s, seed if case["zipf"] else None),
                   flags=rv.FLAG_FP8_EXPERTS if case["fp8"] else 0, backward=False, **_moe_shape_args(s))
    if case["fp8"]:
        blk.quantize_experts()
    y1, x2 = _streams(gen, T, s["d_model"] // 2, 2)
    idx = torch.empty(T, s["top_k"], dtype=torch.int32, device="cuda")
    return dict(run=_run_forward, blk=blk, y1=y1, x2=x2, y2=torch.empty_like(x2), idx=idx)


def _prepare_step(case, gen, seed):
    s, T = SHAPES["large"], case["tokens"]
    w = _moe_weights(gen, s, seed if case["zipf"] else None)
    blk = rv.Block(tokens=T, weight_dtype=rv.BF16, weights=w, **_moe_shape_args(s))
    y1, x2, dy2, g1 = _streams(gen, T, s["d_model"] // 2, 4)
    st = dict(run=_run_step, blk=blk, y1=y1, x2=x2, dy2=dy2, g1=g1, y2=torch.empty_like(x2), x2r=torch.empty_like(x2),
              dy1=torch.empty_like(y1), update=case["update"])
    names = rv.trainable_names(2)[1]       # the router stays frozen
    if case["update"] == "none":
        st["grads"] = _like(w, [n for n in names if n in w])
        return st
    st["grads"] = _like(w, [n for n in names if n in w and n not in UPDATED])
    if case["update"] == "adam":
        st["master"] = {n: w[n].float() for n in UPDATED}
        # moments of a run under way: gradients of order 0.1
        st["mom"] = {n: _normal(gen, w[n].shape, 0.03, dtype=torch.float32) for n in UPDATED}
        st["var"] = {n: torch.empty_like(m).uniform_(0.005, 0.02, generator=gen) for n, m in st["mom"].items()}
        st["t"] = 100
    return st


def _prepare_attention(case, gen, seed):
    s, B, S = SHAPES["large"], case["batch"], case["seq"]
    w = _attn_weights(gen, s, case["kv_heads"])
    br = rv.AttnBranch(batch=B, seq_len=S, d_model=s["d_model"], n_heads=s["n_heads"], n_kv_heads=case["kv_heads"],
                       weight_dtype=rv.BF16, weights=w)
    x1, x2, dy1, g2 = _streams(gen, B * S, s["d_model"] // 2, 4)
    return dict(run=_run_attention, br=br, x1=x1, x2=x2, dy1=dy1, g2=g2, y1=torch.empty_like(x1),
                x1r=torch.empty_like(x1), dx1=torch.empty_like(x1), dx2=torch.empty_like(x1), grads=_like(w, list(w)))


def _prepare_stack(case, gen, seed):
    s, B, S, L = SHAPES[case["shape"]], case["batch"], case["seq"], case["layers"]
    wm = [_moe_weights(gen, s) for _ in range(L)]
    wa = [_attn_weights(gen, s, case["kv_heads"]) for _ in range(L)]
    stk = rv.RevStack(batch=B, seq_len=S, n_heads=s["n_heads"], n_kv_heads=case["kv_heads"], weight_dtype=rv.BF16,
                      attn_weights=wa, moe_weights=wm, **_moe_shape_args(s))
    na, nm = rv.trainable_names(2)
    ga, gm = _like(wa[0], [n for n in na if n in wa[0]], L), _like(wm[0], [n for n in nm if n in wm[0]], L)
    arrays = stk.grads_arrays([{n: t[l] for n, t in ga.items()} for l in range(L)],
                              [{n: t[l] for n, t in gm.items()} for l in range(L)], stage=2)
    inputs = _streams(gen, B * S, s["d_model"] // 2, 4)
    # k different experts for every token of every layer
    idx = torch.rand(L * B * S, s["n_experts"], device="cuda", generator=gen).topk(s["top_k"], dim=1).indices.to(torch.int32)
    return dict(run=_run_stack, stk=stk, arrays=arrays, ga=ga, gm=gm, inputs=inputs, idx=idx,
                work=[torch.empty_like(t) for t in inputs], y=[torch.empty_like(t) for t in inputs[:2]])


_PREPARE = dict(forward=_prepare_forward, step=_prepare_step, attention=_prepare_attention, stack=_prepare_stack)


# --------------------------------------------------------------------------- #
# One pass
# --------------------------------------------------------------------------- #
def run(state):
    return state["run"](state)


def _run_forward(st):
    st["blk"].forward(st["y1"], st["x2"], st["y2"], st["idx"])
    return dict(y2=st["y2"], idx=st["idx"])


def _run_step(st):
    blk = st["blk"]
    blk.forward(st["y1"], st["x2"], st["y2"])
    # the weights have not changed since the forward pass: its folded router is still good
    blk.inverse(st["y1"], st["y2"], st["x2r"], save=True, flags=rv.FLAG_ROUTER_FOLDED)
    st["dy1"].copy_(st["g1"])          # y1 also carries the gradient that comes from above
    upd = None
    if st["update"] == "sgd":
        upd = rv.make_sgd(1e-5, UPDATED)
    elif st["update"] == "adam":
        st["t"] += 1
        upd = rv.make_adam(1e-5, st["t"], UPDATED, st["mom"], st["var"], st["master"], weight_decay=0.01)
    blk.backward(st["y1"], st["dy2"], st["dy1"], st["grads"], reuse=True, sgd=upd)
    out = dict(y2=st["y2"], x2=st["x2r"], dy1=st["dy1"], grads=st["grads"])
    if upd is not None:
        out["weights"] = {n: blk.weights[n] for n in UPDATED}
    if st["update"] == "adam":
        out.update(mom=st["mom"], var=st["var"], master=st["master"])
    return out


def _run_attention(st):
    br = st["br"]
    br.forward(st["x1"], st["x2"], st["y1"])
    br.inverse(st["y1"], st["x2"], st["x1r"], n_iter=1)
    st["dx2"].copy_(st["g2"])
    br.backward(st["x1r"], st["x2"], st["dy1"], st["dx2"], st["dx1"], st["grads"], reuse_kv=True)
    return dict(y1=st["y1"], x1=st["x1r"], dx1=st["dx1"], dx2=st["dx2"], grads=st["grads"])


def _run_stack(st):
    stk, work = st["stk"], st["work"]
    for dst, src in zip(work, st["inputs"]):      # streams from the embedding, their gradients from the loss
        dst.copy_(src)
    s1, s2, g1, g2 = work
    stk.forward(s1, s2)
    st["y"][0].copy_(s1)                          # what the head of the model reads: the sweep overwrites the streams
    st["y"][1].copy_(s2)
    stk.backward(s1, s2, g1, g2, *st["arrays"], topk_idx=st["idx"])
    return dict(y=st["y"], x=[s1, s2], dx=[g1, g2], attn=st["ga"], moe=st["gm"])


# --------------------------------------------------------------------------- #
# Work and tolerance
# --------------------------------------------------------------------------- #
def _moe_counts(s, T):
    """(flops of one evaluation of the branch, weight elements, expert weight elements)"""
    d, h, E, k, I, Is = s["d_model"], s["d_model"] // 2, s["n_experts"], s["top_k"], s["d_expert"], s["d_shared"]
    flops = 2.0 * T * (2 * d * h + 3 * k * d * I + 3 * d * Is + (E + 1) * h)
    return flops, 2 * d * h + 3 * d * Is + (E + 1) * d, 3 * E * d * I


def _attn_counts(s, B, S, kv_heads):
    """(flops of the projections, flops of the causal half of the attention itself, weight elements)"""
    d, h = s["d_model"], s["d_model"] // 2
    dkv = kv_heads * (d // s["n_heads"])
    n = 2 * d * h + 2 * d * d + 2 * d * dkv
    return 2.0 * B * S * (n + d * h), 4.0 * B * d * S * (S + 1) / 2, n


def work(case):
    kind = case["kind"]
    s = SHAPES[case.get("shape", "large")]
    h, k, E = s["d_model"] // 2, s["top_k"], s["n_experts"]
    if kind in ("forward", "step"):
        T = case["tokens"]
        stream = 4.0 * T * h
        flops, dense, experts = _moe_counts(s, T)
        used = experts * (1.0 - (1.0 - k / E) ** T)          # experts that at least one token selects
        if kind == "forward":
            # e4m3 experts: a byte per weight, and one flop counts as half a bf16 flop of tensor time
            fp8 = case["fp8"]
            routed = 2.0 * T * 3 * k * s["d_model"] * s["d_expert"]
            return dict(bytes=2 * dense + (1 if fp8 else 2) * used + 3 * stream + 4.0 * T * k,
                        flops=flops - (routed / 2 if fp8 else 0))
        n = dense + experts
        per_weight = dict(none=4, sgd=2, adam=2 + 3 * 8)[case["update"]]      # gradient, or weight (and Adam's state) rewritten
        return dict(bytes=2 * (dense + used) + per_weight * n + 7 * stream, flops=4 * flops)
    B, S = case["batch"], case["seq"]
    stream = 4.0 * B * S * h
    proj, core, n_attn = _attn_counts(s, B, S, case["kv_heads"])
    # forward and inverse evaluate the branch, the gradient pass takes keys and values from the inverse and computes
    # the query side again; gradients cost twice the projections and two and a half times the attention
    attn_flops = 4.7 * proj + 5.5 * core
    if kind == "attention":
        return dict(bytes=(2 + 4) * n_attn + 8 * stream, flops=attn_flops)
    flops, dense, experts = _moe_counts(s, B * S)
    L = case["layers"]
    return dict(bytes=L * (2 + 4) * (n_attn + dense + experts) + 10 * stream, flops=L * (attn_flops + 4 * flops))


def tolerance(case):
    """Four times what the tensor-core path differs from the library's own CUDA-core evaluation of the same bf16
    problem (other sums, other exponentials): worst outputs 1.9e-3 / 0.037 for a step, 8.8e-3 / 0.03 for attention,
    1.1e-2 / 0.14 for stacks (the key bias, whose gradient nearly cancels; the largest single difference is a token
    of the forward sweep whose routing fell on the other side of a near tie).  A forward pass returns the stream the
    branch is added to, so its error is that of the branch times the branch's share of the stream (0.14); with e4m3
    experts the branch may move by 2.2e-2, a code of an activation that lies next to a rounding boundary."""
    if case["kind"] == "forward":
        return dict(rel=1.2e-2, max=0.1) if case["fp8"] else dict(rel=1e-3, max=2e-2)
    if case["kind"] == "step":
        return dict(rel=7.5e-3, max=0.15)
    return dict(rel=3e-2, max=0.12 if case["kind"] == "attention" else 0.55)
