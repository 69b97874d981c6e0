"""Gradients of the attention branch where its kernels and products are cut: more items than blocks (a block then walks several,
the next one's first products under this one's output), keys and values as one product or as two,
weight gradients split over K.  Against the oracle at the path's stated 2e-2."""
import numpy as np
import pytest
import torch

from oracle import revffn_attn_oracle as orc
from workloads.generate import AttnConfig, make_attn_streams, make_attn_weights

from helpers import dev, rel_l2

pytestmark = pytest.mark.gpu

F32 = ("norm_gamma", "b_q", "b_k", "b_v")


@pytest.mark.parametrize("batch,seq_len,d_model,n_heads,n_kv_heads", [
    (45, 130, 512, 4, 2),        # 360 items of dQ, 180 of dK/dV
    (5, 1000, 512, 4, 4),        # 160 of each, of 1 to 8 steps
    (2, 150, 768, 6, 3),         # three key/value heads: two products
    (2, 150, 256, 2, 2),         # two: one product of one tile per matrix
    (3, 700, 512, 4, 2),         # 2100 tokens: gradients in four slices of K, keys' and values' in one product
])
def test_gradients(batch, seq_len, d_model, n_heads, n_kv_heads):
    import paper_2512_20920_b200 as rv
    cfg = AttnConfig("g", batch=batch, seq_len=seq_len, d_model=d_model, n_heads=n_heads, n_kv_heads=n_kv_heads, weight_dtype="bf16")
    w, s = make_attn_weights(cfg, 7, std=0.05, bias_std=0.05), make_attn_streams(cfg, 7)
    dw = {n: torch.from_numpy(np.ascontiguousarray(v)).to("cuda", torch.float32 if n in F32 else torch.bfloat16) for n, v in w.items()}
    br = rv.AttnBranch(batch=batch, seq_len=seq_len, d_model=d_model, n_heads=n_heads, n_kv_heads=n_kv_heads, weight_dtype=rv.BF16, weights=dw,
                       norm_eps=cfg.norm_eps, rope_theta=cfg.rope_theta)
    grads = {n: torch.full(v.shape, float("nan"), dtype=torch.float32, device="cuda") for n, v in w.items()}
    x1, x2 = dev(s["x1"]), dev(s["x2"])
    dx2 = torch.zeros_like(x2)
    dx1 = br.backward(x1, x2, dev(s["dy1"]), dx2, grads=grads)
    assert br.status() == 0
    g1, g2, G = orc.backward(w, s["x1"], s["x2"], s["dy1"], S=seq_len, n_heads=n_heads, n_kv_heads=n_kv_heads, eps=cfg.norm_eps, theta=cfg.rope_theta)
    assert rel_l2(dx1.cpu().numpy() - s["dy1"], g1 - s["dy1"]) < 2e-2 and rel_l2(dx2.cpu().numpy(), g2) < 2e-2
    for n in w:
        assert rel_l2(grads[n].cpu().numpy(), G[n]) < 2e-2, n


@pytest.mark.parametrize("batch,seq_len", [
    (3, 700),        # four slices of K for every weight's gradient
    (2, 150),        # none: stored by the product itself
])
def test_gradients_added_to_what_is_there_and_a_part_of_them(batch, seq_len):
    """Added to non-zero buffers: the same sums, rounded once more (2^-24 of the larger of sum and start value; fp32 additions in one
    order on both sides).  One of the two key/value gradients alone is a product of its own of the same operands: its fp32 sums are cut
    differently at most, K 2^-24 of the sum of magnitudes, 1e-5 of the result's norm."""
    import paper_2512_20920_b200 as rv
    cfg = AttnConfig("g", batch=batch, seq_len=seq_len, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype="bf16")
    w, s = make_attn_weights(cfg, 8, std=0.05, bias_std=0.05), make_attn_streams(cfg, 8)
    dw = {n: torch.from_numpy(np.ascontiguousarray(v)).to("cuda", torch.float32 if n in F32 else torch.bfloat16) for n, v in w.items()}
    br = rv.AttnBranch(batch=batch, seq_len=seq_len, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype=rv.BF16, weights=dw,
                       norm_eps=cfg.norm_eps, rope_theta=cfg.rope_theta)
    x1, x2, dy1 = dev(s["x1"]), dev(s["x2"]), dev(s["dy1"])

    def run(names, start=None, **kw):
        g = {n: torch.full(w[n].shape, float("nan"), dtype=torch.float32, device="cuda") if start is None else start[n].clone() for n in names}
        dx1 = br.backward(x1, x2, dy1, torch.zeros_like(x2), grads=g, **kw)
        assert br.status() == 0
        return g, dx1
    plain, dx1 = run(w)
    gen = torch.Generator("cuda").manual_seed(9)
    start = {n: torch.randn(w[n].shape, device="cuda", generator=gen) * plain[n].std() for n in w}
    added, dx1_a = run(w, start, accumulate=True)
    assert torch.equal(dx1, dx1_a)
    for n in w:
        want = start[n].double() + plain[n].double()
        assert float((added[n].double() - want).abs().max()) <= 2.0 ** -22 * float(torch.maximum(start[n].abs(), plain[n].abs()).max()), n
    for names in (("w_k",), ("w_v",), ("w_k", "w_o"), ("w_v", "b_k")):
        part, dx1_p = run(names)
        assert torch.equal(dx1, dx1_p)
        part_added, _ = run(names, start, accumulate=True)
        for n in names:
            assert rel_l2(part[n].cpu().numpy(), plain[n].cpu().numpy()) <= 1e-5, n
            assert rel_l2((part_added[n].double() - start[n].double()).cpu().numpy(), part[n].cpu().numpy()) <= 1e-5, n
