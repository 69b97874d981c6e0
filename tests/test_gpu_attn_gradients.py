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
