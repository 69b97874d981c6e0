"""The attention core at the edges of its query tiles, through the branch, against the oracle.

A forward block holds two tiles of 128 query positions and walks the key blocks that they need: sequence lengths on
both sides of one, two, three and four tiles (an odd number of tiles leaves the last block one), grouped key/value
heads; and row maxima that grow along the keys past what the softmax's reference may stay behind (a sum of 64 weights of
2^20, a single weight of 2^14).  Tolerance: the path's stated 2e-2 (bf16 operands, P rounded to bf16, fp32 sums).  The scores
have a standard deviation of (16 std)^2 sqrt(128) = 18.5 at std 0.08; q and k rounded to bf16 (2^-9 / sqrt(3) relative
each) move a score by 18.5 * 2^-9 * sqrt(2/3) = 0.03 and so each unsaturated weight by 3 %, which the sum over keys
brings below 2e-2; at std 0.12 it would be 6.6 %, too much for that tolerance whatever the kernel."""
import numpy as np
import pytest
import torch

from oracle import revffn_attn_oracle as orc
from workloads.generate import AttnConfig, make_attn_streams, make_attn_weights

from helpers import dev, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("std", [0.05, 0.08])
@pytest.mark.parametrize("seq_len", [1, 127, 128, 129, 256, 257, 384, 385, 512, 600])
def test_forward_and_backward_at_tile_edges(seq_len, std):
    import paper_2512_20920_b200 as rv
    cfg = AttnConfig("edge", batch=2, seq_len=seq_len, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype="bf16")
    w, s = make_attn_weights(cfg, 5, std=std, bias_std=std), make_attn_streams(cfg, 5)
    f32 = ("norm_gamma", "b_q", "b_k", "b_v")
    dw = {n: torch.from_numpy(np.ascontiguousarray(v)).to("cuda", torch.float32 if n in f32 else torch.bfloat16) for n, v in w.items()}
    br = rv.AttnBranch(batch=2, seq_len=seq_len, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype=rv.BF16, weights=dw,
                       norm_eps=cfg.norm_eps, rope_theta=cfg.rope_theta)
    oa = dict(S=seq_len, n_heads=4, n_kv_heads=2, eps=cfg.norm_eps, theta=cfg.rope_theta)
    x1, x2 = dev(s["x1"]), dev(s["x2"])
    y1 = br.forward(x1, x2)
    assert br.status() == 0
    want = orc.forward(w, s["x1"], s["x2"], **oa) - s["x1"]
    assert rel_l2(y1.cpu().numpy() - s["x1"], want) < 2e-2
    if std < 0.06:
        dx2 = torch.zeros_like(x2)
        dx1 = br.backward(x1, x2, dev(s["dy1"]), dx2)
        assert br.status() == 0
        g1, g2, _ = orc.backward(w, s["x1"], s["x2"], s["dy1"], **oa)
        assert rel_l2(dx1.cpu().numpy() - s["dy1"], g1 - s["dy1"]) < 2e-2 and rel_l2(dx2.cpu().numpy(), g2) < 2e-2


@pytest.mark.parametrize("seq_len", [200, 256, 600, 1100])
def test_row_maxima_that_grow_along_the_keys(seq_len):
    """Biases in one slowly rotating pair of q and k add 20 cos(0.0029 distance) to every score: towards a late query the
    scores grow by 16 to 39 (23 to 56 in log2) from the first block to its own (600 and 1100 positions), past what the first block's reference may stay.
    q and k rounded to bf16 move such a score by 20 * 2^-9 * sqrt(2/3) = 0.03, which the sum over some hundred keys of
    like weight brings below the path's 2e-2."""
    import paper_2512_20920_b200 as rv
    cfg = AttnConfig("grow", batch=1, seq_len=seq_len, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype="bf16")
    w, s = make_attn_weights(cfg, 6, std=0.03, bias_std=0.03), make_attn_streams(cfg, 6)
    for n in ("b_q", "b_k"):
        w[n] = w[n].copy()
        w[n][27::128] = 15.0
    f32 = ("norm_gamma", "b_q", "b_k", "b_v")
    dw = {n: torch.from_numpy(np.ascontiguousarray(v)).to("cuda", torch.float32 if n in f32 else torch.bfloat16) for n, v in w.items()}
    br = rv.AttnBranch(batch=1, seq_len=seq_len, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype=rv.BF16, weights=dw,
                       norm_eps=cfg.norm_eps, rope_theta=cfg.rope_theta)
    y1 = br.forward(dev(s["x1"]), dev(s["x2"]))
    assert br.status() == 0
    want = orc.forward(w, s["x1"], s["x2"], S=seq_len, n_heads=4, n_kv_heads=2, eps=cfg.norm_eps, theta=cfg.rope_theta) - s["x1"]
    assert rel_l2(y1.cpu().numpy() - s["x1"], want) < 2e-2


@pytest.mark.parametrize("key", [20, 150, 200, 400, 601])
def test_a_dominating_weight_keeps_its_value(key):
    """One key's weight is 2^13.007 times every other one's, a number that bf16 holds to 0.3 % only, and the row's reference
    stays that of the first block when the key comes later.  The weight's rounding must cancel in the output.

    Identities for P_up, W_v, W_o and P_down make Y1 - X1 the first head's output in bf16; X1 = 0 makes the queries b_q, one
    nearly unturned pair (1.2e-6 per position) reads one feature of the keys, and X2 holds +-1.  With w the dominating
    weight's share, rounded weights p (1 + e), |e| <= 2^-8, move the weighted mean of values in [-1, 1] by at most
    2 * 2^-8 * 2 (1 - w), and its rounding to bf16 (below 1) by 2^-9; 1e-4 covers the table, the norm's eps and fp32."""
    import paper_2512_20920_b200 as rv
    S, d, h = 640, 256, 128
    rng = np.random.default_rng(8)
    x2 = np.where(rng.random((S, h)) < 0.5, -1.0, 1.0).astype(np.float32)
    x2[:, 0] = -1.0
    x2[key, 0] = 1.0
    eye = torch.eye(d)
    w = dict(w_up=eye[:, :h], w_down=eye[:h], w_q=torch.zeros(d, d), w_k=torch.zeros(d, d), w_v=eye.clone(), w_o=eye.clone())
    w["w_k"][63, 0] = 1.0
    w = {n: t.to("cuda", torch.bfloat16).contiguous() for n, t in w.items()}
    w["b_q"] = torch.zeros(d, device="cuda")
    w["b_q"][63] = 51.0
    br = rv.AttnBranch(batch=1, seq_len=S, d_model=d, n_heads=2, n_kv_heads=2, weight_dtype=rv.BF16, weights=w, norm_eps=1e-12)
    y1 = br.forward(torch.zeros(S, h, device="cuda"), dev(x2)).cpu().numpy().astype(np.float64)
    assert br.status() == 0
    p = np.exp(51.0 / np.sqrt(128.0) * (x2[:, 0].astype(np.float64) - 1.0))
    want = np.cumsum(p[:, None] * x2, 0) / np.cumsum(p)[:, None]
    share = 1.0 / np.cumsum(p)                  # of the dominating key, for the queries that see it
    err = np.abs(y1 - want).max(1)
    bound = 4 * 2.0 ** -8 * (1 - share) + 2.0 ** -9 + 1e-4
    assert (err[key:] < bound[key:]).all(), (err[key:] / bound[key:]).max()
