"""Row kernels of the gradient passes at the edges of their ranges, and the attention branch's second stream."""
import numpy as np
import pytest
import torch

from workloads import BlockConfig, make_streams, make_weights
from workloads.generate import AttnConfig, make_attn_streams, make_attn_weights

from helpers import dev, make_block, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rv():
    import paper_2512_20920_b200 as rv
    return rv


@pytest.mark.parametrize("tokens,d", [(1, 256), (9, 2048), (70, 2304), (8000, 256)])
def test_norm_backward(rv, tokens, d):
    """dY1 and the scale's gradient from the workspace's own dn (one pass up to 1024 columns, separate passes beyond;
    a warp per row, 444 blocks of eight)."""
    cfg = BlockConfig("N", tokens=tokens, d_model=d, n_experts=4, top_k=2, d_expert=128, d_shared=128, weight_dtype="bf16")
    w, s = make_weights(cfg, 1), make_streams(cfg, 2)
    blk = make_block(cfg, w)
    y1, dy2 = dev(s["y1"]), dev(s["dy2"])
    h = cfg.h
    base = torch.randn(tokens, h, device="cuda")
    dy1, dg = base.clone(), torch.zeros(h, device="cuda")
    blk.backward(y1, dy2, dy1, {"norm_gamma": dg})
    assert blk.status() == 0
    dn = blk.buffer("dn", torch.float32)[: tokens * h].view(tokens, h).cpu().numpy().astype(np.float64)
    y, g = s["y1"].astype(np.float64), w["norm_gamma"].astype(np.float64)
    r = 1.0 / np.sqrt((y * y).mean(axis=1, keepdims=True) + cfg.norm_eps)
    q = g * dn
    want = r * q - y * r ** 3 * (q * y).sum(axis=1, keepdims=True) / h
    # fp32: r and the dot product to a few 2^-24 each; `base` costs its own rounding, 2^-24 of |base|
    got = dy1.cpu().numpy().astype(np.float64) - base.cpu().numpy()
    assert np.abs(got - want).max() <= 1e-5 * np.abs(want).max() + 5e-7
    # a sum of `tokens` products in fp32, in runs of at most tokens / 8: well inside 1e-5
    assert rel_l2(dg.cpu().numpy(), (dn * y * r).sum(axis=0)) <= 1e-5


@pytest.mark.parametrize("batch,seq,kv", [(1, 1, 2), (3, 31, 1), (2, 129, 2), (5, 300, 1)])
def test_attention_second_stream_changes_no_bit(rv, batch, seq, kv):
    cfg = AttnConfig("s", batch=batch, seq_len=seq, d_model=256, n_heads=2, n_kv_heads=kv, weight_dtype="bf16")
    w, s = make_attn_weights(cfg, 4, std=0.05, bias_std=0.05), make_attn_streams(cfg, 4)
    f32 = ("norm_gamma", "b_q", "b_k", "b_v")
    dw = {n: torch.from_numpy(v).cuda().to(torch.float32 if n in f32 else torch.bfloat16).contiguous() for n, v in w.items()}
    x1, x2, dy1, dx2_0 = (dev(s[n]) for n in ("x1", "x2", "dy1", "dx2"))
    want = None
    for flags in (rv.FLAG_SINGLE_STREAM, 0, 0, 0):
        br = rv.AttnBranch(batch=batch, seq_len=seq, d_model=256, n_heads=2, n_kv_heads=kv, weight_dtype=rv.BF16, weights=dw,
                           flags=flags)
        y1 = br.forward(x1, x2)
        xr = br.inverse(y1, x2, n_iter=2)
        dx2 = dx2_0.clone()
        grads = {n: torch.full(v.shape, float("nan"), dtype=torch.float32, device="cuda") for n, v in w.items()}
        dx1 = br.backward(xr, x2, dy1, dx2, grads=grads, reuse_kv=True)
        got = dict(grads, y1=y1, xr=xr, dx1=dx1, dx2=dx2)
        assert br.status() == 0
        if want is None:
            want = got
        for n in want:
            assert torch.equal(got[n], want[n]), n
