"""Passes that share a workspace read nothing that no pass has written: the workspace is filled with 0xFF (NaN in every
floating type) beforehand and the results have to be the bits of a run on a zeroed one.

Experts with 0, 1, 33, 64, 65 and 137 rows: padding is written up to a 64-row boundary past an expert's real rows and
nothing beyond it.  128 columns per expert leave SMs idle and run on row tiles, 4096 (2048 with e4m3 experts) run
transposed."""
import numpy as np
import pytest
import torch

from oracle import revffn_attn_oracle as aorc
from workloads import BlockConfig, make_streams, make_weights, to_bf16_values
from workloads.generate import AttnConfig, make_attn_streams, make_attn_weights

from helpers import dev, grad_buffers, make_block, max_block_rel_l2, rel_l2

pytestmark = pytest.mark.gpu

COUNTS = (0, 1, 33, 64, 65, 137)          # of the first six experts; the second choice falls on the other two


@pytest.fixture(scope="module")
def rv():
    import paper_2512_20920_b200 as rv
    return rv


def _problem(d_expert):
    cfg = BlockConfig("P", tokens=sum(COUNTS), d_model=256, n_experts=8, top_k=2, d_expert=d_expert, d_shared=256, weight_dtype="bf16")
    w = make_weights(cfg, 3)
    for n in w:
        if n not in ("norm_gamma", "b_router"):
            w[n] = to_bf16_values(w[n] * 4.0)
    rng = np.random.default_rng(4)
    first = rng.permutation(np.repeat(np.arange(len(COUNTS)), COUNTS))
    idx = np.stack([first, 6 + rng.integers(0, 2, cfg.tokens)], 1).astype(np.int32)
    return cfg, w, make_streams(cfg, 3), idx


def _step(rv, cfg, w, s, idx, fill, bwd_flags=0):
    blk = make_block(cfg, w)
    blk.ws.fill_(fill)
    y1, y2, dy2, sets = dev(s["y1"]), dev(s["x2"]), dev(s["dy2"]), dev(idx)
    x2 = blk.inverse(y1, y2, topk_idx_in=sets, save=True)
    dy1, g = torch.zeros_like(y1), grad_buffers(cfg, w)
    blk.backward(y1, dy2, dy1, g, topk_idx_in=sets, reuse=True, flags=bwd_flags)
    assert blk.status() == 0
    return dict(g, x2=x2, dy1=dy1)


@pytest.mark.parametrize("d_expert", [128, 4096])
def test_cuda_core_gradients_of_a_saved_tensor_core_evaluation(rv, d_expert):
    """A backward call on the CUDA-core back end takes what an inverse call on the tensor cores has saved."""
    cfg, w, s, idx = _problem(d_expert)
    clean = _step(rv, cfg, w, s, idx, 0, rv.FLAG_FORCE_SIMT)
    got = _step(rv, cfg, w, s, idx, 0xFF, rv.FLAG_FORCE_SIMT)
    for n in clean:
        assert torch.equal(clean[n], got[n]), n
    tensor = _step(rv, cfg, w, s, idx, 0)
    for n in clean:          # both back ends: bf16 operands, fp32 sums
        assert max_block_rel_l2(got[n].cpu().numpy()[None], tensor[n].cpu().numpy()[None]) < 2e-2, n


@pytest.mark.parametrize("d_expert", [128, 4096])
def test_a_step_reads_nothing_that_it_has_not_written(rv, d_expert):
    cfg, w, s, idx = _problem(d_expert)
    clean, got = (_step(rv, cfg, w, s, idx, fill) for fill in (0, 0xFF))
    for n in clean:
        assert torch.equal(clean[n], got[n]), n
    blk, y1, x2 = make_block(cfg, w), dev(s["y1"]), dev(s["x2"])
    y2 = []
    for fill in (0, 0xFF):
        blk.ws.fill_(fill)
        y2.append(blk.forward(y1, x2))
        assert blk.status() == 0
    assert torch.equal(*y2)


@pytest.mark.parametrize("d_expert", [128, 2048])
def test_e4m3_experts_read_nothing_that_the_call_has_not_written(rv, d_expert):
    cfg, w, s, idx = _problem(d_expert)
    blk = make_block(cfg, w, flags=rv.FLAG_FP8_EXPERTS)
    blk.quantize_experts()
    y1, y2, sets, x2 = dev(s["y1"]), dev(s["x2"]), dev(idx), []
    for fill in (0, 0xFF):
        blk.ws.fill_(fill)
        x2.append(blk.inverse(y1, y2, topk_idx_in=sets))
        assert blk.status() == 0
    assert torch.equal(*x2) and torch.isfinite(x2[0]).all()


@pytest.mark.parametrize("seq_len", [128, 200])
@pytest.mark.parametrize("first_simt", [False, True], ids=["tensor_then_cuda", "cuda_then_tensor"])
def test_attention_gradients_take_up_the_other_back_end(rv, first_simt, seq_len):
    """inverse on one back end, backward with the key/value side it left on the other: each needs its own rotary table, and
    the CUDA-core path the tables of its grouped products."""
    cfg = AttnConfig("x", batch=2, seq_len=seq_len, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype="bf16")
    w, s = make_attn_weights(cfg, 2, std=0.05, bias_std=0.05), make_attn_streams(cfg, 2)
    f32 = ("norm_gamma", "b_q", "b_k", "b_v")
    dw = {n: torch.from_numpy(np.ascontiguousarray(v)).to("cuda", torch.float32 if n in f32 else torch.bfloat16) for n, v in w.items()}
    br = rv.AttnBranch(batch=2, seq_len=seq_len, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype=rv.BF16, weights=dw,
                       norm_eps=cfg.norm_eps, rope_theta=cfg.rope_theta)
    br.ws.fill_(0xFF)
    oa = dict(S=seq_len, n_heads=4, n_kv_heads=2, eps=cfg.norm_eps, theta=cfg.rope_theta)
    x1, x2, dy1 = dev(s["x1"]), dev(s["x2"]), dev(s["dy1"])
    br.desc.flags = rv.FLAG_FORCE_SIMT if first_simt else 0
    br.inverse(dev(aorc.forward(w, s["x1"], s["x2"], **oa).astype(np.float32)), x2, n_iter=1)
    br.desc.flags = 0 if first_simt else rv.FLAG_FORCE_SIMT
    grads = {n: torch.full(v.shape, float("nan"), dtype=torch.float32, device="cuda") for n, v in w.items()}
    dx2 = torch.zeros_like(x2)
    dx1 = br.backward(x1, x2, dy1, dx2, grads=grads, reuse_kv=True)
    assert br.status() == 0
    g1, g2, g = aorc.backward(w, s["x1"], s["x2"], s["dy1"], **oa)
    assert rel_l2(dx1.cpu().numpy() - s["dy1"], g1 - s["dy1"]) < 2e-2 and rel_l2(dx2.cpu().numpy(), g2) < 2e-2
    for n in w:
        assert rel_l2(grads[n].cpu().numpy(), g[n]) < 2e-2, n
