"""Passes that share a workspace read nothing that no pass has written: the workspace is filled with 0xFF (NaN in every
floating type) beforehand and the results have to be the bits of a run on a zeroed one.

Experts with 0, 1, 33, 64, 65 and 137 rows: padding is written up to a 64-row boundary past an expert's real rows and
nothing beyond it.  128 columns per expert leave SMs idle and run on row tiles, 4096 (2048 with e4m3 experts) run
transposed."""
import numpy as np
import pytest
import torch

from workloads import BlockConfig, make_streams, make_weights, to_bf16_values

from helpers import dev, grad_buffers, make_block, max_block_rel_l2

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
