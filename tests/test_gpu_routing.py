"""The router and the permutation maps at the edges of their tiles: token counts around a 64-token router tile and
around the map chunks (128 tokens; 256 from 16385 tokens on), one to five passes over the experts, a K range
shorter than the number of slices."""
import numpy as np
import pytest
import torch

from workloads import BlockConfig, make_streams, make_weights

from helpers import dev, make_block

pytestmark = pytest.mark.gpu

SHAPES = [(1, 256, 60, 4), (63, 256, 63, 4), (64, 512, 64, 8), (65, 256, 5, 1), (129, 1024, 130, 3),
          (2049, 256, 256, 8), (16384, 256, 60, 4), (16385, 256, 61, 2), (33000, 256, 7, 7)]


@pytest.fixture(scope="module")
def rv():
    import paper_2512_20920_b200 as rv
    return rv


@pytest.mark.parametrize("tokens,d,E,k", SHAPES)
def test_routing_tables(rv, tokens, d, E, k):
    cfg = BlockConfig("R", tokens=tokens, d_model=d, n_experts=E, top_k=k, d_expert=128, d_shared=128, weight_dtype="bf16")
    w, s = make_weights(cfg, 3), make_streams(cfg, 4)
    blk = make_block(cfg, w)
    y1, x2 = dev(s["y1"]), dev(s["x2"])
    idx = torch.empty(tokens, k, dtype=torch.int32, device="cuda")
    blk.forward(y1, x2, None, idx)
    assert blk.status() == 0
    idx = idx.cpu().numpy()

    # logits, selection and gates in fp64 from the definition
    y = s["y1"].astype(np.float64)
    n = y / np.sqrt((y * y).mean(axis=1, keepdims=True) + cfg.norm_eps) * w["norm_gamma"].astype(np.float64)
    L = (n @ w["w_up"].astype(np.float64).T) @ w["w_router"].astype(np.float64).T
    order = np.argsort(-L, axis=1, kind="stable")
    Ls = np.take_along_axis(L, order, axis=1)
    # two fp64 evaluations of a logit of size ~0.1 differ by about 1e-15: a gap above 1e-12 decides the order
    clear = (np.diff(Ls[:, :k + 1], axis=1) < -1e-12).all(axis=1)
    assert clear.mean() > 0.999
    assert (idx[clear] == order[clear, :k]).all()
    sel = np.take_along_axis(L, idx.astype(np.int64), axis=1)
    g = np.exp(sel - sel.max(axis=1, keepdims=True))
    g /= g.sum(axis=1, keepdims=True)
    gates = blk.buffer("gates", torch.float32)[: tokens * k].view(tokens, k).cpu().numpy()
    # fp32: differences rounded once (2^-24), expf and its sum and quotient a few ulp
    assert np.abs(gates - g).max() <= 2e-6

    # maps: stable counting sort by expert, segments padded to 128 rows
    cnt = np.bincount(idx.reshape(-1), minlength=E)
    off = np.concatenate([[0], np.cumsum((cnt + 127) // 128 * 128)])
    assert (blk.buffer("expert_cnt", torch.int32)[:E].cpu().numpy() == cnt).all()
    assert (blk.buffer("expert_off", torch.int32)[: E + 1].cpu().numpy() == off).all()
    rows_total = blk.buffer("rows_total", torch.int32)[:2].cpu().numpy()
    assert rows_total[0] == off[E] and rows_total[1] == ((cnt + 255) // 256).sum()
    tile_group = blk.buffer("tile_group", torch.int32)[: off[E] // 128].cpu().numpy()
    assert (tile_group == np.repeat(np.arange(E), (cnt + 127) // 128)).all()
    flat = idx.reshape(-1)
    tok_row = np.empty(flat.size, dtype=np.int64)
    by_expert = np.argsort(flat, kind="stable")
    start = np.concatenate([[0], np.cumsum(cnt)])
    tok_row[by_expert] = off[flat[by_expert]] + np.arange(flat.size) - start[flat[by_expert]]
    assert (blk.buffer("tok_row", torch.int32)[: flat.size].cpu().numpy() == tok_row).all()
    row_tok = np.full(off[E], -1)
    row_tok[tok_row] = np.arange(flat.size) // k
    assert (blk.buffer("row_tok", torch.int32)[: off[E]].cpu().numpy() == row_tok).all()
    row_gate = np.zeros(off[E], np.float32)
    row_gate[tok_row] = gates.reshape(-1)
    assert (blk.buffer("row_gate", torch.float32)[: off[E]].cpu().numpy() == row_gate).all()
    # token runs: an expert's rows to a multiple of 32, at most 256 a run; the last run names the rows from there to the
    # next multiple of 64, which products write as zeros
    runs = []
    for e in range(E):
        n = (cnt[e] + 31) // 32 * 32
        runs += [[e, off[e] + r, min(256, n - r), (cnt[e] + 63) // 64 * 64 - n if r + 256 >= n else 0] for r in range(0, n, 256)]
    got = blk.buffer("tok_chunks", torch.int32)[: 4 * len(runs)].view(-1, 4).cpu().numpy()
    assert (got == np.array(runs)).all()


def test_logits_do_not_depend_on_the_batch(rv):
    """Gates of the first tokens are the same bits whatever follows them (the host step splits a batch in two)."""
    cfg = BlockConfig("R", tokens=700, d_model=512, n_experts=60, top_k=4, d_expert=128, d_shared=128, weight_dtype="bf16")
    w, s = make_weights(cfg, 5), make_streams(cfg, 6)
    got = []
    for T in (700, 123):
        blk = make_block(cfg, w, tokens=T)
        blk.forward(dev(s["y1"][:T]), dev(s["x2"][:T]))
        got.append(blk.buffer("gates", torch.float32)[: 123 * 4].clone())
    assert torch.equal(*got)
