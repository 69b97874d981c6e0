"""Products over rows split over K: the partial sums of each slice, with one and two matrices along K, whole and ragged row tiles, K-major and
MN-major weights.  fp32 sums of bf16 products whose order is all that differs: at most K 2^-24 times the sum of magnitudes, 1e-5
of the result's norm here."""
import pytest
import torch

from test_gpu_swiglu_runs import _bf, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("simt", [False, True], ids=["tcgen05", "cuda_cores"])
@pytest.mark.parametrize("M", [1, 127, 512, 700])
@pytest.mark.parametrize("N,K,slices,halves,mn", [
    (256, 256, 2, True, True),        # a slice is a half
    (2048, 1024, 4, True, True),      # two slices to a half
    (256, 512, 4, True, False),
    (384, 256, 4, False, True),       # a ragged last tile; one K step to a slice
    (256, 192, 2, False, False),      # the second slice ends early
    (256, 384, 4, True, True),        # the second slice lies in both halves, the fourth is empty
    (128, 640, 2, True, False),       # whole K steps in each half, an odd number of them
])
def test_partial_sums(M, N, K, slices, halves, mn, simt):
    A = _bf((M, K), 1)
    W = _bf((K, N), 2)                                   # stored [K, N]
    parts = [W[: K // 2].contiguous(), W[K // 2:].contiguous()] if halves else [W]
    if not mn:
        parts = [w.T.contiguous() for w in parts]        # stored [N, K]
    out = torch.full((slices, M, N), float("nan"), device="cuda")
    _run(M=M, N=N, K=K, lda=K, ldb=N if mn else parts[0].shape[1], ldc=N, b_mn_major=int(mn), concat=2 if halves else 0, epilogue=5, group_mode=2,
         n_groups=slices, use_simt=int(simt), c_group_stride=M * N, A=A, B0=parts[0], B1=parts[-1], C=out)
    step = -(-(-(-K // slices)) // 64) * 64
    for s in range(slices):
        k = slice(s * step, min(K, (s + 1) * step))
        want = A[:, k].float() @ W[k].float()
        assert float((out[s] - want).norm()) <= 1e-5 * float(want.norm())


@pytest.mark.parametrize("tokens,d_shared,E,launches", [
    (1, 2048, 6, 2),         # four slices of 1024
    (100, 2048, 6, 2),       # the last block of the sums' kernel has a part of its rows
    (256, 2048, 16, 2),      # whole blocks
    (333, 1024, 8, 2),       # two slices, two row tiles
    (333, 512, 8, 1),        # K = 1024: none
    (2000, 2048, 6, 1),      # the partial sums do not fit: none
])
def test_shared_experts_input_gradient_in_slices(tokens, d_shared, E, launches):
    """The shared expert's input gradient split over K, through the gradient pass, against the oracle and the CUDA cores (which do not
    split) at the path's stated 2e-2."""
    import paper_2512_20920_b200 as rv
    from oracle import revffn_oracle as orc
    from workloads import BlockConfig, make_streams, make_weights, to_bf16_values
    from helpers import dev, grad_buffers, make_block, rel_l2
    cfg = BlockConfig("d", tokens=tokens, d_model=256, n_experts=E, top_k=2, d_expert=128, d_shared=d_shared, weight_dtype="bf16")
    w, s = make_weights(cfg, 3), make_streams(cfg, 3)
    for n in w:
        if n != "norm_gamma":
            w[n] = to_bf16_values(w[n] * (4.0 if not n.startswith("ws_") else 2.0))
    y1, x2, dy2 = dev(s["y1"]), dev(s["x2"]), dev(s["dy2"])
    idx = torch.empty(tokens, 2, dtype=torch.int32, device="cuda")
    make_block(cfg, w).forward(y1, x2, topk_idx_out=idx)

    def run(flags):
        blk = make_block(cfg, w, flags=flags)
        dy1, g = torch.zeros_like(y1), grad_buffers(cfg, w)
        blk.backward(y1, dy2, dy1, g, topk_idx_in=idx)
        assert blk.status() == 0
        return dy1, g
    rv.revffn_prof_enable(True)
    try:
        dy1, g = run(0)
        slots = rv.revffn_prof_collect()
    finally:
        rv.revffn_prof_enable(False)
    assert slots["bwd/gemm_shared_du"][1] == launches, slots
    ref = orc.backward(w, s["y1"], s["dy2"], 2, cfg.norm_eps, route_override=idx.cpu().numpy())
    dy1_c, g_c = run(rv.FLAG_FORCE_SIMT)
    for other, g_other in ((ref["dy1"], {n: ref[n] for n in g}), (dy1_c.cpu().numpy(), {n: t.cpu().numpy() for n, t in g_c.items()})):
        assert rel_l2(dy1.cpu().numpy(), other) < 2e-2
        for n in ("w_up", "norm_gamma"):      # what the input gradient reaches
            assert rel_l2(g[n].cpu().numpy(), g_other[n]) < 2e-2, n
    # the same without timing, where the gradients run on a second stream
    dy1_s, g_s = run(0)
    assert torch.equal(dy1, dy1_s) and all(torch.equal(g[n], g_s[n]) for n in g)
