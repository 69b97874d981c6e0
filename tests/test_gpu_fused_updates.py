"""Fused updates of the experts' weight gradients in both of their forms (row by row while an expert's K range is short,
block by block beyond) against the same update of the written gradient, ragged tiles and empty experts included."""
import pytest
import torch

from workloads import BlockConfig, make_streams, make_weights

from helpers import dev, make_block

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rv():
    import paper_2512_20920_b200 as rv
    return rv


# (tokens, experts, top_k): short K with empty experts; a K range next to the row-wise form's bound for SGD and for Adam; past both
@pytest.mark.parametrize("tokens,E,k", [(5, 6, 1), (300, 5, 2), (1250, 2, 2), (2000, 2, 2), (3000, 2, 2)])
@pytest.mark.parametrize("master", [False, True])
def test_update_equals_the_update_of_the_written_gradient(rv, tokens, E, k, master):
    cfg = BlockConfig("U", tokens=tokens, d_model=256, n_experts=E, top_k=k, d_expert=384, d_shared=0, weight_dtype="bf16")
    w, s = make_weights(cfg, 1), make_streams(cfg, 2)
    names = ("w_gate", "w_upx", "w_downx")
    y1, dy2 = dev(s["y1"]), dev(s["dy2"])
    blk = make_block(cfg, w)
    g = {n: torch.empty(w[n].shape, device="cuda") for n in names}
    blk.backward(y1, dy2, torch.zeros_like(y1), g)
    gen = torch.Generator("cuda").manual_seed(3)
    for rule in ("sgd", "adam"):
        blk = make_block(cfg, w)
        old = {n: blk.weights[n].float() for n in names}
        if master:
            old = {n: t + 1e-4 * torch.randn(t.shape, device="cuda", generator=gen) for n, t in old.items()}
        ms = {n: t.clone() for n, t in old.items()} if master else None
        mom = {n: 0.03 * torch.randn(t.shape, device="cuda", generator=gen) for n, t in old.items()}
        var = {n: 0.005 + 0.01 * torch.rand(t.shape, device="cuda", generator=gen) for n, t in old.items()}
        m0, v0 = {n: t.clone() for n, t in mom.items()}, {n: t.clone() for n, t in var.items()}
        lr = 0.05
        upd = rv.make_sgd(lr, names, ms) if rule == "sgd" else rv.make_adam(lr, 7, names, mom, var, ms, weight_decay=0.1)
        blk.backward(y1, dy2, torch.zeros_like(y1), {}, sgd=upd)
        assert blk.status() == 0
        for n in names:
            if rule == "sgd":
                want = old[n].double() - lr * g[n].double()
            else:
                m, v = 0.9 * m0[n].double() + 0.1 * g[n].double(), 0.999 * v0[n].double() + 0.001 * g[n].double() ** 2
                # a fused multiply-add or two of fp32 rounding: 2^-23 of the larger term
                assert torch.allclose(mom[n].double(), m, rtol=1e-6, atol=1e-8) and torch.allclose(var[n].double(), v, rtol=1e-6, atol=1e-10)
                want = old[n].double() - lr * (m / (1 - 0.9 ** 7) / ((v / (1 - 0.999 ** 7)).sqrt() + 1e-8) + 0.1 * old[n].double())
            if master:
                # a step of size ~lr, its quotient and root to a few 2^-22, then one rounding of the weight
                assert torch.allclose(ms[n].double(), want, rtol=1e-6, atol=2e-6 * lr + 1e-8)
                assert torch.equal(blk.weights[n], ms[n].to(torch.bfloat16))
            else:
                # bf16 weights (8 significant bits): half an ulp is at most 2^-8 of the value, plus the step's own error
                assert torch.allclose(blk.weights[n].double(), want, rtol=2.0 ** -7.99, atol=1e-6)
