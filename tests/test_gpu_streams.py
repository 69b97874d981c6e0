"""The library's second streams: calls on different streams of a caller, and calls under stream capture, do not reach
into each other."""
import ctypes as C

import numpy as np
import pytest
import torch

from workloads import BlockConfig, make_streams, make_weights
from workloads.generate import AttnConfig, make_attn_streams, make_attn_weights

from helpers import dev, grad_buffers, make_block

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rv():
    import paper_2512_20920_b200 as rv
    return rv


class _Attention:
    def __init__(self, rv):
        cfg = AttnConfig("s", batch=2, seq_len=200, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype="bf16")
        w, s = make_attn_weights(cfg, 2, std=0.05, bias_std=0.05), make_attn_streams(cfg, 2)
        f32 = ("norm_gamma", "b_q", "b_k", "b_v")
        dw = {n: torch.from_numpy(np.ascontiguousarray(v)).to("cuda", torch.float32 if n in f32 else torch.bfloat16) for n, v in w.items()}
        self.br = rv.AttnBranch(batch=2, seq_len=200, d_model=512, n_heads=4, n_kv_heads=2, weight_dtype=rv.BF16, weights=dw)
        self.x1, self.x2, self.dy1 = dev(s["x1"]), dev(s["x2"]), dev(s["dy1"])
        self.y1, self.x1r, self.dx1, self.dx2 = (torch.zeros_like(self.x1) for _ in range(4))
        self.g = {n: torch.zeros_like(t, dtype=torch.float32) for n, t in dw.items()}

    def __call__(self):
        self.br.forward(self.x1, self.x2, self.y1)
        self.br.inverse(self.y1, self.x2, self.x1r, n_iter=1)
        self.dx2.zero_()
        self.br.backward(self.x1r, self.x2, self.dy1, self.dx2, self.dx1, self.g, reuse_kv=True)
        return [self.y1, self.x1r, self.dx1, self.dx2, *self.g.values()]


class _Moe:
    def __init__(self, rv):
        cfg = BlockConfig("s", tokens=300, d_model=256, n_experts=6, top_k=2, d_expert=128, d_shared=256, weight_dtype="bf16")
        w, s = make_weights(cfg, 1), make_streams(cfg, 1)
        self.blk = make_block(cfg, w)
        self.y1, self.x2, self.dy2 = dev(s["y1"]), dev(s["x2"]), dev(s["dy2"])
        self.y2, self.x2r, self.dy1 = (torch.zeros_like(self.y1) for _ in range(3))
        self.g = grad_buffers(cfg, w, 0.0)

    def __call__(self):
        self.blk.forward(self.y1, self.x2, self.y2)
        self.blk.inverse(self.y1, self.y2, self.x2r, save=True)
        self.dy1.zero_()
        self.blk.backward(self.y1, self.dy2, self.dy1, self.g, reuse=True)
        return [self.y2, self.x2r, self.dy1, *self.g.values()]


WORK = pytest.mark.parametrize("work", [_Attention, _Moe], ids=["attention", "moe"])


def _bits(out):
    torch.cuda.synchronize()
    return [t.clone() for t in out]


@WORK
def test_a_call_does_not_queue_behind_another_streams_call(rv, work):
    """Stream A is busy for about a second in front of its call; the call on stream B finishes meanwhile."""
    a, b = work(rv), work(rv)
    want = _bits(a())
    assert all(torch.equal(x, y) for x, y in zip(want, _bits(b())))
    for t in a() + b():
        t.zero_()
    torch.cuda.synchronize()
    sa, sb, after_a = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(sa):
        torch.cuda._sleep(2_000_000_000)
        out_a = a()
        after_a.record()
    with torch.cuda.stream(sb):
        out_b = b()
    sb.synchronize()
    assert not after_a.query()
    assert all(torch.equal(x, y) for x, y in zip(want, out_b))
    assert all(torch.equal(x, y) for x, y in zip(want, _bits(out_a)))


class _Graph:
    """A capture of a stream through the driver, so that several can be open at once."""

    def __init__(self, stream):
        self.cu, self.stream, self.graph, self.exe = C.CDLL("libcuda.so.1"), C.c_void_p(stream.cuda_stream), C.c_void_p(), C.c_void_p()
        assert self.cu.cuStreamBeginCapture_v2(self.stream, 2) == 0           # relaxed: the same thread goes on with other work

    def end(self):
        assert self.cu.cuStreamEndCapture(self.stream, C.byref(self.graph)) == 0
        assert self.cu.cuGraphInstantiateWithFlags(C.byref(self.exe), self.graph, C.c_ulonglong(0)) == 0

    def replay(self):
        assert self.cu.cuGraphLaunch(self.exe, self.stream) == 0

    def free(self):
        self.cu.cuGraphExecDestroy(self.exe), self.cu.cuGraphDestroy(self.graph)


@WORK
def test_calls_outside_go_on_while_streams_are_captured(rv, work):
    works = [work(rv) for _ in range(7)]
    for w in works:
        want = _bits(w())
    for w in works:
        for t in w():
            t.zero_()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in works]
    outs, graphs = [], []
    for w, s in zip(works[:-1], streams):           # more captures than the library has second streams for
        with torch.cuda.stream(s):
            graphs.append(_Graph(s))
            outs.append(w())
    with torch.cuda.stream(streams[-1]):            # a call outside all of them
        plain = works[-1]()
    for g in graphs:
        g.end()
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(want, plain))
    for o in outs:
        assert all(float(t.abs().max()) == 0.0 for t in o)                   # captured, not run
    for _ in range(2):
        for g in graphs:
            g.replay()
        for o in outs:
            assert all(torch.equal(x, y) for x, y in zip(want, _bits(o)))
            for t in o:
                t.zero_()
        torch.cuda.synchronize()
    for g in graphs:
        g.free()


@WORK
def test_more_streams_than_the_library_has(rv, work):
    works = [work(rv) for _ in range(11)]
    want = _bits(works[0]())
    for _ in range(2):
        outs = []
        for w in works:
            with torch.cuda.stream(torch.cuda.Stream()):
                outs.append(w())
        for o in outs:
            assert all(torch.equal(x, y) for x, y in zip(want, _bits(o)))
