"""Experts' SwiGLU and its backward with token runs on the MMA N side (weights on M; forward: 16 rows of both matrices in
turn): runs of every kind of length, one and several feature tiles, a last tile of half width, a ragged K step, either
matrix first in memory, with and without the a|b copy, against a plain fp32 evaluation of the same bf16 inputs.  An
expert's padding rows must come out as zeros up to the next multiple of 64; the operands hold NaN beyond it, and there, as past
the last expert, nothing may be written (few tiles go to row tiles of 128 instead, which compute whole tiles).  Tolerance: results are bf16 (half an ulp is 2^-9 relative, as an
RMS 2^-9 / sqrt(3) = 1.1e-3) from fp32 sums whose order is all that differs; 4e-3."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


def _bf(shape, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return (torch.randn(*shape, device="cuda", generator=g) * 0.3).to(torch.bfloat16)


def _layout(counts):
    off, runs = [0], []
    for e, c in enumerate(counts):
        off.append(off[-1] + (c + 127) // 128 * 128)
        n = (c + 31) // 32 * 32
        for r in range(0, n, 256):
            runs.append([e, off[e] + r, min(256, n - r), (c + 63) // 64 * 64 - n if r + 256 >= n else 0])
    t32 = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")
    return off, dict(group_off=t32(off), rows_total=t32([off[-1], len(runs)]),
                     tile_group=t32([e for e in range(len(counts)) for _ in range((off[e + 1] - off[e]) // 128)] + [0] * 8),
                     tok_chunks=t32(runs + [[0, 0, 0, 0]]))


def _transposed(cap, E, feature_tiles):
    """The launcher's rule: token runs where their tiles occupy half the SMs."""
    return ((cap - 127 * E) // 256 + E // 2) * feature_tiles >= torch.cuda.get_device_properties(0).multi_processor_count // 2


def _unset(t, counts, off):
    """NaN in the rows past each expert's 64-row boundary."""
    for e, c in enumerate(counts):
        t[off[e] + (c + 63) // 64 * 64: off[e + 1]] = float("nan")
    return t


def _run(**kw):
    import paper_2512_20920_b200 as rv
    from paper_2512_20920_b200.binding import DbgGemmArgs
    a = DbgGemmArgs()
    a.resid_sign = 1.0
    for k, v in kw.items():
        setattr(a, k, v.data_ptr() if isinstance(v, torch.Tensor) else v)
    status = torch.zeros(64, dtype=torch.int32, device="cuda")
    assert rv.lib.revffn_dbg_gemm(C.byref(a), status.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert int(status[0]) == 0


def _close(x, y, tol=4e-3):
    return float((x.float() - y).norm() / y.norm()) < tol


COUNTS = [[130, 0, 5, 256, 1], [700, 33, 0, 257, 64, 1000], [0, 0, 3], [96, 128, 224] + [40] * 70]


@pytest.mark.parametrize("up_first", [False, True])
@pytest.mark.parametrize("ab", [False, True])
@pytest.mark.parametrize("N,K", [(128, 64), (384, 200), (1408, 512), (6400, 72)])
@pytest.mark.parametrize("counts", COUNTS)
def test_runs(counts, N, K, ab, up_first):
    E, (off, tables) = len(counts), _layout(counts)
    cap = off[-1] + 256
    A = torch.zeros(cap, K, device="cuda", dtype=torch.bfloat16)
    scale = torch.zeros(cap, device="cuda")
    for e, c in enumerate(counts):
        A[off[e]: off[e] + c] = _bf((c, K), 20 + e)
        scale[off[e]: off[e] + c] = torch.rand(c, device="cuda") + 0.5
    _unset(A, counts, off)
    W, tr = _bf((2, E, N, K), 30), _transposed(cap, E, -(-N // 128))
    Wg, Wu = (W[1], W[0]) if up_first else (W[0], W[1])
    H = torch.full((cap, N), 7.0, device="cuda", dtype=torch.bfloat16)
    AB = torch.full((cap, 2 * N), 7.0, device="cuda", dtype=torch.bfloat16)
    _run(M=cap, N=N, K=K, lda=K, ldb=K, ldc=N, ldc1=2 * N, group_mode=1, n_groups=E, b_group_stride=N * K, concat=1, epilogue=1,
         A=A, B0=Wg, B1=Wu, C=H, rowscale=scale, **tables, **(dict(C1=AB) if ab else {}))
    for e, c in enumerate(counts):
        edge = off[e] + (c + 63) // 64 * 64
        real, pad, beyond = slice(off[e], off[e] + c), slice(off[e] + c, edge), slice(edge, off[e + 1])
        if c == 0:
            continue
        assert not tr or ((H[beyond] == 7.0).all() and (AB[beyond] == 7.0).all())
        x = A[real].float()
        g, u = x @ Wg[e].float().T, x @ Wu[e].float().T
        assert _close(H[real], torch.nn.functional.silu(g) * u * scale[real, None])
        assert not H[pad].any()
        if ab:
            assert _close(AB[real, :N], g) and _close(AB[real, N:], u)
            assert not AB[pad].any()
    assert (H[off[-1]:] == 7.0).all() and (AB[off[-1]:] == 7.0).all()


@pytest.mark.parametrize("runs", [False, True])
@pytest.mark.parametrize("N,K", [(128, 64), (384, 192), (1408, 512), (6400, 128)])
@pytest.mark.parametrize("counts", COUNTS)
def test_backward(counts, N, K, runs):
    """Row sums of <dH', H>: fp32 sums of N products in another order, 1e-3 of their norm."""
    E, (off, tables) = len(counts), _layout(counts)
    if not runs:
        del tables["tok_chunks"]
    cap = off[-1] + 256
    A = torch.zeros(cap, K, device="cuda", dtype=torch.bfloat16)
    AB = torch.zeros(cap, 2 * N, device="cuda", dtype=torch.bfloat16)
    AB[off[-1]:] = 7.0
    scale = torch.zeros(cap, device="cuda")
    for e, c in enumerate(counts):
        A[off[e]: off[e] + c] = _bf((c, K), 20 + e)
        AB[off[e]: off[e] + c] = 3 * _bf((c, 2 * N), 70 + e)
        scale[off[e]: off[e] + c] = torch.rand(c, device="cuda") + 0.5
    _unset(A, counts, off), _unset(AB, counts, off)
    W, AB0, ld = _bf((E, K, N), 30), AB.clone(), N // 32
    tr = runs and _transposed(cap, E, -(-N // 256))
    dg = torch.zeros(cap, ld, device="cuda")
    _run(M=cap, N=N, K=K, lda=K, ldb=N, b_mn_major=1, group_mode=1, n_groups=E, b_group_stride=N * K, epilogue=4, A=A, B0=W, ab=AB,
         ld_ab=2 * N, rowscale=scale, dg_part=dg, dg_ld=ld, **tables)
    for e, c in enumerate(counts):
        edge = off[e] + (c + 63) // 64 * 64
        real, pad, beyond = slice(off[e], off[e] + c), slice(off[e] + c, edge), slice(edge, off[e + 1])
        if c == 0:
            continue
        assert not tr or torch.equal(AB[beyond].view(torch.int16), AB0[beyond].view(torch.int16))
        acc, a, b = A[real].float() @ W[e].float(), AB0[real, :N].float(), AB0[real, N:].float()
        s, dh = torch.sigmoid(a), scale[real, None] * acc
        assert _close(AB[real, :N], dh * b * (s * (1 + a * (1 - s)))) and _close(AB[real, N:], dh * a * s)
        assert not AB[pad].any()
        assert _close(dg[real].sum(1), (acc * a * s * b).sum(1), 1e-3)
    assert (AB[off[-1]:] == 7.0).all()
