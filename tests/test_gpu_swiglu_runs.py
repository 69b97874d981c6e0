"""Experts' SwiGLU with token runs on the MMA N side (weights on M, 16 rows of both matrices in turn): runs of every
kind of length, one and several feature tiles, a ragged K step, either matrix first in memory, with and without the
a|b copy and the row scale, against a plain fp32 evaluation of the same bf16 inputs.  An expert's padding rows must come
out as zeros and rows past the last expert untouched.  Tolerance: results are bf16 (half an ulp is 2^-9 relative, as an
RMS 2^-9 / sqrt(3) = 1.1e-3) from fp32 sums whose order is all that differs; 4e-3."""
import ctypes as C

import pytest
import torch

pytestmark = pytest.mark.gpu


def _bf(shape, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    return (torch.randn(*shape, device="cuda", generator=g) * 0.3).to(torch.bfloat16)


@pytest.mark.parametrize("up_first", [False, True])
@pytest.mark.parametrize("ab", [False, True])
@pytest.mark.parametrize("N,K", [(128, 64), (384, 200), (1408, 512)])
@pytest.mark.parametrize("counts", [[130, 0, 5, 256, 1], [700, 33, 0, 257, 64, 1000], [0, 0, 3], [96, 128, 224]])
def test_runs(counts, N, K, ab, up_first):
    import paper_2512_20920_b200 as rv
    from paper_2512_20920_b200.binding import DbgGemmArgs
    E, off, runs = len(counts), [0], []
    for e, c in enumerate(counts):
        off.append(off[-1] + (c + 127) // 128 * 128)
        n = (c + 31) // 32 * 32
        for r in range(0, n, 256):
            runs.append([e, off[e] + r, min(256, n - r), off[e + 1] - off[e] - n if r + 256 >= n else 0])
    cap = off[-1] + 256
    A = torch.zeros(cap, K, device="cuda", dtype=torch.bfloat16)
    scale = torch.zeros(cap, device="cuda")
    for e, c in enumerate(counts):
        A[off[e]: off[e] + c] = _bf((c, K), 20 + e)
        scale[off[e]: off[e] + c] = torch.rand(c, device="cuda") + 0.5
    W = _bf((2, E, N, K), 30)
    Wg, Wu = (W[1], W[0]) if up_first else (W[0], W[1])
    H = torch.full((cap, N), 7.0, device="cuda", dtype=torch.bfloat16)
    AB = torch.full((cap, 2 * N), 7.0, device="cuda", dtype=torch.bfloat16)
    t32 = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")
    tens = dict(A=A, B0=Wg, B1=Wu, C=H, rowscale=scale, group_off=t32(off), rows_total=t32([off[-1], len(runs)]),
                tile_group=t32([e for e in range(E) for _ in range((off[e + 1] - off[e]) // 128)] + [0] * 8),
                tok_chunks=t32(runs + [[0, 0, 0, 0]]))
    if ab:
        tens["C1"] = AB
    a = DbgGemmArgs()
    for k, v in dict(M=cap, N=N, K=K, lda=K, ldb=K, ldc=N, ldc1=2 * N, group_mode=1, n_groups=E, b_group_stride=N * K, concat=1,
                     epilogue=1, resid_sign=1.0).items():
        setattr(a, k, v)
    for k, v in tens.items():
        setattr(a, k, v.data_ptr())
    status = torch.zeros(64, dtype=torch.int32, device="cuda")
    assert rv.lib.revffn_dbg_gemm(C.byref(a), status.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert int(status[0]) == 0
    close = lambda x, y: float((x.float() - y).norm() / y.norm()) < 4e-3
    for e, c in enumerate(counts):
        real, pad = slice(off[e], off[e] + c), slice(off[e] + c, off[e + 1])
        if c == 0:
            continue
        x = A[real].float()
        g, u = x @ Wg[e].float().T, x @ Wu[e].float().T
        assert close(H[real], torch.nn.functional.silu(g) * u * scale[real, None])
        assert not H[pad].any()
        if ab:
            assert close(AB[real, :N], g) and close(AB[real, N:], u)
            assert not AB[pad].any()
    assert (H[off[-1]:] == 7.0).all() and (AB[off[-1]:] == 7.0).all()
