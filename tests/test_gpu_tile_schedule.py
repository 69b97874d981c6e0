"""Tiles taken one by one: every tile is worked exactly once whatever the grid and whoever else holds SMs.  Against an fp32 evaluation of
the same bf16 inputs (results are bf16, half an ulp is 1.1e-3 as an RMS; 4e-3) or bit for bit against the product run alone.  Stores
alone show a tile that was left out, products that add to what is there one that was worked twice."""
import pytest
import torch

from test_gpu_swiglu_runs import _bf, _close, _layout, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [[1000, 0, 33, 700], [96] * 40])
def test_a_table_of_short_runs_has_more_tiles_than_the_grid(counts):
    """The grid is reckoned for runs of 256 rows; runs of 32 are eight times as many tiles."""
    N, K, E = 512, 128, len(counts)
    off, tables = _layout(counts)
    runs = [[e, off[e] + r, 32, 0] for e, c in enumerate(counts) for r in range(0, c, 32)]
    tables["tok_chunks"] = torch.tensor(runs, dtype=torch.int32, device="cuda")
    tables["rows_total"] = torch.tensor([off[-1], len(runs)], dtype=torch.int32, device="cuda")
    A, W = torch.zeros(off[-1], K, device="cuda", dtype=torch.bfloat16), _bf((E, N, K), 3)
    for e, c in enumerate(counts):
        A[off[e]: off[e] + c] = _bf((c, K), 40 + e)
    C = torch.full((off[-1], N), 7.0, device="cuda", dtype=torch.bfloat16)
    _run(M=off[-1], N=N, K=K, lda=K, ldb=K, ldc=N, group_mode=1, n_groups=E, b_group_stride=N * K, epilogue=0, A=A, B0=W, C=C, **tables)
    for e, c in enumerate(counts):
        if c:
            assert _close(C[off[e]: off[e] + c], A[off[e]: off[e] + c].float() @ W[e].float().T)


def _args(**kw):
    from paper_2512_20920_b200.binding import DbgGemmArgs
    return DbgGemmArgs(resid_sign=1.0, **{k: v.data_ptr() if isinstance(v, torch.Tensor) else v for k, v in kw.items()})


@pytest.mark.parametrize("kind", ["store", "accumulate", "couple"])
@pytest.mark.parametrize("no_pair", [0, 1], ids=["pairs", "single"])
@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (2741, 2048, 256), (8192, 5632, 64)])
def test_two_streams_at_once(M, N, K, no_pair, kind):
    """Ten products on each of two streams that take each other's SMs, each with an output of its own that starts as NaN (a tile left out
    stays NaN) or, where the product adds to what is there or rewrites its input in place, from a value that a tile worked
    twice would add its share to twice."""
    import ctypes as C
    import paper_2512_20920_b200 as rv
    n = 10
    Mr = (M + 127) // 128 * 128 if kind == "accumulate" else M      # a weight gradient's rows are columns of A
    A, W = _bf((Mr, K), 1), _bf((N, K), 2)
    f32 = kind != "store"
    start = torch.randn(Mr, N, device="cuda", generator=torch.Generator("cuda").manual_seed(3)) if f32 else None
    out = [[start.clone() if f32 else torch.full((Mr, N), float("nan"), device="cuda", dtype=torch.bfloat16) for _ in range(n if i else 1)]
           for i in range(3)]
    status = torch.zeros(3, 64, dtype=torch.int32, device="cuda")
    streams = [torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()]
    At, Wt = A.T.contiguous(), W.T.contiguous()

    def go(i, j):
        kw = dict(M=Mr, N=N, K=K, lda=K, ldb=K, ldc=N, A=A, B0=W, C=out[i][j], no_pair=no_pair)
        if kind == "accumulate":
            kw.update(epilogue=5, accumulate=1, a_mn_major=1, b_mn_major=1, A=At, lda=Mr, B0=Wt, ldb=N)
        elif kind == "couple":
            kw.update(epilogue=3, resid=out[i][j], ld_resid=N)
        a = _args(**kw)
        assert rv.lib.revffn_dbg_gemm(C.byref(a), status[i].data_ptr(), streams[i].cuda_stream) == 0
    go(0, 0)
    torch.cuda.synchronize()
    for j in range(n):
        go(1, j), go(2, j)
    torch.cuda.synchronize()
    assert not status.any()
    ref = A.float() @ W.float().T
    assert _close(out[0][0] - start if f32 else out[0][0], ref)
    for o in out[1] + out[2]:
        assert torch.equal(out[0][0], o)


def test_a_grid_with_more_tiles_than_there_are():
    """The rows of an expert-grouped product are known on the device only: the grid is planned for four times the rows that there are,
    and what it grants beyond them is no tile.  Rows past the last expert stay as they are; the next product on the stream, of all
    of them, is whole."""
    N, K = 1024, 128
    counts = [200, 0, 90, 640]
    E, (off, tables) = len(counts), _layout(counts)
    cap = 4 * off[-1]
    tables["tile_group"] = torch.cat([tables["tile_group"], torch.zeros(cap // 128, dtype=torch.int32, device="cuda")])
    A, W = torch.zeros(cap, K, device="cuda", dtype=torch.bfloat16), _bf((E, N, K), 3)
    for e, c in enumerate(counts):
        A[off[e]: off[e] + c] = _bf((c, K), 50 + e)
    for runs in (True, False):
        t = dict(tables) if runs else {k: v for k, v in tables.items() if k != "tok_chunks"}
        C = torch.full((cap, N), 7.0, device="cuda", dtype=torch.bfloat16)
        _run(M=cap, N=N, K=K, lda=K, ldb=K, ldc=N, group_mode=1, n_groups=E, b_group_stride=N * K, epilogue=0, A=A, B0=W, C=C, **t)
        for e, c in enumerate(counts):
            if c:
                assert _close(C[off[e]: off[e] + c], A[off[e]: off[e] + c].float() @ W[e].float().T)
        assert torch.equal(C[off[-1]:], torch.full_like(C[off[-1]:], 7.0))
        full = torch.full((cap, N), float("nan"), device="cuda", dtype=torch.bfloat16)
        _run(M=cap, N=N, K=K, lda=K, ldb=K, ldc=N, epilogue=0, A=A, B0=W[0].contiguous(), C=full)
        assert _close(full, A.float() @ W[0].float().T)
