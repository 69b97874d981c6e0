"""Tiles taken one by one: every tile is worked exactly once whatever the grid and whoever else holds SMs.  Against an fp32 evaluation of
the same bf16 inputs (results are bf16, half an ulp is 1.1e-3 as an RMS; 4e-3) or bit for bit against the product run alone."""
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


@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (2741, 2048, 256), (8192, 5632, 64)])
def test_two_streams_at_once(M, N, K):
    import ctypes as C
    import paper_2512_20920_b200 as rv
    from paper_2512_20920_b200.binding import DbgGemmArgs
    A, W = _bf((M, K), 1), _bf((N, K), 2)
    out = [torch.zeros(M, N, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
    status = torch.zeros(3, 64, dtype=torch.int32, device="cuda")
    streams = [torch.cuda.current_stream(), torch.cuda.Stream(), torch.cuda.Stream()]

    def go(i):
        a = DbgGemmArgs()
        for k, v in dict(M=M, N=N, K=K, lda=K, ldb=K, ldc=N, epilogue=0, resid_sign=1.0, A=A.data_ptr(), B0=W.data_ptr(), C=out[i].data_ptr()).items():
            setattr(a, k, v)
        assert rv.lib.revffn_dbg_gemm(C.byref(a), status[i].data_ptr(), streams[i].cuda_stream) == 0
    go(0)
    torch.cuda.synchronize()
    for _ in range(10):
        go(1), go(2)
    torch.cuda.synchronize()
    assert not status.any()
    assert _close(out[0], A.float() @ W.float().T)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
