"""Every tile width of the tcgen05 back end, as CTA pairs and as single CTAs, against a torch fp32 product, and bit for
bit against each other: an element is the same sequence of tensor instructions whatever the tile around it."""
import pytest
import torch

from test_gpu_gemm import EPI, _bf, _call, _close

pytestmark = pytest.mark.gpu

FORMS = [(256, 0), (256, 1), (128, 0), (128, 1), (64, 1), (0, 0)]      # (columns per tile, no_pair); (0, 0): as planned


@pytest.fixture(scope="module")
def rv():
    import paper_2512_20920_b200 as rv
    return rv


def _all(rv, forms, make_out, **kw):
    got = []
    for tile_n, no_pair in forms:
        out = make_out()
        _call(rv, False, tile_n=tile_n, no_pair=no_pair, **{k: v for k, v in dict(kw, **out).items()})
        got.append({k: v.clone() for k, v in out.items() if isinstance(v, torch.Tensor)})
    for g in got[1:]:
        for k in g:
            assert torch.equal(g[k], got[0][k]), k
    return got[0]


def _nan(*shape, dt=torch.bfloat16):
    return torch.full(shape, float("nan"), device="cuda", dtype=dt)


@pytest.mark.parametrize("M,N,K", [(1, 128, 64), (129, 384, 200), (700, 512, 1024)])
def test_store_and_couple_k_major(rv, M, N, K):
    A, B = _bf((M, K), 1), _bf((N, K), 2)
    ref = A.float() @ B.float().T
    base = dict(M=M, N=N, K=K, A=A, B0=B, lda=K, ldb=K, ldc=N)
    _close(_all(rv, FORMS, lambda: dict(C=_nan(M, N)), epilogue=EPI["store"], **base)["C"], ref)
    X = torch.randn(M, N, device="cuda")
    got = _all(rv, FORMS, lambda: dict(C=_nan(M, N, dt=torch.float32)), epilogue=EPI["couple"], resid=X, ld_resid=N, resid_sign=-1.0,
               **base)["C"]
    # fp32 accumulation of K <= 1024 products: 1e-5
    _close(X - got, ref, 1e-5)


@pytest.mark.parametrize("boxes", [0, 1])
@pytest.mark.parametrize("M,N,K", [(130, 128, 64), (300, 384, 320)])
def test_mn_major_operands(rv, M, N, K, boxes):
    A, B0, B1 = _bf((M, 2 * K), 3), _bf((K, N), 4), _bf((K, N), 5)
    got = _all(rv, FORMS, lambda: dict(C=_nan(M, N, dt=torch.float32)), M=M, N=N, K=2 * K, A=A, B0=B0, B1=B1, lda=2 * K, ldb=N,
               b_mn_major=1, concat=2, ldc=N, out_f32=1, epilogue=EPI["store"], mn_boxes=boxes)["C"]
    _close(got, A[:, :K].float() @ B0.float() + A[:, K:].float() @ B1.float(), 1e-5)
    Mw = 256
    At, Bt = _bf((K, Mw), 6), _bf((K, N), 7)
    got = _all(rv, FORMS, lambda: dict(C=_nan(Mw, N, dt=torch.float32)), M=Mw, N=N, K=K, A=At, B0=Bt, lda=Mw, ldb=N, a_mn_major=1,
               b_mn_major=1, ldc=N, epilogue=EPI["wgrad"], mn_boxes=boxes)["C"]
    _close(got, At.float().T @ Bt.float(), 1e-5)


@pytest.mark.parametrize("M,N,K", [(64, 128, 128), (260, 384, 256)])
def test_swiglu_pair_of_matrices(rv, M, N, K):
    A, Bg, Bu = _bf((M, K), 8), _bf((N, K), 9, 0.2), _bf((N, K), 10, 0.2)
    a, b = A.float() @ Bg.float().T, A.float() @ Bu.float().T
    got = _all(rv, [(128, 0), (128, 1), (64, 0), (64, 1), (0, 0)], lambda: dict(C=_nan(M, N), C1=_nan(M, 2 * N)), M=M, N=N, K=K, A=A,
               B0=Bg, B1=Bu, lda=K, ldb=K, concat=1, ldc=N, ldc1=2 * N, epilogue=EPI["swiglu"])
    _close(got["C"], torch.nn.functional.silu(a) * b)
    _close(got["C1"], torch.cat([a, b], dim=1))


@pytest.mark.parametrize("M,N,K", [(77, 384, 256)])
def test_swiglu_backward(rv, M, N, K):
    A, B = _bf((M, K), 11), _bf((K, N), 12, 0.2)
    ab0 = _bf((M, 2 * N), 13)
    got = _all(rv, [(256, 0), (256, 1), (128, 0), (128, 1), (0, 0)], lambda: dict(ab=ab0.clone()), M=M, N=N, K=K, A=A, B0=B, lda=K,
               ldb=N, b_mn_major=1, ld_ab=2 * N, epilogue=EPI["dswiglu"])["ab"]
    dh = A.float() @ B.float()
    a, b = ab0[:, :N].float().requires_grad_(True), ab0[:, N:].float().requires_grad_(True)
    da, db = torch.autograd.grad((torch.nn.functional.silu(a) * b * dh).sum(), (a, b))
    _close(got, torch.cat([da, db], dim=1))


@pytest.mark.parametrize("N,need", [(128, 2), (384, 4), (512, 4)])
def test_too_few_columns_for_the_row_sums_are_rejected(rv, N, need):
    """Two partial sums per row and 256 columns; nothing is launched for fewer, so the product's buffers stay as they are."""
    import ctypes as C
    from paper_2512_20920_b200.binding import DbgGemmArgs
    A, B, ab, dg = _bf((8, 128), 1), _bf((128, N), 2), _bf((8, 2 * N), 3), _nan(8, need, dt=torch.float32)
    before = ab.clone()
    a = DbgGemmArgs(M=8, N=N, K=128, lda=128, ldb=N, b_mn_major=1, A=A.data_ptr(), B0=B.data_ptr(), epilogue=EPI["dswiglu"],
                    ab=ab.data_ptr(), ld_ab=2 * N, dg_part=dg.data_ptr())
    for ld, code in ((need - 1, -2), (0, -2), (need, 0)):
        a.dg_ld = ld
        assert rv.lib.revffn_dbg_gemm(C.byref(a), None, torch.cuda.current_stream().cuda_stream) == code
        torch.cuda.synchronize()
        assert torch.equal(ab, before) == (code != 0)
    assert torch.isfinite(dg).all()
