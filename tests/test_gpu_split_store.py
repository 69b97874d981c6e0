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
