"""Tensor-core GEMMs large enough for CTA pairs against the same rows computed
by single CTAs (a product of few tiles): every output sums the same terms in the
same order, so the results are equal bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu


# pairs from K = 384 (BF16X3, TF32) or 1024 (BF16) on: tiles 256, 192 and 128
# wide with a ragged last column tile, a last row pair whose second half is
# partial or missing, K at a ragged multiple and over several rounds of the ring
@pytest.mark.parametrize("prec", ["tf32", "bf16", "bf16x3"])
@pytest.mark.parametrize("M,N,K", [(20001, 1100, 1030), (26900, 570, 1024), (6912, 576, 1500), (300, 129, 2048),
                                   (20001, 1100, 70)])
def test_pairs_match_single_ctas(prec, M, N, K):
    p = m.PRECS[prec]
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(N, K, dtype=torch.float64, device="cuda", generator=g)
    C = torch.full((M * N,), float("nan"), dtype=torch.float64, device="cuda")
    m.mera_gemm_test(p, A, B, C)
    C = C.reshape(M, N).cpu().numpy()
    for lo, hi in ((0, 128), (M // 2, M // 2 + 100), (M - 128, M)):
        for c0 in range(0, N, 128):  # products of one narrow tile run on single CTAs
            c1 = min(N, c0 + 128)
            D = torch.empty((hi - lo) * (c1 - c0), dtype=torch.float64, device="cuda")
            m.mera_gemm_test(p, A[lo:hi].contiguous(), B[c0:c1].contiguous(), D)
            assert np.array_equal(C[lo:hi, c0:c1], D.cpu().numpy().reshape(hi - lo, c1 - c0))
    assert np.isfinite(C).all()
    assert m.mera_device_status(clear=True) == 0

