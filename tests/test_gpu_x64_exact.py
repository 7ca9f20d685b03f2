"""Outputs of the digit products that are left to the FP64 units: those of rows that the digits cannot represent."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu


def _gemm(A, B):
    """C = A B^T of device matrices, by the tensor-core route (a workspace large enough for it)."""
    (M, K), N = A.shape, B.shape[0]
    C = torch.full((M, N), 7.0, dtype=torch.float64, device="cuda")
    ws = m.workspace(32 * (M + N + 256) * (K + 64) + (24 * M * N * 8 if M * N > 1 << 18 else 1200 * 16 * M * N) + (1 << 20))
    s = torch.cuda.current_stream().cuda_stream
    assert m.library().mera_gemm_test(m.PREC_F64, A.data_ptr(), B.data_ptr(), M, N, K, C.data_ptr(), ws.data_ptr(),
                                      ws.numel(), s) == 0
    torch.cuda.synchronize()
    assert m.mera_device_status(clear=True) == 0
    return C


def _rand(r, c, seed):
    return torch.randn(r, c, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


# tile edges, K splits (long K, few tiles), K below and past the strides of the FP64 sums
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (5, 3, 7), (128, 64, 31), (129, 65, 33), (260, 130, 256), (40, 70, 5000)])
@pytest.mark.parametrize("bad", ["all", "rows", "columns"])
def test_rows_out_of_range(M, N, K, bad):
    A, B = _rand(M, K, 1), _rand(N, K, 2)
    sa = torch.ones(M, 1, dtype=torch.float64, device="cuda")
    sb = torch.ones(N, 1, dtype=torch.float64, device="cuda")
    if bad != "columns":
        sa[slice(None) if bad == "all" else slice(0, None, 3)] = 2.0 ** 450
    if bad != "rows":
        sb[slice(None) if bad == "all" else slice(N - 1, None)] = 2.0 ** -430
    got = (_gemm(A * sa, B * sb) / sa / sb.T).cpu().numpy()
    a, b = A.cpu().numpy().astype(np.longdouble), B.cpu().numpy().astype(np.longdouble)
    # one chain of FMAs, or the digits
    assert np.all(np.abs(got - a @ b.T) <= 2.0 ** -53 * (K + 4) * (np.abs(a) @ np.abs(b).T))


def test_long_sums_finish():
    """152 tiles with K = 331776 (the isometry environment's at chi = 24): a NaN row and an out-of-range column, among
    whole numbers whose sums are exact."""
    M, N, K = 1024, 1216, 331776
    A, B = (torch.round(_rand(r, K, 3 + r) * 100) for r in (M, N))
    nan, far = 5, 100
    A[nan, 7] = float("nan")
    B[far] *= 2.0 ** 450
    C = _gemm(A, B)
    assert torch.isnan(C[nan]).all()
    A[nan], C[nan] = 0.0, 0.0
    assert torch.equal(C[:, far], A @ B[far])
    for r in (0, 6, 500, M - 1):
        assert torch.equal(C[r], B @ A[r])
