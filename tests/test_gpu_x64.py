"""PREC_F64 products on the tensor cores (digit splitting) against numpy and
against the FP64-unit route, which a workspace without room for digits takes."""
import numpy as np
import pytest

import mera_inputs as I

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu


def _cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda().reshape(-1)


def _gemm(A, B):
    """C = A B^T by the tensor-core route (a workspace large enough for it)."""
    (M, K), N = A.shape, B.shape[0]
    C = torch.empty(M * N, dtype=torch.float64, device="cuda")
    ws = m.workspace(64 * (M + N + 256) * (K + 64) + 1200 * 12 * M * N + (1 << 20))
    a, b = _cuda(A), _cuda(B)
    lib = m.library()
    s = torch.cuda.current_stream().cuda_stream
    assert lib.mera_gemm_test(m.PREC_F64, a.data_ptr(), b.data_ptr(), M, N, K, C.data_ptr(), ws.data_ptr(), ws.numel(),
                              s) == 0
    out = C.cpu().numpy().reshape(M, N)
    assert m.mera_device_status(clear=True) == 0
    return out


def _exact(A, B):
    return (A.astype(np.longdouble) @ B.T.astype(np.longdouble)).astype(np.float64)


# one tile and less, tile edges, K at and around the 16-wide steps and the
# 256-blocks, K splits in half and whole blocks, rows of more than 8192
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (16, 16, 16), (127, 63, 15), (128, 64, 17), (129, 65, 255), (300, 70, 256),
                                   (130, 17, 257), (1000, 100, 100), (64, 64, 1000), (100, 10, 8192), (9, 70, 8193),
                                   (20, 20, 16500)])
def test_gemm_shapes(M, N, K):
    rng = np.random.default_rng(M + 7 * N + 13 * K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    got, want = _gemm(A, B), _exact(A, B)
    # dropped digit products and digits: ~2^-55 of the largest entries' product
    # per term, summing at random; one rounding to binary64
    tol = 2.0 ** -52 * np.sqrt(K) * np.abs(A).max() * np.abs(B).max() + 2.0 ** -52 * np.abs(want)
    assert np.all(np.abs(got - want) <= tol)


def test_gemm_exact_on_integers():
    """Sums below 2^53 of integers come out bit for bit, signed zeros aside."""
    rng = np.random.default_rng(3)
    A, B = rng.integers(-2 ** 20, 2 ** 20, (130, 300)).astype(float), rng.integers(-2 ** 20, 2 ** 20, (70, 300)).astype(float)
    A[0] = 0.0
    assert np.array_equal(_gemm(A, B), A @ B.T)
    C = np.full((130, 512), -255.0)  # every product extreme and of one sign
    assert np.array_equal(_gemm(C, C[:70]), C @ C[:70].T)


def test_gemm_scales_and_special_values():
    """Rows graded over 200 decades keep their own accuracy; rows with NaN,
    infinities or entries the digits cannot scale follow the FP64 units."""
    rng = np.random.default_rng(4)
    A, B = rng.standard_normal((140, 200)), rng.standard_normal((70, 200))
    s = 10.0 ** rng.uniform(-100, 100, 140)
    got, want = _gemm(A * s[:, None], B), _exact(A, B) * s[:, None]
    assert np.all(np.abs(got - want) <= 2.0 ** -49 * np.sqrt(200) * 16 * s[:, None])
    A[3, 5], A[7, 0], A[9, 9], B[11, 2] = np.nan, np.inf, -np.inf, np.inf
    A[20] *= 1e200
    A[21] *= 1e-200
    A[22] *= 1e-310
    with np.errstate(all="ignore"):
        want = A @ B.T
    got = _gemm(A, B)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    ok = np.isfinite(want)
    assert np.array_equal(np.sign(got[~ok & ~np.isnan(want)]), np.sign(want[~ok & ~np.isnan(want)]))
    scale = np.linalg.norm(np.where(np.isfinite(A), A, 0), axis=1)[:, None]
    assert np.all(np.abs(got - want)[ok] <= (1e-13 * scale * 16 + 1e-320 + 0 * want)[ok])


def _call(op, hd, rd, ud, wd, cb, ct, ws):
    n = {m.OP_ASCEND: ct ** 6, m.OP_DESCEND: cb ** 6, m.OP_ENV_U: cb ** 4, m.OP_ENV_W: cb * cb * ct}[op]
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    if op == m.OP_ASCEND:
        m.mera_ascend(hd, ud, wd, cb, ct, out, ws=ws)
    elif op == m.OP_DESCEND:
        m.mera_descend(rd, ud, wd, cb, ct, out, ws=ws)
    elif op == m.OP_ENV_U:
        m.mera_env_u(hd, rd, ud, wd, cb, ct, out, ws=ws)
    else:
        m.mera_env_w(hd, rd, ud, wd, cb, ct, out, ws=ws)
    return out.cpu().numpy()


@pytest.mark.parametrize("chi_b,chi_t", [(8, 8), (7, 9), (9, 7), (4, 16), (12, 11)])
@pytest.mark.parametrize("kind", ["random", "large", "tiny", "nan"])
def test_maps_match_the_fp64_route(chi_b, chi_t, kind):
    rng = np.random.default_rng(chi_b * 31 + chi_t)
    h, rho = I.random_operator(rng, chi_b, False), I.random_operator(rng, chi_t, False)
    if kind == "large":
        h = h * 1e150
    if kind == "tiny":
        h = h * 1e-150
    if kind == "nan":
        h[1, 0, 2, 3, 1, 0] = np.nan
    x = [_cuda(v) for v in (h, rho, I.random_u(rng, chi_b), I.random_w(rng, chi_b, chi_t))]
    for op in (m.OP_ASCEND, m.OP_DESCEND, m.OP_ENV_U, m.OP_ENV_W):
        need = m.mera_workspace_size(op, chi_b, chi_t, m.PREC_F64)
        a = _call(op, *x, chi_b, chi_t, m.workspace(need))
        b = _call(op, *x, chi_b, chi_t, m.workspace(need - 256))  # no room for every digit image
        assert np.array_equal(np.isnan(a), np.isnan(b))
        ok = ~np.isnan(b)
        if ok.any():
            # at most nine products deep, each rounding at 2^-53 with sqrt(K) <= 256 terms at random
            assert np.abs(a - b)[ok].max() <= 1e-12 * np.abs(b[ok]).max()
    assert m.mera_device_status(clear=True) == 0
