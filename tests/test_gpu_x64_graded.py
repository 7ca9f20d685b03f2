"""PREC_F64 products whose entries differ by decades within a row: every output is as accurate, relative to the sum of its
terms' magnitudes, as a chain of binary64 FMAs."""
import numpy as np
import pytest

import mera_inputs as I
from test_gpu_x64 import _call, _cuda, _gemm

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu


def _cases(kind, M, N, K, rng):
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    k = np.arange(K) / (K - 1)
    if kind == "opposite":  # along K, in opposite directions
        return A * 10.0 ** (-8 * k), B * 10.0 ** (8 * k)
    if kind == "steep":
        return A * 10.0 ** (-60 * k), B * 10.0 ** (60 * k)
    if kind == "peak":  # one large entry per row, met by a zero
        A[:, 3] = 1e6
        B[:, 3] = 0.0
        return A, B
    if kind == "block":  # a whole block of 256 far above the others, met by zeros
        A[:, :K // 2] *= 2.0 ** 40
        B[:, :K // 2] = 0.0
        return A, B
    if kind == "scattered":  # entries over 30 decades in no order
        return A * 10.0 ** rng.uniform(-15, 15, A.shape), B * 10.0 ** rng.uniform(-15, 15, B.shape)
    if kind == "identity":  # near the identity, and rows of unequal entries
        return A * 10.0 ** rng.uniform(-6, 0, A.shape), np.eye(N, K) + 1e-9 * B
    if kind == "sparse":  # single terms, and exact zeros
        return A * (rng.random(A.shape) < 0.1) * 10.0 ** rng.uniform(-9, 9, A.shape), B * (rng.random(B.shape) < 0.1)
    if kind == "extreme":  # six digits of every entry near their limit, one sign
        return tuple(-sum(rng.integers(115, 128, x.shape) * 2.0 ** (-6 - 8 * p) for p in range(6)) for x in (A, B))
    return A, B


@pytest.mark.parametrize("M,N,K", [(130, 70, 64), (129, 65, 255), (300, 40, 600), (64, 20, 5000)])
@pytest.mark.parametrize("kind", ["plain", "opposite", "steep", "peak", "block", "scattered", "identity", "sparse", "extreme"])
def test_graded_operands(M, N, K, kind):
    A, B = _cases(kind, M, N, K, np.random.default_rng(M + K))
    a, b = A.astype(np.longdouble), B.astype(np.longdouble)
    S = np.abs(a) @ np.abs(b).T
    got = _gemm(A, B)
    # a chain's bound is K 2^-53 S; at random its error, and that of the digits where they are taken, is a few 2^-53 S
    assert np.all(np.abs(got - a @ b.T) <= 2.0 ** -53 * (8 + 4 * np.sqrt(K)) * S)
    assert np.all(got[np.asarray(S == 0)] == 0)


def test_entry_far_below_its_row():
    A, B = np.zeros((40, 32)), np.zeros((40, 32))
    A[:, 0], A[:, 1], B[:, 1] = 1.0, 10.0 ** -np.arange(0.0, 40.0), 1.0
    assert np.array_equal(_gemm(A, B), np.repeat(A[:, 1:2], 40, axis=1))


@pytest.mark.parametrize("op", ["ascend", "descend", "env_u", "env_w"])
def test_maps_of_graded_operators(op):
    """h and rho graded by T (x) 1 (x) 1 and its inverse on the two sides: against the FP64 units, entry by entry."""
    chi = 8
    rng = np.random.default_rng(9)
    t = 10.0 ** (-7 * np.arange(chi) / (chi - 1))
    g = t[:, None, None, None, None, None] / t[None, None, None, :, None, None]
    h, rho = I.random_operator(rng, chi, False) * g, I.random_operator(rng, chi, False) * g
    u = np.eye(chi * chi).reshape((chi,) * 4) + 1e-10 * rng.standard_normal((chi,) * 4)
    w = I.random_w(rng, chi, chi)
    o = getattr(m, "OP_" + op.upper())
    x = [_cuda(v) for v in (h, rho, u, w)]
    with pytest.raises(m.MeraError) as e:  # its text names the least workspace: the FP64 units'
        _call(o, *x, chi, chi, m.workspace(256))
    least = int(str(e.value).split("<")[1].split("needed")[0])
    plan = m.mera_plan_json(o, chi, chi, m.PREC_F64)
    assert any(s.get("ax_buf", -1) >= 0 for dg in plan["diagrams"] for s in dg["steps"]) and least < plan["ws_bytes"]
    a = _call(o, *x, chi, chi, m.workspace(plan["ws_bytes"]))
    b = _call(o, *x, chi, chi, m.workspace(least))
    # the sum of the magnitudes that enter each output
    S = _call(o, *[v.abs() for v in x], chi, chi, m.workspace(least))
    assert np.all(np.abs(a - b) <= 2.0 ** -53 * 64 * S)
