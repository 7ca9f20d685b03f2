"""PREC_F64 maps by digit products against the program without them, which the least workspace gets, and the oracle."""
import numpy as np
import pytest

import mera_inputs as I
from oracle import mera_oracle as O
from test_gpu_x64 import _call, _cuda

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu

ORACLE = {m.OP_ASCEND: lambda h, r, u, w: O.ascend(h, u, w), m.OP_DESCEND: lambda h, r, u, w: O.descend(r, u, w),
          m.OP_ENV_U: O.env_u, m.OP_ENV_W: O.env_w}


def _least(call):
    """Bytes of the least workspace, which a refusal names."""
    with pytest.raises(m.MeraError) as e:
        call(m.workspace(256))
    return int(str(e.value).split("<")[1].split("needed")[0])


@pytest.mark.parametrize("chi_b,chi_t", [(8, 8), (7, 9), (9, 7), (4, 16), (12, 11)])
@pytest.mark.parametrize("kind", ["random", "large", "tiny", "nan", "out of range"])
def test_digits_against_fp64_units(chi_b, chi_t, kind):
    rng = np.random.default_rng(chi_b * 31 + chi_t)
    h, rho = I.random_operator(rng, chi_b, False), I.random_operator(rng, chi_t, False)
    s = {"large": 1e100, "tiny": 1e-100, "out of range": 1e-150}.get(kind, 1.0)
    h, rho = h * s, rho * s
    if kind == "nan":
        h[1, 0, 2, 3, 1, 0] = np.nan
    u, w = I.random_u(rng, chi_b), I.random_w(rng, chi_b, chi_t)
    x = [_cuda(v) for v in (h, rho, u, w)]
    for op in (m.OP_ASCEND, m.OP_DESCEND, m.OP_ENV_U, m.OP_ENV_W):
        plan = m.mera_plan_json(op, chi_b, chi_t, m.PREC_F64)
        held = [sum(dg["bufs"][st[k]]["bytes"] for k in ("a_buf", "b_buf", "ax_buf", "bx_buf", "c_buf", "p_buf") if st[k] >= 0)
                for dg in plan["diagrams"] for st in dg["steps"] if st.get("ax_buf", -1) >= 0]
        need = m.mera_workspace_size(op, chi_b, chi_t, m.PREC_F64)
        least = _least(lambda ws: _call(op, *x, chi_b, chi_t, ws))
        assert held and least < max(held)  # no room for what the largest digit product holds
        a = _call(op, *x, chi_b, chi_t, m.workspace(need))
        b = _call(op, *x, chi_b, chi_t, m.workspace(least))
        assert np.array_equal(np.isnan(a), np.isnan(b))
        ok = ~np.isnan(b)
        # at most nine products deep, each rounding at 2^-53 with sqrt(K) <= 256 terms at random
        if ok.any():
            assert np.abs(a - b)[ok].max() <= 1e-12 * np.abs(b[ok]).max()
        if kind in ("large", "tiny"):
            e = 1.0 if op in (m.OP_ASCEND, m.OP_DESCEND) else 2.0  # powers of s in the output
            want = ORACLE[op](h / s, rho / s, u, w).reshape(-1)
            assert np.abs(a / s ** e - want).max() <= 1e-12 * np.abs(want).max()
    assert m.mera_device_status(clear=True) == 0
