"""PREC_F64 programs whose large products run on the tensor cores: the plan's
layouts, digit images and arena, executed with numpy against the oracle."""
import numpy as np
import pytest

import mera_inputs as I
from oracle import mera_oracle as O
from test_abi_host import _emulate

m = pytest.importorskip("paper_1906_12030_gb300")


@pytest.mark.parametrize("chi_b,chi_t,slice_bytes", [(8, 8, None), (7, 9, None), (7, 7, 0), (8, 8, 8 ** 7 * 22 // 3)])
def test_split_programs_reproduce_oracle(chi_b, chi_t, slice_bytes):
    """slice_bytes: rank-7 intermediates cut value by value, and in blocks."""
    rng = np.random.default_rng(5)
    u, w = I.random_u(rng, chi_b), I.random_w(rng, chi_b, chi_t)
    h, rho = I.random_operator(rng, chi_b, False), I.random_operator(rng, chi_t, False)
    cases = [(m.OP_ASCEND, [h, None, u, w], O.ascend(h, u, w)), (m.OP_DESCEND, [None, rho, u, w], O.descend(rho, u, w)),
             (m.OP_ENV_U, [h, rho, u, w], O.env_u(h, rho, u, w)), (m.OP_ENV_W, [h, rho, u, w], O.env_w(h, rho, u, w))]
    try:
        if slice_bytes is not None:
            m.mera_set_slice_bytes(slice_bytes)
        for op, inputs, want in cases if slice_bytes is None else (cases[1], cases[3]):
            plan = m.mera_plan_json(op, chi_b, chi_t, m.PREC_F64)
            n = 0
            for dg in plan["diagrams"]:
                bufs = dg["bufs"]
                for st in dg["steps"]:
                    if st["kind"] == "gemm" and st["ax_buf"] >= 0:
                        n += 1
                        # the images' live ranges overlap the operands' (rows the digits cannot hold)
                        live = [bufs[k] for k in (st["a_buf"], st["b_buf"], st["ax_buf"], st["bx_buf"])]
                        live += [bufs[k] for k in (st["c_buf"], st["p_buf"]) if k >= 0]
                        spans = sorted((b["offset"], b["offset"] + b["bytes"]) for b in live)
                        assert all(e0 <= s1 for (_, e0), (s1, _) in zip(spans, spans[1:]))
                    if st["kind"] == "split":
                        d, nk = bufs[st["dst_buf"]], (st["K"] + 15) // 16
                        tiles = st["rows"] // st["seg_rows"] * -(-st["seg_rows"] // st["tile"])
                        assert d["bytes"] >= tiles * st["tile"] * nk * 32 * 7 + 4 * st["rows"]
            assert n >= 4
            got = _emulate(plan, inputs, want.size).reshape(want.shape)
            assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max(), op
    finally:
        m.mera_set_slice_bytes(16 << 30)
