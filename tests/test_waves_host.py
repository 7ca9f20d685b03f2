"""Small operations run in waves (one launch for the independent steps of all
diagrams): executed with numpy in wave order, steps of one wave in reverse, the
programs still give the oracle's maps, on first and on repeated runs."""
import numpy as np
import pytest

import mera_inputs as I
from oracle import mera_oracle as O
from test_abi_host import _emulate

m = pytest.importorskip("paper_1906_12030_gb300")


def _in_wave_order(plan):
    """The operation as one diagram whose steps come in wave order."""
    bufs, base = [], []
    for dg in plan["diagrams"]:
        base.append(len(bufs))
        bufs += dg["bufs"]
    steps, seen = [], set()
    for w in plan["waves"]:
        for d, k in reversed(w["steps"]):
            seen.add((d, k))
            st = dict(plan["diagrams"][d]["steps"][k])
            for key in ("a_buf", "b_buf", "c_buf", "p_buf", "ax_buf", "bx_buf", "dst_buf", "op_buf", "raw_buf"):
                if st.get(key, -1) >= 0:
                    st[key] += base[d]
            if st["kind"] == "gemm" and st["c_buf"] < 0:
                st["accumulate"] = 1  # onto zeros: the parts are summed, or the second diagram accumulates
            steps.append(st)
    every = {(d, k) for d, dg in enumerate(plan["diagrams"]) for k, st in enumerate(dg["steps"]) if not st.get("skip")}
    assert seen == every and len(steps) == len(every)
    return {**plan, "diagrams": [{"bufs": bufs, "steps": steps}]}


@pytest.mark.parametrize("prec,chi_b,chi_t", [(p, b, t) for p in (m.PREC_F64, m.PREC_BF16X3, m.PREC_OZ3)
                                              for b, t in ((1, 1), (3, 4), (6, 5))] + [(m.PREC_F64, 8, 8)])
def test_waves_reproduce_oracle(prec, chi_b, chi_t):
    rng = np.random.default_rng(41)
    u, w = I.random_u(rng, chi_b), I.random_w(rng, chi_b, chi_t)
    h, rho = I.random_operator(rng, chi_b, False), I.random_operator(rng, chi_t, False)
    for op, inputs, want in ((m.OP_ASCEND, [h, None, u, w], O.ascend(h, u, w)), (m.OP_DESCEND, [None, rho, u, w], O.descend(rho, u, w)),
                             (m.OP_ENV_U, [h, rho, u, w], O.env_u(h, rho, u, w)), (m.OP_ENV_W, [h, rho, u, w], O.env_w(h, rho, u, w))):
        if chi_b == 8 and op not in (m.OP_DESCEND, m.OP_ENV_W):
            continue
        plan = m.mera_plan_json(op, chi_b, chi_t, prec)
        assert plan["waves"]
        if len(plan["diagrams"]) > 2:
            assert plan["part_off"] + len(plan["diagrams"]) * plan["part_bytes"] <= plan["ws_bytes"]
            assert plan["part_bytes"] == 8 * want.size
            assert all(b["offset"] + b["bytes"] <= plan["part_off"] for dg in plan["diagrams"] for b in dg["bufs"])
        flat = _in_wave_order(plan)
        got, arena = _emulate(flat, inputs, want.size, keep=True)
        assert np.abs(got.reshape(want.shape) - want).max() <= 1e-12 * max(1.0, np.abs(want).max()), op
        if op == m.OP_DESCEND:
            got = _emulate(flat, [None, 2.0 * rho, u, w], want.size, arena=arena, reuse=True)
            assert np.abs(got.reshape(want.shape) - 2.0 * want).max() <= 2e-12 * max(1.0, np.abs(want).max())


def test_diagrams_run_in_pairs_where_all_at_once_take_much_memory():
    """chi = 12 env_w in OZ3: three pairs of diagrams, one after another, on
    the same transient memory."""
    plan = m.mera_plan_json(m.OP_ENV_W, 12, 12, m.PREC_OZ3)
    assert plan["waves"]
    order = [max(d // 2 for d, k in w["steps"] if not plan["diagrams"][d]["steps"][k]["kind"] == "permute") for w in plan["waves"]
             if any(plan["diagrams"][d]["steps"][k]["kind"] != "permute" for d, k in w["steps"])]
    assert order == sorted(order) and set(order) == {0, 1, 2}
