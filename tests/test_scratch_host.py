"""Scratch of sweeps and batches: what each mode asks for, and the lanes that a budget opens."""
import pytest

import mera_inputs as I

m = pytest.importorskip("paper_1906_12030_gb300")

MIB = 1 << 20


def _dims(chis):
    out = []
    for chi in chis:
        d = I.layer_dims(chi)
        out.append(([b for b, _ in d], [t for _, t in d]))
    return out


# scratch of one operation at a time in a reused arena
@pytest.mark.parametrize("prec,chi,mib", [("bf16x3", 8, 24.7), ("bf16x3", 12, 347.5), ("bf16x3", 16, 1917.6), ("oz4", 8, 55.3),
                                          ("oz4", 12, 797.6), ("oz4", 16, 5467.8)])
def test_sweeps_of_the_tensor_core_modes_ask_for_one_arena(prec, chi, mib):
    (b, t), = _dims([chi])
    assert m.mera_sweep_workspace_size(b, t, m.PRECS[prec]) <= (mib + 0.1) * MIB


@pytest.mark.parametrize("prec,chi,n,budget,lanes", [
    ("bf16x3", 12, 1, 512 * MIB, 1), ("bf16x3", 8, 1, 64 * MIB, 1), ("oz4", 8, 4, 256 * MIB, 4), ("bf16x3", 12, 8, 4096 * MIB, 8),
    ("f64", 8, 8, 1024 * MIB, 8), ("f64", 12, 2, 4096 * MIB, 2), ("f64", 8, 1, 40 * MIB, 1)])
def test_budgets_open_lanes(prec, chi, n, budget, lanes):
    p = m.PRECS[prec]
    where, size = m.mera_batch_lanes(_dims([chi] * n), p, budget)
    assert len(size) == lanes and sorted(set(where)) == list(range(lanes)) and sum(size) <= budget


def test_f64_lanes_are_as_fast_as_the_budget_allows():
    """With room for it every lane has the scratch that a sweep asks for."""
    dims = _dims([8, 8, 6])
    need = [m.mera_sweep_workspace_size(b, t, m.PREC_F64) for b, t in dims]
    where, size = m.mera_batch_lanes(dims, m.PREC_F64, sum(need))
    assert [size[k] for k in where] == need


@pytest.mark.parametrize("prec", ["f64", "bf16x3", "oz4"])
@pytest.mark.parametrize("chi_b,chi_t", [(4, 4), (8, 8), (4, 16), (12, 12)])
@pytest.mark.parametrize("op", ["ASCEND", "DESCEND", "ENV_U", "ENV_W"])
def test_buffers_of_a_common_wave_are_apart(prec, chi_b, chi_t, op):
    plan = m.mera_plan_json(getattr(m, "OP_" + op), chi_b, chi_t, m.PRECS[prec])
    if not plan["waves"]:
        pytest.skip("one step at a time")
    live = {}  # (diagram, buffer) -> first and last wave
    for at, wave in enumerate(plan["waves"]):
        for d, k in wave["steps"]:
            st = plan["diagrams"][d]["steps"][k]
            names = {"permute": ("dst_buf",), "split": ("raw_buf", "dst_buf")}.get(
                st["kind"], ("a_buf", "b_buf", "ax_buf", "bx_buf", "c_buf", "p_buf", "m_buf"))
            for name in names:
                if st.get(name, -1) >= 0:
                    lo, hi = live.get((d, st[name]), (at, at))
                    live[d, st[name]] = min(lo, at), max(hi, at)
    spans = []
    for (d, k), (lo, hi) in live.items():
        b = plan["diagrams"][d]["bufs"][k]
        assert b["offset"] % 256 == 0 and b["offset"] + b["bytes"] <= plan["ws_bytes"]
        assert b["resident"] or b["offset"] >= plan["persistent_bytes"]
        if not b["resident"]:
            spans.append((b["offset"], b["offset"] + b["bytes"], lo, hi))
    spans.sort()
    for i, (lo, hi, first, last) in enumerate(spans):
        for lo2, _, first2, last2 in spans[i + 1:]:
            if lo2 >= hi:
                break
            assert last < first2 or last2 < first
