"""Maps whose steps run in waves against the same maps one step at a time
(what a workspace without room for the waves' buffers gets)."""
import numpy as np
import pytest

import mera_inputs as I

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "tf32", "bf16", "bf16x3", "bf16x6", "oz3", "oz4"])
@pytest.mark.parametrize("chi_b,chi_t", [(1, 1), (3, 4), (4, 16), (7, 5), (8, 8)])
def test_waves_match_single_steps(prec, chi_b, chi_t):
    p = m.PRECS[prec]
    rng = np.random.default_rng(chi_b + 17 * chi_t)
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda().reshape(-1)  # noqa: E731
    h, r = d(I.random_operator(rng, chi_b, False)), d(I.random_operator(rng, chi_t, False))
    u, w = d(I.random_u(rng, chi_b)), d(I.random_w(rng, chi_b, chi_t))
    calls = [(m.OP_ASCEND, m.mera_ascend, (h,), chi_t ** 6), (m.OP_DESCEND, m.mera_descend, (r,), chi_b ** 6),
             (m.OP_ENV_U, m.mera_env_u, (h, r), chi_b ** 4), (m.OP_ENV_W, m.mera_env_w, (h, r), chi_b ** 2 * chi_t)]
    for op, fn, ops, n in calls:
        need = m.mera_workspace_size(op, chi_b, chi_t, p)
        out = [torch.full((n,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2)]
        for o, size in zip(out, (need, max(need - 256, 0))):
            fn(*ops, u, w, chi_b, chi_t, o, prec=p, ws=torch.zeros(max(size, 1), dtype=torch.uint8, device="cuda"))
        a, b = (o.cpu().numpy() for o in out)
        if prec == "f64":  # other tile shapes: sums of at most 256 products per step in another order
            assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()
        else:
            assert np.array_equal(a, b)
    assert m.mera_device_status(clear=True) == 0
