"""The same call in scratch of different sizes: steps in waves, or one at a time, give the same bits."""
import numpy as np
import pytest

import mera_inputs as I

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "bf16x3", "oz4"])
@pytest.mark.parametrize("chi_b,chi_t", [(2, 3), (4, 4), (4, 16), (5, 6), (6, 5), (8, 8), (9, 7)])
def test_waves_and_single_steps_agree_bit_for_bit(prec, chi_b, chi_t):
    p = m.PRECS[prec]
    rng = np.random.default_rng(chi_b + 17 * chi_t)
    d = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda().reshape(-1)  # noqa: E731
    h, r = d(I.random_operator(rng, chi_b, False)), d(I.random_operator(rng, chi_t, False))
    u, w = d(I.random_u(rng, chi_b)), d(I.random_w(rng, chi_b, chi_t))
    calls = [(m.OP_ASCEND, m.mera_ascend, (h,), chi_t ** 6), (m.OP_DESCEND, m.mera_descend, (r,), chi_b ** 6),
             (m.OP_ENV_U, m.mera_env_u, (h, r), chi_b ** 4), (m.OP_ENV_W, m.mera_env_w, (h, r), chi_b ** 2 * chi_t)]
    for op, fn, ops, n in calls:
        need = m.mera_workspace_size(op, chi_b, chi_t, p)
        out, launches = [], []
        for size in (need, need - 256):
            n0 = m.mera_launch_count()
            o = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
            fn(*ops, u, w, chi_b, chi_t, o, prec=p, ws=torch.zeros(size, dtype=torch.uint8, device="cuda"))
            out.append(o)
            launches.append(m.mera_launch_count() - n0)
        assert launches[0] < launches[1]  # another form of the call
        assert torch.equal(*out), op
    assert m.mera_device_status(clear=True) == 0
