"""Polar update at the edges of its three forms: fused steps (n <= 320), digit
products, and the FP64 products that a smaller scratch gets."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mm,nn", [(1, 1), (9, 7), (8, 8), (65, 9), (600, 17), (320, 320), (321, 321), (361, 361), (700, 330)])
@pytest.mark.parametrize("less", [0, 256])
def test_polar_matches_svd(mm, nn, less):
    if less and nn <= 320:
        pytest.skip("one form")
    rng = np.random.default_rng(mm + 3 * nn)
    q = lambda r, c: np.linalg.qr(rng.standard_normal((r, c)))[0]  # noqa: E731
    s = 100.0 ** (-np.arange(nn) / max(1, nn - 1))
    env = (q(mm, nn) * s) @ q(nn, nn).T
    ws = m.workspace(m.mera_polar_workspace_size(mm, nn) - less)
    out = torch.empty(mm * nn, dtype=torch.float64, device="cuda")
    m.mera_polar_update(torch.from_numpy(env).cuda().reshape(-1), mm, nn, out, ws=ws)
    u, _, vt = np.linalg.svd(env, full_matrices=False)
    x = out.cpu().numpy().reshape(mm, nn)
    assert m.mera_device_status(clear=True) == 0
    # condition 100, a few roundings per product at 2^-53 sqrt(K)
    assert np.abs(x + u @ vt).max() <= 100 * 2.0 ** -53 * 16 * np.sqrt(mm)
    assert np.abs(x.T @ x - np.eye(nn)).max() <= 2.0 ** -53 * 64 * np.sqrt(mm)


def test_polar_keeps_nan_and_zero_behaviour():
    for env in (np.zeros((9, 9)), np.full((9, 9), np.nan)):
        out = torch.zeros(81, dtype=torch.float64, device="cuda")
        m.mera_polar_update(torch.from_numpy(env).cuda().reshape(-1), 9, 9, out)
        assert torch.isnan(out).all()
    m.mera_device_status(clear=True)
