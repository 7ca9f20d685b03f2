"""Polar update of matrices whose columns differ by decades: the factor of Q D, Q orthonormal and D diagonal
and positive, is Q whatever D."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
m = pytest.importorskip("paper_1906_12030_gb300")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mm,nn,decades", [(65, 40, 8), (400, 330, 8), (400, 330, 12), (800, 721, 8), (1024, 900, 12)])
def test_polar_of_graded_columns(mm, nn, decades):
    rng = np.random.default_rng(mm + nn + decades)
    q = np.linalg.qr(rng.standard_normal((mm, nn)))[0]
    env = q * 10.0 ** (-decades * np.arange(nn) / (nn - 1))
    out = torch.empty(mm * nn, dtype=torch.float64, device="cuda")
    m.mera_polar_update(torch.from_numpy(env).cuda().reshape(-1), mm, nn, out)
    x = out.cpu().numpy().reshape(mm, nn)
    assert m.mera_device_status(clear=True) == 0
    # a step rounds every entry to a few units of 2^-53 of its column's scale; some forty steps
    tol = 2.0 ** -53 * 64 * np.sqrt(mm)
    assert np.abs(x + q).max() <= tol
    assert np.abs(x.T @ x - np.eye(nn)).max() <= tol
