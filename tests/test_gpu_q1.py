"""Compact-WY groups of the back-transformation through Q1: every position of the last, shorter group (1 to
4 panels), a band width that is not a multiple of the block tiles, one panel alone, both element types."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("precision", [egb.PREC_FP64, egb.PREC_FP32_REFINE])
@pytest.mark.parametrize("n,b,k", [(34, 32, 9), (66, 32, 20), (130, 32, 33), (162, 32, 40), (200, 24, 31), (330, 64, 60),
                                   (395, 64, 60), (600, 40, 77), (700, 64, 120)])
def test_q1_groups(n, b, k, precision):
    rng = np.random.default_rng(n + b)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = np.sort(rng.uniform(-3, 3, n))
    lam[k:] += 0.5  # a gap above the wanted states, for the refinement
    h = (q * lam) @ q.T
    h = 0.5 * (h + h.T)
    out = egb.solve_ev(torch.from_numpy(h).cuda(), None, k, overlap_is_unit=True, band_width=b, precision=precision)
    ev, C = out["eval"].cpu().numpy()[:k], out["C"].cpu().numpy()
    np.testing.assert_allclose(ev, lam[:k], rtol=0, atol=1e-12 * n)
    assert np.abs(C.T @ C - np.eye(k)).max() < 1e-10
    assert np.abs(h @ C - C * ev).max() < 1e-10


def test_q1_groups_of_eight():
    """n from 4096: groups of eight panels, a last group of 7 (128 panels of 32, all but one)."""
    n, k = 4130, 40
    a = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    h = a + a.T
    out = egb.solve_ev(h, None, k, overlap_is_unit=True, band_width=32)
    ev, C = out["eval"][:k], out["C"]
    C = C if C.shape[0] == n else C.T
    assert (C.T @ C - torch.eye(k, dtype=torch.float64, device="cuda")).abs().max() < 1e-10
    assert (h @ C - C * ev).abs().max() < 1e-10 * ev.abs().max() * 10
