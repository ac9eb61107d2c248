"""The panel factorisation of the full -> band reduction at the edges of its row split (64 rows
a CTA in binary64, 256 in binary32; 8 and 32 rows a warp), band widths that fill one or two
columns a lane or neither, and more than one exchanging CTA, against LAPACK."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


def _matrix(n):
    a = np.random.default_rng(7 * n).standard_normal((n, n))
    return a + a.T


@pytest.mark.parametrize("n,b", [(10, 8), (41, 16), (66, 64), (67, 64), (90, 24), (128, 64), (129, 64),
                                 (137, 64), (193, 64), (300, 40), (320, 64), (577, 64), (700, 32)])
def test_panel_binary64(n, b):
    h = _matrix(n)
    ref = np.linalg.eigvalsh(h)
    norm = np.abs(ref).max()
    out = egb.solve_ev(torch.from_numpy(h).cuda(), None, n, overlap_is_unit=True, band_width=b)
    ev, C = out["eval"].cpu().numpy(), out["C"].cpu().numpy()
    np.testing.assert_allclose(ev, ref, rtol=0, atol=(1e-13 + 20 * n * 2.2e-16) * norm)
    assert np.abs(C.T @ C - np.eye(n)).max() < 1e-10
    assert np.abs(h @ C - C * ev).max() < 1e-11 * norm


@pytest.mark.parametrize("n,b", [(66, 64), (320, 64), (321, 64), (577, 32), (700, 64), (1100, 40)])
def test_panel_refined(n, b):
    h = _matrix(n)
    k = n // 8
    ref = np.linalg.eigvalsh(h)
    with egb.Handle(n, k, 0.0) as hd:
        hd.use_current_stream()
        hd.set_overlap_is_unit(True)
        hd.set_precision(egb.PREC_FP32_REFINE)
        hd.set_band_width(b)
        ev, _ = hd.ev_real(torch.from_numpy(h).cuda())
        iters, _ = hd.refine_info()
    assert iters > 0  # no binary64 repeat
    np.testing.assert_allclose(ev.cpu().numpy()[:k], ref[:k], rtol=0, atol=1e-11 * np.abs(ref).max())


def test_zero_columns_below_the_diagonal():
    """Diagonal and block-diagonal matrices: columns whose tail is exactly zero (tau = 0)."""
    n = 200
    for h in (np.diag(np.arange(n, dtype=float)), np.kron(np.eye(n // 2), np.array([[0.0, 1.0], [1.0, 0.0]]))):
        out = egb.solve_ev(torch.from_numpy(h).cuda(), None, n, overlap_is_unit=True, band_width=64)
        np.testing.assert_allclose(out["eval"].cpu().numpy(), np.linalg.eigvalsh(h), rtol=0, atol=1e-11)
        C = out["C"].cpu().numpy()
        assert np.abs(C.T @ C - np.eye(n)).max() < 1e-10
