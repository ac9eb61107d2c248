"""Panels whose row split changes on the way down (32 to 64 rows a CTA in binary64, 128 to 256 in
binary32), with one and two columns a lane."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("n,b,precision", [(2200, 32, egb.PREC_FP64), (1200, 64, egb.PREC_FP64),
                                           (4300, 64, egb.PREC_FP32_REFINE), (1700, 32, egb.PREC_FP32_REFINE)])
def test_row_split_changes(n, b, precision):
    k = 50
    g = torch.Generator("cuda").manual_seed(n)
    a = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    h = a + a.T
    out = egb.solve_ev(h, None, k, overlap_is_unit=True, band_width=b, precision=precision)
    ev, C = out["eval"][:k], out["C"]
    C = C if C.shape[0] == n else C.T
    norm = float(ev.abs().max())
    assert (C.T @ C - torch.eye(k, dtype=torch.float64, device="cuda")).abs().max() < 1e-10
    assert (h @ C - C * ev).abs().max() < 1e-10 * norm
