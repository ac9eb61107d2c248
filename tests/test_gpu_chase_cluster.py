"""The bulge chase of up to 16 positions (one cluster, 1 to 16 CTAs and idle ones up to a power of two) and of 17
(through L2), both element types."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("precision", [egb.PREC_FP64, egb.PREC_FP32_REFINE])
@pytest.mark.parametrize("n,b", [(35, 32), (66, 32), (98, 32), (162, 32), (290, 32), (513, 32), (514, 32), (1025, 64),
                                 (1026, 64)])
def test_positions(n, b, precision):
    k = max(1, n // 10)
    g = torch.Generator("cuda").manual_seed(n)
    a = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=g)
    h = a + a.T
    ref = torch.linalg.eigvalsh(h)[:k]
    out = egb.solve_ev(h, None, k, overlap_is_unit=True, band_width=b, precision=precision)
    ev, C = out["eval"][:k], out["C"]
    C = C if C.shape[0] == n else C.T
    norm = float(ref.abs().max())
    assert (ev - ref).abs().max() < (1e-13 + 20 * n * 2.2e-16) * norm
    assert (C.T @ C - torch.eye(k, dtype=torch.float64, device="cuda")).abs().max() < 1e-10
    assert (h @ C - C * ev).abs().max() < 1e-10 * norm
