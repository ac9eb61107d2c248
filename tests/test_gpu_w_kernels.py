"""W of the two-sided update in binary64 on both sides of 8176 rows, where its 16-row blocks pass 512 (the
scratch for their partial products grows from there on), of unit and of large norm."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("n,b,scale", [(8128, 64, 1.0), (8512, 64, 1.0), (8512, 32, 2.0 ** 40)])
def test_lowest_states(n, b, scale):
    k = 12
    g = torch.Generator("cuda").manual_seed(n)
    u = torch.randn(n, 40, dtype=torch.float64, device="cuda", generator=g) / n ** 0.5
    h = (u * torch.linspace(-8, -1, 40, dtype=torch.float64, device="cuda")) @ u.t()
    h = 0.5 * (h + h.t())
    h.diagonal().add_(torch.linspace(0, 1, n, dtype=torch.float64, device="cuda"))
    h *= scale
    with egb.Handle(n, k, 0.0) as hd:
        hd.use_current_stream()
        hd.set_overlap_is_unit(True)
        hd.set_band_width(b)
        ev, C = hd.ev_real(h)
    tol = 9 * n * 2.0 ** -53 * 4  # n roundings of ||H|| <= 9
    assert (h @ C - C * ev[:k]).abs().max() < tol * scale
    assert (C.t() @ C - torch.eye(k, dtype=torch.float64, device="cuda")).abs().max() < tol
