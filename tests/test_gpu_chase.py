"""The bulge chase with the band held on chip (b = 32, 64): orders around its edges (one
position, one row in the last position, several positions), both precision routes, against
LAPACK and against the general chase kernel (another band width of the same problem)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402

SIZES = [(3, 32), (4, 64), (33, 32), (34, 32), (35, 32), (65, 64), (66, 64), (67, 64), (97, 32),
         (130, 64), (193, 64), (260, 32), (451, 64)]


def _matrix(n):
    a = np.random.default_rng(n).standard_normal((n, n))
    return a + a.T


@pytest.mark.parametrize("n,b", SIZES)
def test_resident_chase_binary64(n, b):
    h = _matrix(n)
    ref = np.linalg.eigvalsh(h)
    norm = np.abs(ref).max()
    out = egb.solve_ev(torch.from_numpy(h).cuda(), None, n, overlap_is_unit=True, band_width=b)
    ev, C = out["eval"].cpu().numpy(), out["C"].cpu().numpy()
    # bisection to 1e-13 ||T||, backward error of the reductions a few n eps ||H||
    tol = (1e-13 + 20 * n * 2.2e-16) * norm
    np.testing.assert_allclose(ev, ref, rtol=0, atol=tol)
    assert np.abs(C.T @ C - np.eye(n)).max() < 1e-10
    assert np.abs(h @ C - C * ev).max() < 1e-11 * norm
    gen = egb.solve_ev(torch.from_numpy(h).cuda(), None, n, overlap_is_unit=True, band_width=24)
    np.testing.assert_allclose(ev, gen["eval"].cpu().numpy(), rtol=0, atol=2 * tol)


@pytest.mark.parametrize("n,b", [(4, 32), (67, 64), (97, 32), (451, 64)])
def test_resident_chase_refined(n, b):
    h = _matrix(n)
    k = max(1, n // 4)
    ref = np.linalg.eigvalsh(h)
    out = egb.solve_ev(torch.from_numpy(h).cuda(), None, k, overlap_is_unit=True, band_width=b,
                       precision=egb.PREC_FP32_REFINE)
    np.testing.assert_allclose(out["eval"].cpu().numpy()[:k], ref[:k], rtol=0,
                               atol=1e-11 * np.abs(ref).max())


def test_resident_chase_wait_expires_then_recovers():
    lib = egb.load()
    h = torch.from_numpy(_matrix(100)).cuda()
    with egb.Handle(100, 100, 0.0) as hd:
        hd.use_current_stream()
        hd.set_overlap_is_unit(True)
        hd.set_band_width(32)
        limit = lib.elsi_gb_get_spin_limit()
        assert lib.elsi_gb_set_spin_limit(0) == 0
        try:
            with pytest.raises(egb.ElsiError) as e:
                hd.ev_real(h)
        finally:
            assert lib.elsi_gb_set_spin_limit(limit) == 0
        assert e.value.code == 6
        ev, _ = hd.ev_real(h)
    ref = np.linalg.eigvalsh(h.cpu().numpy())
    np.testing.assert_allclose(ev.cpu().numpy(), ref, rtol=0, atol=1e-12 * np.abs(ref).max())
