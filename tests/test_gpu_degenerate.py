"""States of a degeneracy beyond the clusters of the refinement (32) and the pieces of the tridiagonal solver
(64), exact and up to rounding, with the wanted states ending at, inside or below a degenerate group:
P is a projector of the right trace and energy in both routes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402

SPECTRA = {"three": np.repeat([-1.0, 0.0, 1.0], 40), "zero": np.zeros(100), "one_and_singles": np.concatenate([np.full(40, -1.0), np.linspace(0, 1, 160)]),
           "long": np.concatenate([np.full(70, -1.0), np.linspace(0, 1, 330)]), "pairs": np.repeat(np.linspace(-1, 1, 100), 2)}


@pytest.mark.parametrize("precision", [egb.PREC_FP64, egb.PREC_FP32_REFINE])
@pytest.mark.parametrize("rotated", [False, True])
@pytest.mark.parametrize("name,k", [("three", 40), ("three", 20), ("three", 60), ("zero", 30), ("zero", 100), ("one_and_singles", 40),
                                    ("one_and_singles", 41), ("long", 70), ("long", 30), ("pairs", 50)])
def test_projector(name, k, rotated, precision):
    lam = SPECTRA[name]
    n = len(lam)
    h = np.diag(lam)
    if rotated:
        q, _ = np.linalg.qr(np.random.default_rng(n).standard_normal((n, n)))
        h = (q * lam) @ q.T
        h = 0.5 * (h + h.T)
    with egb.Handle(n, k, 2.0 * k) as hd:
        hd.use_current_stream()
        hd.set_precision(precision)
        P, e = hd.dm_real(torch.from_numpy(h).cuda(), torch.from_numpy(np.eye(n)).cuda())
    P = P.cpu().numpy()
    assert np.isfinite(P).all()
    # the bound of the density matrices of the two routes
    assert np.linalg.norm(P @ P - 2 * P) <= 1e-9 * np.sqrt(n) and abs(np.trace(P) - 2 * k) <= 1e-9 * n
    assert abs(e - 2 * lam[:k].sum()) <= 1e-9 * n and abs((P * h).sum() - e) <= 1e-9 * n
