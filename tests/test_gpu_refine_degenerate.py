"""Refinement of degenerate states beyond its clusters of 32, whose Rayleigh quotients agree to the last bit
across the end of a cluster piece: wanted states next to guard columns of the same eigenvalue (zero),
and more than 32 wanted ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("lam,k", [(np.zeros(100), 30), (np.zeros(100), 100), (np.repeat([-1.0, 0.0, 1.0], 40), 40),
                                   (np.repeat([-1.0, 0.0, 1.0], 40), 20),
                                   (np.concatenate([np.full(40, -1.0), np.linspace(0, 1, 160)]), 40)],
                         ids=["zero_30", "zero_all", "three_40", "three_20", "singles"])
def test_projector(lam, k):
    n = len(lam)
    h = np.diag(lam)
    with egb.Handle(n, k, 2.0 * k) as hd:
        hd.use_current_stream()
        hd.set_precision(egb.PREC_FP32_REFINE)
        P, e = hd.dm_real(torch.from_numpy(h).cuda(), torch.from_numpy(np.eye(n)).cuda())
    P = P.cpu().numpy()
    # the bound of the density matrices of the binary32 route
    assert np.linalg.norm(P @ P - 2 * P) <= 1e-9 * np.sqrt(n) and abs(np.trace(P) - 2 * k) <= 1e-9 * n
    assert abs(e - 2 * lam[:k].sum()) <= 1e-9 * n and abs((P * h).sum() - e) <= 1e-9 * n
