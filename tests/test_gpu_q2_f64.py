"""The pipelined binary64 back-transformation through Q2: every band width it is built for, one
and several pipeline rounds (8 blocks of 64 sweeps), a last round with fewer blocks, ragged
column groups of four, against LAPACK on matrices that need every stage."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("n,b,k", [(3, 8, 3), (66, 8, 5), (67, 64, 67), (130, 24, 6), (200, 40, 9), (515, 48, 30),
                                   (580, 56, 17), (600, 16, 13), (1100, 32, 21), (1300, 64, 11)])
def test_q2_binary64(n, b, k):
    a = np.random.default_rng(n + b).standard_normal((n, n))
    h = a + a.T
    ref = np.linalg.eigvalsh(h)
    norm = np.abs(ref).max()
    out = egb.solve_ev(torch.from_numpy(h).cuda(), None, k, overlap_is_unit=True, band_width=b)
    ev, C = out["eval"].cpu().numpy(), out["C"].cpu().numpy()
    np.testing.assert_allclose(ev, ref, rtol=0, atol=(1e-13 + 20 * n * 2.2e-16) * norm)
    assert np.abs(C.T @ C - np.eye(k)).max() < 1e-10
    assert np.abs(h @ C - C * ev[:k]).max() < 1e-11 * norm
