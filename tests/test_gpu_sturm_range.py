"""Bisection counts of tridiagonals of any scale: the minors of the Sturm recurrence gain or lose the
bits of ||T|| with every step, so their rescaling has to hold at both ends. Binary64 route, all
eigenvalues, orders below and above one piece of the count and with a ragged last piece."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402

EPS = 2.0 ** -53


@pytest.mark.parametrize("n,scale", [(n, s) for n in (7, 100, 403)
                                     for s in (1e-40, 1e-12, 1.4e-9, 1e-8, 1.0, 7e7, 1e8, 1e10, 1e25)]
                         + [(1500, s) for s in (1.4e-9, 1e-8, 1.0, 7e7, 1e8)])
def test_eigenvalues_of_scaled_matrices(n, scale):
    a = np.random.default_rng(n).standard_normal((n, n))
    h = (a + a.T) * scale
    ev = egb.solve_ev(torch.from_numpy(h).cuda(), None, n, overlap_is_unit=True)["eval"].cpu().numpy()
    ref = np.linalg.eigvalsh(h)
    # backward error of the reduction: 20 n roundings of ||H||
    np.testing.assert_allclose(ev, ref, rtol=0, atol=40 * n * EPS * np.abs(ref).max())


def test_eigenvalues_of_a_graded_standard_form():
    """A diagonal overlap with entries 2^-30: H~ is formed exactly, ||H~|| is 2^30 ||H|| on a fifth of
    the basis and most of the spectrum is far below it."""
    n = 500
    d = np.ones(n)
    d[::5] = 2.0 ** -15
    a = np.random.default_rng(9).standard_normal((n, n)) / np.sqrt(n)
    h = a + a.T
    ev = egb.solve_ev(torch.from_numpy(h).cuda(), torch.from_numpy(np.diag(d * d)).cuda(), n)["eval"].cpu().numpy()
    ref = np.linalg.eigvalsh(h / d[:, None] / d[None, :])
    np.testing.assert_allclose(ev, ref, rtol=0, atol=40 * n * EPS * np.abs(ref).max())
