"""The two-sided update as one digit product holds V (unit columns) and W (the size of H~) in the
same rows: eigenvalues of matrices far from unit norm, at an order where it runs."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402

EPS = 2.0 ** -53


@pytest.mark.parametrize("scale", [1e-40, 1e-12, 1e10, 1e25])
def test_eigenvalues_of_scaled_matrices(scale):
    n = 1500
    a = np.random.default_rng(n).standard_normal((n, n))
    h = (a + a.T) * scale
    ev = egb.solve_ev(torch.from_numpy(h).cuda(), None, n, overlap_is_unit=True)["eval"].cpu().numpy()
    ref = np.linalg.eigvalsh(h)
    # backward error of the reduction: 20 n roundings of ||H||
    np.testing.assert_allclose(ev, ref, rtol=0, atol=40 * n * EPS * np.abs(ref).max())

