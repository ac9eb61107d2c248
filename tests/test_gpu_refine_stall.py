"""Refinement that stalls: a graded matrix, whose spectrum ends in hundreds of eigenvalues that the binary32
route cannot tell apart. The corrections of the lowest states stay near 5e-9 there instead of
converging, below the size that used to be taken for convergence, with P off by as much."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("n,k,digits", [(636, 12, 9.0), (400, 10, 6.0), (900, 30, 11.0)])
@pytest.mark.parametrize("seed", [0, 1])
def test_graded_matrix(n, k, digits, seed):
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((n, n))
    d = np.logspace(0, -digits, n)
    h = (a + a.T) / np.sqrt(2 * n) * d[:, None] * d
    w, c = np.linalg.eigh(h)
    ref = 2 * c[:, :k] @ c[:, :k].T
    P = egb.solve_dm(torch.from_numpy(h).cuda(), torch.from_numpy(np.eye(n)).cuda(), k, 2.0 * k,
                     precision=egb.PREC_FP32_REFINE)["P"].cpu().numpy()
    # the bound of the binary32 route's density matrices, or what the gap leaves of 64 bits
    assert np.linalg.norm(P - ref) <= max(1e-9, 1e-14 / (w[k] - w[k - 1])) * np.linalg.norm(ref)
