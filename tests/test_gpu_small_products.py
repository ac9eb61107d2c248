"""Shapes at which a product changes kernel: the small-tile SIMT kernels (binary32 and binary64),
their tile remainders, the in-place product with a diagonal block's inverse, and the sizes just
around the tensor-core limits, through density matrices of problems of those orders (the
Cholesky factor, both triangular solves and the back-substitution) against LAPACK."""
import numpy as np
import pytest

import ksinputs

torch = pytest.importorskip("torch")
sla = pytest.importorskip("scipy.linalg")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("prec,tol", [(egb.PREC_FP64, 1e-11), (egb.PREC_FP32_REFINE, 1e-9)])
@pytest.mark.parametrize("n", [5, 63, 64, 65, 127, 129, 191, 255, 256, 257, 320, 449, 513, 705])
def test_orders_around_block_edges(n, prec, tol):
    p = ksinputs.cluster_problem(n, seed=60 + n)
    k = p.n_state
    w, v = sla.eigh(p.h, p.s)
    if k < n and w[k] - w[k - 1] < 1e-4:
        pytest.skip("no gap above the occupied states")
    c = v[:, :k]
    f = np.clip(p.n_electron - 2.0 * np.arange(k), 0.0, 2.0)
    ref = (c * f) @ c.T
    with egb.Handle(n, k, p.n_electron) as hd:
        hd.use_current_stream()
        hd.set_precision(prec)
        P, e = hd.dm_real(torch.from_numpy(np.ascontiguousarray(p.h)).cuda(),
                          torch.from_numpy(np.ascontiguousarray(p.s)).cuda())
    assert np.linalg.norm(P.cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
    assert abs(e - (f * w[:k]).sum()) <= 1e-10 * max(1.0, abs(e))
