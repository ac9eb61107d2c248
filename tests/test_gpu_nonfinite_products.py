"""Infinities and NaNs through the binary64 products that run as digit products: the product itself
against IEEE sums, the eigenpair adjoint and batched density matrices below and above the size
where the digit products begin."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ksinputs  # noqa: E402
import paper_1705_11191_gb300 as egb  # noqa: E402
from test_gpu_ozaki_wide import EPS, _wide  # noqa: E402


@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 1)])
@pytest.mark.parametrize("k,spare", [(3, 0), (200, 0), (1000, 1 << 22)])
def test_product(ta, tb, k, spare):
    rng = np.random.default_rng(k)
    m, n = 150, 70
    A, B, C = rng.standard_normal((m, k)), rng.standard_normal((k, n)), rng.standard_normal((m, n))
    A[3, 2], A[140, 0], A[17, k - 1], A[17, 0] = np.nan, np.inf, np.inf, -np.inf
    A[60, 1] = np.array([0xFFF8000000000000], dtype=np.uint64).view(np.float64)[0]  # of inf - inf
    B[1, 66], B[k - 1, 5], B[0, 9] = np.inf, -np.inf, 0.0  # A[140, 0] B[0, 9] is NaN
    got = _wide(ta, tb, np.asfortranarray(A.T if ta else A), np.asfortranarray(B.T if tb else B), C, -2.0, 0.5, 0, spare)
    with np.errstate(invalid="ignore"):
        ref = sum(-2.0 * A[:, [q]] * B[[q], :] for q in range(k)) + 0.5 * C
    finite = np.isfinite(ref)
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(got[np.isinf(ref)], ref[np.isinf(ref)])
    ok = np.isfinite(A).all(1)[:, None] & np.isfinite(B).all(0)[None, :]
    assert finite[ok].all()
    mag = np.abs(np.where(np.isfinite(A), A, 0)) @ np.abs(np.where(np.isfinite(B), B, 0))
    # one rounding per part of a divided K and the additions, against k of the reference
    assert (np.abs(got - ref)[ok] <= ((2 * k + 12) * EPS * (2 * mag + np.abs(C)))[ok]).all()


@pytest.mark.parametrize("n", [100, 600])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_eigenpair_adjoint_of_a_cotangent_that_is_not_finite(n, bad):
    rng = np.random.default_rng(n)
    C = torch.from_numpy(rng.standard_normal((n, n))).cuda()
    ev = torch.from_numpy(np.sort(rng.uniform(-1, 1, n))).cuda()
    g = torch.from_numpy(rng.standard_normal((n, n // 4))).cuda()
    g[3, 2] = bad
    with egb.Handle(n, n, 0.0) as hd:
        hd.use_current_stream()
        hb, sb = hd.ev_adjoint(ev, C, None, g)
    # column 2 of C^T G reaches every entry of both gradients
    assert not torch.isfinite(hb).any() and not torch.isfinite(sb).any()


@pytest.mark.parametrize("n", [100, 600])
def test_batched_density_of_an_occupation_that_is_not_finite(n):
    p = ksinputs.cluster_problem(n, seed=3)
    H, S = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (p.h, p.s))
    with egb.Handle(n, p.n_state, p.n_electron) as hd:
        hd.use_current_stream()
        hd.set_batch_autotune(False)
        hd.batch_ev([H], [S], [p.n_state])
        occ = torch.full((p.n_state,), 2.0, dtype=torch.float64, device="cuda")
        good = hd.batch_dm(occ)[0][0].clone()
        occ[1] = float("nan")
        bad = hd.batch_dm(occ)[0][0]
    assert torch.isfinite(good).all()
    assert torch.isnan(bad).all()
