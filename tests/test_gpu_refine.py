"""GPU parity of the FP32 reduction + refinement route against the FP64 CPU oracle.

Tolerances: the refined result must meet the same bar as the binary64 route:
eigenvalues of the wanted states within 1e-10 * max(1, |eps|max), P and W within 1e-9
relative Frobenius error, the band energy within 1e-9 relative, and the final
S-orthonormality defect max|X^T S X - I| <= 1e-12.
"""
import numpy as np
import pytest

import ksinputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n,seed,b", [(64, 31, 16), (150, 32, 32), (257, 33, 64), (400, 34, 32)])
def test_refined_dm_matches_oracle(n, seed, b):
    p = ksinputs.cluster_problem(n, seed=seed)
    ref = oracle.solve(p.h, p.s, p.n_state, p.n_electron)
    with egb.Handle(p.n, p.n_state, p.n_electron) as hd:
        hd.use_current_stream()
        hd.set_precision(egb.PREC_FP32_REFINE)
        hd.set_band_width(b)
        P, e = hd.dm_real(dev(p.h), dev(p.s))
        W = hd.get_edm()
        iters, orth = hd.refine_info()
    assert rel(P.cpu().numpy(), ref["P"]) <= 1e-9
    assert rel(W.cpu().numpy(), ref["W"]) <= 1e-9
    assert abs(e - ref["energy"]) <= 1e-9 * abs(ref["energy"])
    assert orth <= 1e-11
    assert 1 <= iters <= 8


@pytest.mark.parametrize("n,seed", [(200, 35), (333, 36)])
def test_refined_ev_matches_oracle(n, seed):
    p = ksinputs.cluster_problem(n, seed=seed)
    k = p.n_state
    ref = oracle.solve(p.h, p.s, k, p.n_electron, want_pw=False)
    out = egb.solve_ev(dev(p.h), dev(p.s), k, precision=egb.PREC_FP32_REFINE, band_width=32)
    ev = out["eval"].cpu().numpy()
    C = out["C"].cpu().numpy()
    np.testing.assert_allclose(ev[:k], ref["eval"][:k], rtol=0, atol=1e-10)
    # the rest come from the binary32 route
    np.testing.assert_allclose(ev[k:], ref["eval"][k:], rtol=0, atol=1e-4)
    np.testing.assert_allclose(C.T @ p.s @ C, np.eye(k), atol=1e-12)
    r = p.h @ C - (p.s @ C) * ev[None, :k]
    assert np.abs(r).max() < 1e-9


@pytest.mark.parametrize("tau", [1e-2, 1e-4, 1e-6])
def test_overlap_conditioning_sweep(tau):
    """lambda_min(S) in {1e-2, 1e-4, 1e-6}: the refined route against the oracle. At
    lambda_min = 1e-6 the binary64 floor itself is about kappa(S) eps ~ 1e-10, so P is
    only required within 1e-8 there."""
    p = ksinputs.cluster_problem(300, seed=37, tau=tau, force_tau=True)
    assert abs(p.lambda_min_s - tau) < 1e-3 * tau + 1e-12
    ref = oracle.solve(p.h, p.s, p.n_state, p.n_electron)
    with egb.Handle(p.n, p.n_state, p.n_electron) as hd:
        hd.use_current_stream()
        hd.set_precision(egb.PREC_FP32_REFINE)
        hd.set_band_width(32)
        P, e = hd.dm_real(dev(p.h), dev(p.s))
    tol = 1e-9 if tau >= 1e-4 else 1e-8
    assert rel(P.cpu().numpy(), ref["P"]) <= tol


def test_refined_route_not_pd_then_reuse():
    """S not positive definite: the binary32 factorisation fails, the binary64 one fails at
    the same pivot, and the error names it; the handle then solves a valid problem."""
    p = ksinputs.cluster_problem(64, seed=24)
    s = p.s.copy()
    s[40, 40] = -1.0
    ref = oracle.solve(p.h, p.s, p.n_state, p.n_electron)
    with egb.Handle(p.n, p.n_state, p.n_electron) as hd:
        hd.use_current_stream()
        hd.set_precision(egb.PREC_FP32_REFINE)
        hd.set_band_width(16)
        with pytest.raises(egb.ElsiError) as e:
            hd.dm_real(dev(p.h), dev(s))
        assert e.value.code == 3 and "pivot 40" in str(e.value)
        P, _ = hd.dm_real(dev(p.h), dev(p.s))
    assert rel(P.cpu().numpy(), ref["P"]) <= 1e-9


def test_refined_route_nonfinite_hamiltonian():
    p = ksinputs.cluster_problem(64, seed=25)
    h = p.h.copy()
    h[3, 7] = np.nan
    with egb.Handle(p.n, p.n_state, p.n_electron) as hd:
        hd.use_current_stream()
        hd.set_precision(egb.PREC_FP32_REFINE)
        hd.set_band_width(16)
        with pytest.raises(egb.ElsiError) as e:
            hd.dm_real(dev(h), dev(p.s))
    assert e.value.code == 4


def test_binary64_cholesky_fallback_nearly_dependent_pair():
    """Two basis functions i, j with overlap c = 1 - 2e-8 (lambda_min(S) = 2e-8) and no
    overlap or coupling with the rest, H on the pair = h0 S on the pair (both of its
    eigenvalues h0, above the whole spectrum of the rest). c rounds to 1 in binary32, so
    the binary32 Cholesky meets a zero pivot at the later of i, j and the route factors S
    in binary64; its binary32 standard form is still wrong on the pair by O(h0), so the
    refinement must not return the pair's state among the wanted ones. P must equal the
    oracle's (the pair is unoccupied and decoupled, so P is that of the rest)."""
    sla = pytest.importorskip("scipy.linalg")
    base = ksinputs.cluster_problem(198, seed=38)
    h0 = float(sla.eigh(base.h, base.s, eigvals_only=True)[-1]) + 1.0
    n, i, j = 200, 17, 150
    c = 1.0 - 2e-8
    assert np.float32(c) == np.float32(1.0)
    rest = [q for q in range(n) if q not in (i, j)]
    H = np.zeros((n, n))
    S = np.zeros((n, n))
    H[np.ix_(rest, rest)] = base.h
    S[np.ix_(rest, rest)] = base.s
    S[i, i] = S[j, j] = 1.0
    S[i, j] = S[j, i] = c
    H[i, i] = H[j, j] = h0
    H[i, j] = H[j, i] = h0 * c
    ref = oracle.solve(H, S, base.n_state, base.n_electron)
    ref_rest = oracle.solve(base.h, base.s, base.n_state, base.n_electron)
    # the oracle itself: P vanishes on the pair and equals the smaller problem's elsewhere
    assert np.abs(ref["P"][[i, j], :]).max() < 1e-9
    assert rel(ref["P"][np.ix_(rest, rest)], ref_rest["P"]) < 1e-8
    with egb.Handle(n, base.n_state, base.n_electron) as hd:
        hd.use_current_stream()
        hd.set_precision(egb.PREC_FP32_REFINE)
        hd.set_band_width(32)
        P, e = hd.dm_real(dev(H), dev(S))
        iters, _ = hd.refine_info()
    assert rel(P.cpu().numpy(), ref["P"]) <= 1e-7
    assert abs(e - ref["energy"]) <= 1e-7 * abs(ref["energy"])
    assert iters == -1 or iters >= 1


@pytest.mark.parametrize("gap", [1e-3, 1e-5, 1e-7])
def test_small_gap_above_the_wanted_states(gap):
    """The k-th and (k+1)-th eigenvalues 'gap' apart, below the error of the binary32 route for
    the smallest: the wanted states are the lowest k, without a binary64 repeat (the guard
    columns keep the edge of the refined block away from the wanted states)."""
    n, k = 400, 50
    rng = np.random.default_rng(11)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lam = np.sort(rng.uniform(-4.0, 6.0, n))
    lam[k] = lam[k - 1] + gap
    lam = np.sort(lam)
    h = (q * lam) @ q.T
    h = 0.5 * (h + h.T)
    ref = np.linalg.eigvalsh(h)
    with egb.Handle(n, k, 0.0) as hd:
        hd.use_current_stream()
        hd.set_overlap_is_unit(True)
        hd.set_precision(egb.PREC_FP32_REFINE)
        ev, C = hd.ev_real(dev(h))
        iters, orth = hd.refine_info()
    C = C.cpu().numpy()
    assert iters > 0 and orth < 1e-10
    # eigenvalues are accurate to second order in the vectors' error, and to eps ||H||
    np.testing.assert_allclose(ev.cpu().numpy()[:k], ref[:k], rtol=0, atol=1e-12)
    assert np.abs(h @ C - C * ref[:k]).max() < 1e-10
