"""Calls whose products are large enough for the digit products of the binary64 route, against the oracle
or extended sums: the eigenpair adjoint, batched density matrices, and the binary64 route with a
nearly singular overlap (its standard form is graded over six decades)."""
import numpy as np
import pytest

import ksinputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402

EPS = 2.0 ** -53


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n,k,with_ev", [(257, 60, True), (500, 500, False), (611, 37, True)])
def test_eigenpair_adjoint(n, k, with_ev):
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    ev = np.linspace(-1, 1, n)
    g, eb = rng.standard_normal((n, k)), rng.standard_normal(n) if with_ev else None
    ref = oracle.ev_adjoint(ev, q, eb, g)
    with egb.Handle(n, n, 0.0) as hd:
        hd.use_current_stream()
        got = hd.ev_adjoint(dev(ev), dev(q), None if eb is None else dev(eb), dev(g))
    for a, b in zip(got, ref):
        assert rel(a.cpu().numpy(), b) <= 1e-11


def test_batched_density_matrices():
    probs = [ksinputs.cluster_problem(n, seed=n) for n in (600, 431)]
    with egb.Handle(5, 5, 1.0) as hd:
        hd.use_current_stream()
        hd.set_batch_autotune(False)
        P, W, E, _ = hd.dm_batched([dev(p.h) for p in probs], [dev(p.s) for p in probs], [p.n_state for p in probs],
                                   [p.n_electron for p in probs], shared_mu=False)
    for p, a, b, e in zip(probs, P, W, E):
        ref = oracle.solve(p.h, p.s, p.n_state, p.n_electron)
        assert rel(a.cpu().numpy(), ref["P"]) <= 1e-9 and rel(b.cpu().numpy(), ref["W"]) <= 1e-9
        assert abs(e - ref["energy"]) <= 1e-9 * abs(ref["energy"])


def test_nearly_singular_overlap():
    p = ksinputs.cluster_problem(600, seed=37, tau=1e-6, force_tau=True)
    ref = oracle.solve(p.h, p.s, p.n_state, p.n_electron)
    out = egb.solve_dm(dev(p.h), dev(p.s), p.n_state, p.n_electron)
    # n roundings, amplified by 1 / lambda_min(S) on either side of the comparison
    assert rel(out["P"].cpu().numpy(), ref["P"]) <= 2 * 600 * EPS * 1e6
