"""Basis functions scaled by powers of two, diag(S) over up to 24 decimals: every operation of the
binary64 route scales with them exactly, so D P D of the scaled problem is P of the plain one up to
what the digit products leave out (2^-64 of the largest entries of a row and a column: 1e-15 with
n terms and the condition of S), and likewise for the eigenpair adjoint."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ksinputs  # noqa: E402
import paper_1705_11191_gb300 as egb  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def scaling(n, decades):
    """Powers of two with squares over that many decades."""
    return np.ldexp(1.0, np.round(np.random.default_rng(1).uniform(-0.5, 0.5, n) * decades / 2 * np.log2(10)).astype(int))


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n", [250, 601, 1000])
@pytest.mark.parametrize("decades", [12, 24])
def test_density_matrices(n, decades):
    p = ksinputs.cluster_problem(n, seed=5)
    d = scaling(n, decades)
    out = egb.solve_dm(dev(p.h), dev(p.s), p.n_state, p.n_electron)
    sc = egb.solve_dm(dev(p.h * d[:, None] * d), dev(p.s * d[:, None] * d), p.n_state, p.n_electron)
    for key in ("P", "W"):
        assert rel(sc[key].cpu().numpy() * d[:, None] * d, out[key].cpu().numpy()) < 1e-14


@pytest.mark.parametrize("n,k", [(600, 150), (601, 601)])
def test_eigenpair_adjoint(n, k):
    rng = np.random.default_rng(n)
    ev, C, g = np.sort(rng.uniform(-1, 1, n)), rng.standard_normal((n, n)), rng.standard_normal((n, k))
    d = scaling(n, 24)
    with egb.Handle(n, n, 0.0) as hd:
        hd.use_current_stream()
        ref = hd.ev_adjoint(dev(ev), dev(C), None, dev(g))
        got = hd.ev_adjoint(dev(ev), dev(C / d[:, None]), None, dev(g * d[:, None]))
    for a, b in zip(got, ref):
        assert rel(a.cpu().numpy() * d[:, None] * d, b.cpu().numpy()) < 1e-13
