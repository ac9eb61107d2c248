"""Chemical potential and occupations where the counts are at their limits: no electron, a hundredth of one,
all states full, next to levels far above and below, against the oracle's bisection."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("k", [1, 10, 40])
@pytest.mark.parametrize("fill", [0.0, 1e-2, 1.0, "half", "full"])
def test_fermi(k, fill):
    kt = 0.02
    eps = np.sort(np.random.default_rng(k).uniform(-2, 2, k))
    n_el = {"half": float(k), "full": 2.0 * k - 1e-3}.get(fill, fill)
    ref = oracle.occupation(eps, n_el, oracle.SCHEME_FERMI, kt)
    with egb.Handle(k, k, n_el) as hd:
        hd.use_current_stream()
        hd.set_overlap_is_unit(True)
        hd.set_broadening(egb.OCC_FERMI, kt)
        hd.dm_real(torch.from_numpy(np.diag(eps)).cuda())
        mu, f = hd.get_mu(), hd.get_occ().cpu().numpy()
    # the bisection stops at an accuracy of 1e-12 electrons, and the levels are good to 1e-15
    f_ref, mu_ref = ref[0], ref[1]
    assert abs(mu - mu_ref) < 1e-9
    assert np.abs(f - f_ref).max() < 1e-11
