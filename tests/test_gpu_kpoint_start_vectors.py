"""Start vectors of the refinement for complex k-points: a last bisection interval that is too
wide leaves vectors of close eigenvalues far from orthogonal, and the refinement ends at its
iteration limit and is repeated in binary64."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ksinputs  # noqa: E402
import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("index,band", [(8, 64), (43, 64), (12, 32)])
def test_kpoint_refines_without_fallback(index, band):
    n, kt = 2048, 0.01
    _, h, s, _ = list(ksinputs.kpoint_set(n, grid=4, seed=3, device="cuda"))[index]
    with egb.Handle(n, 640, 512.0) as handle:
        handle.use_current_stream()
        handle.set_precision(1)
        handle.set_broadening(egb.OCC_FERMI, kt)
        handle.set_band_width(band)
        p, _ = handle.dm_complex(h, s)
        assert handle.refine_info()[0] >= 0
    # the refinement is accepted at a defect of 1e-10 a state: Tr(P S) is off by 1e-10 of the electrons at most
    electrons = torch.einsum("ij,ji->", p, s.to(p.dtype)).real.item()
    assert abs(electrons - 512.0) < 512.0 * 1e-10
