"""k-point problems in their real form, where every state is a pair and the second vector of a pair is
regenerated: in the binary32 route it is accepted at the rounding of binary32, since it is refined."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ksinputs  # noqa: E402
import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("band", [64])
def test_all_kpoints_of_a_grid(band):
    n, k, kt = 2048, 640, 0.01
    kset = ksinputs.kpoint_set(n, grid=4, seed=3, device="cuda")
    nel = float(n // 4)
    with egb.Handle(n, k, nel) as hd:
        hd.use_current_stream()
        hd.set_precision(egb.PREC_FP32_REFINE)
        hd.set_broadening(egb.OCC_FERMI, kt)
        hd.set_band_width(band)
        hd.set_batch_autotune(False)
        P, _, E, mu = hd.dm_batched([h.t().contiguous() for _, h, _, _ in kset], [s.t().contiguous() for _, _, s, _ in kset],
                                    [k] * len(kset), nel, weights=[1.0 / len(kset)] * len(kset), shared_mu=True,
                                    inputs_colmajor=True)
    for (_, h, s, _), p, e in zip(kset, P, E):
        # Tr(P H) is the band energy, and sum of Tr(P S) the electrons
        assert abs(float(torch.einsum("ij,ji->", p, h).real) - e) <= 1e-9 * n
    count = sum(float(torch.einsum("ij,ji->", p, s).real) for (_, _, s, _), p in zip(kset, P)) / len(kset)
    assert abs(count - nel) <= 1e-9 * nel
