"""Memory of a batch of one large and several small problems: one large workspace, whatever the number
of solver instances."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import ksinputs  # noqa: E402
import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("precision", [egb.PREC_FP64, egb.PREC_FP32_REFINE])
def test_one_large_and_several_small_problems(precision):
    probs = [ksinputs.cluster_problem(n, seed=20 + n) for n in (200, 2000, 150, 120)]
    hs, ss = ([torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in y] for y in zip(*[(p.h, p.s) for p in probs]))
    ks, nel = [p.n_state for p in probs], [p.n_electron for p in probs]

    def used(which, streams):
        torch.cuda.empty_cache()
        with egb.Handle(probs[1].n, probs[1].n_state, probs[1].n_electron) as hd:
            hd.use_current_stream()
            hd.set_precision(precision)
            hd.set_batch_autotune(False)
            hd.set_batch_streams(streams)
            free = torch.cuda.mem_get_info()[0]
            out = hd.dm_batched([hs[i] for i in which], [ss[i] for i in which], [ks[i] for i in which],
                                [nel[i] for i in which], shared_mu=False)
            del out
            torch.cuda.empty_cache()
            return free - torch.cuda.mem_get_info()[0]

    used([1], 1)  # what the context itself takes on a first call
    alone, together = used([1], 1), used([0, 1, 2, 3], 4)
    assert together < 1.6 * alone


def test_band_width_goes_by_the_order_of_the_problem():
    """... and not by that of the handle, which solves none of its own here."""
    n = 2999  # a size class that no other test tunes
    a = torch.randn(n, n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    with egb.Handle(25000, 10, 10.0) as hd:
        hd.use_current_stream()
        hd.set_overlap_is_unit(True)
        hd.set_batch_autotune(False)
        hd.batch_ev([a + a.T], None, [10])
        assert hd.batch_tuning(n)[0] == 32
