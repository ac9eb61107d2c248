"""Back-transformation through Q2 as a pipeline over the sweep blocks: many column groups and blocks
under way at a time, column groups that end ragged, more columns than rows (binary32, progress words for
n columns at a time), and every number of lanes per column of the binary64 kernel (2, 4, 8 by size)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402
from test_gpu_q2 import _apply_ref, _lib, _reflectors  # noqa: E402


@pytest.mark.parametrize("n,b,k", [(3, 64, 3), (900, 64, 650), (700, 24, 700), (400, 16, 401), (130, 64, 600)])
def test_q2_binary32_units(n, b, k):
    lib = _lib()
    v2, tau, S = _reflectors(n, b, n + k)
    z0 = np.random.default_rng(n).standard_normal((n, k)).astype(np.float32)
    v32, t32 = v2.astype(np.float32), tau.astype(np.float32)
    ref = _apply_ref(n, b, v32.astype(np.float64), t32.astype(np.float64), S, z0.astype(np.float64))
    dv, dt = torch.from_numpy(v32).cuda().contiguous(), torch.from_numpy(t32).cuda()
    work = torch.full((lib.elsi_gb_q2_work(n, b) + 16,), 1e30, dtype=torch.float32, device="cuda")
    st = torch.zeros(8, dtype=torch.int32, device="cuda")
    outs = []
    for _ in range(2):  # the progress words are set up again for each call
        zt = torch.from_numpy(z0.T.copy()).cuda()
        rc = lib.elsi_gb_q2_apply_f32(n, b, dv.data_ptr(), dt.data_ptr(), k, zt.data_ptr(), n, work.data_ptr(),
                                      work.numel(), st.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert rc == 0 and int(st[0]) == 0
        outs.append(zt.cpu().numpy().T.astype(np.float64))
    assert np.array_equal(outs[0], outs[1])
    # three TF32 products per group keep about 2^-21 a group; 2e-5 is the bound of the single-CTA shapes
    assert np.linalg.norm(outs[0] - ref) / np.linalg.norm(ref) < 2e-5


@pytest.mark.parametrize("n,b,k", [(1500, 32, 1499), (900, 32, 850), (600, 32, 597), (1400, 64, 1400), (333, 64, 5)])
def test_q2_binary64_lanes(n, b, k):
    a = np.random.default_rng(n + b).standard_normal((n, n))
    h = a + a.T
    out = egb.solve_ev(torch.from_numpy(h).cuda(), None, k, overlap_is_unit=True, band_width=b)
    ev, C = out["eval"].cpu().numpy(), out["C"].cpu().numpy()
    norm = np.abs(ev).max()
    assert np.abs(C.T @ C - np.eye(k)).max() < 1e-10
    assert np.abs(h @ C - C * ev[:k]).max() < 1e-11 * norm
