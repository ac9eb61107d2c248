"""The update factors w = tau (P_j + scl d) of a binary32 panel: the sums d over all CTAs are kept to twice
the working precision and w is rounded once. Integer columns (every partial sum is exact) under a
first row of full significands, so that row 0 of R is known to the last bit: P_0 - fl(w)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


@pytest.mark.parametrize("m,b", [(300, 8), (300, 32), (1000, 64), (5000, 40), (9000, 64)])
def test_first_row_of_r(m, b):
    lib, v, i = egb.load(), ctypes.c_void_p, ctypes.c_int
    lib.elsi_gb_panel_qr_f32_work.argtypes = [i]
    lib.elsi_gb_panel_qr_f32_work.restype = ctypes.c_size_t
    lib.elsi_gb_panel_qr_f32.argtypes = [i, i, v, i, v, i, v, i, i, v, ctypes.c_size_t, v, v]
    words = lib.elsi_gb_panel_qr_f32_work(m)
    work = torch.empty(words, dtype=torch.int64, device="cuda")
    st = torch.zeros(8, dtype=torch.int32, device="cuda")
    for seed in range(8):
        rng = np.random.default_rng(seed)
        A = rng.integers(-60, 61, (m, b)).astype(np.float32)
        A[:, 0] = rng.integers(-4, 5, m)
        A[1, 0] = 8.0  # v = 8 scl there: scl is read off exactly
        A[0] = rng.standard_normal(b)
        d = A[1:, 0].astype(np.float64) @ A[1:].astype(np.float64)  # sums below 2^24
        P = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()
        V, T = torch.empty_like(P), torch.empty((b, b), dtype=torch.float32, device="cuda")
        rc = lib.elsi_gb_panel_qr_f32(m, b, P.data_ptr(), m, V.data_ptr(), m, T.data_ptr(), b, 152, work.data_ptr(), words,
                                      st.data_ptr(), None)
        torch.cuda.synchronize()
        assert rc == 0 and int(st[0]) == 0
        tau, scl = float(T[0, 0]), float(V[0, 1]) / 8.0
        w = (tau * (A[0].astype(np.float64) + scl * d)).astype(np.float32)
        assert np.array_equal(P[:, 0].cpu().numpy()[1:], (A[0] - w)[1:])
