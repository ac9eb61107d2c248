"""Binary64 panels with more rows than one launch takes with two columns a lane (38 656 on 152 SMs): with
one column a lane and 512 rows a CTA up to 32 columns, as two panels above. Also on few SMs, where short
panels take the same forms."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402

EPS = 2.0 ** -53


def run(m, b, sms):
    lib, v, i = egb.load(), ctypes.c_void_p, ctypes.c_int
    lib.elsi_gb_panel_qr_f64_work.argtypes = [i]
    lib.elsi_gb_panel_qr_f64_work.restype = ctypes.c_size_t
    lib.elsi_gb_panel_qr_f64.argtypes = [i, i, v, i, v, i, v, i, i, v, ctypes.c_size_t, v, v]
    if m > 1000 and torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the limits are those of 152 SMs")
    P0 = torch.randn(b, m, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(m + b))
    P = P0.clone()
    V, T = torch.full_like(P, 7.0), torch.full((b, b), 7.0, dtype=torch.float64, device="cuda")
    words = lib.elsi_gb_panel_qr_f64_work(m)
    work = torch.empty(words, dtype=torch.int64, device="cuda")
    st = torch.zeros(8, dtype=torch.int32, device="cuda")
    rc = lib.elsi_gb_panel_qr_f64(m, b, P.data_ptr(), m, V.data_ptr(), m, T.data_ptr(), b, sms, work.data_ptr(), words,
                                  st.data_ptr(), None)
    torch.cuda.synchronize()
    return rc, int(st[0]), P0, P, V, T


@pytest.mark.parametrize("m,b,sms", [(513, 33, 2), (77344, 40, 152)])
def test_more_rows_than_fit(m, b, sms):
    assert run(m, b, sms)[0] == 7  # ELSI_ERR_CUDA: invalid configuration


@pytest.mark.parametrize("m,b,sms", [(700, 64, 3), (512, 33, 2), (700, 40, 3), (512, 40, 2), (1000, 32, 3),
                                     (38656, 64, 152), (38657, 64, 152), (40001, 40, 152), (60000, 56, 152),
                                     (38657, 32, 152), (77312, 32, 152), (77312, 8, 152), (77312, 40, 152)])
def test_tall_panel(m, b, sms):
    rc, status, P0, P, V, T = run(m, b, sms)
    assert rc == 0 and status == 0
    P0, P, V, T = P0.t(), P.t(), V.t(), T.t()
    R, Vt = torch.triu(P[:b]), torch.tril(V[:b], -1)
    assert torch.equal(torch.tril(P[:b], -1), Vt) and torch.equal(P[b:], V[b:])
    assert torch.equal(torch.diagonal(V[:b]), torch.ones(b, dtype=torch.float64, device="cuda"))
    assert not torch.triu(V[:b], 1).any() and not torch.tril(T, -1).any()
    # Q R = P0, column by column, and T + T^T = T V^T V T^T: a few roundings for each of the b reflectors
    QR = torch.zeros_like(P0)
    QR[:b] = R
    QR -= V @ (T @ (V[:b].t() @ R))
    assert torch.linalg.norm(QR - P0) <= 20 * b * EPS * torch.linalg.norm(P0)
    G = V.t() @ V
    assert torch.linalg.norm(T + T.t() - T @ G @ T.t()) <= 20 * b * EPS * torch.linalg.norm(T) * max(1.0, float(torch.linalg.norm(T)))
