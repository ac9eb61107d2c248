"""The wide digit product of the binary64 route (eight 9-bit digits, 128-bit sums) against
products in extended precision, at ragged sizes around its 128 x 64 tiles and 64-long k-tiles,
with and without room to divide K over CTAs, and on graded operands, where its error must stay
at the level of a binary64 product sum by sum and not of the row's largest entry."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402

EPS = 2.0 ** -53


def _wide(ta, tb, A, B, C, alpha, beta, uplo, spare=0):
    lib, v = egb.load(), ctypes.c_void_p
    lib.elsi_gb_gemm_f64_wide_planes.argtypes = [ctypes.c_int] * 3
    lib.elsi_gb_gemm_f64_wide_planes.restype = ctypes.c_size_t
    lib.elsi_gb_gemm_f64_digits_exps.argtypes = [ctypes.c_int] * 2
    lib.elsi_gb_gemm_f64_digits_exps.restype = ctypes.c_size_t
    lib.elsi_gb_gemm_f64_wide.argtypes = (
        [ctypes.c_int] * 5 + [ctypes.c_double, v, ctypes.c_int, v, ctypes.c_int, ctypes.c_double, v, ctypes.c_int,
                              ctypes.c_int, v, ctypes.c_size_t, v, ctypes.c_size_t, v, v])
    m = A.shape[1] if ta else A.shape[0]
    k = A.shape[0] if ta else A.shape[1]
    n = B.shape[0] if tb else B.shape[1]
    dA, dB, dC = (torch.from_numpy(np.ascontiguousarray(x.T)).cuda() for x in (A, B, C))
    planes = torch.zeros(lib.elsi_gb_gemm_f64_wide_planes(m, n, k) + 8 + spare, dtype=torch.bfloat16, device="cuda")
    exps = torch.zeros(lib.elsi_gb_gemm_f64_digits_exps(m, n), dtype=torch.int32, device="cuda")
    st = torch.zeros(8, dtype=torch.int32, device="cuda")
    rc = lib.elsi_gb_gemm_f64_wide(ta, tb, m, n, k, alpha, dA.data_ptr(), A.shape[0], dB.data_ptr(), B.shape[0],
                                   beta, dC.data_ptr(), m, uplo, planes.data_ptr(), planes.numel(), exps.data_ptr(),
                                   exps.numel(), st.data_ptr(), None)
    torch.cuda.synchronize()
    assert rc == 0 and int(st[0]) == 0
    return dC.cpu().numpy().T


@pytest.mark.parametrize("ta,tb,m,n,k", [(0, 0, 1, 1, 1), (0, 1, 128, 64, 64), (1, 0, 129, 65, 65), (0, 0, 200, 63, 17),
                                         (1, 1, 70, 130, 200), (0, 1, 127, 127, 1000)])
@pytest.mark.parametrize("spare", [0, 1 << 22])
def test_wide_product(ta, tb, m, n, k, spare):
    rng = np.random.default_rng(m + 3 * n + k)
    A = rng.standard_normal((k, m) if ta else (m, k))
    B = rng.standard_normal((n, k) if tb else (k, n))
    C = rng.standard_normal((m, n))
    opA, opB = A.T if ta else A, B.T if tb else B
    got = _wide(ta, tb, A, B, C, -1.0, 1.0, 0, spare)
    ref = C.astype(np.longdouble) - opA.astype(np.longdouble) @ opB.astype(np.longdouble)
    # at most 8 partial products of a divided K (k <= 1000: 16 k-tiles, two or more each): one
    # rounding each, their 7 additions, the factors and the addition of C
    bound = 12 * EPS * (np.abs(C) + np.abs(opA) @ np.abs(opB))
    assert (np.abs(got - ref) <= bound).all()
    half = _wide(ta, tb, A, B, C, 0.3, -0.5, 0, spare)
    ref = 0.3 * (opA.astype(np.longdouble) @ opB.astype(np.longdouble)) - 0.5 * C.astype(np.longdouble)
    assert (np.abs(half - ref) <= bound).all()


def test_wide_product_graded():
    """Entries that fall by 2^-12 along K on both sides (2^-12 .. 2^-60 against the row maximum)."""
    rng = np.random.default_rng(5)
    m, n, k = 140, 70, 90
    g = 2.0 ** -rng.integers(0, 31, size=k)
    A, B = rng.standard_normal((m, k)) * g, rng.standard_normal((k, n)) * g[::-1][:, None]
    got = _wide(0, 0, A, B, np.zeros((m, n)), 1.0, 0.0, 0)
    ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    assert (np.abs(got - ref) <= 2 * EPS * k * (np.abs(A) @ np.abs(B))).all()


def test_wide_product_lower_triangle_and_zero_rows():
    rng = np.random.default_rng(6)
    m, k = 190, 130
    A = rng.standard_normal((m, k))
    A[7] = 0.0
    A[:, 3] *= 1e-300
    C = rng.standard_normal((m, m))
    got = _wide(0, 1, A, A, C, 1.0, 0.0, 1)
    ref = (A.astype(np.longdouble) @ A.T.astype(np.longdouble)).astype(np.float64)
    low = np.tril(np.ones((m, m), dtype=bool))
    assert (np.abs(got - ref)[low] <= 4 * EPS * (np.abs(A) @ np.abs(A.T))[low]).all()
    assert np.array_equal(got[~low], C[~low])
