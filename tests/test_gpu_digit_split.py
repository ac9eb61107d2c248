"""The cut into digits at the ends of its range, through the wide product: rows of powers of two (ties and
carries through every digit), full significands next to the row's largest entry, entries far below it,
rows of subnormal numbers and zero rows, along memory and across."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_ozaki_wide import EPS, _wide  # noqa: E402


@pytest.mark.parametrize("ta", [0, 1])
@pytest.mark.parametrize("k", [3, 70, 300])
def test_digits_at_the_ends_of_the_range(ta, k):
    rng = np.random.default_rng(k)
    m, n = 12, 9
    A = rng.standard_normal((m, k))
    A[0] = 0.0
    A[1] = np.ldexp(1.0, rng.integers(-60, 1, k))                      # powers of two
    A[2] = np.ldexp(1.0 - EPS, rng.integers(-12, 1, k))                # all bits set
    A[3] = -A[2]
    A[4] = np.ldexp(rng.choice([257.0, 255.0, 256.5], k), rng.integers(-30, 1, k))
    A[5] = np.ldexp(rng.integers(1, 1 << 40, k).astype(float), -1074)  # subnormal rows
    A[6] = np.ldexp(rng.integers(1, 8, k).astype(float), -1074)
    A[7] = A[7] * 1e300
    A[8, 0] = 1e18
    A[9] = np.ldexp(A[9], rng.integers(-90, 1, k))
    B = np.ldexp(rng.standard_normal((k, n)), 0)
    B[:, :3] = np.ldexp(B[:, :3], 600)  # subnormal rows give normal products here
    C = np.zeros((m, n))
    got = _wide(ta, 0, np.asfortranarray(A.T if ta else A), B, C, 1.0, 0.0, 0)
    ref = np.zeros((m, n), dtype=np.longdouble)
    with np.errstate(over="ignore"):
        ref = A.astype(np.longdouble) @ B.astype(np.longdouble)
    # per term 2^-71 of the largest entries for each factor (they are 2 to 4 times smaller than their
    # power of two) and 14 2^-71 for the seven dropped pairs, then one rounding; subnormal results
    # to half their unit
    big = np.abs(A).max(1)[:, None].astype(np.longdouble) * np.abs(B).max(0)[None, :]
    bound = 2 * EPS * np.abs(ref) + 20 * k * np.ldexp(np.longdouble(1), -71) * big + np.longdouble(2.0 ** -1074)
    ok = np.abs(ref) < 1e307  # what passes the range is not compared
    assert (np.abs(got - ref)[ok] <= bound[ok]).all()
    assert (got[0] == 0).all()
