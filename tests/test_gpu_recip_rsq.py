"""The reciprocal and reciprocal square root of the reflectors, Cholesky pivots and twisted factorisations
over the whole range of either precision: every exponent with random significands, both ends of a
binade, both sides of every limit at which the library's operations take over, and the
special values. Bounds: the last rounding (half an ulp), and for the square root another half
from the rounding of x r; what the iteration leaves is below a tenth (2^-57 in binary64)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1705_11191_gb300 as egb  # noqa: E402


def run(x):
    lib, v = egb.load(), ctypes.c_void_p
    lib.elsi_gb_recip_rsq.argtypes = [ctypes.c_int, ctypes.c_int, v, v, v, v]
    d = torch.from_numpy(x).cuda()
    r, s = torch.empty_like(d), torch.empty_like(d)
    assert lib.elsi_gb_recip_rsq(x.size, int(x.dtype == np.float64), d.data_ptr(), r.data_ptr(), s.data_ptr(), None) == 0
    torch.cuda.synchronize()
    return r.cpu().numpy(), s.cpu().numpy()


def arguments(dtype):
    f = np.finfo(dtype)
    rng = np.random.default_rng(0)
    one = dtype(1)
    edge = [one, np.nextafter(one, dtype(2)), np.nextafter(dtype(2), one), dtype(1.5), np.nextafter(dtype(1.5), one)]
    x = []
    for e in range(f.minexp - f.nmant, f.maxexp):  # subnormal numbers too
        m = np.concatenate([edge, rng.uniform(1, 2, 40).astype(dtype)])
        x.append(np.ldexp(m, e).astype(dtype))
    x = np.concatenate(x)
    for lim in (1e-36, 1e36) if dtype == np.float32 else [np.ldexp(1.0, e - 1023) for e in (1, 40, 41, 2000, 2044)]:
        a = dtype(lim)
        for _ in range(3):
            x = np.append(x, [a, np.nextafter(dtype(lim), dtype(0))])
            a = np.nextafter(a, dtype(np.inf))
    return x[(x > 0) & np.isfinite(x)].astype(dtype)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_error_in_ulps(dtype):
    x = arguments(dtype)
    wide = np.longdouble
    f = np.finfo(dtype)
    for sign in (1, -1):
        y = (sign * x).astype(dtype)
        r, s = run(y)
        with np.errstate(over="ignore"):
            ref = (wide(1) / y.astype(wide))
            big = np.abs(ref) > wide(f.max)
            assert np.isinf(r[np.abs(ref) >= wide(f.max) * (1 + wide(f.eps))]).all()
            ulp = np.spacing(np.abs(ref[~big]).astype(dtype)).astype(wide)
            assert (np.abs(r[~big].astype(wide) - ref[~big]) <= ulp).all()
        if sign < 0:
            assert np.isnan(s).all()
            continue
        ref = wide(1) / np.sqrt(y.astype(wide))
        ulp = np.spacing(ref.astype(dtype)).astype(wide)
        assert (np.abs(s.astype(wide) - ref) <= wide(1.25) * ulp).all()


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_special_values(dtype):
    r, s = run(np.array([0.0, -0.0, np.inf, -np.inf, np.nan], dtype=dtype))
    assert r[0] == np.inf and r[1] == -np.inf and r[2] == 0 and r[3] == 0 and np.isnan(r[4])
    assert s[0] == np.inf and np.isinf(s[1]) and s[2] == 0 and np.isnan(s[3]) and np.isnan(s[4])
