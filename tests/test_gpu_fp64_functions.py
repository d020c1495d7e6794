"""The FP64 reciprocal, square root and damping exponential of the stage kernels against correctly rounded
or CUDA's own results, in units in the last place over their ranges.

The bounds: with a starting value good to 2^-20 the reciprocal's third-order step leaves 2^-60 (0.01 ulp) and
the root's series 2^-61, the root's product a quarter of an ulp, and each result is rounded once (0.5): less
than one ulp from the true value, so at most one from the correctly rounded one. The exponential's
polynomials leave 2^-69 and at most 0.57 ulp of rounding, CUDA's function one ulp: at most one ulp apart in
the polynomials' range, two beyond it."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2407_19169_gb300 import _native as N

pytestmark = pytest.mark.gpu


def _run(fn, x):
    x = np.ascontiguousarray(x, dtype=np.float64)
    y = np.empty_like(x)
    dp = C.POINTER(C.c_double)
    assert N.load().dg_probe_fp64(fn, x.size, x.ctypes.data_as(dp), y.ctypes.data_as(dp)) == 0
    return y


def _ulps(a, b):
    """Steps between a and b, of one sign and finite."""
    assert np.isfinite(a).all() and np.isfinite(b).all() and np.array_equal(np.signbit(a), np.signbit(b))
    return np.abs(a.view(np.int64) - b.view(np.int64)).max()


def _values(lo, hi, seed):
    """2^lo to 2^hi: every binade, random and extreme significands, and a dense set around one."""
    r = np.random.default_rng(seed)
    e = np.arange(lo, hi)
    ends = np.ldexp(np.array([1.0, 1.0 + 2.0**-52, 1.5, 2.0 - 2.0**-52])[:, None], e[None]).ravel()
    wide = np.ldexp(r.uniform(1.0, 2.0, 1 << 19), r.integers(lo, hi, 1 << 19))
    return np.concatenate([ends, wide, np.exp(r.uniform(-9.0, 9.0, 1 << 19))])


def test_reciprocal():
    x = _values(-1021, 1021, 1)
    for v in (x, -x):
        assert _ulps(_run(0, v), 1.0 / v) <= 1
    assert not np.isfinite(_run(0, [0.0, -0.0, np.nan])).any()


def test_square_root():
    x = _values(-1021, 1024, 2)
    assert _ulps(_run(1, x), np.sqrt(x)) <= 1
    # zero and below 2^-1021: the correctly rounded function
    tiny = np.concatenate([[0.0, -0.0, 5e-324, 2.0**-1022, np.nextafter(2.0**-1021, 0.0)],
                           np.ldexp(np.random.default_rng(3).uniform(0.0, 1.0, 1000), -1022)])
    assert np.array_equal(_run(1, tiny), np.sqrt(tiny))
    assert not np.isfinite(_run(1, [-1.0, -5e-324, -np.inf, np.nan, np.inf])).any()


def _exp(x):
    return torch.exp(torch.as_tensor(x, device="cuda")).cpu().numpy()


@pytest.mark.parametrize("top", [-9, -4, 0, 9])
def test_damping_exponential(top):
    # warps within each polynomial's range, up to its last number, and beyond; 709 is near the underflow
    r = np.random.default_rng(10 + top)
    last = np.nextafter(2.0**top, 0.0)
    x = -np.minimum(np.concatenate([2.0 ** r.uniform(top - 60, top, 1 << 18), r.uniform(0.0, 2.0**top, 1 << 18),
                                    np.full(32, last), np.zeros(32)]), last)
    x = np.maximum(x, -708.0)
    assert _ulps(_run(2, x), _exp(x)) <= (1 if top <= -4 else 2)


def test_damping_exponential_of_a_mixed_warp():
    # one larger argument takes its whole warp to the function; NaN stays NaN, -inf damps to zero
    x = np.full(96, -1e-5)
    x[40] = -3.0
    assert _ulps(_run(2, x), _exp(x)) <= 1 + (x < -0.0625).any()
    y = _run(2, np.array([np.nan, -np.inf, -1e-5, 0.0]))
    assert np.isnan(y[0]) and y[1] == 0.0 and y[3] == 1.0
