"""The float64 reciprocal and inverse square root of the step kernels (Newton's iteration
and the binomial series from the hardware's approximations) over the exponent range,
beside powers of two and at the ends, against extended precision.

Bounds: the reciprocal is rounded once (2^-53) plus less than 2^-70 of the second
iteration; the inverse square root is 1.6 x 2^-53 (its final rounding, half of the rounding
of x r in the residual, and 5/16 e^3 with e about 2^-19)."""
import ctypes

import numpy as np
import pytest

import device_checks as D

pytestmark = pytest.mark.gpu


def _run(x):
    torch = pytest.importorskip("torch")
    d = [torch.tensor(np.asarray(x, dtype=np.float64), device="cuda")]
    d += [torch.empty_like(d[0]) for _ in range(2)]
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(t.data_ptr()) for t in d]
    assert D.load().check_reciprocals(p[0], ctypes.c_int64(d[0].numel()), p[1], p[2]) == 0
    return d[1].cpu().numpy(), d[2].cpu().numpy()


def _rel(got, want):
    return np.abs((got.astype(np.longdouble) - want) / want).max()


def test_over_the_exponent_range():
    r = np.random.default_rng(3)
    m = 1.0 + r.uniform(size=(8, 2044))
    x = np.ldexp(m, np.arange(-1022, 1022)[None, :]).ravel()
    x = x[x <= 2.0 ** 1022]
    p2 = np.ldexp(1.0, np.arange(-1021, 1022))
    x = np.concatenate([x, p2, np.nextafter(p2, 0), np.nextafter(p2, np.inf), 1.0 - 2.0 ** -np.arange(1, 54), 1.0 + r.uniform(size=200000)])
    rcp, rsq = _run(x)
    one = np.longdouble(1)
    assert _rel(rcp, one / x) <= 2.0 ** -53 * (1 + 2.0 ** -10)
    assert _rel(rsq, one / np.sqrt(x.astype(np.longdouble))) <= 1.6 * 2.0 ** -53
    assert np.array_equal(_run(-x)[0], -rcp)


def test_at_the_ends():
    inf = np.inf
    rcp, rsq = _run([0.0, -0.0, inf, -inf, np.nan, 1e-310, -1e-310, 1.7e308, -1.0])
    assert np.array_equal(rcp[:4], [inf, -inf, 0.0, 0.0]) and np.array_equal(np.signbit(rcp[:4]), [False, True, False, True])
    assert np.isnan(rcp[4]) and np.array_equal(rcp[5:9], [inf, -inf, 0.0, -1.0])
    assert np.array_equal(rsq[[0, 2]], [inf, 0.0]) and rsq[5] == inf
    assert np.isnan(rsq[[3, 4, 8]]).all()
    assert rsq[7] == pytest.approx(1.0 / np.sqrt(1.7e308), rel=2.0 ** -52)
