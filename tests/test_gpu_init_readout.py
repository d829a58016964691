"""The initial state formed in float32 pairs, and the moments widened on the integer
pipes, against the float64 run of the same fields (whose own kernels are held to the
oracle elsewhere).

Tolerances: a float32 population is its float64 deviation rounded once (2^-24 of the
deviation; the deviation of a direction is at most twice its spread over cells that
surround the mean state), so 2^-22 of the spread leaves a factor two; J of a float32
run is what float64 arithmetic gives from its float32 fields, rounded at 1e-16 per
term, so 1e-13 of the terms' scale."""
import numpy as np
import pytest

from paper_1508_03452_gb300 import lbrmhd as L

pytestmark = pytest.mark.gpu


def _fields(nx, ny, nz, seed, zero):
    r = np.random.default_rng(seed)
    N = nx * ny * nz
    n, p = 1.0 + 0.3 * r.uniform(-1, 1, N), 1.0 + 0.3 * r.uniform(-1, 1, N)
    u, B = 0.4 * r.uniform(-1, 1, (3, N)), 0.5 + 0.3 * r.uniform(-1, 1, (3, N))
    if zero:  # exact zeros of either sign and tiny values take the conversions' other branches
        u[0] = 0.0
        u[1, ::2] = -0.0
        B[2] = 0.0
        B[0, ::3] = 1e-30
    return n, p, u, B


def _solver(shape, precision, fields):
    s = L.Solver(L.make_params(*shape, sigma=50.0, precision=precision))
    s.init_fields(0, *fields)
    return s


@pytest.mark.parametrize("shape", [(33, 1, 1), (13, 9, 1), (130, 7, 1), (9, 7, 5)])
@pytest.mark.parametrize("zero", [False, True])
def test_initial_populations_are_the_float64_ones_rounded(shape, zero):
    fields = _fields(*shape, 3, zero)
    a, b = _solver(shape, L.FP32, fields), _solver(shape, L.FP64, fields)
    for x, y in zip(a.populations(), b.populations()):
        spread = np.abs(y - y.mean(axis=1, keepdims=True)).max(axis=1, keepdims=True)
        assert np.all(np.abs(x - y) <= 2.0 ** -22 * spread + 1e-13 * np.abs(y).max())
    a.close()
    b.close()


@pytest.mark.parametrize("precision", [L.FP64, L.FP32, L.FP16_DEV])
@pytest.mark.parametrize("shape", [(1, 1, 1), (129, 3, 1), (7, 5, 6)])
@pytest.mark.parametrize("zero", [False, True])
def test_moments_are_float64_of_the_stored_fields(precision, shape, zero):
    s = _solver(shape, precision, _fields(*shape, 4, zero))
    m = s.moments()
    s.close()
    n, p, eps, u, E, B, rho, J = m[0], m[1], m[2], m[3:6], m[6:9], m[9:12], m[12], m[13:16]
    if precision != L.FP64:
        for row in (n, eps, *u, *E, *B, rho):
            assert np.array_equal(row, row.astype(np.float32).astype(np.float64))
    assert np.allclose(p, (4.0 / 3.0 - 1.0) * (eps - n), rtol=1e-14, atol=1e-15)
    g = 1.0 / np.sqrt(1.0 - (u * u).sum(0))
    terms = 50.0 * g * (np.abs(E).sum(0) + np.abs(u).sum(0) * np.abs(B).sum(0)) + np.abs(rho)
    want = 50.0 * g * (E + np.cross(u, B, axis=0) - (E * u).sum(0) * u) + rho * u
    assert np.all(np.abs(J - want) <= 1e-13 * terms + 1e-300)
