"""The initial state of float32 and float16 runs where its terms cancel: small
perturbations of a uniform state, ideal fields (E = -u x B) at large conductivity, a cold
gas, fields too small for float32. Against the float64 run of the same fields, whose
differences from the reference state are formed by the same float64 operations.

Tolerance, per population: the stored deviation is float64's rounded once (2^-24 of at
most twice its spread over the cells; for the Maxwell populations also of the current's
part, sqrt(2) / 16 (|J_1| + |J_2|), which has no reference), and adding the reference state back rounds either
value once in float64, after at most four float64 roundings of terms of the population's
size (6 x 2^-53 of its largest value). Differences taken in 48 bits instead miss it by 2^-48 of the
terms they are taken of: 16 times the second part, whatever the perturbation's size."""
import numpy as np
import pytest

from paper_1508_03452_gb300 import lbrmhd as L

pytestmark = pytest.mark.gpu

SHAPE = (33, 9, 1)
N = 33 * 9


def _check(fields, **kw):
    n, p, u, B, E = fields
    out = []
    for precision in (L.FP32, L.FP16_DEV, L.FP64):
        s = L.Solver(L.make_params(*SHAPE, precision=precision, **kw))
        s.init_fields(0, n, p, u, B, E)
        out.append(s.populations())
        J = np.abs(s.moments()[13:16]).max()
        s.close()
    for which, x, h, y in zip("fgh", *out):
        spread = np.abs(y - y.mean(axis=1, keepdims=True)).max(axis=1, keepdims=True)
        current = np.sqrt(2.0) / 8.0 * J if which == "h" else 0.0
        tol = 2.0 ** -23 * spread + 2.0 ** -24 * current + 6 * 2.0 ** -53 * np.abs(y).max(axis=1, keepdims=True)
        assert np.all(np.isfinite(x)) and np.all(np.abs(x - y) <= tol), (which, (np.abs(x - y) / (tol + 1e-300)).max())
        if which == "h":  # float32 in both formats
            assert np.array_equal(h, x)


@pytest.mark.parametrize("d", [1e-6, 1e-8, 1e-10])
@pytest.mark.parametrize("seed", [1, 2])
def test_small_perturbations(d, seed):
    r = np.random.default_rng(seed)
    n0, p0, B0 = 0.7 + r.uniform(), 0.7 + r.uniform(), 0.3 + 0.2 * r.uniform(size=(3, 1))
    wave = lambda *s: d * r.uniform(-1, 1, s)
    E = np.zeros((3, N)) + 0.1 * (1 + wave(3, N))
    _check((n0 * (1 + wave(N)), p0 * (1 + wave(N)), wave(3, N), B0 * (1 + wave(3, N)), E), sigma=10.0)


@pytest.mark.parametrize("sigma", [1e2, 1e6, 1e8, 1e10])
@pytest.mark.parametrize("seed", [1, 2])
def test_ideal_fields_at_large_conductivity(sigma, seed):
    r = np.random.default_rng(seed)
    n, p = 1.0 + 0.3 * r.uniform(-1, 1, N), 1.0 + 0.3 * r.uniform(-1, 1, N)
    _check((n, p, 0.1 * r.uniform(-1, 1, (3, N)), 0.1 * r.uniform(-1, 1, (3, N)), None), sigma=sigma)


def test_cold_gas():
    r = np.random.default_rng(5)
    n, p = 1.0 + 0.3 * r.uniform(-1, 1, N), 1e-7 * (1.0 + 0.3 * r.uniform(-1, 1, N))
    _check((n, p, np.zeros((3, N)), np.zeros((3, N)), np.zeros((3, N))), sigma=10.0)


@pytest.mark.parametrize("tiny", [1e-40, 1e-310])
def test_fields_below_the_float32_range(tiny):
    r = np.random.default_rng(6)
    n, p = 1.0 + 0.3 * r.uniform(-1, 1, N), 1.0 + 0.3 * r.uniform(-1, 1, N)
    u, B = 0.1 * r.uniform(-1, 1, (3, N)), 0.1 * r.uniform(-1, 1, (3, N))
    B[0] = tiny
    u[1, ::2] = -tiny
    _check((n, p, u, B, None), sigma=100.0)


def test_pressure_over_its_exponent_rounds_as_the_division():
    """eps = n c^2 + p / (Gamma - 1) in float64, c = 1: a sum of two values rounded once each."""
    r = np.random.default_rng(7)
    n, p = 1e-3 * (1.0 + r.uniform(size=N)), 10.0 ** r.uniform(-3, 6, N)
    for gamma_ad in (4.0 / 3.0, 5.0 / 3.0, 1.1):
        s = L.Solver(L.make_params(*SHAPE, precision=L.FP64, gamma_ad=gamma_ad))
        s.init_fields(0, n, p, np.zeros((3, N)), np.zeros((3, N)))
        eps = s.moments()[2]
        s.close()
        gm1 = np.float64(gamma_ad) - 1.0
        assert np.all((eps == n + p / gm1) | (eps == (n.astype(np.longdouble) + p / gm1).astype(np.float64)))
