"""A population that is not a number spoils the same cells in every storage format. The
float64 and float32 limiters choose differently when one of their arguments is not a number
(the other argument; the smaller of the middle difference and 0), which changes
finite values beside a lost cell but not which cells are lost: those whose first-order
flux or viscosity reads it."""
import numpy as np
import pytest

from paper_1508_03452_gb300 import lbrmhd as L

pytestmark = pytest.mark.gpu

NX, NY, X, Y = 40, 12, 17, 5


def _lost(precision, which):
    N = NX * NY
    r = np.random.default_rng(2)
    s = L.Solver(L.make_params(NX, NY, precision=precision, sigma=50.0))
    s.init_fields(0, 1 + 0.1 * r.uniform(size=N), 1 + 0.1 * r.uniform(size=N), 0.02 * r.uniform(-1, 1, (3, N)),
                  0.2 + 0.05 * r.uniform(-1, 1, (3, N)))
    pop, other = {L.FP64: (np.float64, 8), L.FP32: (np.float32, 4), L.FP16_DEV: (np.float16, 4)}[precision]
    blob = bytearray(s.get_state())
    # f and g group by group (4 values a cell; the first group's are f, g of +x and of -x),
    # their rest pairs, then h (25 a cell), the primitives (12) and the initial E^z (1)
    start = len(blob) - 38 * N * np.dtype(pop).itemsize - (25 + 12 + 1) * N * other
    values = np.frombuffer(blob, dtype=pop, count=4 * N, offset=start)
    values[4 * (X + NX * Y) + (0 if which == "f" else 1)] = np.nan
    s.set_state(bytes(blob))
    before = s.populations()
    assert [int((~np.isfinite(p)).sum()) for p in before] == ([1, 0, 0] if which == "f" else [0, 1, 0])
    assert not np.isfinite(before[0 if which == "f" else 1][1, X + NX * Y])
    s.step(1)
    lost = ~np.isfinite(np.concatenate(s.populations())).all(axis=0).reshape(NY, NX)
    s.close()
    return {(int(y), int(x)) for y, x in np.argwhere(lost)}


@pytest.mark.parametrize("which", ["f", "g"])
def test_every_format_loses_the_same_cells(which):
    want = {(Y, X), (Y, X + 1)}
    if which == "f":  # the viscosity's Laplacian
        want |= {(Y, X - 1), (Y - 1, X), (Y + 1, X)}
    for precision in (L.FP64, L.FP32, L.FP16_DEV):
        assert _lost(precision, which) == want, precision
