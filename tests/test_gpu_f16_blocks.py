"""Float16 2-D runs take a kernel of four resident blocks an SM where the grid fits them, one
of five otherwise. Both make the same update: a state uniform along y steps alike in a
grid of exactly four blocks an SM and in one of a block more, in every schedule.

Tolerance: the variants are compiled separately, so a value may be stored one rounding away:
2^-10 of a float16 population's deviation (at most twice its spread), 2^-22 of a float32
one's, a step."""
import numpy as np
import pytest

from paper_1508_03452_gb300 import lbrmhd as L
from paper_1508_03452_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 4


@pytest.mark.parametrize("kind", [L.SCHED_PER_RUN, L.SCHED_BATCH, L.SCHED_PERSISTENT])
@pytest.mark.parametrize("recovery", [L.RECOVERY_PLAIN, L.RECOVERY_COLD])
@pytest.mark.parametrize("open_x", [False, True])
def test_both_block_counts_step_alike(kind, recovery, open_x):
    torch = pytest.importorskip("torch")
    if open_x and kind == L.SCHED_PERSISTENT:
        pytest.skip("the persistent schedule takes periodic runs")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = []
    for ny in (4 * sms, 4 * sms + 1):  # a block per row of 128 cells
        F = W.current_sheet(128, ny, 1, delta=4.0)
        bc = (L.OPEN, L.OPEN) + (L.PERIODIC,) * 4 if open_x else (L.PERIODIC,) * 6
        s = L.Solver(L.make_params(128, ny, precision=L.FP16_DEV, recovery=recovery, bc=bc, sigma=100.0))
        s.init_fields(0, F.n, F.p, F.u, F.B, F.E)
        s.set_schedule(kind=kind, bx=128)
        s.step(STEPS)
        assert s.status()["rc"] == L.OK
        out.append([p.reshape(len(p), ny, 128) for p in s.populations()])
        s.close()
    for which, a, b in zip("fgh", *out):
        row = a[:, :1]
        spread = np.abs(row - row.mean(axis=2, keepdims=True)).max(axis=2, keepdims=True)
        tol = STEPS * ((2.0 ** -22 if which == "h" else 2.0 ** -10) * 2 * spread + 1e-7 * np.abs(row).max(axis=2, keepdims=True))
        assert np.all(np.abs(a - row) <= tol) and np.all(np.abs(b - row) <= tol), which
