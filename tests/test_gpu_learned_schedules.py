"""The learned seed is the same in every launch schedule. The one-run step kernel takes
the network through tensor memory (tcgen05), the batched and persistent ones through
warp-level products (mma.sync); the eigen-solve starts from its output, so a seed that
differs in one bf16 rounding lets a run's states and iteration counts depend on the
schedule (and so on what the autotuner picks)."""
import ctypes

import numpy as np
import pytest

import device_checks as D
from oracle import mlp_ref as M
from paper_1508_03452_gb300 import lbrmhd as L
from paper_1508_03452_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _params(seed, bias):
    """Initial weights with biases of the given scale: of 24 significant bits, so that all
    three bf16 parts of a bias count."""
    P = W.mlp_init_params(seed).astype(np.float64)
    r, o = np.random.default_rng(seed + 100), 0
    for name, shape in M.SHAPES:
        k = int(np.prod(shape))
        if name.startswith("b"):
            P[o:o + k] = bias * r.normal(size=k)
        o += k
    return P.astype(np.float32)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 100003])
@pytest.mark.parametrize("bias", [0.0, 1e-3, 0.1, 3.0])
def test_tensor_memory_network_is_the_warp_level_one(n, bias):
    """Bit for bit on rows that all differ, and near the float64 sums of the bf16 operands
    (the bound of the standalone inference's test: a bf16 rounding of a hidden unit that
    falls otherwise)."""
    torch = pytest.importorskip("torch")
    P, r = _params(3, bias), np.random.default_rng(n)
    X = r.normal(0, 0.5, size=(n, M.N_IN)).astype(np.float32)
    X[:, 19] = 1
    dP, dX = torch.tensor(P, device="cuda"), torch.tensor(X, device="cuda")
    y = torch.full((n, M.N_OUT), float("nan"), device="cuda")
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(t.data_ptr()) for t in (dP, dX, y)]
    assert D.load().check_seed(p[0], p[1], ctypes.c_int64(n), p[2]) == 0
    got = y.cpu().numpy()
    assert np.array_equal(got, L.mlp_infer(L.mlp_pack(dP), dX).cpu().numpy())
    want = M.forward_bf16(P.astype(np.float64), X.astype(np.float64))
    d, scale = np.abs(got - want).max(1), np.abs(want).max()
    assert d.max() <= 1e-2 * scale and np.median(d) <= 1e-4 * scale


@pytest.mark.parametrize("tol", [0.0, 1e-3])
def test_learned_float64_runs_agree_bit_for_bit(tol):
    """States, iteration counts and failures of the three schedules, also with a loose
    recovery tolerance, whose result still depends on where the solve started."""
    torch = pytest.importorskip("torch")
    fields = [W.kelvin_helmholtz(nx, ny, 1, V=0.3, ratio=3.0, B0=0.5, a=2.0, noise=1e-2, seed=60 + i)
              for i, (nx, ny) in enumerate([(100, 60), (130, 33)])]
    P, ref = torch.tensor(_params(3, 0.05), device="cuda"), None
    for sc in (dict(kind=L.SCHED_PER_RUN), dict(kind=L.SCHED_BATCH, bx=128), dict(kind=L.SCHED_BATCH, bx=32, waves=1, order=1),
               dict(kind=L.SCHED_PERSISTENT, bx=64)):
        s = L.Solver([L.make_params(F.nx, F.ny, sigma=1e3, alpha=0.02, precision=L.FP64, recovery=L.RECOVERY_MLP, tol=tol)
                      for F in fields], stream=torch.cuda.current_stream())
        for r, F in enumerate(fields):
            s.init_fields(r, F.n, F.p, F.u, F.B, F.E)
        s.set_schedule(**sc)
        s.set_mlp_weights(P)
        s.step(7)
        out = [(np.concatenate([*s.populations(r), s.moments(r)]), s.stats(r)) for r in range(2)]
        s.close()
        ref = ref or out
        for (x, sx), (y, sy) in zip(out, ref):
            assert np.array_equal(x, y) and sx == sy, sc
