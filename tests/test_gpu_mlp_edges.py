"""The network's gradient, training and inference kernels at the edges of their
tiles (8 samples a training block, 456 blocks; 32 rows an inference warp, 456
blocks of 4 warps), with parameters and rows that are not 16-byte aligned,
against the float64 reference of oracle/mlp_ref.py.

Tolerances: a float32 sum of n <= 64 products and a batch sum of up to 4,000
samples in 8 shares keep ~1e-6 relative, held to 1e-5 per layer as the larger
batches are; an inference differs from the bf16 forward pass where a float32
sum falls on the other side of a bf16 rounding of a hidden unit (2^-8 of one of
64 inputs)."""
import numpy as np
import pytest

from oracle import mlp_ref as M
from paper_1508_03452_gb300 import lbrmhd as L
from paper_1508_03452_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _rows(n, seed):
    r = np.random.default_rng(seed)
    X = r.normal(0, 0.5, size=(n, M.N_IN))
    X[:, 19] = 1
    return np.concatenate([X, r.normal(0, 0.2, size=(n, M.N_OUT))], 1).astype(np.float32)


def _device(a, shift):
    """The array on the device, `shift` floats past a 256-byte boundary."""
    torch = pytest.importorskip("torch")
    a = np.asarray(a, dtype=np.float32)
    buf = torch.zeros(a.size + shift, device="cuda")
    v = buf[shift:].view(a.shape)
    v.copy_(torch.from_numpy(a))
    return v


@pytest.mark.parametrize("n", [1, 7, 8, 9, 3647, 3649])
@pytest.mark.parametrize("shift", [0, 1])
def test_gradient_at_tile_edges(n, shift):
    P, data = W.mlp_init_params(2), _rows(n, n)
    loss, g = L.mlp_grad(_device(P, shift), _device(data, shift))
    Lw, gw = M.loss_and_grad(P.astype(np.float64), data[:, :20].astype(np.float64), data[:, 20:].astype(np.float64))
    g = g.cpu().numpy().astype(np.float64)
    assert loss == pytest.approx(Lw, rel=1e-5)
    o = 0
    for name, shape in M.SHAPES:
        k = int(np.prod(shape))
        assert np.linalg.norm(g[o:o + k] - gw[o:o + k]) <= 1e-5 * np.linalg.norm(gw[o:o + k]), name
        o += k


@pytest.mark.parametrize("batch", [1, 9, 3649])
@pytest.mark.parametrize("shift", [0, 1])
def test_training_at_tile_edges(batch, shift):
    torch = pytest.importorskip("torch")
    P0, data, steps, lr, seed = W.mlp_init_params(5), _rows(500, 6), 5, 1e-3, 17
    v0 = np.full(M.NPARAM, 1e-3)  # a second moment that keeps the step linear in the gradient
    P, adam = _device(P0, shift), _device(np.concatenate([np.zeros(M.NPARAM), v0]), shift)
    losses = L.mlp_train(P, adam, _device(data, shift), steps, batch, lr, seed=seed)
    torch.cuda.synchronize()
    Pw, mw, vw, lw = M.train(P0.astype(np.float64), np.zeros(M.NPARAM), v0, data.astype(np.float64), steps, batch, lr,
                             seed)
    assert np.allclose(losses.cpu().numpy(), lw, rtol=1e-5, atol=0)
    got = adam.cpu().numpy()
    assert np.linalg.norm(got[:M.NPARAM] - mw) <= 1e-5 * np.linalg.norm(mw)
    # the parameters' change carries the float32 rounding of the parameters (6e-8 of ~0.2 a step)
    step_gpu, step_ref = P.cpu().numpy() - P0, Pw - P0
    floor = steps * 6e-8 * np.linalg.norm(P0)
    assert np.linalg.norm(step_gpu - step_ref) <= 1e-4 * np.linalg.norm(step_ref) + floor


@pytest.mark.parametrize("n", [1, 31, 32, 33, 129, 58368, 58369])
@pytest.mark.parametrize("shift", [0, 1])
def test_inference_at_tile_edges(n, shift):
    P, X = W.mlp_init_params(3), _rows(n, n)[:, :M.N_IN]
    y = L.mlp_infer(L.mlp_pack(_device(P, 0)), _device(np.ascontiguousarray(X), shift)).cpu().numpy()
    want = M.forward_bf16(P.astype(np.float64), X.astype(np.float64))
    assert y.shape == want.shape
    d, scale = np.abs(y - want).max(1), np.abs(want).max()
    assert d.max() <= 1e-2 * scale and np.median(d) <= 1e-4 * scale
