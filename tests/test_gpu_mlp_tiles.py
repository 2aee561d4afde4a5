"""Training-step kernels of the controller network at the edges of their tiles
and of the batch sizes where they change form, with rows that are not 16-byte
aligned and with the gradient written over the outputs, against the FP64
reference of oracle/mlp_oracle.py on the same BF16 weights."""
import numpy as np
import pytest

from test_gpu_mlp import P, _dev, _setup  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("batch", [15, 16, 33, 4096, 4097, 4863, 4865, 9727, 9729, 19455, 19457])
def test_training_step_matches_oracle(P, batch, shift, in_place):
    import torch
    from oracle import mlp_oracle as M
    if in_place and batch not in (33, 4097, 19457):
        pytest.skip("one size per form")
    _, wq, X, wb = _setup(21, batch)
    rng = np.random.default_rng(22)
    T = rng.normal(size=(batch, 2)).astype(np.float32)
    wt = rng.uniform(0.0, 2.0, batch).astype(np.float32)

    def buf(rows, cols):  # `shift` floats past an aligned base
        return torch.zeros(rows * cols + 4, device="cuda")[shift:shift + rows * cols].view(rows, cols)

    x = buf(batch, 16)
    x.copy_(_dev(X))
    y, cache = buf(batch, 2), buf(batch, 128)
    P.mlp_forward(wb, x, y, cache)
    Yr, cr = M.forward(wq, X.astype(np.float64))
    assert np.allclose(y.cpu().numpy(), Yr, rtol=1e-5, atol=1e-5)
    got = cache.cpu().numpy()
    assert np.allclose(got[:, :64], cr["Z1"], rtol=1e-5, atol=1e-5)
    assert np.allclose(got[:, 64:], cr["Z2"], rtol=1e-5, atol=1e-5)
    dy = y if in_place else buf(batch, 2)
    loss = torch.zeros(1, device="cuda")
    P.mlp_wmse(y, _dev(T), _dev(wt), dy, loss)
    Lr, dYr = M.wmse(Yr, T.astype(np.float64), wt.astype(np.float64))
    assert abs(loss.item() - Lr) <= 1e-5 * max(1.0, Lr)
    # FP32 rounding of y, t and their product: 4 units of 2^-24 of |y| + |t| <= 8, times 2 w / sum w.
    assert np.abs(dy.cpu().numpy() - dYr).max() <= 8 * 4 * 6e-8 * 2 * 2.0 / wt.sum() + 1e-5 * np.abs(dYr).max()
    grad = torch.zeros(P.mlp_param_count(), device="cuda")
    scratch = torch.full((((batch + 15) // 16) * P.mlp_param_count() + 64,), 7.0, device="cuda")
    P.mlp_backward(wb, x, cache, dy, grad, scratch)
    gr = M.backward(wq, cr, dYr)
    assert np.abs(grad.cpu().numpy() - gr).max() <= 1e-4 * np.abs(gr).max()
    assert bool((scratch[-64:] == 7.0).all())  # nothing written past ceil(batch / 16) rows
