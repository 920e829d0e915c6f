"""Training steps that draw the next batch beside the network's products: every run length (the last step
alone, two steps, pairs replayed from a graph) gives the weights, moments and losses of one step per
call, bit for bit; and the first convolution's products at batches around a tile."""
import numpy as np
import pytest
import torch

from oracle import cnn as ocnn
from oracle import proposal as oprop

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_run", [1, 2, 3, 4, 7])
def test_run_lengths_equal_single_steps(lib, n_run):
    p = lib.cnn_train_params(batch=33, n_steps=50, warmup=5, seed=8)
    w = lib.cnn_init(2)
    one, many = [w.clone(), torch.zeros(2 * w.numel(), device="cuda")], [w.clone(), torch.zeros(2 * w.numel(), device="cuda")]
    hist = np.concatenate([lib.cnn_train(one[0], one[1], p, 3 + k, 1) for k in range(n_run)])
    assert np.array_equal(lib.cnn_train(many[0], many[1], p, 3, n_run), hist)
    assert torch.equal(one[0], many[0]) and torch.equal(one[1], many[1])


@pytest.mark.parametrize("batch", [1, 2, 9])
def test_first_layer_gradient(lib, batch):
    """Each element of the first convolution's gradient within 3e-2 of the layer's norm of FP64 (the
    normwise tolerance of test_gpu_cnn.py: BF16 operands)."""
    w = oprop.init_params(4)
    x, y, _, _ = oprop.make_batch(4, 1, batch)
    f32 = dict(dtype=torch.float32, device="cuda")
    _, g = lib.cnn_loss_grad(torch.tensor(w, **f32), torch.tensor(x, **f32), torch.tensor(y, **f32))
    _, ref = ocnn.loss_and_grad(w, x, y)
    g, ref = g.cpu().numpy()[:704].astype(np.float64), ref[:704]
    assert np.linalg.norm(g - ref) <= 3e-2 * np.linalg.norm(ref)
