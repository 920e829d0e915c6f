"""AdamW over the range of its second moment: gradients from 1e-18 to 1e18 with moments to match, zero, and
second moments that have overflowed FP32 to infinity (a gradient above 6e20 once), after which a weight
only decays. Tolerance as in test_gpu_cnn.py: the update is FP64, the stored weight FP32."""
import numpy as np
import pytest
import torch

from oracle import cnn as ocnn
from oracle import proposal as op

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps", [1e-8, 1e-30])
def test_adamw_over_the_range_of_its_moments(lib, eps):
    N = ocnn.N_PARAMS
    rng = np.random.default_rng(1)
    size = 10.0 ** rng.uniform(-18, 18, N)
    w = rng.normal(size=N).astype(np.float32)
    g = (size * rng.normal(size=N)).astype(np.float32)
    m = (size * rng.normal(size=N)).astype(np.float32)
    v = (size * size * rng.uniform(0.1, 1, N)).astype(np.float32)
    g[::7] = m[::7] = v[::7] = 0.0
    v[3::7] = np.inf
    p = lib.cnn_train_params(lr=3e-3, n_steps=100, warmup=10, eps=eps)
    wt = torch.tensor(w, device="cuda")
    st = torch.tensor(np.concatenate([m, v]), device="cuda")
    lib.cnn_adamw(wt, st, torch.tensor(g, device="cuda"), p, 7)
    w2, _, v2 = op.adamw(*(a.astype(np.float64) for a in (w, m, v, g)), 7, op.lr_at(7, 100, 10, 3e-3), eps=eps)
    assert np.isfinite(w2).all() and np.isinf(v2[3::7]).all()
    np.testing.assert_allclose(wt.cpu().numpy(), w2, rtol=1e-6, atol=1e-7)
