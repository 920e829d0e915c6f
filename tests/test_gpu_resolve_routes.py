"""The batched fitter's two ways through its MIXED re-solve queue (csrc/batch.cu): a lane per epoch when the
queue is longer than the block has threads, six epochs per warp otherwise. The same fit in blocks of 64 and
of 512 threads takes one or the other; the epochs and their FP32 solutions are the same (16 threads per
candidate in both)."""
import numpy as np
import pytest
import torch

from paper_1208_4830_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_pop,n_ep", [(64, 97), (200, 300), (256, 700)])
def test_long_and_short_queues_agree(lib, n_pop, n_ep):
    """Both routes return magnifications within 1e-9 of the exact ones (1e-10 where |det J| >= 1e-3), so
    chi^2 of curves with sigma = 2% and a population far from the truth agrees to 1e-7."""
    b = synth.heldout_batch(5, seed=31, n_ep=n_ep)
    t = torch.tensor(b.t, device="cuda")
    A = torch.cat([
        lib.magnification(torch.tensor(b.truth[i : i + 1], device="cuda"), t[b.offsets[i] : b.offsets[i + 1]], "fp64")[0]
        for i in range(5)
    ])
    off = torch.tensor(b.offsets, device="cuda")
    p = lib.params(n_pop=n_pop, n_gen=1, precision="mixed", seed=3)
    out = [lib.fit_batch(t, A, 0.02 * A, off, synth.FIT_LO, synth.FIT_HI, p, tuning=(16, block)) for block in (64, 512)]
    assert np.allclose(out[0][1], out[1][1], rtol=1e-7, atol=0.0)
    assert np.array_equal(out[0][0], out[1][0])
