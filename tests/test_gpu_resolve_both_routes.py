"""The two ways through a MIXED block queue of the batched fitter (csrc/batch.cu: a lane per epoch when the queue is
longer than the block has threads, six epochs per warp otherwise), row by row: a population within 1% of a
caustic-crossing event, so that its rows hold re-solved epochs, their number between the two block sizes. An
image with |det J| below 5e-4 takes the general solver on both ways; the others round by 2^-53 / det^2 = 4.4e-10
times a constant of order ten, and the observed flux lies 30% off, so that chi^2 takes over no more than ten
times A's error: 1e-7."""
import numpy as np
import pytest
import torch

from paper_1208_4830_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ep,half", [(40, 0.3), (64, 0.5), (97, 1.0), (150, 1.0)])
def test_every_row_on_both_routes(lib, n_ep, half):
    n_pop = 64
    one, _, t_cross = synth.force_caustics(synth.prior_theta(1, 5), 1.0, 6)
    genes = one[0].copy()
    genes[5] = np.log10(genes[5])
    lo, hi = genes - 0.01 * np.abs(genes), genes + 0.01 * np.abs(genes)
    t = torch.tensor(t_cross[0] + one[0, 1] * np.linspace(-half, half, n_ep), device="cuda")
    flux = 1.3 * lib.magnification(torch.tensor(one, device="cuda"), t, "fp64")[0]
    off = torch.tensor([0, n_ep], device="cuda")
    p = lib.params(n_pop=n_pop, n_gen=1, precision="mixed", seed=3)
    P = torch.empty((n_pop, 6), dtype=torch.float64, device="cuda")
    lib.ea_init(P, 6, p, 0, lib.new_state_buffer("cuda"))
    theta = lo + (hi - lo) * P.cpu().numpy()
    theta[:, 5] = 10.0 ** theta[:, 5]
    _, flags = lib.magnification(torch.tensor(theta, device="cuda"), t, "mixed", flags=True)
    assert 64 < ((flags & 2) != 0).sum().item() <= 512
    lanes, groups = (lib.fit_batch_archived(t, flux, 0.02 * flux, off, lo, hi, p, size=n_pop, radius=1e-9,
                                            tuning=(16, block)) for block in (64, 512))
    assert lanes[4][0] == groups[4][0] == n_pop
    assert not np.array_equal(lanes[3], groups[3])  # they round differently: both ways were taken
    np.testing.assert_allclose(lanes[3], groups[3], rtol=1e-7)
    np.testing.assert_allclose(lanes[2], groups[2], rtol=1e-12)
