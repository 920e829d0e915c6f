"""FP64 batched fits evaluate a population in passes of as many rows as hold 2^18 epochs: populations that fit
one pass, end on it, and leave a few rows for another one, and the scratch they take."""
import numpy as np
import pytest
import torch

from paper_1208_4830_gb300 import synth

pytestmark = pytest.mark.gpu


def curves(lib, n_lc, n_ep, seed):
    b = synth.heldout_batch(n_lc, seed=seed, n_ep=n_ep)
    t, off = torch.tensor(b.t, device="cuda"), torch.tensor(b.offsets, device="cuda")
    A = torch.cat([lib.magnification(torch.tensor(b.truth[i : i + 1], device="cuda"),
                                     t[b.offsets[i] : b.offsets[i + 1]], "fp64")[0] for i in range(n_lc)])
    return t, A, 0.02 * A, off


@pytest.mark.parametrize("n_pop", [130, 160, 161, 333])
def test_passes_equal_the_forward_model(lib, n_pop):
    """1611 epochs: 160 rows (five passes of the block's 32 groups) to an emptying of the queue. The 64 fittest
    rows against sblm_chi2_genes: the same epochs from other FP32 starts, within 1e-9 of the exact magnifications."""
    t, flux, sigma, off = curves(lib, 1, 1611, 5)
    p = lib.params(n_pop=n_pop, n_gen=1, precision="fp64", seed=6)
    got = lib.fit_batch_archived(t, flux, sigma, off, synth.FIT_LO, synth.FIT_HI, p, size=64, radius=1e-9)
    P = torch.empty((n_pop, 6), dtype=torch.float64, device="cuda")
    lib.ea_init(P, 6, p, 0, lib.new_state_buffer("cuda"))
    c = np.sort(lib.chi2_genes(P, t, flux, sigma, synth.FIT_LO, synth.FIT_HI, "fp64").cpu().numpy())[:64]
    np.testing.assert_allclose(got[3][0], c, rtol=1e-7)


def test_scratch_does_not_grow_with_the_population(lib):
    """152 curves, 4096 rows of 3000 epochs: 15 GB of chi^2 terms if all had a place; 2^18 epochs of 60 bytes
    per block, the populations and a quarter of spare room are 3.1 GB."""
    t, flux, sigma, off = curves(lib, 152, 3000, 7)
    p = lib.params(n_pop=4096, n_gen=1, precision="fp64", seed=6)
    with torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        best, chi = lib.fit_batch(t, flux, sigma, off, synth.FIT_LO, synth.FIT_HI, p)
        torch.cuda.synchronize()
        assert before - torch.cuda.mem_get_info()[0] < 4e9
    assert np.isfinite(np.asarray(chi)).all()
