"""FP64 magnifications from FP32 roots (csrc/refine.cuh) at the sizes where their bookkeeping can go
wrong: re-solve queues that end inside a warp's six epochs, calls cut into several chunks of
candidates, full queues, and lenses and sources outside the refined range. Tolerance: relative 1e-10
where the oracle's smallest |det J| over the images is at least 1e-3, as in test_gpu_forward.py."""
import numpy as np
import pytest
import torch

from oracle import sblm as osb
from paper_1208_4830_gb300 import synth

pytestmark = pytest.mark.gpu


def dev(x):
    return torch.tensor(x, device="cuda")


def _check(A, theta, t, share=0.5):
    A_ref, info = osb.magnification(theta, t, return_info=True)
    ok = (info["min_det"] >= 1e-3) & ~info["flag"]
    assert ok.mean() >= share
    err = np.abs(A - A_ref) / A_ref
    assert err[ok].max() <= 1e-10, err[ok].max()


@pytest.mark.parametrize("n_cand,n_ep", [(1, 1), (1, 13), (2, 97), (7, 331), (33, 64)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_short_queues(lib, n_cand, n_ep, prec):
    """Every trajectory crosses a caustic: queues of a few epochs, most not a multiple of six."""
    theta = synth.force_caustics(synth.prior_theta(n_cand, 51), 1.0, 52)[0]
    t = synth.uniform_epochs(n_ep, 53)
    A, fl = lib.magnification(dev(theta), dev(t), prec, flags=True)
    A, fl = A.cpu().numpy(), fl.cpu().numpy()
    if prec == "fp64":
        return _check(A, theta, t)
    A_ref, info = osb.magnification(theta, t, return_info=True)
    re = ((fl & 2) != 0) & ~info["flag"] & (info["min_det"] >= 1e-3)  # the epochs re-solved in FP64
    assert np.all(np.abs(A - A_ref)[re] <= 1e-10 * A_ref[re])


def test_chunked_call(lib):
    """More epochs than one chunk of candidates holds (2^22): rows on both sides of the cut, and chi^2."""
    n, m = 2200, 2000
    sw = synth.forward_sweep(n_cand=n, n_ep=m, seed=61)
    th, t = dev(sw.theta), dev(sw.t)
    A = lib.magnification(th, t, "fp64")
    cut = (1 << 22) // m
    rows = [0, cut - 1, cut, n - 1]
    _check(A[rows].cpu().numpy(), sw.theta[rows], sw.t, share=0.9)
    flux, sigma = A[5].clone(), 0.01 * A[5]
    c = lib.chi2(th, t, flux, sigma, "fp64")
    ref = (((flux - A) / sigma) ** 2).sum(1)
    # the same terms in another order of summation: 2000 roundings of 2^-53 at most
    assert torch.all((c - ref).abs() <= 2000 * 2.0**-53 * ref + 1e-300)


def test_full_queue(lib):
    """Every epoch of every candidate next to a caustic: far more re-solves than the queue holds."""
    theta, _, t_cross = synth.force_caustics(synth.prior_theta(3, 71), 1.0, 72)
    k = 1
    t = t_cross[k] + theta[k, 1] * np.linspace(-2e-4, 2e-4, 801)
    A = lib.magnification(dev(np.repeat(theta[k : k + 1], 96, 0)), dev(t), "fp64").cpu().numpy()
    _check(A[[0, 50, 95]], np.repeat(theta[k : k + 1], 3, 0), t, share=0.2)


@pytest.mark.parametrize("d,q", [(12.0, 0.3), (0.2, 0.5), (1.2, 45.0)])
def test_lens_outside_the_refined_range(lib, d, q):
    theta = synth.prior_theta(5, 81)
    theta[:, 4], theta[:, 5] = d, q
    t = synth.uniform_epochs(211, 82)
    _check(lib.magnification(dev(theta), dev(t), "fp64").cpu().numpy(), theta, t)


def test_sources_at_the_lenses(lib):
    """Epochs with the source on the primary, on the secondary and within 1e-7 of them."""
    theta = np.array([[0.0, 20.0, 0.0, 0.0, 1.2, 0.05], [0.0, 20.0, 0.0, 0.5 * np.pi, 1.2, 0.05]])
    t = np.array([-24.0, -24.0 + 2e-6, -1e-6, 0.0, 1e-6, 24.0, 24.0 - 2e-6, 7.0])
    A = lib.magnification(dev(theta), dev(t), "fp64").cpu().numpy()
    A_ref, info = osb.magnification(theta, t, return_info=True)
    ok = (info["min_det"] >= 1e-3) & ~info["flag"]
    assert np.all(np.isfinite(A)) and ok.any()
    assert np.all(np.abs(A - A_ref)[ok] <= 1e-10 * A_ref[ok])
