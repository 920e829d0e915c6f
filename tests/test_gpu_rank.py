"""Ranking and reproduction at the sizes where the register / shuffle / shared-memory sort changes form
(elements per thread 1, 2, 4, 8; populations below a warp; odd sizes) and at both lane counts per
pairing, bit for bit against the oracle's generation; ties, NaN, infinities and signed zeros."""
import numpy as np
import pytest
import torch

from oracle import ea as oea

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_pop", [2, 3, 31, 33, 64, 1000, 1025, 2049, 4097, 8192])
def test_generation_sizes(lib, n_pop):
    rng = np.random.default_rng(n_pop)
    op = oea.EAParams(n_pop=n_pop, seed=9, stream=4)
    p = lib.params(n_pop=n_pop, seed=9)
    P0 = oea.init_population(n_pop, 6, op, 0)
    chi = np.round(rng.uniform(-2, 2, n_pop), 1)  # many ties, negative values, zeros of both signs
    chi[rng.integers(0, n_pop, max(1, n_pop // 9))] = -0.0
    chi[rng.integers(0, n_pop, max(1, n_pop // 11))] = np.nan
    chi[rng.integers(0, n_pop, max(1, n_pop // 13))] = np.inf
    P = torch.tensor(P0, device="cuda")
    state = lib.new_state_buffer("cuda")
    lib.ea_init(torch.empty_like(P), 6, p, 4, state)
    lib.ea_generation(P, torch.tensor(chi, device="cuda"), p, 4, 0, state)
    st = oea.new_state(op)
    ref = oea.generation(P0, chi, st, op, 0)
    assert np.allclose(P.cpu().numpy(), ref, rtol=0, atol=1e-15)


@pytest.mark.parametrize("n_pops,n_pop", [(3, 130), (40, 2048)])
def test_batch_equals_single_populations(lib, n_pops, n_pop):
    """Eight lanes per pairing (a few populations) and two (many) give the same genes bit for bit."""
    g = np.random.default_rng(n_pops)
    p = lib.params(n_pop=n_pop, seed=3)
    P0 = torch.tensor(g.uniform(size=(n_pops, n_pop, 6)), device="cuda")
    chi = torch.tensor(g.uniform(1, 9, n_pops * n_pop), device="cuda")
    states = torch.stack([lib.new_state_buffer("cuda") for _ in range(n_pops)])
    for k in range(n_pops):
        lib.ea_init(torch.empty_like(P0[k]), 6, p, k, states[k])
    P, S = P0.clone(), states.clone()
    lib.ea_generation_batch(P, chi, p, 0, 0, S)
    for k in {0, 1, n_pops - 1}:
        Q, T = P0[k].clone(), states[k].clone()
        lib.ea_generation(Q, chi[k * n_pop : (k + 1) * n_pop].contiguous(), p, k, 0, T)
        assert torch.equal(P[k], Q) and torch.equal(S[k], T)
