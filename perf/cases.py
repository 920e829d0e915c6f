"""Performance cases: the work a user of the fitter has it do, through its public entry points.

A case is a dict of plain values; ``kind`` names the entry point, the rest its sizes and options.
Inputs come from the seed alone: parameter rows, epochs and noise from the repository's synthetic
workloads (``synth``), observed fluxes from the reference magnification below, which is plain
torch in 64 bits and shares no code with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1208_4830_gb300 import sblm, synth

DEV = "cuda"

# gene domains of the sweep (wide enough for the trajectories re-aimed at caustics)
SWEEP_LO = np.array([-600.0, 5.0, 0.0, 0.0, 0.3, -4.0])
SWEEP_HI = np.array([600.0, 100.0, 8.0, 2.0 * np.pi, 3.0, 0.0])

# floating-point operations one magnification cannot do without: the quintic's coefficients (123),
# one correction of each of five roots from its neighbour's (value and derivative of the quintic
# 80, correction 20), the lens equation and its Jacobian at each root (60), the sum (12)
MAG_FLOP = 123 + 5 * (80 + 20 + 60) + 12

# proposal network: layers (fan in, fan out), output positions of the four convolutions
CNN_LAYERS = ((10, 64), (320, 64), (320, 64), (320, 64), (2048, 128), (128, 12))
CNN_POSITIONS = (256, 128, 64, 32, 1, 1)
CNN_PARAMS = sum((k + 1) * n for k, n in CNN_LAYERS)
CNN_FORWARD_FLOP = sum(2 * p * k * n for p, (k, n) in zip(CNN_POSITIONS, CNN_LAYERS))
# backward: weight and input gradients (the first layer has no input gradient)
CNN_STEP_FLOP = 3 * CNN_FORWARD_FLOP - 2 * 256 * 10 * 64


# ------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------
def listed():
    return [
        # the model curve of one event (a truth, a fitted best): the smallest call there is
        dict(name="curve_fp64", kind="magnification", n_cand=1, n_ep=400, precision="fp64"),
        # a library of template curves, odd sizes
        dict(name="templates_mixed", kind="magnification", n_cand=2999, n_ep=509, precision="mixed"),
        # fitness of the paper's population (1000 rows) against a 100-point curve, default precision:
        # one generation of an EA driven from the host
        dict(name="paper_population_mixed", kind="chi2_genes", n_cand=1000, n_ep=100, precision="mixed"),
        # the benchmark's step without its operators: 32 populations of 4096 on a 2000-epoch curve
        dict(name="sweep_mixed", kind="chi2_genes", n_cand=131072, n_ep=2000, precision="mixed"),
        # the forward sweep in full FP64 (the arithmetic of the plain FP64 fitter)
        dict(name="sweep_fp64", kind="chi2", n_cand=4096, n_ep=2000, precision="fp64"),
        # blended events (Section 4.4): chi^2 with the blending fraction profiled out, ragged sizes
        dict(name="blend_mixed", kind="chi2_blend", n_cand=997, n_ep=487, precision="mixed"),
        # the EA operators of 32 populations of 4096 (the other half of the benchmark's step)
        dict(name="generation_32x4096", kind="generation", n_pops=32, n_pop=4096),
        # one whole fit of the single-lightcurve configuration: N_pop 64 x 100 generations, FP64
        dict(name="fit_fp64", kind="fit", n_ep=400, n_pop=64, n_gen=100, precision="fp64"),
        # batched fits of held-out curves of uneven length, one curve per SM, first generations
        dict(name="fit_batch_mixed", kind="fit_batch", n_lc=152, n_lo=300, n_hi=700, n_pop=1024, n_gen=6,
             precision="mixed"),
        # amoeba fine-tuning of many solutions
        dict(name="polish_mixed", kind="polish", n_lc=64, n_ep=500, maxfev=200, precision="mixed"),
        # loss and gradients of the proposal network at its default batch
        dict(name="proposal_gradient", kind="cnn_gradient", batch=256),
        # training steps of the proposal network at the benchmark's batch (generator, network, AdamW)
        dict(name="proposal_training", kind="cnn_train", batch=1024, n_run=8),
    ]


def _log(rng, lo, hi):
    """An integer whose logarithm is uniform over [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["magnification", "magnification", "chi2", "chi2", "chi2_genes", "chi2_genes", "chi2_blend",
                       "generation", "fit", "fit_batch", "polish", "cnn_gradient", "cnn_train"])
    if kind in ("magnification", "chi2", "chi2_genes", "chi2_blend"):
        precision = rng.choice(["fp64", "mixed", "fp32"])
        n_ep = _log(rng, 100, 3000)
        # magnifications write 8 bytes per value; FP64 is sixty times dearer than FP32
        most = {"fp64": 4_000_000, "mixed": 32_000_000, "fp32": 32_000_000}[precision]
        n_cand = _log(rng, 1 if kind == "magnification" else 32, max(64, most // n_ep))
        return dict(kind=kind, n_cand=n_cand, n_ep=n_ep, precision=precision)
    if kind == "generation":
        n_pop = _log(rng, 64, 8192)
        return dict(kind=kind, n_pops=_log(rng, 1, max(1, 131072 // n_pop)), n_pop=n_pop)
    if kind == "fit":
        precision = rng.choice(["fp64", "mixed"])
        return dict(kind=kind, n_ep=_log(rng, 100, 1000), n_pop=_log(rng, 64, 1000 if precision == "mixed" else 200),
                    n_gen=rng.randint(10, 60), precision=precision)
    if kind == "fit_batch":
        precision = rng.choice(["mixed", "mixed", "mixed+blend", "fp64"])
        n_lo = _log(rng, 100, 500)
        return dict(kind=kind, n_lc=_log(rng, 16, 304), n_lo=n_lo, n_hi=n_lo + rng.randint(0, 400),
                    n_pop=_log(rng, 64, 1024 if precision != "fp64" else 128), n_gen=rng.randint(3, 8),
                    precision=precision)
    if kind == "polish":
        return dict(kind=kind, n_lc=_log(rng, 1, 304), n_ep=_log(rng, 100, 1000), maxfev=_log(rng, 30, 300),
                    precision=rng.choice(["mixed", "mixed+blend", "fp64"]))
    if kind == "cnn_gradient":
        return dict(kind=kind, batch=_log(rng, 1, 2048))
    return dict(kind=kind, batch=_log(rng, 32, 1024), n_run=rng.randint(1, 8))


# ------------------------------------------------------------------------------------------
# reference magnification: quintic roots by Aberth iteration in 64 bits, torch on the GPU
# ------------------------------------------------------------------------------------------
def _poly_mul(a, b):
    out = [None] * (len(a) + len(b) - 1)
    for i, x in enumerate(a):
        for j, y in enumerate(b):
            out[i + j] = x * y if out[i + j] is None else out[i + j] + x * y
    return out


def _norm2(z):
    return z.real * z.real + z.imag * z.imag


def _point_magnification(zeta, d, q):
    """Magnification at source positions zeta (complex128 [n]) of lenses (d, q) (float64 [n])."""
    one = torch.ones_like(zeta)
    zero = torch.zeros_like(zeta)
    dc, qc, zb = d.to(zeta.dtype), q.to(zeta.dtype), zeta.conj().resolve_conj()
    D = [zero, -dc, one]  # z (z - d), ascending powers
    N = [-dc, one + qc - zb * dc, zb]  # conj(zeta) D + (1 + q) z - d
    M = [n - dc * x for n, x in zip(N, D)]
    p = _poly_mul([-zeta, one], _poly_mul(N, M))
    for poly, m in ((_poly_mul(D, M), one), (_poly_mul(D, N), qc)):
        p = [a - m * poly[k] if k < len(poly) else a for k, a in enumerate(p)]
    # five starting points around the roots' centroid
    centre = -0.2 * p[4] / p[5]
    v = p[5]
    for k in (4, 3, 2, 1, 0):
        v = v * centre + p[k]
    radius = torch.pow(_norm2(v / p[5]), 0.1)
    ang = torch.arange(5, dtype=torch.float64, device=zeta.device) * (2.0 * math.pi / 5.0) + 0.4
    spokes = torch.complex(torch.cos(ang), torch.sin(ang))[:, None]
    z = centre[None, :] + radius[None, :] * spokes
    for it in range(96):
        f, df = p[5].expand_as(z), torch.zeros_like(z)
        for k in (4, 3, 2, 1, 0):
            df = df * z + f
            f = f * z + p[k]
        newton = f / df
        near = torch.zeros_like(z)
        for s in range(1, 5):
            near = near + 1.0 / (z - torch.roll(z, s, 0))
        w = newton / (1.0 - newton * near)
        w = torch.where(torch.isfinite(w.real) & torch.isfinite(w.imag), w, torch.zeros_like(w))
        z = z - w
        if it % 8 == 7 and bool((_norm2(w) <= 1e-28 * _norm2(z)).all()):
            break
    gap = torch.full(z.shape, math.inf, dtype=torch.float64, device=z.device)
    for s in range(1, 5):
        gap = torch.minimum(gap, _norm2(z - torch.roll(z, s, 0)))
    z0 = z
    for it in range(5):  # Newton steps on the lens equation, then its residual
        zc = z.conj().resolve_conj()
        a, b = 1.0 / zc, 1.0 / (dc - zc)
        f = z - a + qc * b - zeta
        K = a * a + qc * b * b
        det = 1.0 - _norm2(K)
        if it == 4:
            break
        step = (K * f.conj().resolve_conj() - f) / det
        z = torch.where(_norm2(z + step - z0) <= 0.25 * gap, z + step, z)
    size = _norm2(z).sqrt() + _norm2(a).sqrt() + q * _norm2(b).sqrt() + _norm2(zeta).sqrt()
    res = _norm2(f).sqrt() / size
    order = torch.argsort(torch.nan_to_num(res, nan=math.inf), 0)
    rank = torch.empty_like(order)
    rank.scatter_(0, order, torch.arange(5, device=z.device)[:, None].expand_as(order))
    five = torch.nan_to_num(res, nan=math.inf).amax(0) <= 1e-9
    image = (rank < 3) | five[None, :]
    return torch.where(image, 1.0 / det.abs(), torch.zeros_like(det)).sum(0)


def _magnification(theta, t):
    """A [n, m] of parameter rows theta [n, 6] at epochs t [m] or [n, m], float64 on the GPU."""
    n, m = theta.shape[0], t.shape[-1]
    t = t.expand(n, m) if t.ndim == 1 else t
    out = torch.empty(n, m, dtype=torch.float64, device=theta.device)
    rows = max(1, 1_000_000 // m)
    for i in range(0, n, rows):
        th = theta[i : i + rows]
        tau = (t[i : i + rows] - th[:, 0:1]) / th[:, 1:2]
        sa, ca = torch.sin(th[:, 3:4]), torch.cos(th[:, 3:4])
        zeta = torch.complex(tau * sa + th[:, 2:3] * ca, th[:, 2:3] * sa - tau * ca)
        d, q = th[:, 4:5].expand_as(tau), th[:, 5:6].expand_as(tau)
        out[i : i + rows] = _point_magnification(zeta.reshape(-1), d.reshape(-1), q.reshape(-1)).reshape(tau.shape)
    return out


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _cuda(x):
    return torch.as_tensor(x, device=DEV)


def _rows(n, seed):
    """Candidate rows of the sweep: its priors, 10% of the trajectories through a caustic."""
    theta = synth.prior_theta(n, seed)
    return synth.force_caustics(theta, 0.1, seed + 1)[0]


def _curve(n_ep, seed, sigma_frac=0.01):
    """(t, flux, sigma) of one prior draw's lightcurve with noise of 1% of the flux."""
    t = _cuda(synth.uniform_epochs(n_ep, seed + 2))
    truth = _cuda(synth.prior_theta(1, seed + 3))
    A = _magnification(truth, t)[0]
    z = _cuda(np.random.Generator(np.random.Philox(seed + 4)).standard_normal(n_ep))
    sigma = sigma_frac * A
    return t, A + sigma * z, sigma


def _genes(theta, lo, hi):
    a = np.array(theta, copy=True)
    a[:, 5] = np.log10(a[:, 5])
    return (a - lo) / (hi - lo)


def _batch(n_lc, n_lo, n_hi, seed):
    """Concatenated held-out curves of n_lo..n_hi epochs each (2% noise) with their truths."""
    g = np.random.Generator(np.random.Philox(seed + 5))
    n = g.integers(n_lo, n_hi + 1, n_lc)
    b = synth.heldout_batch(n_lc, seed=seed, n_ep=int(n.max()))
    t = b.t.reshape(n_lc, -1)
    z = b.z.reshape(n_lc, -1)
    A = _magnification(_cuda(b.truth), _cuda(t))
    keep = np.zeros(t.shape, dtype=bool)
    for i in range(n_lc):  # a random subset of the epochs, in order
        keep[i, g.choice(t.shape[1], size=int(n[i]), replace=False)] = True
    k = _cuda(keep.ravel())
    sigma = 0.02 * A.reshape(-1)
    flux = A.reshape(-1) + sigma * _cuda(z.ravel())
    offsets = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
    return dict(t=_cuda(t.ravel())[k].contiguous(), flux=flux[k].contiguous(), sigma=sigma[k].contiguous(),
                offsets=offsets, truth=b.truth)


def _network(seed):
    """FP32 weights like an initialised network's: per layer W [fan in][fan out] and its bias."""
    g = torch.Generator().manual_seed(seed)
    parts = []
    for k, n in CNN_LAYERS:
        parts += [torch.randn(k * n, generator=g) * math.sqrt((2.0 if n != 12 else 0.01) / k),
                  0.02 * torch.randn(n, generator=g)]
    return torch.cat(parts).to(DEV)


def _network_batch(batch, seed):
    """Normalised curves [B, 256, 2] (flux, mask) and targets [B, 6] of the training prior's ranges."""
    g = torch.Generator().manual_seed(seed + 1)
    s = torch.linspace(-1.0, 1.0, 256)
    t0 = torch.rand(batch, 1, generator=g) * 0.8 - 0.4
    tE = torch.exp(torch.rand(batch, 1, generator=g) * 3.6 - 3.2)
    u0 = torch.rand(batch, 1, generator=g)
    u2 = u0 * u0 + ((s[None, :] - t0) / tE) ** 2
    A = (u2 + 2.0) / torch.sqrt(u2 * (u2 + 4.0)).clamp_min(1e-3)
    F = A * (1.0 + 0.02 * torch.randn(batch, 256, generator=g))
    mask = (torch.rand(batch, 256, generator=g) >= 0.7 * torch.rand(batch, 1, generator=g)).float()
    med = F.median(1, keepdim=True).values
    x = torch.stack([torch.asinh(10.0 * (F / med - 1.0)) / 3.0 * mask, mask], 2)
    y = torch.cat([t0, torch.log(tE), u0, torch.rand(batch, 1, generator=g),
                   torch.rand(batch, 1, generator=g) * 2.3 - 1.2, -4.0 * torch.rand(batch, 1, generator=g)], 1)
    return x.contiguous().to(DEV), y.contiguous().to(DEV)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind in ("magnification", "chi2", "chi2_genes", "chi2_blend"):
        theta = _rows(case["n_cand"], seed)
        s["theta"] = _cuda(theta)
        if kind == "magnification":
            s["t"] = _cuda(synth.uniform_epochs(case["n_ep"], seed + 2))
        else:
            s["t"], s["flux"], s["sigma"] = _curve(case["n_ep"], seed)
        if kind == "chi2_blend":
            f = 0.3 + 0.7 * np.random.Generator(np.random.Philox(seed + 6)).uniform()
            s["flux"] = f * s["flux"] + (1.0 - f)
        if kind == "chi2_genes":
            s["P"] = _cuda(_genes(theta, SWEEP_LO, SWEEP_HI))
        return s
    if kind == "generation":
        n_pops, n_pop = case["n_pops"], case["n_pop"]
        g = np.random.Generator(np.random.Philox(seed))
        s["P"] = _cuda(g.uniform(size=(n_pops, n_pop, 6)))
        s["chi2"] = _cuda(np.exp(g.normal(10.0, 2.0, size=n_pops * n_pop)))  # wide, as a first population's
        s["params"] = sblm.params(n_pop=n_pop, n_gen=100, seed=seed)
        s["states"] = torch.stack([sblm.new_state_buffer(DEV) for _ in range(n_pops)])
        for k in range(n_pops):
            sblm.ea_init(torch.empty_like(s["P"][k]), 6, s["params"], k, s["states"][k])
        s["P_next"], s["states_next"] = torch.empty_like(s["P"]), torch.empty_like(s["states"])
        return s
    if kind == "fit":  # one observed curve, host arrays as a user reads them from a file
        t, flux, sigma = _curve(case["n_ep"], seed)
        s["t"], s["flux"], s["sigma"] = t.cpu().numpy(), flux.cpu().numpy(), sigma.cpu().numpy()
        s["params"] = sblm.params(n_pop=case["n_pop"], n_gen=case["n_gen"], precision=case["precision"], seed=seed)
        return s
    if kind in ("fit_batch", "polish"):
        s.update(_batch(case["n_lc"], case.get("n_lo", case.get("n_ep")), case.get("n_hi", case.get("n_ep")), seed))
        if kind == "fit_batch":
            s["params"] = sblm.params(n_pop=case["n_pop"], n_gen=case["n_gen"], precision=case["precision"], seed=seed)
        else:  # starts near the truths, as an EA leaves them
            g = np.random.Generator(np.random.Philox(seed + 7))
            genes = _genes(s["truth"], synth.FIT_LO, synth.FIT_HI)
            s["genes"] = _cuda(np.clip(genes + g.normal(0.0, 0.01, genes.shape), 0.0, 1.0))
        return s
    s["w0"] = _network(seed)
    if kind == "cnn_gradient":
        s["x"], s["y"] = _network_batch(case["batch"], seed)
        return s
    s["params"] = sblm.cnn_train_params(batch=case["batch"], n_steps=1024, warmup=100, seed=seed)
    s["w"], s["state"] = torch.empty_like(s["w0"]), torch.empty(2 * CNN_PARAMS, dtype=torch.float32, device=DEV)
    return s


def run(s):
    kind, c = s["kind"], s["case"]
    if kind == "magnification":
        return sblm.magnification(s["theta"], s["t"], c["precision"])
    if kind == "chi2":
        return sblm.chi2(s["theta"], s["t"], s["flux"], s["sigma"], c["precision"])
    if kind == "chi2_genes":
        return sblm.chi2_genes(s["P"], s["t"], s["flux"], s["sigma"], SWEEP_LO, SWEEP_HI, c["precision"])
    if kind == "chi2_blend":
        return sblm.chi2_blend(s["theta"], s["t"], s["flux"], s["sigma"], c["precision"])
    if kind == "generation":  # on a copy: the evaluated populations are kept, as Appendix A returns them
        s["P_next"].copy_(s["P"])
        s["states_next"].copy_(s["states"])
        sblm.ea_generation_batch(s["P_next"], s["chi2"], s["params"], 0, 0, s["states_next"])
        return s["P_next"], s["states_next"]
    if kind == "fit":
        return sblm.fit(s["t"], s["flux"], s["sigma"], synth.FIT_LO, synth.FIT_HI, s["params"], trace=True)
    if kind == "fit_batch":
        return sblm.fit_batch(s["t"], s["flux"], s["sigma"], s["offsets"], synth.FIT_LO, synth.FIT_HI, s["params"])
    if kind == "polish":
        return sblm.polish_batch(s["t"], s["flux"], s["sigma"], s["offsets"], synth.FIT_LO, synth.FIT_HI, s["genes"],
                                 c["maxfev"], c["precision"])
    if kind == "cnn_gradient":
        return sblm.cnn_loss_grad(s["w0"], s["x"], s["y"])
    s["w"].copy_(s["w0"])  # training starts from the same weights and moments on every pass
    s["state"].zero_()
    losses = sblm.cnn_train(s["w"], s["state"], s["params"], 0, c["n_run"])
    return s["w"], s["state"], losses


def work(case):
    kind = case["kind"]
    if kind in ("magnification", "chi2", "chi2_genes", "chi2_blend"):
        n, m = case["n_cand"], case["n_ep"]
        out = {"magnification": 8 * n * m, "chi2_blend": 16 * n}.get(kind, 8 * n)
        return {"bytes": 48 * n + 8 * m * (1 if kind == "magnification" else 3) + out, "flops": MAG_FLOP * n * m}
    if kind == "generation":
        rows = case["n_pops"] * case["n_pop"]
        # genes and fitness in, genes out; per gene a weighted pair, a creep step and a jump
        return {"bytes": rows * (48 + 8 + 48), "flops": rows * 6 * 30}
    if kind == "fit":
        m = case["n_ep"]
        return {"bytes": 24 * m + 56 + 32 * case["n_gen"], "flops": MAG_FLOP * m * case["n_pop"] * case["n_gen"]}
    if kind == "fit_batch":
        m = case["n_lc"] * (case["n_lo"] + case["n_hi"]) / 2
        return {"bytes": 24 * m + 56 * case["n_lc"], "flops": MAG_FLOP * m * case["n_pop"] * case["n_gen"]}
    if kind == "polish":
        m = case["n_lc"] * case["n_ep"]
        return {"bytes": 24 * m + 104 * case["n_lc"], "flops": MAG_FLOP * m * case["maxfev"]}
    B = case["batch"]
    if kind == "cnn_gradient":
        return {"bytes": 4 * (2 * CNN_PARAMS + B * (512 + 6)), "flops": CNN_STEP_FLOP * B}
    return {"bytes": 4 * 6 * CNN_PARAMS, "flops": case["n_run"] * B * (CNN_STEP_FLOP + 256 * MAG_FLOP)}


# ------------------------------------------------------------------------------------------
# 64-bit values
# ------------------------------------------------------------------------------------------
def _exact_network(w, x, y):
    """(loss, gradient) of the proposal network in float64."""
    w = w.double().requires_grad_(True)
    h, at = x.double(), 0
    for layer, (k, n) in enumerate(CNN_LAYERS):
        W, b = w[at : at + k * n].reshape(k, n), w[at + k * n : at + (k + 1) * n]
        at += (k + 1) * n
        if layer < 4:  # kernel 5, padding 2, stride 1 then 2: windows [B, positions, 5, channels]
            pad = torch.nn.functional.pad(h, (0, 0, 2, 2))
            h = pad.unfold(1, 5, 1 if layer == 0 else 2).transpose(2, 3)
            h = h.reshape(h.shape[0], h.shape[1], -1) @ W + b
        else:
            h = h.reshape(h.shape[0], -1) @ W + b
        if layer < 5:
            h = torch.nn.functional.gelu(h)
    mu, s = h[:, :6], h[:, 6:]
    loss = (0.5 * ((y.double() - mu) ** 2 * torch.exp(-s) + s)).sum(1).mean()
    (grad,) = torch.autograd.grad(loss, w)
    return float(loss.detach()), grad


def exact(case, seed):
    kind = case["kind"]
    if kind in ("magnification", "chi2", "chi2_genes", "chi2_blend"):
        # over 20 seconds; or plain FP32, which loses image pairs next to caustics: 64 bits say nothing
        # about it there
        if case["n_cand"] * case["n_ep"] > 40_000_000 or case["precision"] == "fp32":
            return None
        s = prepare(case, seed)
        A = _magnification(s["theta"], s["t"])
        if kind == "magnification":
            return A
        if kind != "chi2_blend":
            return (((s["flux"] - A) / s["sigma"]) ** 2).sum(1)
        wt, a, b = s["sigma"] ** -2, A - 1.0, s["flux"] - 1.0
        f = ((wt * a * b).sum(1) / (wt * a * a).sum(1)).clamp(1e-3, 1.0)
        return (wt * (b - f[:, None] * a) ** 2).sum(1), f
    if kind == "cnn_gradient":
        s = prepare(case, seed)
        return _exact_network(s["w0"], s["x"], s["y"])
    return None  # whole searches and training runs
