"""The FP32 log-likelihood of posterior populations against 64 bits, and the
gate transform it rests on.

Models about one earth share their roundings, so the population's error does
not average out, and the late gates (which cancel to about a hundredth of
their terms) amplify it.  The bars are derived from the inputs:
  * log-likelihood: an FP32 chain whose spectrum is exact but for one rounding
    to a float, with T rounded to a float and a serial FP32 dot product, has
    some error on these models; the kernel, which has the recursion's error
    besides, has to stay under 3/4 of it (root mean square over all models).
  * gates: the kernel's spectrum is a float pair of which the caller sees the
    rounded value, so a gate is T x (that value) to sum |T| |x| 2^-24, plus
    its own rounding; a plain FP32 sum's error grows with the frequencies."""
import numpy as np
import pytest

import oracle as O
from paper_2109_00661_gb300 import inputs as I
from parity_util import oracle_system

pytestmark = pytest.mark.gpu
EPS_AN = 1e-11


def _posterior(P, lmax, seed, spread=1.0):
    """About one earth of moderate conductivity, weakly chargeable from its third layer down."""
    rng = np.random.default_rng(seed)
    at = np.arange(lmax)[None, :]
    n = lambda sd: spread * sd * rng.standard_normal((P, lmax))  # noqa: E731
    m = dict(nlayers=rng.integers(1, lmax + 1, size=P).astype(np.int8), logsig=-1.5 + 0.3 * np.sin(1.3 * at) + n(0.1),
             logh=1.2 + n(0.1), m=np.where(at >= 2, np.clip(0.15 + n(0.03), 0, 1), 0.0), logtau=-3.0 + n(0.1),
             c=np.clip(0.5 + n(0.03), 0.1, 1.0))
    return {k: v if k == "nlayers" else np.float32(v).astype(np.float64) for k, v in m.items()}


def _fp32_chain(imh, T):
    """Gates of an exact spectrum rounded once, T rounded, fused FP32 multiply-adds in order."""
    x, t = np.float32(imh), np.float32(T)
    acc = np.zeros((x.shape[0], t.shape[0]), np.float32)
    for j in range(t.shape[1]):  # an FP32 product is exact in 64 bits
        acc = np.float32(acc.astype(np.float64) + x[:, j:j + 1].astype(np.float64) * t[None, :, j].astype(np.float64))
    return acc.astype(np.float64)


@pytest.mark.parametrize("name, lmax, P, draws", [
    ("sounding-g20-f40-k120", 8, 1, 96), ("sounding-g20-f40-k120", 8, 16, 8), ("sounding-g20-f40-k120", 8, 256, 6),
    ("sounding-g20-f40-k120", 3, 256, 6), ("forward-g30-f60-k200", 10, 16, 8), ("forward-g30-f60-k200", 10, 256, 6),
    ("forward-g30-f60-k200", 14, 700, 2)])
def test_loglik_of_a_posterior_population(name, lmax, P, draws):
    import torch
    import paper_2109_00661_gb300 as L
    sysg, so = L.System(**I.system_kwargs(name)), oracle_system(name)
    earth = _posterior(1, lmax, 0, spread=0.0)
    earth["nlayers"][:] = lmax
    truth = O.forward(earth, so, mode=O.HANKEL_RULE)[0]
    here = chain = 0.0
    for seed in range(draws):
        models = _posterior(P, lmax, 1 + seed)
        y = I.noisy(truth, seed=seed, eps_an=EPS_AN)
        gates, imh = O.forward(models, so, mode=O.HANKEL_RULE, want_imh=True)
        ref = O.loglik(gates, y, EPS_AN, I.EPS_MN)
        got = L.loglik_f32(sysg, I.to_torch(models, torch.float32), y, EPS_AN, I.EPS_MN).cpu().numpy()
        here += np.sum((got - ref) ** 2)
        chain += np.sum((O.loglik(_fp32_chain(imh, so["T"]), y, EPS_AN, I.EPS_MN) - ref) ** 2)
    assert np.sqrt(here) < 0.75 * np.sqrt(chain), np.sqrt(here / chain)


@pytest.mark.parametrize("G, F, K, lmax", [(1, 2, 8, 1), (1, 40, 120, 8), (20, 3, 120, 8), (31, 41, 121, 3),
                                           (32, 40, 120, 20), (33, 57, 163, 9), (64, 128, 512, 20), (64, 5, 9, 2)])
def test_gates_are_the_transform_of_the_spectrum(G, F, K, lmax):
    import torch
    import paper_2109_00661_gb300 as L
    sysg = L.System(n_freq=F, gate_times=np.logspace(-5, -2, G) if G > 1 else [1e-3], n_hankel=K)
    T = sysg.tables()[3]
    models = I.to_torch(I.random_models(37, seed=G + F, lmax=lmax, layers_max=lmax), torch.float32)
    gates, imh = L.forward_f32(sysg, models, want_imh=True)
    gates, imh = gates.cpu().numpy().astype(np.float64), imh.cpu().numpy().astype(np.float64)
    bound = 2.0 ** -24 * (np.abs(imh) @ np.abs(T).T + np.abs(gates)) * (1 + 1e-3)
    assert np.all(np.abs(gates - imh @ T.T) <= bound)
