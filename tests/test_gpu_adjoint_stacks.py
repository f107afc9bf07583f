"""The gradient on twenty thick alternating layers: a 10^3 conductivity contrast drives
the downgoing amplitude of some items beyond the adjoint kernel's unscaled range
(|D_0|^2 > 10^30, both sweeps are then scaled layer by layer), thin layers of a
small contrast stay within it.  Bars: those of the adjoint tests (test_gpu_adjoint.check)."""
import numpy as np
import pytest

import oracle as O
from paper_2109_00661_gb300 import inputs as I
from parity_util import oracle_ref, oracle_system
from test_gpu_adjoint import NAME, check, gbounds

pytestmark = pytest.mark.gpu


def _stacks(P, resistive, conductive, decades, seed):
    rng = np.random.default_rng(seed)
    L = 20
    odd = np.arange(L) % 2 == 1
    m = dict(nlayers=np.full(P, L, dtype=np.int8),
             logsig=np.where(odd, -2.0 + decades / 2, -2.0 - decades / 2) + rng.uniform(-0.2, 0.2, (P, L)),
             logh=np.log10(np.where(odd, conductive, resistive)) + rng.uniform(-0.1, 0.1, (P, L)),
             m=rng.uniform(0.05, 0.3, (P, L)), logtau=rng.uniform(-3.3, -2.7, (P, L)), c=rng.uniform(0.3, 0.9, (P, L)))
    return {k: (v if k == "nlayers" else np.float32(v).astype(np.float64)) for k, v in m.items()}


def _d0(models, s):
    """max and min over items of |D_0| of the first model in FP64 (D doubles per
    interface, as the kernel carries it)."""
    lam = np.asarray(O.hankel_rule(s["K"], s["a"], s["h"])[0])[None, :]
    om = 2 * np.pi * np.asarray(s["freqs"], dtype=np.float64)[:, None]
    sig, h = 10.0 ** models["logsig"][0], 10.0 ** models["logh"][0]
    w = [np.sqrt(2 * (lam**2 + 1j * om * 4e-7 * np.pi * v)) for v in sig]
    e, hh = 1.0, w[-1]
    for n in range(len(w) - 2, -1, -1):
        g = 2 * hh / w[n]
        N, D = e - g / 2, e + g / 2
        P = N * np.exp(-np.sqrt(2) * w[n] * h[n])
        e, hh = D + P, w[n] * (D - P)
    d = np.abs(e + hh / (np.sqrt(2) * lam))
    return d.max(), d.min()


@pytest.mark.parametrize("resistive, conductive, decades", [(300.0, 100.0, 3.0), (2.0, 1.0, 1.0)])
def test_alternating_stacks(resistive, conductive, decades):
    import torch
    import paper_2109_00661_gb300 as L
    sysg, s = L.System(**I.system_kwargs(NAME)), oracle_system(NAME)
    sysg.set_depth_cutoff(0.0)
    models = _stacks(4, resistive, conductive, decades, seed=5)
    hi, lo = _d0(models, s)
    assert lo < 1e15 and (hi > 1e15) == (decades > 1)
    y_model, _, _, kap = oracle_ref(models, NAME)
    y_obs = I.noisy(y_model[0], seed=1)
    _, g_ref = O.loglik_grad_fd(models, s, y_obs, I.EPS_AN, I.EPS_MN)
    _, g = L.loglik_grad_f32(sysg, I.to_torch(models, torch.float32), y_obs, I.EPS_AN, I.EPS_MN)
    _, J = O.forward_jacobian_fd(models, s)
    check(g.cpu().numpy().astype(np.float64), g_ref, "alternating stacks", *gbounds(y_model, J, y_obs, kap, sysg.F))
