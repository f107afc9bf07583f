"""The double-precision form where its split and its functions part: batches on
either side of each cluster size, layer counts from one to the largest, odd
numbers of frequencies, gates past a warp, very thick layers (the exponential's
underflow) and very thin ones.  Bound: the spectrum within 1e-12 of A_f, the
forward tests' FP64 accuracy."""
import numpy as np
import pytest

import oracle as O
from paper_2109_00661_gb300 import inputs as I
from parity_util import DELTA_S64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("models, F, K, G, lmax, logh", [
    (1, 40, 120, 20, 20, None), (3, 41, 121, 33, 1, None), (7, 2, 8, 1, 5, None), (310, 9, 33, 20, 4, None),
    (700, 17, 40, 64, 6, None), (1300, 5, 24, 20, 3, None), (2500, 3, 16, 20, 2, None), (12, 40, 120, 20, 6, 4.5),
    (12, 40, 120, 20, 6, -2.0)])
def test_double_form_edges(models, F, K, G, lmax, logh):
    import torch
    import paper_2109_00661_gb300 as L
    times = np.logspace(-5, -2, G)
    sysg = L.System(loop_radius=13.0, height=30.0, n_freq=F, gate_times=times, n_hankel=K)
    so = dict(I.oracle_system("sounding-g20-f40-k120"), times=times, K=K,
              freqs=np.exp(np.linspace(0.0, np.log(1e7), F)))
    so["T"] = O.tmatrix(so["freqs"], so["times"])
    m = I.random_models(models, seed=models, lmax=lmax, layers_max=lmax)
    if logh is not None:
        m["logh"] = np.full_like(m["logh"], logh)
    y, ref, absh = O.forward(m, so, mode=O.HANKEL_RULE, want_imh=True, want_absh=True)
    gates, imh = L.forward_f64(sysg, I.to_torch(m, torch.float64), want_imh=True)
    assert np.max(np.abs(imh.cpu().numpy() - ref) / absh) < DELTA_S64
    # the transform of the spectrum, in FP64 (the system's own table)
    T = sysg.tables()[3]
    assert np.max(np.abs(gates.cpu().numpy() - imh.cpu().numpy() @ T.T) / (np.abs(imh.cpu().numpy()) @ np.abs(T).T)) < 1e-14
    y_obs = y[0]
    ll = L.loglik_f64(sysg, I.to_torch(m, torch.float64), y_obs, 1e-11, 0.03).cpu().numpy()
    g = gates.cpu().numpy()
    v = 1e-22 + (0.03 * g) ** 2
    want = -0.5 * np.sum((y_obs - g) ** 2 / v + np.log(2 * np.pi * v), axis=1)
    assert np.allclose(ll, want, rtol=1e-12)
