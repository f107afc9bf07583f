"""The double-precision spectrum keeps its digits where conductive layers lie
under resistive ones, also for a small loop near the ground, whose abscissae
hardly see them.  Bound, of A_f = sum_k |w_k| |R_0|: some ten rounded
operations in each of up to ten layers on either side, 2 x 100 x 2^-53 =
2.2e-14, rounded up to 2^-45."""
import numpy as np
import pytest

import oracle as O
from paper_2109_00661_gb300 import inputs as I
from parity_util import spectrum_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("height, radius, f_max", [(0.5, 0.2, 1e5), (5.0, 2.0, 1e5), (30.0, 13.0, 1e7)])
@pytest.mark.parametrize("kind", ["random", "contrast", "sea ice"])
def test_spectrum_of_contrasting_layers(height, radius, f_max, kind):
    import torch
    import paper_2109_00661_gb300 as L
    kw = dict(I.system_kwargs("sounding-g20-f40-k120"), height=height, loop_radius=radius, f_max_hz=f_max)
    sysg = L.System(**kw)
    so = dict(I.oracle_system("sounding-g20-f40-k120"), h=height, a=radius,
              freqs=np.exp(np.linspace(np.log(I.F_MIN_HZ), np.log(f_max), 40)))
    so["T"] = np.zeros((20, 40))
    if kind == "contrast":
        models = I.contrast_models(24, seed=5)
    else:
        models = I.random_models(24, seed=5, lmin=2)
        if kind == "sea ice":  # a resistive cover (down to 1e-9 S/m) on sea water
            rng = np.random.default_rng(1)
            models["logsig"] = rng.uniform(-9.0, -7.0, models["logsig"].shape)
            models["logsig"][np.arange(24), models["nlayers"] - 1] = np.log10(4.0)
            models["m"][:] = 0.0
    _, ref, absh = O.forward(models, so, mode=O.HANKEL_RULE, want_imh=True, want_absh=True)
    imh = L.forward_f64(sysg, I.to_torch(models, torch.float64), want_imh=True)[1].cpu().numpy()
    assert spectrum_err(imh, ref, absh).max() < 2.0 ** -45
