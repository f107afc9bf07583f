"""The FP32 form where a power of the conductivity or the abscissa comes near
the ends of its range: very conductive layers under a high loop, and nearly
insulating ones.  Bound: the spectrum within 2^-17 of A_f, the forward tests'
component accuracy.  (It is for layers of some wavelength's thickness: under a
loop at 200 km insulating layers of 2 to 200 m are 1e-5 of one, and the FP32
recursion is 1e-5 of A_f off whatever its form, so that corner is left out.)"""
import numpy as np
import pytest

import oracle as O
from paper_2109_00661_gb300 import inputs as I
from parity_util import DELTA_S32, spectrum_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("height, radius", [(0.5, 0.2), (30.0, 13.0), (3000.0, 100.0), (200000.0, 1000.0)])
@pytest.mark.parametrize("lo, hi", [(6.0, 10.0), (-4.0, 8.0), (-9.0, -7.0)])
def test_ends_of_the_conductivity_range(height, radius, lo, hi):
    if height > 1e5 and hi < 0:
        pytest.skip("layers of a hundred-thousandth of a wavelength")
    import torch
    import paper_2109_00661_gb300 as L
    kw = dict(I.system_kwargs("sounding-g20-f40-k120"), height=height, loop_radius=radius)
    sysg = L.System(**kw)
    so = dict(I.oracle_system("sounding-g20-f40-k120"), h=height, a=radius)
    so["T"] = np.zeros((20, 40))
    models = I.random_models(48, seed=11, lmax=6, layers_max=6)
    models["logsig"] = np.random.default_rng(2).uniform(lo, hi, models["logsig"].shape)
    models = {k: (v if k == "nlayers" else np.float32(v).astype(np.float64)) for k, v in models.items()}
    _, ref, absh = O.forward(models, so, mode=O.HANKEL_RULE, want_imh=True, want_absh=True)
    for cutoff in (20.0, 0.0):
        sysg.set_depth_cutoff(cutoff)
        imh = L.spectrum_f32(sysg, I.to_torch(models, torch.float32)).cpu().numpy().astype(np.float64)
        assert spectrum_err(imh, ref, absh).max() < DELTA_S32
    _, grad = L.loglik_grad_f32(sysg, I.to_torch(models, torch.float32), np.full(20, 1e-9), 1e-11, 0.03)
    assert torch.isfinite(grad).all()
