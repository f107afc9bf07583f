"""The double-precision form where an exponent is not a number: a NaN parameter
of either sign (a host's 0 / 0 has the sign bit set) gives NaN, as does an
infinite thickness, for that model only."""
import numpy as np
import pytest

from paper_2109_00661_gb300 import inputs as I

pytestmark = pytest.mark.gpu

NEGATIVE_NAN = np.array([0xFFF8000000000000], dtype=np.uint64).view(np.float64)[0]
LOW_BITS_NAN = np.array([0xFFF8000012345600], dtype=np.uint64).view(np.float64)[0]


@pytest.mark.parametrize("name", ["logsig", "logh", "m", "logtau", "c"])
@pytest.mark.parametrize("value", [np.nan, NEGATIVE_NAN, LOW_BITS_NAN, np.inf])
def test_not_a_number_stays(name, value):
    import torch
    import paper_2109_00661_gb300 as L
    if np.isinf(value) and name != "logh":
        pytest.skip("the thickness alone forms an exponent of -inf")
    sysg = L.System(**I.system_kwargs("sounding-g20-f40-k120"))
    y = np.full(20, 1e-9)
    models = I.random_models(12, seed=4, lmax=5, lmin=5, layers_max=5)
    ref = L.loglik_f64(sysg, I.to_torch(models, torch.float64), y, 1e-11, 0.03).cpu().numpy()
    bad = [2, 5, 9]
    for at, layer in zip(bad, (0, 2, 3)):
        models[name][at, layer] = value
    got = L.loglik_f64(sysg, I.to_torch(models, torch.float64), y, 1e-11, 0.03).cpu().numpy()
    assert np.all(np.isnan(got[bad]))
    keep = np.delete(np.arange(12), bad)
    assert np.array_equal(got[keep], ref[keep])
