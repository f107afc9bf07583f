"""The FP32 recursion where its paths part: every remainder of the two-layer
loop and the last unrolled count (10), both code forms bit for bit, and
geometries at the ends of the length scale.  Bound: the spectrum within 2^-17
of A_f = sum_k |w_k| |R_0|, the forward tests' component accuracy."""
import numpy as np
import pytest

import oracle as O
from paper_2109_00661_gb300 import inputs as I
from parity_util import DELTA_S32, spectrum_err

pytestmark = pytest.mark.gpu


def _models(P, L, seed):
    m = I.random_models(P, seed=seed, lmax=max(L, 1), lmin=L, layers_max=L)
    return {k: (v if k == "nlayers" else np.float32(v).astype(np.float64)) for k, v in m.items()}


@pytest.mark.parametrize("layers", [1, 2, 3, 4, 5, 10, 11, 12, 19, 20])
def test_layer_counts_looped_and_unrolled(layers):
    import torch
    import paper_2109_00661_gb300 as L
    name = "sounding-g20-f40-k120"
    sysg, so = L.System(**I.system_kwargs(name)), I.oracle_system(name)
    so["T"] = O.tmatrix(so["freqs"], so["times"])
    models = _models(9, layers, seed=100 + layers)
    _, ref, absh = O.forward(models, so, mode=O.HANKEL_RULE, want_imh=True, want_absh=True)
    sysg.set_depth_cutoff(0.0)
    got = []
    for shape in (1, 3):  # looped, unrolled
        sysg.set_forward_shape(layers, shape)
        got.append(L.spectrum_f32(sysg, I.to_torch(models, torch.float32)))
    assert torch.equal(got[0], got[1])
    assert spectrum_err(got[0].cpu().numpy().astype(np.float64), ref, absh).max() < DELTA_S32


@pytest.mark.parametrize("height, radius", [(0.5, 0.2), (30.0, 13.0), (3000.0, 100.0), (200000.0, 1000.0)])
def test_length_scales(height, radius):
    import torch
    import paper_2109_00661_gb300 as L
    kw = dict(I.system_kwargs("sounding-g20-f40-k120"), height=height, loop_radius=radius)
    sysg = L.System(**kw)
    so = dict(I.oracle_system("sounding-g20-f40-k120"), h=height, a=radius)
    so["T"] = O.tmatrix(so["freqs"], so["times"])
    models = _models(9, 6, seed=7)
    _, ref, absh = O.forward(models, so, mode=O.HANKEL_RULE, want_imh=True, want_absh=True)
    imh = L.spectrum_f32(sysg, I.to_torch(models, torch.float32)).cpu().numpy().astype(np.float64)
    assert spectrum_err(imh, ref, absh).max() < DELTA_S32


@pytest.mark.parametrize("name, lmax, models", [("sounding-g20-f40-k120", 8, 305), ("sounding-g20-f40-k120", 8, 1217),
                                                ("sounding-g20-f40-k120", 20, 5001), ("throughput", 10, 609),
                                                ("throughput", 1, 3000), ("throughput", 10, 4100)])
def test_models_taken_from_the_grid(name, lmax, models):
    """Launches without a recorded shape claim their models from the grid once
    there are more of them than resident CTAs: the fixed order's results bit
    for bit, also under capture and from two streams at once."""
    import torch
    import paper_2109_00661_gb300 as L
    kw = I.system_kwargs("sounding-g20-f40-k120")
    if name == "throughput":
        kw = dict(kw, n_freq=60, n_hankel=200)
    sysg, fixed = L.System(**kw), L.System(**kw)
    fixed.set_forward_shape(lmax, 1)
    m = I.to_torch(I.random_models(models, seed=models, lmax=lmax, layers_max=lmax), torch.float32)
    want = L.spectrum_f32(fixed, m)
    assert torch.equal(L.spectrum_f32(sysg, m), want)
    side = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = []
    torch.cuda.synchronize()
    for _ in range(3):
        for s in side:
            with torch.cuda.stream(s):
                out.append(L.spectrum_f32(sysg, m))
    torch.cuda.synchronize()
    assert all(torch.equal(o, want) for o in out)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        got = L.spectrum_f32(sysg, m)
    for _ in range(2):
        got.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, want)
