"""The tensor-core transform at the edges of its staging and pipeline: tiles
partly filled, one and several tiles per CTA, frequencies that are and are not
whole 16-byte rows, beyond the prefetch registers, gates either side of an
accumulator, blocks at any offset in a tile, and values the likelihood's
fast form leaves to the exact one.  Bounds: gates within the split's term bound
3 u^2 plus FP32 accumulation of sum |T| |x| (u = 2^-11, 2^-8), the likelihood
of the kernel's own gates within 2^-22 of the sum of its terms' magnitudes (a
quotient and the logarithms' product, each 2^-24 per gate, with a factor of
four)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _system(L, F, G):
    return L.System(n_freq=F, gate_times=np.logspace(-5, -2, G), n_hankel=16)


@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("P, F, G", [(1, 60, 30), (127, 41, 21), (128, 64, 32), (129, 63, 33), (700, 3, 1), (40000, 60, 30),
                                     (60001, 41, 21), (500, 65, 64), (500, 128, 48), (300, 66, 20)])
def test_transform_tiles(P, F, G, mode):
    import torch
    import paper_2109_00661_gb300 as L
    sysg = _system(L, F, G)
    g = torch.Generator(device="cuda")
    g.manual_seed(P + F)
    imh = -10.0 ** (torch.rand((P, F), generator=g, device="cuda") * 4 - 8)
    y = torch.as_tensor(4e-7 * (1 + np.logspace(-5, -2, G) / 1e-4) ** -2.5, device="cuda")
    gates, ll = L.gates_from_spectrum(sysg, imh, mode=mode, y_obs=y, eps_an=1e-11, eps_mn=0.03)
    assert L.system_status(sysg) == 0
    T = torch.as_tensor(sysg.tables()[3], device="cuda")
    want = imh.double() @ T.T
    scale = imh.double().abs() @ T.abs().T
    u = 2.0 ** -11 if mode == 1 else 2.0 ** -8
    # + the table's own rounding to FP32
    assert float(((gates.double() - want).abs() / scale).max()) < 3 * u * u + (3 * F + 2) * 2.0 ** -24
    gd = gates.double()
    v = 1e-22 + (0.03 * gd) ** 2
    terms = (y - gd) ** 2 / v
    logs = torch.log(2 * np.pi * v)
    got = (ll + 0.5 * (terms + logs).sum(1)).abs()
    # the residual's and variance's own FP32 rounding moves a quotient by 6 units
    assert bool((got <= 0.5 * (8 * terms + logs.abs() + 1).sum(1) * 2.0 ** -24 * 4).all())
    alone, _ = L.gates_from_spectrum(sysg, imh, mode=mode)
    assert torch.equal(alone, gates)


@pytest.mark.parametrize("eps_an", [1e-25, 1e-19, 1e-13, 1e14])
def test_likelihood_outside_the_fast_range(eps_an):
    """Variances below 2^-100 and above 2^100, residuals that vanish and a NaN
    spectrum: finite where the FP64 form is, NaN only for the NaN."""
    import torch
    import paper_2109_00661_gb300 as L
    sysg = _system(L, 60, 30)
    imh = torch.zeros((300, 60), device="cuda")
    imh[100:200] = -1e-6
    imh[250, 7] = float("nan")
    gates, ll = L.gates_from_spectrum(sysg, imh, mode=1)[0], None
    y = gates[150].double()
    gates, ll = L.gates_from_spectrum(sysg, imh, mode=1, y_obs=y, eps_an=eps_an, eps_mn=0.03)
    gd = gates.double()
    v = eps_an ** 2 + (0.03 * gd) ** 2
    want = -0.5 * ((y - gd) ** 2 / v + torch.log(2 * np.pi * v)).sum(1)
    bad = torch.zeros(300, dtype=torch.bool, device="cuda")
    bad[250] = True
    assert bool(torch.isnan(ll[bad]).all()) and bool(torch.isnan(gates[250]).all())
    if eps_an ** 2 > 1.2e-38:  # eps_an^2 in FP32's normal range
        assert torch.allclose(ll[~bad], want[~bad], rtol=1e-5, atol=1e-3)


@pytest.mark.parametrize("N, S", [(200, 9), (1, 300), (64, 10)])
def test_rows_do_not_depend_on_their_tile(N, S):
    """A block of spectra gives the same gates alone as inside a batch, at any offset in a tile."""
    import torch
    import paper_2109_00661_gb300 as L
    sysg = _system(L, 60, 30)
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    imh = -10.0 ** (torch.rand((N * S, 60), generator=g, device="cuda") * 3 - 7)
    whole, _ = L.gates_from_spectrum(sysg, imh, mode=1)
    for s in (0, S // 2, S - 1):
        part, _ = L.gates_from_spectrum(sysg, imh[s * N:(s + 1) * N].contiguous(), mode=1)
        assert torch.equal(whole[s * N:(s + 1) * N], part)
