"""Reweighting and resampling at the edges of their splits: populations
smaller than a CTA's warps, the largest one, one model and a hundred, weights
on one particle, few halvings, populations partly at -inf, and the step where
the screening hands over to FP64.  The reweight bounds are those of the
existing oracle comparison (the step to 1e-10 of itself); the ancestors equal
the integer rule exactly."""
import numpy as np
import pytest

from oracle import rjsmc as R

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, models, spread, g0, alpha, iters, lost", [
    (2, 1, 5.0, 0.0, 0.5, 60, 0.0), (17, 3, 20.0, 0.0, 0.5, 60, 0.0), (33, 20, 3.0, 0.5, 0.7, 60, 0.0),
    (1023, 100, 1e3, 0.0, 0.5, 60, 0.2), (1024, 100, 1e6, 0.0, 0.9, 60, 0.0), (9600, 20, 50.0, 0.0, 0.5, 7, 0.0),
    (16384, 1, 300.0, 0.1, 0.5, 60, 0.0), (16384, 100, 1e4, 0.0, 0.5, 60, 0.3), (4096, 9, 1e-3, 0.2, 0.5, 60, 0.0),
    (300, 4, 10.0, 0.0, 0.9, 20, 0.4)])
def test_reweight_edges(n, models, spread, g0, alpha, iters, lost):
    import torch
    from paper_2109_00661_gb300 import smc as S
    rng = np.random.default_rng(n + models)
    model = rng.integers(0, models, n)
    ll = -40.0 - spread * rng.exponential(1.0, n) ** 2
    ll[rng.random(n) < lost] = -np.inf
    ll[0] = -30.0
    dg, done, inc, W = S.reweight(torch.as_tensor(ll, device="cuda"),
                                  torch.as_tensor(model.astype(np.int32), device="cuda"), models, g0, alpha, iters)
    # the same halvings with FP64 sums throughout
    top = np.full(models, -np.inf)
    np.maximum.at(top, model, ll)
    live = np.isfinite(ll)

    def sums(x):
        e = np.zeros(n)
        e[live] = np.exp(x * (ll[live] - top[model[live]]))
        return e, np.bincount(model, e, models), np.bincount(model, e * e, models)

    def tess(x):
        _, s1, s2 = sums(x)
        return float(np.sum(s1[s2 > 0] ** 2 / s2[s2 > 0]))

    lo, hi, ref_done = 0.0, 1.0 - g0, tess(1.0 - g0) >= alpha * n
    for _ in range(0 if ref_done else iters):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if tess(mid) >= alpha * n else (lo, mid)
    ref = 1.0 - g0 if ref_done else (lo if lo > 0.0 else hi)
    assert int(done.item()) == int(ref_done)
    assert abs(dg.item() - ref) <= 1e-10 * ref + 1e-15
    e, s1, _ = sums(ref)
    some = s1[model] > 0
    assert np.allclose(W.cpu().numpy()[some], (e / np.where(s1[model] > 0, s1[model], 1.0))[some], rtol=1e-8, atol=1e-14)
    cnt = np.bincount(model, minlength=models)
    k = np.isfinite(top)
    assert np.allclose(inc.cpu().numpy()[k], (ref * top + np.log(np.where(s1 > 0, s1, 1.0)) - np.log(np.maximum(cnt, 1)))[k],
                       rtol=1e-9, atol=1e-9)
    assert np.all(inc.cpu().numpy()[cnt == 0] == 0.0)


@pytest.mark.parametrize("n, models", [(1, 1), (2, 2), (31, 1), (33, 5), (1024, 3), (1025, 100), (9600, 20), (16384, 1)])
@pytest.mark.parametrize("kind", ["spread", "one", "equal"])
def test_resample_edges(n, models, kind):
    import torch
    from paper_2109_00661_gb300 import smc as S
    rng = np.random.default_rng(n)
    model = rng.integers(0, models, n)
    W = np.zeros(n)
    for k in range(models):
        idx = np.nonzero(model == k)[0]
        if idx.size == 0:
            continue
        w = np.ones(idx.size)
        if kind == "spread":
            w = rng.exponential(1.0, idx.size) ** 6
        elif kind == "one":
            w[:] = 0.0
            w[rng.integers(idx.size)] = 1.0
        W[idx] = w / w.sum()
    one = 1 << R.CDF_BITS
    u40 = rng.integers(0, one, models, dtype=np.int64)
    u40[0] = one - 1
    if models > 1:
        u40[1] = 0
    got = S.resample_systematic(torch.as_tensor(W, device="cuda"),
                                torch.as_tensor(model.astype(np.int32), device="cuda"), models,
                                torch.as_tensor(u40, device="cuda")).cpu().numpy()
    ref = np.arange(n)
    for k in range(models):
        idx = np.nonzero(model == k)[0]
        m = idx.size
        if m == 0:
            continue
        C = np.cumsum(np.rint(W[idx] * one).astype(np.int64))
        C[-1] = one
        C = np.maximum.accumulate(C)  # the smallest index whose C exceeds thr
        thr = np.array([(j * one + int(u40[k])) // m for j in range(m)], dtype=np.int64)
        ref[idx] = idx[np.searchsorted(C, thr, side="right")]
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("n", [1024, 1300, 1396, 4001, 9600])
@pytest.mark.parametrize("shift", [0, 1, 7, 31])
def test_models_beginning_past_a_slice(n, shift):
    """Models that begin `shift` positions past the end of each of the eight
    cluster slices, after another population's sums went through the same
    shared memory: such a model has no share in that slice."""
    import torch
    from paper_2109_00661_gb300 import smc as S
    rng = np.random.default_rng(n)
    at = np.unique(np.minimum(np.arange(1, 8) * n // 8 + shift, n - 1))
    models = at.size + 1
    model = np.searchsorted(at, np.arange(n), side="right")
    ll = -20.0 / rng.random(n)

    def call(ll, model, models, alpha):
        return S.reweight(torch.as_tensor(ll, device="cuda"), torch.as_tensor(model.astype(np.int32), device="cuda"),
                          models, 0.0, alpha)

    def sums(x):
        top = np.full(models, -np.inf)
        np.maximum.at(top, model, ll)
        e = np.exp(x * (ll - top[model]))
        return e, np.bincount(model, e, models), np.bincount(model, e * e, models)

    lo, hi = 0.0, 1.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        _, s1, s2 = sums(mid)
        lo, hi = (mid, hi) if np.sum(s1**2 / s2) >= 0.9 * n else (lo, mid)
    big = -rng.random(16384)  # leaves exponentials near one behind on every SM
    for _ in range(64):
        call(big, rng.integers(0, 20, 16384), 20, 0.5)
        dg, _, _, W = call(ll, model, models, 0.9)
        assert abs(dg.item() - lo) <= 1e-10 * lo
    e, s1, _ = sums(lo)
    assert np.allclose(W.cpu().numpy(), e / s1[model], rtol=1e-8, atol=1e-14)
