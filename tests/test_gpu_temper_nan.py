"""A NaN log-likelihood in the standalone tempering step, of either sign (a
host's 0 / 0 has the sign bit set): its model counts for nothing in TESS, its
weights are NaN, the other models' step is the crossing without it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NEGATIVE_NAN = np.array([0xFFF8000000000000], dtype=np.uint64).view(np.float64)[0]


@pytest.mark.parametrize("N", [500, 2000])  # one CTA; a cluster
@pytest.mark.parametrize("at", [[0], [7, 11], list(range(0, 400, 100))])
def test_nan_of_either_sign(N, at):
    import torch
    from paper_2109_00661_gb300 import smc as S
    rng = np.random.default_rng(N + len(at))
    M, alpha = 6, 0.5
    ll, model = rng.normal(-50, 20, N), rng.integers(0, M, N).astype(np.int32)
    model[at] = 2
    out = []
    for nan in (np.nan, NEGATIVE_NAN):
        bad = ll.copy()
        bad[at] = nan
        out.append([v.cpu().numpy() for v in S.reweight(torch.as_tensor(bad, device="cuda"),
                                                        torch.as_tensor(model, device="cuda"), M, 0.0, alpha)])
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)
    dg, done, inc, W = out[0]
    keep = model != 2
    top = np.full(M, -np.inf)
    np.maximum.at(top, model[keep], ll[keep])
    lo, hi = 0.0, 1.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        e = np.exp(mid * (ll[keep] - top[model[keep]]))
        s1, s2 = np.bincount(model[keep], e, M), np.bincount(model[keep], e * e, M)
        lo, hi = (mid, hi) if np.sum(s1[s2 > 0] ** 2 / s2[s2 > 0]) >= alpha * N else (lo, mid)
    assert int(done[0]) == 0 and abs(dg[0] / lo - 1) < 1e-12
    assert np.isnan(inc[2]) and np.all(np.isfinite(np.delete(inc, 2)))
    assert np.all(np.isnan(W[~keep])) and np.all(np.isfinite(W[keep]))
