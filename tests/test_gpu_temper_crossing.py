"""The tempering step against the exact crossing of TESS = alpha N, up to alpha
= 0.999 where TESS is nearly flat: as near to it as 60 halvings in FP64 come.
Both rest on an FP64 TESS with independent roundings of the same kind, so over
the draws the root mean square of one error is within 4 of the other's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _tess(x, d, model, M, dtype=np.float64):
    e = np.exp(dtype(x) * d.astype(dtype))
    s1, s2 = np.zeros(M, dtype), np.zeros(M, dtype)
    np.add.at(s1, model, e)
    np.add.at(s2, model, e * e)
    ok = s2 > 0
    return np.sum(s1[ok] ** 2 / s2[ok])


def _slope(x, d, model, M):
    e = np.exp(x * d)
    s1, s2, d1, d2 = (np.bincount(model, v, M) for v in (e, e * e, d * e, d * e * e))
    ok = s2 > 0
    r = s1[ok] / s2[ok]
    return np.sum(2 * r * (d1[ok] - r * d2[ok]))


@pytest.mark.parametrize("alpha", [0.5, 0.9, 0.99, 0.999])
@pytest.mark.parametrize("N, M", [(200, 5), (4096, 20)])
def test_crossing_is_as_exact_as_fp64_halvings(N, M, alpha):
    import torch
    from paper_2109_00661_gb300 import smc as S
    rng = np.random.default_rng(int(1000 * alpha) + N)
    here = halved = 0.0
    for draw in range(16):
        ll = -20.0 / rng.uniform(0, 1, N) if draw % 2 else rng.normal(-100, 30, N)
        model = rng.integers(0, M, N).astype(np.int32)
        top = np.full(M, -np.inf)
        np.maximum.at(top, model, ll)
        d, target = ll - top[model], alpha * N
        lo, hi = 0.0, 1.0
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if _tess(mid, d, model, M) >= target else (lo, mid)
        # one Newton step in extended precision from there: its error is the square of the halvings'
        step = (_tess(lo, d, model, M, np.longdouble) - np.longdouble(target)) / _slope(lo, d, model, M)
        dg, done, _, _ = S.reweight(torch.as_tensor(ll, device="cuda"), torch.as_tensor(model, device="cuda"), M, 0.0,
                                    alpha)
        assert int(done) == 0
        halved += (float(step) / lo) ** 2
        here += (float(np.longdouble(dg.item()) - np.longdouble(lo) + step) / lo) ** 2
    assert np.sqrt(here) <= 4 * np.sqrt(halved), np.sqrt(here / halved)
