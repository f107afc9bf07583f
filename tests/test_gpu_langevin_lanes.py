"""The Langevin proposal's eight lanes per particle: every remainder of its
components (3 + 2 kappa + 2 lambda, up to 39) and particle counts that leave a
warp partly filled, against the oracle's serial form.  Bounds: those of the
proposal test in test_gpu_langevin.py."""
import numpy as np
import pytest

from oracle import rjsmc as R
from test_gpu_langevin import env, gpu_smc, gpu_theta_grad, settings, to_host, to_oracle  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 5, 67])
def test_proposals_of_every_dimension(env, n):  # noqa: F811
    S, gsys, s, data = env
    st = settings(n_particles=n, kappa_max=9, lambda_max=9, langevin_h=0.002, seed=17 + n)
    parts = [R.sample_prior(st, i) for i in range(n)]
    gamma, stage, sweep = 1e-6, 2, 1
    sm = gpu_smc(S, gsys, data, st)
    sm.set_particles(to_host(S, parts), gamma=np.array([gamma]), stage=stage)
    g = sm.grad_current()
    sm.langevin_propose(stage, sweep)
    prop = sm.get_particles(1)
    for i, p in enumerate(parts):
        p = to_oracle(sm.get_particles(0), i)
        q, _ = R.langevin_propose(p, gpu_theta_grad(g[i], p), st, i, stage, sweep, gamma)
        assert bool(prop.valid[i]) == (q is not None), i
        q = p if q is None else q
        got = np.array([prop.phib[i], *prop.phic[i, :p.kappa], *prop.zc[i, :p.kappa], *prop.zm[i, :p.lam],
                        *prop.mv[i, :p.lam], prop.tau[i], prop.c[i]], dtype=np.float64)
        ref = np.array([q.phib, *q.phic, *q.zc, *q.zm, *q.mv, q.tau, q.c]).astype(np.float32).astype(np.float64)
        assert np.allclose(got, ref, rtol=2.5e-7, atol=0), (i, got, ref)
