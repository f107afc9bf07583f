"""Performance cases: calls of the framework's public entry points over the
sizes, types and options its users run, with the work each cannot do without
and what it returns in 64 bits.

Systems, layer-count ranges and value distributions are those of the tests, the
benchmark and ``paper_2109_00661_gb300.inputs``: a central loop of radius 13 m at
30 m height, off-time gates from 1e-5 to 1e-2 s, sounding system 20 gates x 40
frequencies x 120 Hankel points, throughput system 30 x 60 x 200, and odd sizes
beside them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2109_00661_gb300 as L
from paper_2109_00661_gb300 import smc as S

LOOP, HEIGHT, F_MIN, F_MAX = 13.0, 30.0, 1.0, 1e7
EPS_MN = 0.03
# additive noise floors, T/s per A: data an inversion has converged on, data scored
# against prior draws (whose late gates change sign), stored spectra, and the sampler's default
EPS_AN = {"posterior": 1e-11, "random": 1e-8, "spectra": 1e-9, "sampler": 1e-13}
MU0 = 4e-7 * math.pi
PARAMS = ("logsig", "logh", "m", "logtau", "c")

# (gates, frequencies, Hankel points): the sounding system, the throughput
# system and two with odd sizes
SOUNDING, THROUGHPUT, ODD, ODD2 = (20, 40, 120), (30, 60, 200), (21, 41, 121), (33, 57, 163)


def _models_case(name, kind, system, models, lmax, lmin=1, form=L.CC_PAPER, draw="posterior", tuned=False, **more):
    c = dict(kind=kind, G=system[0], F=system[1], K=system[2], P=models, lmax=lmax, lmin=lmin, form=form, draw=draw,
             tuned=tuned, **more)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one earth model through the forward model: an interactive what-if, the smallest call
        _models_case("one-model", "forward", SOUNDING, 1, 3, lmin=3),
        # the population of one sounding, evaluated by a program's own sampler (256 particles, 1..8 merged layers)
        _models_case("population-256", "loglik", SOUNDING, 256, 8),
        # a batch of odd sizes in Pelton's form with the spectra kept, more layers than the usual ten
        _models_case("ragged-forward", "forward", ODD, 3001, 14, form=L.CC_PELTON, draw="random", imh=True),
        # a sampler's sweep over 128 soundings x 256 particles, evaluated directly, launch shape tuned once
        _models_case("sweep-32768", "loglik", SOUNDING, 32768, 8, tuned=True),
        # the headline workload: 2^20 random models of 1..10 layers, gate transform on the tensor cores
        _models_case("throughput-1m", "loglik_tc", THROUGHPUT, 1 << 20, 10, draw="random", tuned=True,
                     mode=L.GATES_TF32_SPLIT),
        # spectra kept from an earlier pass, scored against new data: the transform and the likelihood alone
        dict(name="gates-tf32-1m", kind="gates", G=30, F=60, P=1 << 20, mode=L.GATES_TF32_SPLIT, want_gates=False),
        # predictions of a posterior sample in the BF16 split, odd batch, gates kept
        dict(name="gates-bf16-odd", kind="gates", G=21, F=41, P=100003, mode=L.GATES_BF16_SPLIT, want_gates=True),
        # gradients of the log-likelihood with torch.autograd: a batch of gradient-based inversions
        _models_case("gradient-16384", "gradient", THROUGHPUT, 16384, 10, tuned=True),
        # the plain double-precision form: the reference a user checks the FP32 results with
        _models_case("double-1024", "loglik64", THROUGHPUT, 1024, 10),
        # sampler: prior draw and ten mutation sweeps, 128 soundings x 256 particles
        dict(name="sampler-128x256", kind="sampler", S=128, N=256, kappa_max=3, lambda_max=4, sweeps=10, langevin=0),
        # sampler with gradient-informed moves: two Langevin sweeps on 2 x 2048 particles of up to 19 merged layers
        dict(name="langevin-2x2048", kind="sampler", S=2, N=2048, kappa_max=9, lambda_max=9, sweeps=0, langevin=2),
        # tempering and resampling of one sounding's 9600 particles over 20 models by a program's own sampler
        dict(name="temper-9600", kind="temper", N=9600, M=20, alpha=0.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "loglik", "loglik", "loglik_tc", "gates", "gradient", "loglik64", "sampler", "temper"])
    system = rng.choice([SOUNDING, THROUGHPUT, ODD, ODD2])
    lmax = rng.randint(3, 14)
    if kind == "forward":
        return _models_case(None, kind, system, _log_int(rng, 1, 100000), lmax, form=rng.choice([0, 1, 2]),
                            draw=rng.choice(["random", "posterior"]), imh=rng.random() < 0.5)
    if kind == "loglik":
        return _models_case(None, kind, system, _log_int(rng, 1, 200000), lmax, tuned=rng.random() < 0.5)
    if kind == "loglik_tc":
        return _models_case(None, kind, rng.choice([SOUNDING, THROUGHPUT]), _log_int(rng, 4096, 400000), 10,
                            draw="random", tuned=True, mode=rng.choice([L.GATES_TF32_SPLIT, L.GATES_BF16_SPLIT]))
    if kind == "gates":
        return dict(kind=kind, G=system[0], F=system[1], P=_log_int(rng, 1000, 1 << 20),
                    mode=rng.choice([L.GATES_TF32_SPLIT, L.GATES_BF16_SPLIT]), want_gates=rng.random() < 0.5)
    if kind == "gradient":
        return _models_case(None, kind, system, _log_int(rng, 64, 20000), lmax, tuned=rng.random() < 0.5)
    if kind == "loglik64":
        return _models_case(None, kind, system, _log_int(rng, 1, 3000), lmax)
    if kind == "sampler":
        lang = rng.random() < 0.3
        km, lm = rng.randint(0, 6), rng.randint(1, 6)
        N = _log_int(rng, 64, 4096)
        return dict(kind=kind, S=max(1, _log_int(rng, 2000, 60000) // N), N=N, kappa_max=km, lambda_max=lm,
                    sweeps=0 if lang else rng.randint(1, 10), langevin=rng.randint(1, 3) if lang else 0)
    return dict(kind="temper", N=_log_int(rng, 64, 16384), M=rng.randint(1, 100), alpha=rng.choice([0.5, 0.7, 0.9]))


# ------------------------------------------------------------------ inputs
_systems = {}


def _system(G, F, K, form=L.CC_PAPER):
    """One system per geometry, kept for the whole program as a survey's is."""
    key = (G, F, K, form)
    if key not in _systems:
        _systems[key] = L.System(loop_radius=LOOP, height=HEIGHT, current=1.0, n_freq=F, f_min_hz=F_MIN,
                                 f_max_hz=F_MAX, gate_times=np.logspace(-5, -2, G), n_hankel=K, cc_form=form)
    return _systems[key]


_tuned = set()


def _tune(system, models, key):
    """The launch shape for this row stride, chosen once per system on a sample, as the benchmark does."""
    if key not in _tuned:
        _tuned.add(key)
        system.autotune({k: v[:65536].contiguous() for k, v in models.items()}, repeats=3)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + 17)
    return g


def _uniform(g, shape, lo, hi, dtype):
    return (torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo).to(dtype)


def _posterior(n, lmax):
    """About one earth of moderate conductivity, weakly chargeable from its third layer down."""
    at = torch.arange(lmax, device="cuda", dtype=torch.float64)[None, :]
    return dict(logsig=-1.5 + 0.3 * torch.sin(1.3 * at) + n(0.1), logh=1.2 + n(0.1),
                m=torch.where(at >= 2, (0.15 + n(0.03)).clamp(0.0, 1.0), torch.zeros_like(at)),
                logtau=-3.0 + n(0.1), c=(0.5 + n(0.03)).clamp(0.1, 1.0))


def _models(case, seed, dtype=torch.float32):
    """draw "random": every property drawn per layer over the prior's ranges.
    draw "posterior": models about one earth, as a converged inversion holds them."""
    g, shape = _generator(seed), (case["P"], case["lmax"])
    u = lambda lo, hi: _uniform(g, shape, lo, hi, torch.float64)  # noqa: E731
    n = lambda sd: sd * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    nl = torch.randint(case["lmin"], case["lmax"] + 1, shape[:1], generator=g, device="cuda").to(torch.int8)
    if case["draw"] == "random":
        p = dict(logsig=u(-4.0, 0.0), logh=u(math.log10(2.0), math.log10(200.0)), m=u(0.0, 1.0), logtau=u(-6.0, -1.0),
                 c=u(0.1, 1.0))
    else:
        p = _posterior(n, case["lmax"])
    # float32 values in either type, so that the two forms see the same earth
    return dict(nlayers=nl, **{k: p[k].to(torch.float32).to(dtype).contiguous() for k in PARAMS})


def _data(case, seed, rows=None):
    """Observed gates with noise: the response of the posterior's earth, or a
    smooth late-time decay where no model is meant."""
    G, kind = case["G"], case.get("draw", "sampler" if case["kind"] == "sampler" else "spectra")
    rng = np.random.default_rng(int(seed) + 77)
    if kind == "posterior":
        key = (G, case["F"], case["K"], case["form"], case["lmax"])
        if key not in _responses:
            p = _posterior(lambda sd: torch.zeros((1, case["lmax"]), device="cuda", dtype=torch.float64),
                           case["lmax"])
            p["nlayers"] = torch.tensor([case["lmax"]], device="cuda", dtype=torch.int8)
            _responses[key] = (_spectrum64(case, p) @ _tables64(G, case["F"], case["K"])[1].T)[0].cpu().numpy()
        y = _responses[key]
    else:
        y = 4e-7 * (1.0 + np.logspace(-5, -2, G) / 1e-4) ** -2.5
    n = rng.standard_normal((rows, G) if rows else G)
    return y + np.sqrt(EPS_AN[kind] ** 2 + (EPS_MN * y) ** 2) * n


_responses = {}


def _spectra(case, seed):
    """Im Hz spectra with the shape of layered-earth responses: three relaxations per model."""
    g, P, F = _generator(seed), case["P"], case["F"]
    w = 2 * math.pi * torch.logspace(0, 7, F, device="cuda", dtype=torch.float64)
    h = torch.zeros((P, F), device="cuda", dtype=torch.float32)
    for _ in range(3):
        a, tau = 10 ** _uniform(g, (P, 1), -7, -5, torch.float64), 10 ** _uniform(g, (P, 1), -7, -3, torch.float64)
        wt = w[None, :] * tau
        h -= (a * wt / (1 + wt * wt)).to(torch.float32)
    return h


def prepare(case, seed):
    kind = case["kind"]
    if kind == "gates":
        return dict(case=case, system=_system(case["G"], case["F"], 120), imh=_spectra(case, seed),
                    y=torch.as_tensor(_data(case, seed), device="cuda"))
    if kind == "sampler":
        y = _data(dict(case, G=SOUNDING[0]), seed, rows=case["S"])
        sm = S.SMC(_system(*SOUNDING), y, EPS_AN["sampler"], EPS_MN, n_particles=case["N"], n_soundings=case["S"],
                   kappa_max=case["kappa_max"], lambda_max=case["lambda_max"], seed=int(seed),
                   r_max=max(case["sweeps"], 1))
        return dict(case=case, smc=sm)
    if kind == "temper":
        g, N, M = _generator(seed), case["N"], case["M"]
        ll = -_uniform(g, (N,), 0.0, 1.0, torch.float64) ** -1.0 * 20.0
        model = torch.randint(0, M, (N,), generator=g, device="cuda", dtype=torch.int32)
        u40 = torch.randint(0, 1 << 40, (M,), generator=g, device="cuda", dtype=torch.int64)
        return dict(case=case, ll=ll, model=model, u40=u40)
    system = _system(case["G"], case["F"], case["K"], case["form"])
    models = _models(case, seed, torch.float64 if kind == "loglik64" else torch.float32)
    if case["tuned"]:
        _tune(system, models, (case["G"], case["F"], case["K"], case["form"], case["lmax"]))
    if kind == "gradient":
        for k in PARAMS:
            models[k].requires_grad_(True)
    return dict(case=case, system=system, models=models, y=torch.as_tensor(_data(case, seed), device="cuda"))


# -------------------------------------------------------------------- runs
# The FP32 forms form the log-likelihood from FP32 predictions: a program that
# works in the models' type keeps it in that type.
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "forward":
        return L.forward_f32(state["system"], state["models"], want_imh=case["imh"]) if case.get("imh") else \
            L.forward_f32(state["system"], state["models"])
    if kind == "loglik":
        ll, gates = L.loglik_f32(state["system"], state["models"], state["y"], EPS_AN[case["draw"]], EPS_MN,
                                 want_gates=True)
        return dict(ll=ll.float(), gates=gates)
    if kind == "loglik_tc":
        ll, gates = L.loglik_f32_tc(state["system"], state["models"], state["y"], EPS_AN[case["draw"]], EPS_MN,
                                    mode=case["mode"], want_gates=True)
        return dict(ll=ll.float(), gates=gates)
    if kind == "gates":
        gates, ll = L.gates_from_spectrum(state["system"], state["imh"], mode=case["mode"], y_obs=state["y"],
                                          eps_an=EPS_AN["spectra"], eps_mn=EPS_MN, want_gates=case["want_gates"])
        return dict(ll=ll.float(), gates=gates)
    if kind == "gradient":
        models = state["models"]
        ll = L.loglik(state["system"], models, state["y"], EPS_AN[case["draw"]], EPS_MN)
        return torch.autograd.grad(ll.sum(), [models[k] for k in PARAMS])
    if kind == "loglik64":
        return L.loglik_f64(state["system"], state["models"], state["y"], EPS_AN[case["draw"]], EPS_MN,
                            want_gates=True)
    if kind == "temper":
        dg, done, inc, W = S.reweight(state["ll"], state["model"], case["M"], 0.0, case["alpha"])
        anc = S.resample_systematic(W, state["model"], case["M"], state["u40"])
        return dict(dgamma=dg, done=done, logz_inc=inc, W=W, ancestors=anc)
    sm = state["smc"]
    sm.init()
    if case["sweeps"]:
        sm.mutate(case["sweeps"])
    if case["langevin"]:
        sm.langevin(case["langevin"])
    # the population; each particle's log-likelihood at a prior draw is left to the
    # cases above, since its largest values are gates at their zero crossings
    p = sm.get_particles()
    return {n: getattr(p, n) for n, _, _ in S.Particles.FIELDS if n != "ll"}


# -------------------------------------------------------------------- work
def _layer_bytes(case, size):
    return case["P"] * (5 * size * case["lmax"] + 1)


def work(case):
    """Bytes: every input and output once.  Flops: 60 per (layer, abscissa,
    frequency) of the whole stacks' recursion (230 more for its reverse sweep),
    the transform's multiply-adds and about 30 per gate of likelihood."""
    kind = case["kind"]
    if kind == "temper":
        return dict(bytes=case["N"] * (8 + 4 + 8 + 4), flops=case["N"] * 61 * 25)
    if kind == "gates":
        P, G, F = case["P"], case["G"], case["F"]
        return dict(bytes=P * (4 * F + 8 + (4 * G if case["want_gates"] else 0)), flops=P * G * (2 * F + 30))
    if kind == "sampler":
        P, (G, F, K) = case["S"] * case["N"], SOUNDING
        layers = (case["kappa_max"] + case["lambda_max"]) / 2 + 1
        passes = 1 + case["sweeps"] + (case["langevin"] + 1 if case["langevin"] else 0)
        per = 60 * F * K * layers + 2 * G * F
        flops = P * (passes * per + (case["langevin"] + 1 if case["langevin"] else 0) * 230 * F * K * layers)
        return dict(bytes=passes * P * 200, flops=flops)
    P, G, F, K = case["P"], case["G"], case["F"], case["K"]
    layers = (case["lmin"] + case["lmax"]) / 2
    size = 8 if kind == "loglik64" else 4
    flops = P * (60 * F * K * layers + 2 * G * F + 30 * G)
    out = P * G * size + (P * 8 if kind != "forward" else P * F * 4 if case.get("imh") else 0)
    if kind == "gradient":
        flops += P * 230 * F * K * layers
        out = P * 5 * 4 * case["lmax"]
    return dict(bytes=_layer_bytes(case, size) + out, flops=flops)


# ------------------------------------------------- the same results in 64 bits
_tables = {}


def _legendre_panels(lo, hi, count, x, w):
    """Nodes and weights of the composite Gauss-Legendre rule on count equal panels."""
    r = 0.5 * (hi - lo) / count
    c = lo + r * (2 * torch.arange(count, device="cuda", dtype=torch.float64) + 1)
    return (c[:, None] + r * x[None, :]).reshape(-1), (r * w).repeat(count)


def _transform(G, F):
    """T [G, F]: -(2 mu0 / pi) Int Im H(w) sin(w t) dw of the clamped cubic
    spline in ln w (Im H proportional to w below the first node and to w^-1/2
    above the last one) for every unit spectrum."""
    dev = dict(device="cuda", dtype=torch.float64)
    x = torch.linspace(math.log(F_MIN), math.log(F_MAX), F, **dev) + math.log(2 * math.pi)
    h, omega, times = x[1:] - x[:-1], torch.exp(x), np.logspace(-5, -2, G)
    A, R, I = torch.zeros((F, F), **dev), torch.zeros((F, F), **dev), torch.eye(F, **dev)
    slope = (I[1:] - I[:-1]) / h[:, None]  # divided differences of every unit vector
    for i in range(F):
        if i > 0:
            A[i, i - 1] += h[i - 1] / 6
            A[i, i] += h[i - 1] / 3
            R[i] -= slope[i - 1]
        if i < F - 1:
            A[i, i + 1] += h[i] / 6
            A[i, i] += h[i] / 3
            R[i] += slope[i]
    R[0] -= I[0]
    R[F - 1] += -0.5 * I[F - 1]
    M = torch.linalg.solve(A, R)  # second derivatives at the nodes, column per unit vector
    gx, gw = np.polynomial.legendre.leggauss(16)
    gx, gw = torch.as_tensor(gx, **dev), torch.as_tensor(gw, **dev)
    T = torch.zeros((G, F), **dev)
    for g, t in enumerate(times):
        row = torch.zeros(F, **dev)
        for j in range(F - 1):
            lo, hi = float(omega[j]), float(omega[j + 1])
            by_phase, by_x = math.ceil((hi - lo) * t / (0.5 * math.pi)), math.ceil(float(h[j]) / 0.05)
            if by_phase > by_x:
                w, wt = _legendre_panels(lo, hi, by_phase, gx, gw)
                d = torch.log(w) - x[j]
            else:
                xx, wt = _legendre_panels(float(x[j]), float(x[j + 1]), by_x, gx, gw)
                w, d = torch.exp(xx), xx - x[j]
                wt = wt * w
            s = wt * torch.sin(w * t)
            m0, m1, m2, m3 = s.sum(), (s * d).sum(), (s * d * d).sum(), (s * d * d * d).sum()
            b = slope[j] - h[j] * (2 * M[j] + M[j + 1]) / 6
            row += I[j] * m0 + b * m1 + 0.5 * M[j] * m2 + (M[j + 1] - M[j]) / (6 * h[j]) * m3
        w0, wF = float(omega[0]), float(omega[-1])
        row[0] += (math.sin(w0 * t) - w0 * t * math.cos(w0 * t)) / (w0 * t * t)
        # Int_X^inf u^-1/2 sin u du: panels to 200, then repeated integration by parts
        X, X0 = wF * t, max(wF * t, 200.0)
        tail = 0.0
        if X < X0:
            u, wt = _legendre_panels(X, X0, math.ceil((X0 - X) / 0.5), gx, gw)
            tail = float((wt * torch.sin(u) / torch.sqrt(u)).sum())
        acc, term = 0j, 1 + 0j
        for n in range(40):
            acc += term
            nxt = term * -1j * (0.5 + n) / X0
            if abs(nxt) > abs(term) or abs(nxt) < 1e-20:
                break
            term = nxt
        tail += (1j * complex(math.cos(X0), math.sin(X0)) * X0 ** -0.5 * acc).imag
        row[F - 1] += math.sqrt(wF / t) * tail
        T[g] = -(2 * MU0 / math.pi) * row
    return omega, T


def _tables64(G, F, K):
    """omega [F], T [G, F], and the Hankel rule's abscissae and weights [K]: a
    trapezoid in ln lambda with the loop's geometry in the weights."""
    if (G, F) not in _tables:
        _tables[(G, F)] = _transform(G, F)
    omega, T = _tables[(G, F)]
    x0, x1 = math.log(1e-5 / (2 * HEIGHT + LOOP)), math.log(20 / HEIGHT)
    dx = (x1 - x0) / (K - 1)
    lam = torch.exp(x0 + dx * torch.arange(K, device="cuda", dtype=torch.float64))
    wt = torch.full((K,), dx, device="cuda", dtype=torch.float64)
    wt[0] = wt[-1] = 0.5 * dx
    hw = wt * 0.5 * LOOP * lam * lam * torch.special.bessel_j1(lam * LOOP) * torch.exp(-2 * lam * HEIGHT)
    return omega, T, lam, hw


def _spectrum64(case, p):
    """Im H [P, F] of models p (float64 tensors) by the textbook recursion."""
    omega, _, lam, hw = _tables64(case["G"], case["F"], case["K"])
    lmax = p["logsig"].shape[1]
    n = torch.arange(lmax, device="cuda")[None, :]
    last = (p["nlayers"].long() - 1)[:, None]
    at = torch.minimum(n, last)  # rows past the basement repeat it: no reflection there
    sig, m, tau, c = (p[k].gather(1, at)[:, None, :] for k in ("logsig", "m", "logtau", "c"))
    lw = torch.log(omega)[None, :, None] + tau * math.log(10.0)
    x = torch.exp(torch.complex(c * lw, (c * (0.5 * math.pi)).expand_as(lw)))
    if case["form"] == L.CC_PAPER:
        cc = 1 - m / (1 + x)
    elif case["form"] == L.CC_PELTON:
        cc = (1 + x) / (1 + (1 - m) * x)
    else:
        cc = (1 + (1 - m) * x) / (1 + x)
    s = (1j * MU0) * omega[None, :, None] * 10 ** sig * cc  # [P, F, lmax]
    th = 10 ** p["logh"]
    lam2 = (lam * lam)[None, None, :]
    ub, R = torch.sqrt(lam2 + s[:, :, -1:]), None
    for j in range(lmax - 1, -1, -1):
        sb = s[:, :, j:j + 1]
        if j > 0:
            sa = s[:, :, j - 1:j]
            ua = torch.sqrt(lam2 + sa)
        else:
            sa, ua = torch.zeros_like(sb), lam[None, None, :].to(torch.complex128)
        r = (sa - sb) / (ua + ub) ** 2
        if R is None:
            R = r
        else:
            RE = R * torch.exp(-2 * ub * th[:, j, None, None])
            R = (r + RE) / (1 + r * RE)
        ub = ua
    return (R.imag * hw).sum(dim=2)


def _loglik64(gates, y, eps_an):
    v = eps_an ** 2 + (EPS_MN * gates) ** 2
    return -0.5 * ((y - gates) ** 2 / v + torch.log(2 * math.pi * v)).sum(dim=1)


def _temper64(case, state):
    """Reweighting by bisection on the total effective sample size, and the
    integer systematic resampling of the ancestors."""
    N, M = case["N"], case["M"]
    ll, model, u40 = (state[k].cpu().numpy() for k in ("ll", "model", "u40"))
    top = np.full(M, -np.inf)
    np.maximum.at(top, model, ll)
    n = np.bincount(model, minlength=M)

    def weights(dg):
        e = np.exp(dg * (ll - top[model]))
        s1, s2 = np.bincount(model, e, M), np.bincount(model, e * e, M)
        return e, s1, float(np.sum(s1[n > 0] ** 2 / s2[n > 0]))

    lo, hi, done = 0.0, 1.0, weights(1.0)[2] >= case["alpha"] * N
    for _ in range(0 if done else 60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if weights(mid)[2] >= case["alpha"] * N else (lo, mid)
    dg = 1.0 if done else (lo if lo > 0 else hi)
    e, s1, _ = weights(dg)
    inc = np.zeros(M)
    inc[n > 0] = dg * top[n > 0] + np.log(s1[n > 0]) - np.log(n[n > 0])
    return dict(dgamma=np.array([dg]), done=np.array([int(done)], dtype=np.int32), logz_inc=inc, W=e / s1[model],
                ancestors=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sampler" or (kind in ("forward", "loglik", "loglik_tc") and
                             case["P"] * case["F"] * case["K"] * case["lmax"] > 1.2e10):
        return None
    state = prepare(case, seed)
    if kind == "temper":
        return _temper64(case, state)
    if kind == "gates":
        gates = state["imh"].double() @ _tables64(case["G"], case["F"], 120)[1].T
        return dict(ll=_loglik64(gates, state["y"], EPS_AN["spectra"]), gates=gates if case["want_gates"] else None)
    models = {k: v.detach().double() if k in PARAMS else v for k, v in state["models"].items()}
    T = _tables64(case["G"], case["F"], case["K"])[1]
    chunk = max(1, int((3e6 if kind == "gradient" else 2e7) / (case["F"] * case["K"])))
    out = []
    for i in range(0, case["P"], chunk):
        p = {k: v[i:i + chunk] for k, v in models.items()}
        if kind == "gradient":
            leaves = [p[k].clone().requires_grad_(True) for k in PARAMS]
            p.update(zip(PARAMS, leaves))
            ll = _loglik64(_spectrum64(case, p) @ T.T, state["y"], EPS_AN[case["draw"]])
            out.append(torch.autograd.grad(ll.sum(), leaves))
        else:
            imh = _spectrum64(case, p)
            out.append((imh @ T.T, imh))
    parts = [torch.cat(v) for v in zip(*out)]
    if kind == "gradient":
        return parts
    gates, imh = parts
    if kind == "forward":
        return (gates, imh) if case.get("imh") else gates
    ll = _loglik64(gates, state["y"], EPS_AN[case["draw"]])
    return (ll, gates) if kind == "loglik64" else dict(ll=ll, gates=gates)
