"""The work that a user of the simulator has it do, as cases that can be timed.

A case is one call (or the few calls that belong together) through the package's
public entry points.  Kinds:

  loglik  log likelihood, log prior and end state of a particle cloud
  rw      one random-walk Metropolis iteration of the M phase
  mala    one Langevin (MALA) iteration: likelihood, adjoint gradient, decision
  grad    the likelihood as a torch function: value and gradient by autograd
  cs      the steps around the M phase: power search, S phase, proposal covariance
  run     a whole adaptive run (C, S and M phases to the posterior) with its
          log marginal likelihood and posterior moments
  batch   many datasets of different length and model run as one batch

Sizes are those of the package's own workloads (``inputs.WORKLOADS``,
``inputs.batched_workloads``) and tests.  Returns are simulated from the model.
The clouds of single steps are posterior-like: the simulating parameters plus
normal noise, with a power of the likelihood at which a good part of the
proposals is accepted, as in the middle of a run.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1304_4334_gb300 import autograd as A
from paper_1304_4334_gb300 import inputs as I
from paper_1304_4334_gb300 import smc as S

F64 = torch.float64
CLOUD = 0.05       # standard deviation of a cloud's parameters


# ------------------------------------------------------------------------ cases
def listed():
    return [
        # Initial evaluation of a wide mixture model in double precision, odd sizes.
        {"name": "loglik_f64_k3i4", "kind": "loglik", "precision": "f64", "K": 3, "I": 4, "gamma": True,
         "T": 3089, "P": 10007},
        # The smallest run's M-phase iteration: EGARCH(1,1), 4 groups of 256, double precision.
        {"name": "rw_f64_k1i1_1k", "kind": "rw", "precision": "f64", "K": 1, "I": 1, "gamma": False,
         "T": 500, "P": 1024, "phi": 0.5},
        # The plain double-precision random walk at the paper's own shape (64 groups of 1024).
        {"name": "rw_f64_k2i2_64k", "kind": "rw", "precision": "f64", "K": 2, "I": 2, "gamma": True,
         "T": 5000, "P": 65536, "phi": 0.05},
        # The same iteration in the single-precision recursion that most runs use.
        {"name": "rw_f32_k2i2_64k", "kind": "rw", "precision": "f32", "K": 2, "I": 2, "gamma": True,
         "T": 5000, "P": 65536, "phi": 0.05},
        # The largest iteration: 1M particles, 23 parameters, 20000 observations.
        {"name": "rw_f32_k3i4_1m", "kind": "rw", "precision": "f32", "K": 3, "I": 4, "gamma": True,
         "T": 20000, "P": 1048576, "phi": 0.02},
        # A Langevin iteration at the MALA workload's shape.
        {"name": "mala_f32_k2i2_256k", "kind": "mala", "precision": "f32", "K": 2, "I": 2, "gamma": True,
         "T": 5000, "P": 262144, "phi": 0.05},
        # Scores for an optimiser or another sampler through torch, odd sizes, double precision.
        {"name": "grad_f64_k2i2", "kind": "grad", "precision": "f64", "K": 2, "I": 2, "gamma": True,
         "T": 1037, "P": 2049},
        # C and S phase of the smallest run: latency.
        {"name": "cs_1k", "kind": "cs", "J": 4, "N": 256, "d": 4},
        # C and S phase of the largest run.
        {"name": "cs_1m", "kind": "cs", "J": 128, "N": 8192, "d": 23},
        # A whole small run in double precision.
        {"name": "run_f64_k1i1", "kind": "run", "precision": "f64", "tempering": "power", "K": 1, "I": 1,
         "gamma": False, "T": 500, "J": 4, "N": 256, "rbar": 10, "kappa": 1},
        # The paper's own simulator: observations one at a time, 64 groups of 1024.
        {"name": "run_f32_k2i2_data", "kind": "run", "precision": "f32", "tempering": "data", "K": 2, "I": 2,
         "gamma": True, "T": 5000, "J": 64, "N": 1024, "rbar": 7, "kappa": 3},
        # Several datasets and model variants in one batch.
        {"name": "batch8_f32", "kind": "batch", "n": 8, "J": 16, "N": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["loglik", "rw", "rw", "rw", "mala", "grad", "cs", "run"])
    if kind == "cs":
        J, N = _log_int(rng, 2, 128), _log_int(rng, 33, 8192)
        return {"kind": kind, "J": J, "N": N, "d": rng.randint(2, 26)}
    precision = rng.choice(["f32", "f64"])
    if kind == "run":
        # within the cost of the largest listed run
        K, I_ = rng.randint(1, 2), rng.randint(1, 2)
        most = 2.5e5 if precision == "f64" else 2e7
        J, N = rng.choice([4, 8]) if precision == "f64" else rng.choice([4, 16, 32]), _log_int(rng, 64, 256)
        T = _log_int(rng, 100, max(110, min(3000, most / (J * N))))
        return {"kind": kind, "precision": precision, "tempering": rng.choice(["power", "data"]), "K": K, "I": I_,
                "gamma": rng.random() < 0.7, "T": T, "J": J, "N": N, "rbar": 7, "kappa": rng.choice([1, 3])}
    K, I_ = rng.randint(1, 3), rng.randint(1, 4)
    T = _log_int(rng, 37, 5000)
    # particle x observation evaluations, within the cost of the largest listed cases
    most = {("loglik", "f32"): 2e9, ("loglik", "f64"): 1e8, ("rw", "f32"): 2e9, ("rw", "f64"): 1e8,
            ("mala", "f32"): 5e8, ("mala", "f64"): 1e7, ("grad", "f32"): 2e7, ("grad", "f64"): 5e6}[kind, precision]
    P = _log_int(rng, 129, max(200, min(400000, most / T)))
    c = {"kind": kind, "precision": precision, "K": K, "I": I_, "gamma": rng.random() < 0.7, "T": T, "P": P}
    if kind in ("rw", "mala"):
        c["phi"] = round(min(1.0, 250.0 / T), 4)
    return c


# ----------------------------------------------------------------------- inputs
def _truth(K, I_):
    """The simulating process: the workload's where one has these K and I."""
    for w in I.WORKLOADS.values():
        if (w.K, w.I) == (K, I_):
            return w.truth
    if I_ == 1:
        p, mu, sg = (1.0,), (0.0,), (1.0,)
    else:
        p, mu, sg = I.normalized_mixture(np.linspace(1.0, 0.3, I_), np.linspace(-0.2, 0.3, I_),
                                         np.linspace(0.8, 2.5, I_))
    return I.EgarchTruth(0.0003, 0.01, tuple(np.linspace(0.97, 0.6, K)), tuple(np.linspace(0.08, 0.15, K)),
                         tuple(np.linspace(-0.05, 0.01, K)), p, mu, sg)


def _cloud(c, seed):
    """Returns (host [T]), the cloud (device [d][P], float64) and, for the
    mutation kinds, the Cholesky factor of (0.3)^2 V (device [d][d])."""
    truth = _truth(c["K"], c["I"])
    y = I.simulate_egarch(truth, c["T"], 7000 + seed)
    th = torch.tensor(I.theta_of_truth(truth, I_model=c["I"], gamma=c["gamma"]), dtype=F64, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed)
    theta = th[:, None] + CLOUD * torch.randn((len(th), c["P"]), dtype=F64, device="cuda", generator=g)
    L = None
    if c["kind"] in ("rw", "mala"):
        L = (0.3 * torch.linalg.cholesky(torch.cov(theta).reshape(len(th), -1).cpu())).contiguous().cuda()
    return y, theta.contiguous(), L


def _search_inputs(c, seed):
    """Log likelihoods of a prior-like population (quadratic forms with a few
    dead particles) and the particles' parameters."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    P, d = c["J"] * c["N"], c["d"]
    x = torch.randn((d, P), dtype=F64, device="cuda", generator=g)
    theta = (0.5 * x + torch.linspace(-2.0, 2.0, d, dtype=F64, device="cuda")[:, None]).contiguous()
    ll = 15000.0 - 60.0 * x.square().sum(0)
    ll[torch.rand(P, dtype=F64, device="cuda", generator=g) < 2e-4] = -math.inf
    return ll.contiguous(), theta


def _model(c):
    return S.model_egarch(c["K"], c["I"], c["gamma"])


def _obs(y, precision):
    return torch.tensor(y, dtype=torch.float32 if precision == "f32" else F64, device="cuda")


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"kind": kind, "case": c, "seed": seed}
    if kind == "cs":
        P, d = c["J"] * c["N"], c["d"]
        st["ll"], st["theta"] = _search_inputs(c, seed)
        st["idx"] = torch.zeros(P, dtype=torch.int32, device="cuda")
        st["mean"], st["cov"], st["L"] = (torch.zeros(s, dtype=F64, device="cuda") for s in ((d,), (d, d), (d, d)))
        return st
    if kind == "batch":
        ws = I.batched_workloads(n=c["n"], J=c["J"], N=c["N"])
        models = [S.model_egarch(w.K, w.I, w.gamma) for w in ws]
        cfgs = [S.config_default(J=w.J, N=w.N, precision=S.FP32, seed=100 + i) for i, w in enumerate(ws)]
        st["theta0"] = [S.draw_prior(m, seed * 64 + i, w.P) for i, (m, w) in enumerate(zip(models, ws))]
        ys = [I.simulate_egarch(w.truth, w.T, w.data_seed + 64 * seed) for w in ws]
        st["batch"] = S.Batch(models, cfgs, ys, [t.t().cpu().numpy() for t in st["theta0"]])
        st["batch"].autotune()
        return st
    m = st["model"] = _model(c)
    prec = st["prec"] = S.FP32 if c["precision"] == "f32" else S.FP64
    if kind == "run":
        y = I.simulate_egarch(_truth(c["K"], c["I"]), c["T"], 7000 + seed)
        st["theta0"] = S.draw_prior(m, seed, c["J"] * c["N"])
        cfg = S.config_default(J=c["J"], N=c["N"], precision=prec, rbar=c["rbar"], kappa=c["kappa"], seed=seed,
                               tempering=S.DATA if c["tempering"] == "data" else S.POWER)
        st["ctx"] = S.init(m, cfg, y, st["theta0"], theta0_on_device=True)
        st["ctx"].autotune()
        return st
    y, st["theta"], st["L"] = _cloud(c, seed)
    st["obs"] = _obs(y, c["precision"])
    d, P = st["theta"].shape
    st["ll"], st["lp"] = (torch.zeros(P, dtype=F64, device="cuda") for _ in range(2))
    st["state"] = torch.zeros((c["K"] + 1, P), dtype=F64, device="cuda")
    if kind == "grad":
        st["theta"] = st["theta"].t().contiguous()
    elif kind in ("rw", "mala"):
        st["it"] = 0
        S.loglik(m, prec, st["obs"], st["theta"], st["ll"], st["lp"], st["state"])
        if kind == "mala":
            st["grad"] = torch.zeros((d, P), dtype=F64, device="cuda")
            S.loglik_grad(m, prec, st["obs"], st["theta"], st["ll"], st["grad"], st["state"])
    return st


# -------------------------------------------------------------------- one pass
def run(st):
    c, kind = st["case"], st["kind"]
    if kind == "loglik":
        S.loglik(st["model"], st["prec"], st["obs"], st["theta"], st["ll"], st["lp"], st["state"])
        return {"ll": st["ll"], "lp": st["lp"], "state": st["state"]}
    if kind == "rw":
        n = S.mutate_rw(st["model"], st["prec"], st["obs"], st["theta"], st["ll"], st["lp"], st["state"], st["L"],
                        c["phi"], st["seed"], 1, st["it"])
        st["it"] += 1
        return {"theta": st["theta"], "ll": st["ll"], "lp": st["lp"], "state": st["state"], "accepted": n}
    if kind == "mala":
        n = S.mutate_mala(st["model"], st["prec"], st["obs"], st["theta"], st["ll"], st["lp"], st["grad"],
                          st["state"], st["L"], c["phi"], st["seed"], 1, st["it"])
        st["it"] += 1
        return {"theta": st["theta"], "ll": st["ll"], "lp": st["lp"], "grad": st["grad"], "state": st["state"],
                "accepted": n}
    if kind == "grad":
        theta = st["theta"].detach().requires_grad_(True)
        ll = A.loglik(theta, st["model"], st["prec"], st["obs"])
        (g,) = torch.autograd.grad(ll.sum(), theta)
        return {"ll": ll.detach(), "grad": g}
    if kind == "cs":
        J, N = c["J"], c["N"]
        dphi, rss = S.power_search(st["ll"], 0.0)
        lwbar = S.resample_logw(dphi * st["ll"], J, N, st["idx"], seed=st["seed"], cycle=1)
        S.cov_chol(st["theta"], 5, st["mean"], st["cov"], st["L"])
        return {"dphi": dphi, "rss": rss, "idx": st["idx"], "lwbar": lwbar, "mean": st["mean"], "cov": st["cov"],
                "L": st["L"]}
    if kind == "run":
        x = st["ctx"]
        x.reset(st["theta0"], st["seed"], theta0_on_device=True)
        x.run()
        return {"log_ml": x.log_ml(), "moments": x.moments(), "groups": x.group_estimators(),
                "particles": x.particles()}
    b = st["batch"]
    b.reset(st["theta0"], st["seed"])
    b.run()
    members = [b.member(i) for i in range(c["n"])]
    return {"log_ml": [x.log_ml()[0] for x in members], "moments": [x.moments() for x in members],
            "particles": [x.particles()[:2] for x in members]}


# ------------------------------------------------------------------ least work
def _ops(K, I_, gamma):
    """Operations of one particle and observation: |eps|, the factor updates,
    log h and its sum, the shock with its exponential, the mixture."""
    mix = {1: 1, 2: 9}.get(I_, 6 * I_)
    return 1 + (3 if gamma else 2) * K + K + 1 + 3 + mix


def _dim(K, I_, gamma):
    return 2 + (3 if gamma else 2) * K + (3 * I_ if I_ > 1 else 0)


def work(case):
    c, kind = case, case["kind"]
    if kind == "cs":
        P, d = c["J"] * c["N"], c["d"]
        # log likelihoods for the search and the weights, indices, particles for the covariance
        return {"bytes": 8 * P + 4 * P + 8 * P * d, "flops": P * (d * (d + 1) + 6 * 2 * 32)}
    if kind == "batch":
        # 16384 particles per dataset, 5250 observations and about 16 cycles of 7 iterations on average
        return {"bytes": c["n"] * c["J"] * c["N"] * 8 * 12, "flops": c["n"] * c["J"] * c["N"] * 5250 * 16 * 7 * _ops(2, 2, True)}
    K, I_, g = c["K"], c["I"], c["gamma"]
    d, size = _dim(K, I_, g), 4 if c["precision"] == "f32" else 8
    if kind == "run":
        P = c["J"] * c["N"]
        # data tempering: about 60 cycles at half the observations on average; power tempering: 12 cycles
        evals = P * c["T"] * c["rbar"] * (30 if c["tempering"] == "data" else 12)
        return {"bytes": 2 * 8 * P * d, "flops": evals * _ops(K, I_, g)}
    P, T = c["P"], c["T"]
    evals = P * T * _ops(K, I_, g)
    if kind == "loglik":
        return {"bytes": size * T + 8 * P * (d + 2 + K + 1), "flops": evals}
    if kind == "rw":
        return {"bytes": size * T + 2 * 8 * P * (d + 2 + K + 1), "flops": evals}
    if kind == "mala":
        return {"bytes": size * T + 2 * 8 * P * (2 * d + 2 + K + 1), "flops": 4 * evals}
    return {"bytes": size * T + 8 * P * (2 * d + 1), "flops": 4 * evals}


# ------------------------------------------------- the same in plain 64 bits
def _split(th, K, I_, gamma):
    """Model parameters of full parameter rows th [d][P] (Table 1's transforms
    and the mixture's normalisation to mean 0, variance 1)."""
    j = 2 + 2 * K
    q = {"mu": th[0] / 1000.0, "lsy": th[1], "al": torch.tanh(th[2:2 + K]), "be": torch.exp(th[2 + K:j]),
         "ga": torch.zeros_like(th[2:2 + K])}
    if gamma:
        q["ga"] = th[j:j + K]
        j += K
    if I_ > 1:
        p = torch.tanh(th[j:j + I_]) + 1.0
        p = p / p.sum(0)
        mu, s = th[j + I_:j + 2 * I_], torch.exp(th[j + 2 * I_:j + 3 * I_])
        mu = mu - (p * mu).sum(0)
        k = 1.0 / torch.sqrt((p * (mu * mu + s * s)).sum(0))
        q |= {"lp": torch.log(p) - torch.log(k * s), "m": k * mu, "a": 1.0 / (k * s)}
    return q


def _loglik64(th, y, K, I_, gamma):
    q = _split(th, K, I_, gamma)
    y = [float(v) for v in y]
    v = torch.zeros_like(q["al"])
    acc = torch.zeros_like(q["mu"])
    for t, yt in enumerate(y):
        if t:
            v = q["al"] * v + q["be"] * (eps.abs() - math.sqrt(2.0 / math.pi)) + q["ga"] * eps
        lh = q["lsy"] + 0.5 * v.sum(0)
        eps = (yt - q["mu"]) * torch.exp(-lh)
        if I_ == 1:
            acc = acc - 0.5 * eps * eps - lh
        else:
            z = (eps - q["m"]) * q["a"]
            acc = acc + torch.logsumexp(q["lp"] - 0.5 * z * z, 0) - lh
    return acc - 0.5 * math.log(2.0 * math.pi) * len(y), torch.cat([v, eps[None]])


def _grad64(th, y, K, I_, gamma):
    th = th.detach().requires_grad_(True)
    ll, state = _loglik64(th, y, K, I_, gamma)
    (g,) = torch.autograd.grad(ll.sum(), th)
    return ll.detach(), g, state.detach()


def _prior64(c, th, with_grad=False):
    mean, sd, lo = (torch.tensor(np.asarray(a), dtype=F64, device=th.device)[:, None] for a in S.model_prior(_model(c)))
    z = (th - mean) / sd
    lp = (-0.5 * z * z - 0.5 * math.log(2.0 * math.pi) - torch.log(sd)).sum(0)
    lp = torch.where((th >= lo).all(0), lp, torch.full_like(lp, -math.inf))
    return (lp, -z / sd) if with_grad else lp


def _philox(c0, c1, c2, c3, key):
    """Philox4x64-10 (Salmon et al. 2011) over arrays of counters c0."""
    mask, low = (1 << 64) - 1, np.uint64(0xFFFFFFFF)

    def mulhi(a, b):
        a, b32 = np.uint64(a), np.uint64(32)
        al, ah, bl, bh = a & low, a >> b32, b & low, b >> b32
        m = ah * bl + ((al * bl) >> b32)
        n = al * bh + (m & low)
        return ah * bh + (m >> b32) + (n >> b32)

    c = [np.array(c0, dtype=np.uint64)] + [np.full(len(c0), v, dtype=np.uint64) for v in (c1, c2, c3)]
    k0, k1 = key, 0
    m0, m1 = 0xD2E7470EE14C6C93, 0xCA5A826395121157
    with np.errstate(over="ignore"):
        for _ in range(10):
            h0, l0, h1, l1 = mulhi(m0, c[0]), np.uint64(m0) * c[0], mulhi(m1, c[2]), np.uint64(m1) * c[2]
            c = [h1 ^ c[1] ^ np.uint64(k0), l1, h0 ^ c[3] ^ np.uint64(k1), l0]
            k0, k1 = (k0 + 0x9E3779B97F4A7C15) & mask, (k1 + 0xBB67AE8584CAA73B) & mask
    return [((x >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53 for x in c]


def _normals64(seed, P, cycle, it, d):
    z = []
    for b in range((d + 3) // 4):
        u = _philox(np.arange(P), it, cycle, (1 << 32) | b, seed)
        for k in (0, 2):
            r = np.sqrt(-2.0 * np.log(u[k]))
            z += [r * np.cos(2.0 * np.pi * u[k + 1]), r * np.sin(2.0 * np.pi * u[k + 1])]
    return torch.tensor(np.stack(z[:d]), dtype=F64, device="cuda")


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("run", "batch"):
        return None      # every draw of a run depends on all decisions before it
    if kind == "cs":
        ll, theta = _search_inputs(c, seed)
        x, lo, hi = ll - ll.max(), 0.0, 1.0

        def rss(p):
            w = torch.exp(p * x)
            return float(w.sum() ** 2 / (w.square().sum() * len(w)))

        for _ in range(60):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if rss(mid) >= 0.5 else (lo, mid)
        lw = (hi * ll).reshape(c["J"], c["N"])
        cov = torch.cov(theta).reshape(c["d"], c["d"])
        return {"dphi": hi, "rss": None, "idx": None, "lwbar": (torch.logsumexp(lw, 1) - math.log(c["N"])).cpu().numpy(),
                "mean": theta.mean(1), "cov": cov, "L": 0.5 * torch.linalg.cholesky(cov.cpu()).cuda()}
    K, I_, gamma, P, T = c["K"], c["I"], c["gamma"], c["P"], c["T"]
    # about 60 torch operations an observation, each at least a launch or P values in 64 bits; with the
    # backward pass three times as many, whose inputs are all kept
    if T * max(1.0, P / 1e5) > (10000 if kind in ("loglik", "rw") else 2500):
        return None
    if kind in ("mala", "grad") and 8.0 * 60 * P * T > 6e10:
        return None
    y, theta, L = _cloud(c, seed)
    y = np.asarray(y, dtype=np.float32).astype(float) if c["precision"] == "f32" else y
    if kind == "loglik":
        ll, state = _loglik64(theta, y, K, I_, gamma)
        return {"ll": ll, "lp": _prior64(c, theta), "state": state}
    if kind == "grad":
        ll, g, _ = _grad64(theta, y, K, I_, gamma)
        return {"ll": ll, "grad": g.t().contiguous()}
    phi, d = c["phi"], theta.shape[0]
    z = _normals64(seed, P, 1, 0, d)
    logu = torch.log(torch.tensor(_philox(np.arange(P), 0, 1, 2 << 32, seed)[0], dtype=F64, device="cuda"))
    if kind == "rw":
        ll, state = _loglik64(theta, y, K, I_, gamma)
        prop = theta + L @ z
        ll2, state2 = _loglik64(prop, y, K, I_, gamma)
        lp, lp2 = _prior64(c, theta), _prior64(c, prop)
        acc = logu < (lp2 + phi * ll2) - (lp + phi * ll)
    else:
        ll, g, state = _grad64(theta, y, K, I_, gamma)
        lp, pg = _prior64(c, theta, True)
        prop = theta + 0.5 * L @ (L.t() @ (pg + phi * g)) + L @ z
        ll2, g2, state2 = _grad64(prop, y, K, I_, gamma)
        lp2, pg2 = _prior64(c, prop, True)
        back = theta - prop - 0.5 * L @ (L.t() @ (pg2 + phi * g2))
        u = torch.linalg.solve_triangular(L, back, upper=False)
        acc = logu < (lp2 + phi * ll2) - (lp + phi * ll) - 0.5 * u.square().sum(0) + 0.5 * z.square().sum(0)
    out = {"theta": torch.where(acc, prop, theta), "ll": torch.where(acc, ll2, ll), "lp": torch.where(acc, lp2, lp),
           "state": torch.where(acc, state2, state), "accepted": None}
    if kind == "mala":
        out["grad"] = torch.where(acc, g2, g)
    return out
