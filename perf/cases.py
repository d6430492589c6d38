"""Performance cases: what a user of the sampler has it do, through its public entry points.

The listed cases are this repository's own workloads (the benchmark's configurations, its observation-length sweep and
its tests' sizes): Metropolis sweeps of one chain from short to long paths in both precisions, the paper's own setting,
streaming windows, a batched launch, whole-path HMC, and the differentiable action.  `draw` gives more of the same kinds
over the same ranges.  `exact` replays a case in plain torch FP64 without this repository's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1103_4887_gb300 import pimc, synth
from paper_1103_4887_gb300.autograd import path_action

N_SKIP = 10                                   # sweeps per record or adaptation step
FREE = {3: ("gNa", "gK", "gL"), 7: "all"}     # the two parameter sets of the benchmark
PREC = {"fp64": pimc.FP64, "fp32": pimc.FP32_MIXED}


def listed():
    return [
        # The plain method at its first configuration: FP64 (the default precision), M = 1000, gNa, gK and gL free,
        # during burn-in (the steps adapt every 10 sweeps).
        {"name": "sweep_fp64_M1000", "kind": "sweep", "precision": "fp64", "M": 1000, "n_free": 3, "sweeps": 100,
         "burn_in": True},
        # The short end of the observation-length sweep in the fast precision.
        {"name": "sweep_fp32_M1024", "kind": "sweep", "precision": "fp32", "M": 1024, "n_free": 7, "sweeps": 200,
         "burn_in": False},
        # The paper's own setting: tanh kinetics, trapezoid rule, uniform proposals, M = 8000.
        {"name": "paper_fp32_M8000", "kind": "paper", "precision": "fp32", "M": 8000, "sweeps": 200},
        # The benchmark workload: M = 32768, all parameters free, FP32-mixed, recording statistics.
        {"name": "sweep_fp32_M32768", "kind": "sweep", "precision": "fp32", "M": 32768, "n_free": 7, "sweeps": 200,
         "burn_in": False},
        # The same workload in plain FP64, the precision it is compared with.
        {"name": "sweep_fp64_M32768", "kind": "sweep", "precision": "fp64", "M": 32768, "n_free": 7, "sweeps": 20,
         "burn_in": False},
        # The long end of the observation-length sweep: one long run over M = 2^20, then the path is read.
        {"name": "sweep_fp32_M1048576", "kind": "sweep", "precision": "fp32", "M": 1 << 20, "n_free": 7, "sweeps": 400,
         "burn_in": False},
        # Streaming: a new window of observations from pinned memory, ten sweeps, parameters and path read back.
        {"name": "stream_fp32_M4000", "kind": "stream", "precision": "fp32", "M": 4000, "n_free": 7, "sweeps": 10},
        # The batched configuration's 512 chains (64 data sets of uneven length, 8 chains each) in one launch, at an
        # eighth of its lengths.
        {"name": "batch_fp32_512", "kind": "batch", "precision": "fp32", "n_sets": 64, "per_set": 8, "M_lo": 1024,
         "M_hi": 8192, "sweeps": 400},
        # Whole-path HMC of L = 20 leapfrog steps at the length of the differentiation configuration, both precisions.
        {"name": "hmc_fp32_M16384", "kind": "hmc", "precision": "fp32", "M": 16384, "n_traj": 20, "n_leap": 20},
        {"name": "hmc_fp64_M16384", "kind": "hmc", "precision": "fp64", "M": 16384, "n_traj": 4, "n_leap": 20},
        # The differentiable action, forward and backward through autograd: the configuration's length in FP64, and a
        # long ragged path in FP32-mixed.
        {"name": "action_fp64_M16384", "kind": "action", "precision": "fp64", "M": 16384},
        {"name": "action_fp32_M1000001", "kind": "action", "precision": "fp32", "M": 1000001},
    ]


def _between(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "paper", "stream", "batch", "hmc", "action"])
    prec = rng.choice(["fp32", "fp64"])
    if kind == "sweep":
        M = _between(rng, 200, 1 << 20 if prec == "fp32" else 1 << 17)
        most = (1 << 27) // M if prec == "fp32" else (1 << 20) // M  # no more site moves than the largest listed
        return {"kind": kind, "precision": prec, "M": M, "n_free": rng.choice([3, 7]),
                "sweeps": max(4, _between(rng, 10, 200) if most >= 200 else most), "burn_in": rng.random() < 0.3}
    if kind == "paper":
        return {"kind": kind, "precision": prec, "M": _between(rng, 500, 12000), "sweeps": _between(rng, 10, 100)}
    if kind == "stream":
        return {"kind": kind, "precision": "fp32", "M": _between(rng, 1000, 40000), "n_free": rng.choice([3, 7]),
                "sweeps": rng.choice([5, 10, 20])}
    if kind == "batch":
        lo = _between(rng, 500, 4096)
        return {"kind": kind, "precision": "fp32", "n_sets": rng.randint(4, 48), "per_set": rng.choice([4, 8]),
                "M_lo": lo, "M_hi": lo * rng.randint(2, 6), "sweeps": rng.randint(20, 200)}
    if kind == "hmc":
        return {"kind": kind, "precision": prec, "M": _between(rng, 500, 40000), "n_traj": rng.randint(1, 4),
                "n_leap": rng.randint(8, 24)}
    return {"kind": kind, "precision": prec, "M": _between(rng, 500, 1 << 20 if prec == "fp32" else 300000)}


# ---- a user's program ------------------------------------------------------------------------------------------------

def _problem(case, seed, M=None, **kw):
    if case["kind"] == "paper":
        return synth.paper_problem(case["M"], data_seed=seed, substeps=1)
    return synth.hh_problem(M or case["M"], data_seed=seed, free=FREE[case.get("n_free", 7)], substeps=2, **kw)


def _sampler(case, prob):
    return pimc.Sampler.from_problem(prob, precision=PREC[case["precision"]])


def _perturbed(prob, seed):
    """A path about as far from the data as a chain's own: the true path with the proposal scales' noise."""
    return synth.random_path_near(prob, prob.X_true, prob.sig_x, seed)


def _inv_mass(prob):
    return np.concatenate([np.repeat([5e-3, 5e-5, 5e-5, 5e-5], prob.M + 1), 1e-6 * prob.p_true ** 2])


def _batch_problems(case, seed):
    Ms = np.random.default_rng(2024).integers(case["M_lo"], case["M_hi"] + 1, size=case["n_sets"])
    rng = np.random.default_rng([seed, 2024])
    out = []
    for d, M in enumerate(Ms):
        q = synth.HH_TRUTH.copy()
        q[:3] *= 1.0 + 0.2 * rng.uniform(-1.0, 1.0, 3)
        out.append(synth.hh_problem(int(M), data_seed=1000 * (seed % 100000) + d, free=FREE[3], p_true=q, substeps=2))
    return out


def prepare(case, seed):
    kind, st = case["kind"], {"case": case, "seed": seed}
    if kind == "batch":
        st["samplers"] = []
        for prob in _batch_problems(case, seed):
            for k in range(case["per_set"]):
                s = _sampler(case, prob)
                s.set_chain(k)
                s.set_schedule(n_init=10 ** 6, n_skip=N_SKIP, f_acc=0.4, alpha=0.5)
                st["samplers"].append(s)
        st["batch"] = pimc.Batch(st["samplers"])
        return st
    prob = _problem(case, seed)
    s = st["sampler"] = _sampler(case, prob)
    if kind in ("sweep", "paper", "stream"):
        s.set_schedule(n_init=10 ** 9 if case.get("burn_in") else 0, n_skip=N_SKIP, f_acc=0.4, alpha=0.5)
    if kind == "stream":
        st["y"] = torch.from_numpy(prob.y.copy()).pin_memory()
        st["I"] = torch.from_numpy(prob.I.copy()).pin_memory()
        st["p"] = torch.zeros(s.Np, dtype=torch.float64).pin_memory()
    if kind in ("hmc", "action"):
        X = _perturbed(prob, seed)
        s.set_params(prob.p_true, prob.lo, prob.hi, prob.free)
        if kind == "hmc":
            s.set_path(X)
            s.set_schedule(n_init=0, n_skip=N_SKIP)
            st["inv_mass"] = _inv_mass(prob)
        else:
            st["X"] = torch.tensor(X, dtype=torch.float64, device="cuda", requires_grad=True)
            st["p"] = torch.tensor(prob.p_true, dtype=torch.float64, device="cuda", requires_grad=True)
    return st


EPS = 0.05  # leapfrog step


def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind in ("sweep", "paper"):
        s = state["sampler"]
        s.sweep(case["sweeps"], seed)
        X, p = s.state()
        out = {"X": X, "p": p}
        if not case.get("burn_in") and case["M"] <= 40000:
            out["mean"], out["var"], _ = s.moments()
        return out
    if kind == "stream":
        s = state["sampler"]
        s.load_data(state["y"].data_ptr(), state["I"].data_ptr())
        s.sweep(case["sweeps"], seed, sync=False)
        s.params_async(state["p"].data_ptr())
        return {"X": s.state()[0], "p": state["p"]}
    if kind == "batch":
        state["batch"].sweep(case["sweeps"], seed)
        got = [s.state() for s in state["samplers"]]
        return {"X": np.concatenate([X.ravel() for X, _ in got]), "p": np.stack([p for _, p in got])}
    if kind == "hmc":
        s = state["sampler"]
        n = s.hmc(case["n_traj"], case["n_leap"], EPS, state["inv_mass"], seed)
        X, p = s.state()
        return {"X": X, "p": p, "accepted": n}
    A = path_action(state["X"], state["p"], state["sampler"])
    gX, gp = torch.autograd.grad(A, (state["X"], state["p"]))
    return {"A": A.detach(), "gX": gX, "gp": gp}


# Floating-point operations of the HH map (one RK4 step): four fields of 34 single operations and 16 multiply-adds, 5
# transcendental operations each, and 28 stage combinations.
MAP_FLOPS = 316


def work(case):
    """Maps: one a site move and one a site and parameter move (a leapfrog step or gradient: a forward and a reverse
    pass, three maps' worth).  Bytes: data, path, proposal scales in, path out."""
    es = 4 if case["precision"] == "fp32" else 8
    kind = case["kind"]
    if kind == "batch":
        n = case["n_sets"] * case["per_set"] * (case["M_lo"] + case["M_hi"] + 2) // 2
        return {"bytes": 14.0 * es * n, "flops": 4.0 * MAP_FLOPS * n * case["sweeps"]}
    n = case["M"] + 1
    if kind == "hmc":
        return {"bytes": 10.0 * es * n, "flops": 3.0 * MAP_FLOPS * n * case["n_traj"] * (case["n_leap"] + 1)}
    if kind == "action":
        return {"bytes": 8.0 * 8 * n + 2.0 * es * n, "flops": 4.0 * MAP_FLOPS * n}
    # the trapezoid rule of the paper's setting takes one field a value, not four
    per = MAP_FLOPS / 4 if kind == "paper" else MAP_FLOPS
    return {"bytes": 14.0 * es * n, "flops": per * (1.0 + case.get("n_free", 7)) * n * case["sweeps"]}


# ---- the same in plain torch FP64 ------------------------------------------------------------------------------------

_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox-4x32-10 over int64 tensors holding 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        a, b = 0xD2511F53 * c0, 0xCD9E8D57 * c2  # the low 64 bits of the products
        c0, c1, c2, c3 = (((b >> 32) & _M32) ^ c1 ^ k0, b & _M32, ((a >> 32) & _M32) ^ c3 ^ k1, a & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _block(seed, chain, sweep, idx, kind, blk):
    z = torch.zeros_like(idx)
    return _philox(idx, z + (sweep & _M32), z + ((kind << 24) | blk), z + chain, seed)


def _uni(hi, lo):
    return (((hi >> 6) << 26 | (lo >> 6)).double() + 0.5) * 2.0 ** -52


def _normals(w):
    r, t = torch.sqrt(-2.0 * torch.log(_uni(w[0], w[1]))), 2.0 * math.pi * _uni(w[2], w[3])
    return r * torch.cos(t), r * torch.sin(t)


def _psi(u):
    small = u.abs() < 1e-4
    v = torch.where(small, torch.ones_like(u), u)
    return torch.where(small, 1.0 + u / 2 + u * u / 12, -v / torch.expm1(-v))


def _rates(V):
    a = (_psi((V + 40) / 10), 0.07 * torch.exp(-(V + 65) / 20), 0.1 * _psi((V + 55) / 10))
    return a, (4 * torch.exp(-(V + 65) / 18), 1 / (1 + torch.exp(-(V + 35) / 10)), 0.125 * torch.exp(-(V + 65) / 80))


def _field(model, x, q, I):
    V, m, h, n = x
    if model == pimc.MODEL_HH:
        a, b = _rates(V)
        dV = (I - q[0] * m ** 3 * h * (V - q[3]) - q[1] * n ** 4 * (V - q[4]) - q[2] * (V - q[5])) / q[6]
        return torch.stack([dV] + [a[g] * (1 - x[1 + g]) - b[g] * x[1 + g] for g in range(3)])
    dV = q[0] * I + q[1] * m ** 3 * h * (q[2] - V) + q[3] * n ** 4 * (q[4] - V) + q[5] * (q[6] - V)
    F = [dV]
    for g, (Va, dVa, t0, t1) in enumerate(((25.0, 15.0, 0.1, 0.4), (5.0, -15.0, 1.0, 7.0), (10.0, 30.0, 1.0, 5.0))):
        t = torch.tanh((V - Va) / dVa)
        F.append((0.5 + 0.5 * t - x[1 + g]) / (t0 + t1 * (1 - t * t)))
    return torch.stack(F)


class _Plain:
    """The action, sweeps and HMC of one chain, vectorised over the sites, in FP64."""

    def __init__(self, prob, chain=0):
        d = self.d = dict(dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
        self.prob, self.model, self.M, self.chain, self.trap = prob, prob.model, prob.M, chain, prob.scheme == 1
        self.y, self.I = torch.tensor(prob.y, **d), torch.tensor(prob.I, **d)
        self.In = torch.cat([self.I, self.I[-1:]])
        self.Rf = torch.tensor(prob.Rf, **d)[:, None]
        self.p = torch.tensor(prob.p_init, **d)
        if self.model == pimc.MODEL_HH:
            a, b = _rates(self.y)
            self.X = torch.stack([self.y] + [a[g] / (a[g] + b[g]) for g in range(3)])
        else:
            zero = torch.zeros_like(self.y)
            t = [torch.tanh((self.y - Va) / dVa) for Va, dVa in ((25.0, 15.0), (5.0, -15.0), (10.0, 30.0))]
            self.X = torch.stack([self.y] + [0.5 + 0.5 * v + zero for v in t])
        self.sx = torch.tensor(prob.sig_x, **d)[:, None].repeat(1, self.M + 1)
        self.sp = torch.tensor(prob.sig_p, **d)

    def value(self, x, q, I):
        """What a site's cache holds: the RK4 map, or the field under the trapezoid rule."""
        if self.trap:
            return _field(self.model, x, q, I)
        dt = self.prob.dt
        k1 = _field(self.model, x, q, I)
        k2 = _field(self.model, x + 0.5 * dt * k1, q, I)
        k3 = _field(self.model, x + 0.5 * dt * k2, q, I)
        k4 = _field(self.model, x + dt * k3, q, I)
        return x + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4)

    def eps(self, x0, x1, g0, g1):
        return x1 - x0 - 0.5 * self.prob.dt * (g0 + g1) if self.trap else x1 - g0

    def action(self, X, p):
        g = self.value(X, p, self.In)
        e = self.eps(X[:, :-1], X[:, 1:], g[:, :-1], g[:, 1:])
        return 0.5 * self.prob.Rm * ((X[0, 1:] - self.y[1:]) ** 2).sum() + 0.5 * (self.Rf * e * e).sum()

    def grad(self):
        X, p = self.X.clone().requires_grad_(), self.p.clone().requires_grad_()
        A = self.action(X, p)
        return (A.detach(),) + torch.autograd.grad(A, (X, p))

    def sweeps(self, n, seed, s0=0, burn_in=False, samples=None):
        prob, M, X, p = self.prob, self.M, self.X, self.p
        G = self.value(X, p, self.In)
        dev = X.device
        free = [l for l in range(prob.Np) if prob.free[l]]
        acc_x, acc_p = torch.zeros(M + 1, **self.d), torch.zeros(prob.Np, **self.d)
        lidx = torch.arange(prob.Np, device=dev)
        for s in range(s0, s0 + n):
            for par in (0, 1):
                j = torch.arange(par, M + 1, 2, device=dev)
                z = []
                for pair in (0, 1):
                    w = _block(seed, self.chain, s, j, 0, pair)
                    z += [2 * _uni(w[0], w[1]) - 1, 2 * _uni(w[2], w[3]) - 1] if prob.proposal else list(_normals(w))
                w = _block(seed, self.chain, s, j, 0, 2)
                E = -torch.log(_uni(w[0], w[1]))
                xo, go = X[:, j], G[:, j]
                xn = xo + self.sx[:, j] * torch.stack(z)
                gn = self.value(xn, p, self.In[j])
                dA = torch.zeros_like(E)
                lf, rt = j >= 1, j < M  # the terms to the left and to the right of a site
                jl, jr = (j - 1).clamp(min=0), (j + 1).clamp(max=M)
                sq = lambda a, b: (0.5 * self.Rf * (a - b) * (a + b)).sum(0)  # noqa: E731
                dA += lf * 0.5 * prob.Rm * (xn[0] - xo[0]) * (xn[0] + xo[0] - 2 * self.y[j])
                dA += lf * sq(self.eps(X[:, jl], xn, G[:, jl], gn), self.eps(X[:, jl], xo, G[:, jl], go))
                dA += rt * sq(self.eps(xn, X[:, jr], gn, G[:, jr]), self.eps(xo, X[:, jr], go, G[:, jr]))
                ok = dA < E
                X[:, j], G[:, j] = torch.where(ok, xn, xo), torch.where(ok, gn, go)
                acc_x[j] += ok
            w, v = _block(seed, self.chain, s, lidx, 1, 0), _block(seed, self.chain, s, lidx, 1, 1)
            zp = 2 * _uni(w[0], w[1]) - 1 if prob.proposal else _normals(w)[0]
            pn, Ep = (p + self.sp * zp).tolist(), (-torch.log(_uni(v[0], v[1]))).tolist()
            for l in free:
                if not prob.lo[l] <= pn[l] <= prob.hi[l]:
                    continue
                q = p.clone()
                q[l] = pn[l]
                Gq = self.value(X, q, self.In)
                en, eo = (self.eps(X[:, :-1], X[:, 1:], g[:, :-1], g[:, 1:]) for g in (Gq, G))
                if float((0.5 * self.Rf * (en - eo) * (en + eo)).sum()) < Ep[l]:
                    p, G = q, Gq
                    acc_p[l] += 1
            if not burn_in and s % N_SKIP == 0 and samples is not None:
                samples.append(torch.cat([X.reshape(-1), p]))
            if burn_in and (s + 1) % N_SKIP == 0:
                self.sx *= 1 + 0.5 * (acc_x / N_SKIP - 0.4)
                self.sp *= torch.where(torch.tensor(prob.free, device=dev) > 0, 1 + 0.5 * (acc_p / N_SKIP - 0.4), 1.0)
                acc_x.zero_()
                acc_p.zero_()
        self.p = p

    def hmc(self, n_traj, n_leap, eps, inv_mass, seed):
        nx, acc = self.X.numel(), 0
        im = torch.tensor(inv_mass, **self.d)
        move = torch.cat([torch.ones(nx, **self.d), torch.tensor(self.prob.free, **self.d)])
        lo, hi = (torch.tensor(v, **self.d) for v in (self.prob.lo, self.prob.hi))
        pairs = torch.arange((im.numel() + 1) // 2, device=im.device)
        for t in range(n_traj):
            P = torch.stack(_normals(_block(seed, self.chain, t, pairs, 2, 0)), 1).reshape(-1)[:im.numel()]
            P = move * P / torch.sqrt(im)
            w = _block(seed, self.chain, t, pairs[:1], 3, 0)
            h, E = eps * (0.8 + 0.4 * float(_uni(w[2], w[3]))), -math.log(float(_uni(w[0], w[1])))
            X0, p0, K0, inside = self.X, self.p, 0.5 * float((P * P * im).sum()), True
            for k in range(n_leap + 1):
                A, gX, gp = self.grad()
                A0 = float(A) if k == 0 else A0
                P = P - (0.5 if k in (0, n_leap) else 1.0) * h * move * torch.cat([gX.reshape(-1), gp])
                if k < n_leap:
                    dq = h * im * P
                    self.X, self.p = self.X + dq[:nx].reshape(self.X.shape), self.p + dq[nx:]
                    inside &= bool(((self.p >= lo) & (self.p <= hi) | (move[nx:] == 0)).all())
            if inside and float(A) + 0.5 * float((P * P * im).sum()) - A0 - K0 < E:
                acc += 1
            else:
                self.X, self.p = X0, p0
        return acc


def exact(case, seed):
    """FP64 replay of the same draws.  None where it would take too long (long chains, batches) -- and for FP32-mixed
    chains of many decisions, whose outputs have no 64-bit value: accept decisions are discrete, and one decision at its
    threshold that FP32 rounding takes the other way makes another, equally valid chain."""
    kind = case["kind"]
    if kind == "batch":
        return None
    moves = case["M"] * (1 + case.get("n_free", 7)) * case.get("sweeps", 0)
    if kind in ("sweep", "paper", "stream") and (moves > 1 << 23 or case["sweeps"] > 300
                                                 or case["precision"] == "fp32" and case["M"] * case["sweeps"] > 1 << 18):
        return None
    prob = _problem(case, seed)
    c = _Plain(prob)
    if kind in ("sweep", "paper", "stream"):
        samples = []
        c.sweeps(case["sweeps"], seed, burn_in=case.get("burn_in", False), samples=samples)
        out = {"X": c.X, "p": c.p}
        if kind != "stream" and not case.get("burn_in") and case["M"] <= 40000:
            out["mean"] = torch.stack(samples).mean(0)
            out["var"] = torch.stack(samples).var(0) if len(samples) > 1 else torch.full_like(samples[0], math.nan)
        return out
    c.X, c.p = torch.tensor(_perturbed(prob, seed), **c.d), torch.tensor(prob.p_true, **c.d)
    if kind == "hmc":
        n = c.hmc(case["n_traj"], case["n_leap"], EPS, _inv_mass(prob), seed)
        return {"X": c.X, "p": c.p, "accepted": n}
    A, gX, gp = c.grad()
    return {"A": A, "gX": gX, "gp": gp}
