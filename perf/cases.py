"""What the performance of this framework is measured on.

Each case is one kind of call that a program using the framework makes, through the public entry
points (``api.simulate``, ``api.Batch``, ``api.LogLik``), at sizes taken from the configurations of
``workloads.py``, the tests and the benchmark, or of the same order.  A case names its family (how
the network is made and which entry point runs it) and its sizes; the seed given to ``prepare``
makes the inputs: rates, initial counts and the seed of the simulation's random numbers.

  listed()            the listed cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) the network or batch handle and the device inputs a program has in hand
  run(state)          one call, outputs whole
  work(case)          operations and bytes the call cannot do without
  exact(case, seed)   the same outputs from plain torch in 64 bits (small cases)
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2103_00405_gb300 import _lib as L
from paper_2103_00405_gb300 import api
from paper_2103_00405_gb300 import workloads as W

UNBOUNDED = 1.0e6  # a horizon no trajectory reaches: the event cap ends the run


def listed():
    return [
        # an interactive call: a few hundred short birth-death trajectories, every sample kept
        dict(name="bd_small_grid", family="birth_death", n_traj=250, t_end=1.0, sample_dt=0.05, grid="traj"),
        # Table 4's Lotka-Volterra run as the paper plots it: 64 trajectories, sampled paths
        dict(name="lv_64_paths", family="lotka_volterra", n_traj=64, t_end=5.0, sample_dt=0.01, grid="traj"),
        # ensemble means and variances of Lotka-Volterra over a large ensemble (ragged count)
        dict(name="lv_ensemble", family="lotka_volterra", n_traj=250001, t_end=1.0, sample_dt=0.01, grid="moments"),
        # the same of the dimerisation network, run to its slow phase
        dict(name="dimer_ensemble", family="dimerisation", n_traj=1 << 20, t_end=10.0, sample_dt=0.1, grid="moments"),
        # a small model of a dozen reactions (thread mapping), final states of many trajectories
        dict(name="small_model_m12", family="random", m=12, n=6, x0_mean=200.0, c_sigma=0.5, n_traj=100000,
             t_end=2.0, max_events=4000, grid="none"),
        # rate inference: log-likelihood of a 64-reaction network and its gradient, one training step
        dict(name="grad_m64", family="grad", m=64, n=16, x0_mean=200.0, c_sigma=0.5, n_traj=65536, t_end=5.0,
             max_events=20000),
        # a mid-size pathway model: moments over a sampling grid (warp mapping)
        dict(name="pathway_m200", family="random", m=200, n=50, x0_mean=100.0, c_sigma=0.5, n_traj=10000,
             t_end=5.0, max_events=3000, sample_dt=0.25, grid="moments"),
        # a network of a few thousand reactions, some hundred trajectories (block mapping)
        dict(name="network_m2000", family="random", m=2000, n=500, x0_mean=50.0, c_sigma=1.0, n_traj=500,
             t_end=10.0, max_events=5000, grid="none"),
        # a screen over many networks of uneven size in one launch
        dict(name="batch_512", family="batch", n_nets=512, m_lo=4, m_hi=4096, x0_mean=50.0, c_sigma=1.0,
             n_traj=1, max_events=20000),
        # the large network of a million reactions in internal times (every channel every event)
        dict(name="large_internal", family="random", m=1000000, n=10000, x0_mean=100.0, c_sigma=1.0, n_traj=16,
             t_end=UNBOUNDED, max_events=500, grid="none"),
        # the large network in absolute times with the dependency graph (touched channels only)
        dict(name="large_absolute", family="random", m=1000000, n=10000, x0_mean=100.0, c_sigma=1.0, n_traj=16,
             t_end=UNBOUNDED, max_events=20000, grid="none", form="absolute"),
        # time-dependent rates: ramped channels in a network of some dozen reactions
        dict(name="ramped_m48", family="ramped", m=48, n=12, x0_mean=100.0, c_sigma=0.5, n_traj=10000,
             t_end=1.0, max_events=2000, grid="none"),
    ]


def _log_int(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["birth_death", "lotka_volterra", "dimerisation", "thread", "grad", "warp", "block", "batch",
                       "bundle", "tree", "ramped"])
    if kind == "birth_death":
        return dict(family=kind, n_traj=_log_int(rng, 1, 100000), t_end=rng.choice([1.0, 2.0, 5.0]),
                    sample_dt=rng.choice([0.05, 0.1]), grid=rng.choice(["traj", "moments"]))
    if kind == "lotka_volterra":
        return dict(family=kind, n_traj=_log_int(rng, 16, 250000), t_end=rng.choice([0.25, 0.5, 1.0]),
                    sample_dt=0.01, grid=rng.choice(["none", "moments"]))
    if kind == "dimerisation":
        return dict(family=kind, n_traj=_log_int(rng, 100, 1 << 20), t_end=rng.choice([2.0, 5.0, 10.0]),
                    sample_dt=0.1, grid=rng.choice(["none", "moments"]))
    if kind == "thread":
        m = rng.randint(3, 16)
        return dict(family="random", m=m, n=max(5, m // 2), x0_mean=200.0, c_sigma=0.5,
                    n_traj=_log_int(rng, 100, 100000), t_end=2.0, max_events=4000, grid="none")
    if kind == "grad":
        m = rng.randint(17, 128)
        return dict(family="grad", m=m, n=max(4, m // 4), x0_mean=200.0, c_sigma=0.5,
                    n_traj=_log_int(rng, 100, 30000), t_end=2.0, max_events=4000)
    if kind == "warp":
        m = rng.randint(17, 256)
        return dict(family="random", m=m, n=m // 4, x0_mean=100.0, c_sigma=0.5, n_traj=_log_int(rng, 100, 10000),
                    t_end=5.0, max_events=3000, sample_dt=0.25, grid=rng.choice(["none", "moments"]))
    if kind == "block":
        m = _log_int(rng, 257, 4096)
        return dict(family="random", m=m, n=m // 4, x0_mean=50.0, c_sigma=1.0, n_traj=_log_int(rng, 10, 500),
                    t_end=10.0, max_events=5000, grid="none")
    if kind == "batch":
        return dict(family="batch", n_nets=_log_int(rng, 32, 512), m_lo=4, m_hi=_log_int(rng, 300, 4096),
                    x0_mean=50.0, c_sigma=1.0, n_traj=1, max_events=20000)
    if kind == "ramped":
        m = rng.randint(17, 200)
        return dict(family="ramped", m=m, n=m // 4, x0_mean=100.0, c_sigma=0.5, n_traj=_log_int(rng, 100, 10000),
                    t_end=1.0, max_events=1000, grid="none")
    m = _log_int(rng, 5000, 1000000)
    case = dict(family="random", m=m, n=max(100, m // 100), x0_mean=100.0, c_sigma=1.0,
                n_traj=rng.randint(1, 16), t_end=UNBOUNDED, grid="none")
    if kind == "tree":
        return dict(case, max_events=_log_int(rng, 1000, 20000), form="absolute")
    return dict(case, max_events=_log_int(rng, 100, 500))


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _structure(n, m, c_sigma):
    """The reactions of a random network: the model a program works on, the same for every seed."""
    return W.random_mass_action(n, m, W.GEN_SEED_BASE + m, c_sigma)


def _spec(case, rng):
    """The case's network, its rates varied a little by the seed's generator."""
    if case["family"] == "birth_death":
        s = W.birth_death()
    elif case["family"] == "lotka_volterra":
        s = W.lotka_volterra()
    elif case["family"] == "dimerisation":
        s = W.dimerisation()
    else:
        s = _structure(case["n"], case["m"], case["c_sigma"])
    return s.with_rates(s.c * rng.uniform(0.98, 1.02, s.n_reactions))


def _x0(case, rng, n):
    if case["family"] == "birth_death":
        return np.zeros(1, np.int32)
    if case["family"] == "lotka_volterra":
        return rng.poisson(1000.0, 2).astype(np.int32)
    if case["family"] == "dimerisation":
        return np.array([rng.poisson(1000.0), 0], np.int32)
    return rng.poisson(case["x0_mean"], n).astype(np.int32)


def _slopes(rng, m):
    """Rate slopes beta_k: three channels in ten constant, the others ramped."""
    return np.where(rng.random(m) < 0.3, 0.0, rng.uniform(0.1, 3.0, m))


def _inputs(case, seed):
    rng = np.random.default_rng([20210301, int(seed)])
    spec = _spec(case, rng)
    x0 = _x0(case, rng, spec.n_species)
    beta = _slopes(rng, spec.n_reactions) if case["family"] == "ramped" else None
    return spec, x0, beta, int(rng.integers(1, 2**31))


@functools.lru_cache(maxsize=4)
def _batch_structure(n_nets, m_lo, m_hi, c_sigma):
    return tuple(i.net for i in W.batched_networks(n_nets, m_lo, m_hi, c_sigma=c_sigma))


def _batch_inputs(case, seed):
    """The networks of a batch (the same reactions for every seed) with their rates varied, the initial
    counts and the horizons."""
    rng = np.random.default_rng([20210301, int(seed)])
    specs = [s.with_rates(s.c * rng.uniform(0.98, 1.02, s.n_reactions))
             for s in _batch_structure(case["n_nets"], case["m_lo"], case["m_hi"], case["c_sigma"])]
    x0 = np.concatenate([rng.poisson(case["x0_mean"], s.n_species) for s in specs]).astype(np.int32)
    return specs, x0, rng.uniform(1.0, 10.0, len(specs)), int(rng.integers(1, 2**31))


def prepare(case, seed):
    st = dict(case=case)
    if case["family"] == "batch":
        specs, x0, t_end, st["seed"] = _batch_inputs(case, seed)
        st["batch"] = api.Batch(specs)
        st["x0"] = torch.from_numpy(x0).cuda()
        st["t_end"] = torch.from_numpy(t_end).cuda()
        return st
    spec, x0, beta, st["seed"] = _inputs(case, seed)
    st["x0"] = torch.from_numpy(x0).cuda()
    if case["family"] == "grad":
        st["spec"] = spec
        st["c"] = torch.from_numpy(spec.c).cuda().requires_grad_(True)
    else:
        st["net"] = api.Network(spec)
        if beta is not None:
            st["net"].set_rate_slopes(beta)
    return st


def run(state):
    case = state["case"]
    if case["family"] == "batch":
        return state["batch"].run(state["x0"], state["t_end"], case["n_traj"], state["seed"], case["max_events"])
    if case["family"] == "grad":
        # one training step: path log-likelihoods, their mean as the objective, the gradient
        c = state["c"]
        c.grad = None
        ll = api.LogLik.apply(c, state["spec"], state["x0"], case["t_end"], case["n_traj"], state["seed"], 0,
                              case["max_events"])
        ll.mean().backward()
        return dict(loglik=ll.detach(), grad=c.grad)
    out = api.simulate(state["net"], state["x0"], case["t_end"], case["n_traj"], seed=state["seed"],
                       max_events=case.get("max_events", W.ENSEMBLE_MAX_EVENTS), sample_dt=case.get("sample_dt", 0.0),
                       grid=case["grid"],
                       form=L.RT_FORM_ABSOLUTE if case.get("form") == "absolute" else L.RT_FORM_INTERNAL)
    return {k: v for k, v in out.items() if not k.startswith("_")}


# ------------------------------------------------------------------------------------------
# Work
# ------------------------------------------------------------------------------------------

def _reactant_index(spec):
    """Per reaction (s0, s1): reactant species, s0 = -1 for none, s1 = -1 for one molecule of s0,
    s1 = -2 for two molecules of s0."""
    s0 = np.full(spec.n_reactions, -1)
    s1 = np.full(spec.n_reactions, -1)
    for r, s, k in zip(spec.reac_rxn.tolist(), spec.reac_sp.tolist(), spec.reac_coef.tolist()):
        if s0[r] < 0:
            s0[r] = s
            s1[r] = -2 if k == 2 else -1
        else:
            s1[r] = s
    return s0, s1


def _mean_field_events(spec, x0, t_end, cap):
    """Events of one trajectory to t_end from the rate equations (at most cap)."""
    s0, s1 = _reactant_index(spec)
    v = spec.dense_stoich().astype(np.float64)
    x, t, ev = x0.astype(np.float64), 0.0, 0.0
    for _ in range(4000):
        h = np.where(s0 < 0, 1.0, x[np.maximum(s0, 0)])
        h = np.where(s1 >= 0, h * x[np.maximum(s1, 0)], np.where(s1 == -2, h * np.maximum(h - 1, 0) / 2, h))
        a = spec.c * h
        tot = a.sum()
        if tot <= 0 or t >= t_end or ev >= cap:
            break
        drift = a @ v
        dt = min(t_end - t, 0.05 * float(np.min((x + 10.0) / (np.abs(drift) + 1e-9))), t_end / 100)
        ev += tot * dt
        x = np.maximum(x + drift * dt, 0.0)
        t += dt
    return min(ev, cap)


@functools.lru_cache(maxsize=64)
def _events(key):
    case = dict(key)
    if case.get("t_end") == UNBOUNDED:
        return float(case["max_events"])
    spec, x0, _, _ = _inputs(case, 0)
    return _mean_field_events(spec, x0, case["t_end"], case.get("max_events", W.ENSEMBLE_MAX_EVENTS))


def work(case):
    """Per event and channel: the remaining internal time (a subtraction and a quotient) and the advance
    of the internal time (a product and a sum); in absolute times only of the touched channels.  Bytes:
    the network and the initial counts read once, the outputs written once."""
    if case["family"] == "batch":
        m = (case["m_lo"] + case["m_hi"]) / 2
        n, ev, nt = m / 4, case["max_events"] * 0.85, case["n_traj"]
        return dict(flops=case["n_nets"] * nt * ev * (4 * m + 2), bytes=case["n_nets"] * (40 * m + nt * (4 * n + 20)))
    ev = _events(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    small = dict(birth_death=(2, 1), lotka_volterra=(3, 2), dimerisation=(2, 2))
    m, n = small.get(case["family"]) or (case["m"], case["n"])
    nt = case["n_traj"]
    per_event = 4 * m + 2
    if case.get("form") == "absolute":
        per_event = 5 * min(m, 2.5 * 1.5 * m / n) + 2  # 2.5 changed species, 1.5 m / n readers of each
    bytes_ = 40 * m + 4 * n + nt * (4 * n + 20)
    if case["family"] == "grad":
        bytes_ += 2 * nt * (12 * m + 8)
    if case.get("grid") == "traj":
        bytes_ += 4 * nt * n * (case["t_end"] / case["sample_dt"] + 1)
    if case.get("grid") == "moments":
        bytes_ += (16 * n + 8) * (case["t_end"] / case["sample_dt"] + 1)
    return dict(flops=float(nt * ev * per_event), bytes=float(bytes_))


# ------------------------------------------------------------------------------------------
# The same outputs from plain torch
# ------------------------------------------------------------------------------------------

_LOW = 0xFFFFFFFF


def _draws(seed, traj, chan, n):
    """Exp(1) increments -ln u of draw n of a channel: Philox4x32-10 (Salmon et al., SC'11), in int64."""
    c = [n >> 1, traj, chan, torch.zeros_like(n)]
    k0, k1 = seed & _LOW, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & _LOW) ^ c[1] ^ k0, p1 & _LOW, ((p0 >> 32) & _LOW) ^ c[3] ^ k1, p0 & _LOW]
        k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
    odd = (n & 1) == 1
    w0, w1 = torch.where(odd, c[2], c[0]), torch.where(odd, c[3], c[1])
    v = (w1 << 20) | (w0 >> 12)
    return -torch.log((2 * v + 1).to(torch.float64) * 2.0**-53)


# Above this many events per trajectory the event-by-event loop below takes too long.
_EXACT_EVENTS = 4500


def exact(case, seed):
    if case["family"] == "batch" or case["family"] == "lotka_volterra" or case.get("t_end") == UNBOUNDED:
        return None
    n_traj = case["n_traj"]
    spec, x0, beta, sim_seed = _inputs(case, seed)
    m, n = spec.n_reactions, spec.n_species
    cap = case.get("max_events", W.ENSEMBLE_MAX_EVENTS)
    ev_est = _events(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    if ev_est > _EXACT_EVENTS or ev_est * n_traj * m > 1.5e10:
        return None
    dev, f64, i64 = torch.device("cuda" if torch.cuda.is_available() else "cpu"), torch.float64, torch.int64
    s0, s1 = (torch.from_numpy(a).to(dev) for a in _reactant_index(spec))
    v = torch.from_numpy(spec.dense_stoich()).to(dev)
    c = torch.from_numpy(spec.c).to(dev)
    bt = torch.zeros(m, dtype=f64, device=dev) if beta is None else torch.from_numpy(beta).to(dev)
    t_end = case["t_end"]
    grid = case.get("grid", "none")
    ng = int(math.floor(t_end / case["sample_dt"] * (1 + 1e-12))) + 1 if grid != "none" else 0
    gt = torch.arange(ng + 1, dtype=f64, device=dev) * case.get("sample_dt", 0.0)
    gt[ng:] = math.inf

    rows = torch.arange(n_traj, device=dev)
    x = torch.from_numpy(x0.astype(np.int64)).to(dev).repeat(n_traj, 1)

    def propensities():
        a0 = x[:, s0.clamp(min=0)]
        h = torch.where(s0 < 0, torch.ones_like(a0), a0)
        h = torch.where(s1 >= 0, h * x[:, s1.clamp(min=0)], torch.where(s1 == -2, h * (h - 1) // 2, h))
        return c * h.to(f64)

    def integral(t, d):  # of 1 + beta s over [t, t + d]
        d = d[:, None]
        return d if beta is None else d * (1 + bt * t[:, None]) + bt * d * d * 0.5

    P = _draws(sim_seed, rows[:, None].expand(-1, m), torch.arange(m, device=dev)[None].expand(n_traj, -1),
               torch.zeros((n_traj, m), dtype=i64, device=dev))
    T = torch.zeros_like(P)
    cnt = torch.zeros((n_traj, m), dtype=i64, device=dev)
    t = torch.zeros(n_traj, dtype=f64, device=dev)
    t_last, ll = t.clone(), t.clone()
    ev = torch.zeros(n_traj, dtype=i64, device=dev)
    status = torch.zeros(n_traj, dtype=i64, device=dev)
    gi = torch.zeros(n_traj, dtype=i64, device=dev)
    live = torch.ones(n_traj, dtype=torch.bool, device=dev)
    paths = torch.full((n_traj, ng, n), -1, dtype=torch.int32, device=dev) if grid == "traj" else None
    msum = torch.zeros((ng + 1, n), dtype=i64, device=dev)
    msq, mcnt = torch.zeros_like(msum), torch.zeros(ng + 1, dtype=i64, device=dev)

    def sample(until):  # the grid points before `until` (of trajectories still sampled)
        while ng:
            due = gt[gi.clamp(max=ng)] < until
            if not bool(due.any()):
                return
            r = rows[due]
            if paths is not None:
                paths[r, gi[r]] = x[r].to(torch.int32)
            else:
                msum.index_add_(0, gi[r], x[r])
                msq.index_add_(0, gi[r], x[r] * x[r])
                mcnt.index_add_(0, gi[r], torch.ones_like(gi[r]))
            gi[r] += 1

    while True:
        a = propensities()
        rem = torch.clamp(P - T, min=0.0)
        if beta is None:
            w = rem / a
        else:
            b = a * (1 + bt * t[:, None])
            w = torch.where(bt == 0, rem / a, 2 * rem / (b + torch.sqrt(b * b + 2 * a * bt * rem)))
        w = torch.where(a > 0, w, torch.full_like(w, math.inf))
        dt, mu = w.min(dim=1)
        tn = t + dt
        absorbed = live & torch.isinf(dt)
        ended = live & ~absorbed & (tn > t_end)
        capped = live & ~absorbed & ~ended & (ev >= cap)
        status = torch.where(absorbed, 2, torch.where(capped, 1, status))
        live = live & ~(absorbed | ended | capped)
        if not bool(live.any()):
            break
        sample(torch.where(live, tn, torch.full_like(tn, -1.0)))
        d = torch.where(live, dt, torch.zeros_like(dt))
        T = torch.where(live[:, None], T + a * integral(t, d), T)
        t = torch.where(live, tn, t)
        amu = a[rows, mu] * (1 + bt[mu] * t)
        ll = torch.where(live, ll + torch.log(amu), ll)
        x = x + v[mu] * live[:, None]
        cnt[rows, mu] += live.to(i64)
        ev += live.to(i64)
        P[rows, mu] += torch.where(live, _draws(sim_seed, rows, mu, cnt[rows, mu]), torch.zeros_like(t))
    known = status != 1
    sample(torch.where(known, torch.full_like(t, math.inf), torch.full_like(t, -1.0)))
    if case["family"] == "grad":
        rest = torch.where(known, t_end - t, torch.zeros_like(t))
        T = T + propensities() * rest[:, None]
        return dict(loglik=ll - T.sum(dim=1), grad=((cnt.to(f64) - T) / c).mean(dim=0))
    out = dict(x_final=x.to(torch.int32), n_events=ev, status=status.to(torch.int32), t_last=t)
    if grid == "traj":
        out["grid"] = paths
    if grid == "moments":
        out.update(grid_sum=msum[:ng], grid_sumsq=msq[:ng], grid_count=mcnt[:ng])
    return out
