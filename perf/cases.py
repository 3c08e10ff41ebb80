"""The calls this library is timed on.

A case names one inference call of a user's program: a model's structure, who shares it, how many
agents and steps, and the entry point.  ``listed()`` gives the fixed ones, ``draw(rng)`` one more of
the same ranges, ``prepare`` what the program holds before the call (the packed model and the device
tensors), ``run`` the call.

Fields of a case
  n, m, U     states per factor, outcomes per modality, actions per factor ("8,8,6")
  dep         per modality the factors it depends on, one digit each ("012 01")
  bdep        the same per factor for transitions that read other factors' states; "" = its own only
  own         every agent has a model of its own (else all share one)
  agents, steps, iters
  algo        filter, vmp or mmp
  call        "batch"  whole trajectories from the model's prior
              "tick"   filtering continued from the previous belief (one or a few steps per call)
              "slide"  a window continued from the previous belief and started from the last window's
              "soft"   observations as categorical vectors
  arith       f64 (the default arithmetic) or f32 (the fast mode, used with damped updates)
  damping     step of the update on the log-beliefs; 1 = the plain iteration
  sparsity    share of zeros in A
  sticky      transitions that mostly stay (Dirichlet(1/2) plus half the identity), else Dirichlet(1)
  prior       initial states drawn from a Dirichlet, else uniform
  extras      log-beliefs and most probable states are asked for too
"""
from __future__ import annotations

import math

import torch

import paper_2607_17855_b200 as bi

_BASE = {"bdep": "", "own": False, "iters": 16, "call": "batch", "arith": "f64", "damping": 1.0, "sparsity": 0.0,
         "sticky": False, "prior": True, "extras": False}


def _case(**kw):
    c = dict(_BASE)
    c.update(kw)
    return c


def _ints(text):
    return [int(v) for v in text.split(",")]


def _lists(text):
    return [[int(d) for d in word] for word in text.split()]


def listed():
    return [
        # one agent in a control loop: a belief update per sensor reading; latency of a call is all there is
        _case(name="tick_one_agent", n="4,3", m="5,4", U="2,2", dep="01 01", agents=1, steps=1, algo="filter",
              call="tick", prior=False, extras=True),
        # a handful of small agents over a short episode (the benchmark's first configuration)
        _case(name="filter_small", n="4,3", m="5,4", U="2,2", dep="01 01", agents=8, steps=10, algo="filter",
              prior=False),
        # thousands of simulated agents sharing one model (the benchmark's headline workload)
        _case(name="filter_shared", n="8,8,6", m="16,8,8", U="4,4,4", dep="012 012 012", agents=4096, steps=50,
              algo="filter", sticky=True, prior=False),
        # the same use at odd sizes in the fast arithmetic, with the damping that makes it accurate
        _case(name="filter_odd_f32", n="7,9,5", m="11,6,9", U="3,2,4", dep="012 01 012", agents=1000, steps=25,
              algo="filter", arith="f32", damping=0.5),
        # a structure of the randomised sweep with coupled groups of two to four factors, filtered
        _case(name="filter_sweep", n="4,5,15,21,9", m="23,12,45,26,9", U="3,3,4,2,1", dep="0124 02 024 0134 34",
              agents=256, steps=10, algo="filter"),
        # smoothing windows on a shared model with mixed dependencies (the benchmark's third configuration)
        _case(name="vmp_shared", n="10,10,8,6", m="20,16,12,8", U="3,3,3,3", dep="01 12 023 0123", agents=1024, steps=20,
              algo="vmp"),
        # every agent has learned a sparse model of its own (the benchmark's fourth configuration)
        _case(name="mmp_own_models", n="16,12,8", m="32,16", U="2,2,2", dep="012 012", own=True, agents=2048, steps=20,
              algo="mmp", sparsity=0.7, prior=False),
        # two more structures of the sweep: a large group beside small ones; pairs of large factors
        _case(name="vmp_sweep", n="18,29,11", m="25,35,32,56,7,17", U="4,2,4", dep="2 02 01 12 012 2", agents=256,
              steps=10, algo="vmp"),
        _case(name="mmp_pairs", n="25,27,6,28,17", m="14,46,50,30,47", U="4,3,2,3,4", dep="03 2 4 3 01", agents=256,
              steps=10, algo="mmp"),
        # sensors that report distributions instead of outcomes
        _case(name="filter_soft", n="8,8,6", m="16,8,8", U="4,4,4", dep="012 012 012", agents=2000, steps=30,
              algo="filter", call="soft", sticky=True, prior=False),
        # a sliding inference window advanced by one step: continued, warm-started, few iterations, all outputs
        _case(name="mmp_slide", n="9,6,12", m="13,20,7", U="3,2,3", dep="01 12 012", agents=500, steps=15, iters=6,
              algo="mmp", call="slide", extras=True),
        # transitions that read a neighbouring factor's state
        _case(name="vmp_coupled", n="10,10,8,6", m="12,10,8,6", U="3,3,3,3", dep="01 12 023 0123", bdep="01 12 23 30",
              agents=1024, steps=20, algo="vmp", prior=False),
    ]


# ---- more cases of the same ranges -----------------------------------------------------------------

_A_ENTRIES = 1 << 18      # largest A of one modality, as in the benchmark's sweep
_FLOPS = 4e9              # most arithmetic of a drawn case
_UNITS = 200_000          # most (agent, step) pairs
_OWN_ENTRIES = 150_000_000   # most entries of A over all agents' own models
_SOFT_ENTRIES = 30_000_000   # most slice entries of a call with observation vectors


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _structure(rng, joint, small=False):
    """n, m, dep: every modality on every factor (joint), or the sweep's random subsets of up to five factors."""
    while True:
        if joint:
            F = rng.randint(2, 3 if small else 4)
            n = [rng.randint(2, 8 if small else 16) for _ in range(F)]
            M = rng.randint(1, 4)
            dep = [list(range(F))] * M
        else:
            F = rng.randint(1, 5)
            n = [rng.randint(2, 12 if small else 32) for _ in range(F)]
            M = rng.randint(1, 6)
            dep = []
            for _ in range(M):
                d = [f for f in range(F) if rng.random() < 0.5]
                dep.append(d or [rng.randrange(F)])
        m = [rng.randint(2, 64) for _ in range(M)]
        if all(m[i] * math.prod(n[f] for f in d) <= _A_ENTRIES and len(d) <= 4 for i, d in enumerate(dep)):
            return n, m, dep


def draw(rng):
    while True:
        kind = rng.choices(["tick", "filter", "window", "own", "soft", "slide", "coupled"],
                           [12, 30, 30, 8, 8, 8, 4])[0]
        n, m, dep = _structure(rng, rng.random() < 0.5, small=kind in ("tick", "coupled"))
        F = len(n)
        c = _case(n=",".join(map(str, n)), m=",".join(map(str, m)), U=",".join(str(rng.randint(1, 4)) for _ in n),
                  dep=" ".join("".join(map(str, d)) for d in dep), sticky=rng.random() < 0.3, prior=rng.random() < 0.5,
                  extras=rng.random() < 0.25)
        c["sparsity"] = rng.choice([0.0, 0.0, 0.5])
        c["algo"] = rng.choice(["vmp", "mmp"])
        if kind == "tick":
            c.update(call="tick", algo="filter", agents=_log_int(rng, 1, 64), steps=rng.choice([1, 1, 1, 2, 4]))
        elif kind == "filter":
            c.update(algo="filter", agents=_log_int(rng, 8, 4096), steps=rng.randint(5, 50))
        elif kind == "window":
            c.update(agents=_log_int(rng, 32, 2048), steps=rng.randint(4, 32))
        elif kind == "own":
            c.update(own=True, algo=rng.choice(["filter", "vmp", "mmp"]), agents=_log_int(rng, 64, 2048),
                     steps=rng.randint(4, 24), sparsity=rng.choice([0.0, 0.7]))
        elif kind == "soft":
            c.update(call="soft", algo=rng.choice(["filter", "filter", "vmp", "mmp"]), agents=_log_int(rng, 16, 2000),
                     steps=rng.randint(4, 32))
        elif kind == "slide":
            c.update(call="slide", agents=_log_int(rng, 16, 1024), steps=rng.randint(4, 24), iters=rng.randint(4, 12))
        else:
            if F < 2:
                continue
            c.update(algo=rng.choice(["filter", "vmp"]), agents=_log_int(rng, 32, 1024), steps=rng.randint(4, 20),
                     bdep=" ".join(f"{f}{(f + 1) % F}" for f in range(F)))
        if kind in ("filter", "window", "slide") and rng.random() < 0.2:
            c.update(arith="f32", damping=0.5)
        NT = c["agents"] * c["steps"]
        entries = sum(m[i] * math.prod(n[f] for f in d) for i, d in enumerate(dep))
        if NT > _UNITS or work(c)["flops"] > _FLOPS or (c["own"] and c["agents"] * entries > _OWN_ENTRIES):
            continue
        if kind == "soft" and (NT * sum(math.prod(n[f] for f in g) for g in _groups(n, dep)) > _SOFT_ENTRIES or sum(m) > 384):
            continue
        return c


# ---- what a call cannot do without ----------------------------------------------------------------

def _groups(n, dep):
    """The distinct sets of coupled factors (modalities on the same set share one contraction)."""
    return {tuple(sorted(f for f in d if n[f] > 1)) for d in dep} - {()}


def work(case):
    n, m, U, dep = _ints(case["n"]), _ints(case["m"]), _ints(case["U"]), _lists(case["dep"])
    N, T, K, S, F, M = case["agents"], case["steps"], case["iters"], sum(n), len(n), len(m)
    par = _lists(case["bdep"]) if case["bdep"] else [[f] for f in range(F)]
    trans = [n[f] * math.prod(n[g] for g in par[f]) for f in range(F)]   # entries of a transition per action
    slices = [math.prod(n[f] for f in d) for d in dep]                   # entries of one outcome's slice
    # all leave-one-out messages of a group of P states: two multiply-adds per entry and iteration
    flops = 4.0 * sum(math.prod(n[f] for f in g) for g in _groups(n, dep) if len(g) > 1) * N * T * K
    flops += 2.0 * sum(trans) * N * T if case["algo"] == "filter" else 4.0 * sum(trans) * N * T * K
    if case["call"] == "soft":
        flops += 2.0 * N * T * sum(a * b for a, b in zip(m, slices))
        bytes_ = 4.0 * N * T * sum(m)
    else:
        bytes_ = 4.0 * N * T * M
    bytes_ += 4.0 * N * (T - 1) * F
    bytes_ += 4.0 * N * T * (S * (2 if case["extras"] else 1) + (F if case["extras"] else 0))
    if case["call"] in ("tick", "slide"):
        bytes_ += 4.0 * N * (S + F) + (4.0 * N * T * S if case["call"] == "slide" else 0.0)
    if case["own"]:   # each agent's observed slices and taken transitions, or all of them if fewer
        bytes_ += 4.0 * N * sum(p * min(T, k) for p, k in zip(slices, m))
        bytes_ += 4.0 * N * (sum(e * min(T, u) for e, u in zip(trans, U)) + S)
    else:
        bytes_ += 4.0 * (sum(a * b for a, b in zip(m, slices)) + sum(e * u for e, u in zip(trans, U)) + S)
    return {"bytes": bytes_, "flops": flops}


# ---- inputs ---------------------------------------------------------------------------------------

def _simplex(shape, axis, gen, half=False):
    """Dirichlet(1), or Dirichlet(1/2) (half), along an axis: normalised exponential or squared normal draws."""
    x = torch.empty(shape, device="cuda")
    x = x.normal_(generator=gen).square_() if half else x.exponential_(generator=gen)
    return x.div_(x.sum(dim=axis, keepdim=True).clamp_min_(1e-30))


def _sparse(a, share, axis, gen):
    """The given share of entries zeroed, columns renormalised, empty columns uniform."""
    if share <= 0.0:
        return a
    a.mul_(torch.rand(a.shape, device="cuda", generator=gen) >= share)
    tot = a.sum(dim=axis, keepdim=True)
    return torch.where(tot > 0, a / tot.clamp_min(1e-30), 1.0 / a.shape[axis]).contiguous()


def _model(case, gen):
    n, m, U, dep = _ints(case["n"]), _ints(case["m"]), _ints(case["U"]), _lists(case["dep"])
    G = case["agents"] if case["own"] else 1
    bdep = _lists(case["bdep"]) if case["bdep"] else None
    A = [_sparse(_simplex((G, m[i]) + tuple(n[f] for f in d), 1, gen), case["sparsity"], 1, gen)
         for i, d in enumerate(dep)]
    B, D = [], []
    for f, nf in enumerate(n):
        par = tuple(n[g] for g in bdep[f]) if bdep else (nf,)
        b = _simplex((G, nf) + par + (U[f],), 1, gen, half=case["sticky"])
        if case["sticky"] and not bdep:
            b = 0.5 * b + 0.5 * torch.eye(nf, device="cuda").reshape(1, nf, nf, 1)
        B.append(b.contiguous())
        D.append(_simplex((G, nf), 1, gen) if case["prior"] else torch.full((G, nf), 1.0 / nf, device="cuda"))
    return n, m, U, dep, bdep, G, A, B, D


def _sample(case, n, m, U, dep, bdep, G, A, B, D, gen):
    """Observation and action streams sampled from the model (and the action before the first step)."""
    N, T, F = case["agents"], case["steps"], len(n)
    rows = torch.arange(N, device="cuda") if G > 1 else torch.zeros(N, dtype=torch.int64, device="cuda")

    def pick(p):
        return torch.multinomial(p, 1, generator=gen)[:, 0]

    def flat(factors, s):
        k = torch.zeros(N, dtype=torch.int64, device="cuda")
        for f in factors:
            k = k * n[f] + s[f]
        return k

    a_flat = [A[i].reshape(G, m[i], -1) for i in range(len(m))]
    b_flat = [B[f].reshape(G, n[f], -1) for f in range(F)]
    act = torch.stack([torch.randint(0, U[f], (N, T), device="cuda", generator=gen) for f in range(F)], 2)
    obs = torch.empty((N, T, len(m)), dtype=torch.int32, device="cuda")
    s = [pick(D[f][rows]) for f in range(F)]
    for t in range(T):
        for i, d in enumerate(dep):
            obs[:, t, i] = pick(a_flat[i][rows, :, flat(d, s)])
        if t + 1 < T:
            s = [pick(b_flat[f][rows, :, flat(bdep[f] if bdep else [f], s) * U[f] + act[:, t + 1, f]]) for f in range(F)]
    act = act.to(torch.int32)
    return obs, act[:, 1:].contiguous(), act[:, 0].contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, m, U, dep, bdep, G, A, B, D = _model(case, gen)
    obs, act, act_prev = _sample(case, n, m, U, dep, bdep, G, A, B, D, gen)
    N, T, S = case["agents"], case["steps"], sum(n)
    st = {"case": case, "obs": obs, "act": act if T > 1 else None, "act_prev": act_prev}
    if case["call"] == "soft":
        # a detector's confidence: most of the weight on the outcome, the rest spread over all of them
        parts = []
        for i, mi in enumerate(m):
            w = _simplex((N, T, mi), 2, gen)
            hot = torch.nn.functional.one_hot(obs[:, :, i].long(), mi)
            parts.append(0.8 * hot + 0.2 * w)
        st["obs"] = torch.cat(parts, 2).to(torch.float32).contiguous()
    if case["call"] in ("tick", "slide"):
        st["q_prev"] = torch.cat([_simplex((N, k), 1, gen) for k in n], 1).contiguous()
    if case["call"] == "slide":
        st["q_init"] = torch.cat([_simplex((N, T, k), 2, gen) for k in n], 2).contiguous()
    st["model"] = bi.Model(n, m, dep, U, G, A, B, D, arith=case["arith"], bdep=bdep)
    if case["damping"] != 1.0:
        st["model"].set_damping(case["damping"])
    st["out"] = {"q": torch.empty((N, T, S), device="cuda")}
    if case["extras"]:
        st["out"]["logq"] = torch.empty((N, T, S), device="cuda")
        st["out"]["argmax"] = torch.empty((N, T, len(n)), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()   # A, B and D are released here; the model keeps its packed copies
    return st


def run(state):
    c, md, out = state["case"], state["model"], state["out"]
    to = {"q_out": out["q"], "logq_out": out.get("logq"), "argmax_out": out.get("argmax")}
    if c["call"] == "tick":
        md.bi_filter_from(state["obs"], state["act"], state["q_prev"], state["act_prev"], c["iters"], **to)
    elif c["call"] == "slide":
        md.run_from(c["algo"], state["obs"], state["act"], state["q_prev"], state["act_prev"], c["iters"],
                    q_init=state["q_init"], **to)
    elif c["call"] == "soft":
        md.run_soft(c["algo"], state["obs"], state["act"], c["iters"], **to)
    else:
        md.run(c["algo"], state["obs"], state["act"], c["iters"], **to)
    return out


def tolerance(case):
    """Outputs are float32.  Float64 arithmetic leaves them their own rounding (6e-8) and little else on dense
    models; float32 arithmetic carries sums of logarithms (about -50, so 3e-6 absolute) and is used damped.  The
    undamped iteration on a sparse A amplifies the last bit of single agents by factors up to 1e9 (1e-14 of
    a table-driven exponential to 1e-5), so single values may be further off there.  Most probable
    states differ only where two states tie to that accuracy."""
    tol = {"rel": 1e-5} if case["arith"] == "f32" else {"rel": 1e-6}
    if case["sparsity"] > 0.0:
        tol = {"rel": 1e-5, "max": 0.02}
    if case["extras"]:
        tol["differ"] = 1e-4
    return tol
