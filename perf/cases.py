"""What the performance of this library is measured on: calls that its users make, over the sizes they
make them at.  Everything goes through the public binding (``Simulation`` and its methods).

A case is a dict of plain values; ``listed`` names the fixed ones, ``draw`` makes others of the same
ranges, ``prepare`` builds what a program holds before the call, ``run`` is one pass, ``work`` the bytes
and operations that no implementation of the pass can do without, ``exact`` plain 64-bit values where
there is a closed form.

Kinds of pass:
  run         advance a system by ``steps`` steps on the device, then read its state into the caller's
              page-locked buffers (a trajectory sampled every so many steps).  The A+B<->C systems start
              at their mass-action composition and the network changes slowly, so passes on one state
              are alike.
  exchange    one step between host programs: state uploaded from host arrays, one step, state back
  pair_probs  p_enc and p_reac of a batch of separations
  propagate   new separation vectors of encountered pairs drawn from the full propagator
  first_passage  first-contact bins of encountered pairs
"""
import math

import numpy as np
import torch

import paper_1107_0270_gb300 as rd
import workloads as W

PER_UM3 = W.PER_UM3_PER_UM * 10.0      # particles per um^3 at 10 uM, the density of the 3D A+B<->C system


def listed():
    return [
        # a small box in the default mode (FP64, directions from the full propagator): tests, teaching
        # examples, one replica of a parameter scan on its own
        {"name": "small_fp64", "kind": "run", "system": "reversible", "n": 1000, "dt": 1e-5, "precision": "fp64",
         "angle": "exact", "steps": 10},
        # the same box in the fast mode over many steps: nothing but latency and launches
        {"name": "small_mixed", "kind": "run", "system": "reversible", "n": 1000, "dt": 1e-5, "precision": "mixed",
         "angle": "free_step", "steps": 200},
        # the benchmark's system, fast mode
        {"name": "reversible_mixed", "kind": "run", "system": "reversible", "n": 100_000, "dt": 1e-5,
         "precision": "mixed", "angle": "free_step", "steps": 50},
        # the benchmark's system in the default mode
        {"name": "reversible_fp64", "kind": "run", "system": "reversible", "n": 100_000, "dt": 1e-5,
         "precision": "fp64", "angle": "exact", "steps": 4},
        # crowded 2D membrane with excluded volume: many encounters, conflicts and directions per step
        {"name": "membrane_mixed", "kind": "run", "system": "membrane", "n": 200_000, "dt": 1e-4,
         "precision": "mixed", "angle": "exact", "steps": 20},
        # a small membrane patch in the default mode: quadrature per pair
        {"name": "membrane_fp64", "kind": "run", "system": "membrane", "n": 1500, "dt": 1e-4, "precision": "fp64",
         "angle": "exact", "steps": 1},
        # a batch of thousands of independent boxes of very different sizes (parameter inference)
        {"name": "ensemble_mixed", "kind": "run", "system": "ensemble", "n": 4096, "dt": 1e-5, "precision": "mixed",
         "angle": "exact", "steps": 8},
        # one large box of a five-species network, ten million particles
        {"name": "network_mixed", "kind": "run", "system": "network", "n": 10_000_000, "dt": 1e-5,
         "precision": "mixed", "angle": "free_step", "steps": 8},
        # coupling to a host program that owns the state, an odd size
        {"name": "exchange_mixed", "kind": "exchange", "system": "reversible", "n": 99_991, "dt": 1e-5,
         "precision": "mixed", "angle": "free_step", "steps": 1},
        # probability batches of another simulator's candidate pairs, larger than any cache, a ragged end
        {"name": "pair_probs_mixed", "kind": "pair_probs", "n": (1 << 25) + 3, "dt": 1e-5, "precision": "mixed",
         "dim": 3},
        # another simulator's encountered pairs moved by the full propagator
        {"name": "propagate_mixed", "kind": "propagate", "n": 500_001, "dt": 1e-5, "precision": "mixed", "dim": 3},
        # first-contact times of encountered pairs to a thousandth of the step
        {"name": "first_passage_mixed", "kind": "first_passage", "n": 1 << 20, "dt": 1e-5, "precision": "mixed",
         "levels": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "exchange", "pair_probs", "propagate", "first_passage"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    dt = 10.0 ** rng.choice([-6, -5.5, -5, -4.5, -4])
    if kind in ("run", "exchange"):
        c = {"kind": kind, "system": "reversible", "dt": dt, "precision": precision,
             "angle": rng.choice(["exact", "free_step"])}
        if kind == "run":
            c["system"] = rng.choice(["reversible", "reversible", "membrane", "ensemble", "network"])
        if c["system"] == "ensemble":
            c.update(n=_log(rng, 16, 4096), dt=1e-5, precision="mixed")
        elif c["system"] == "network":
            c.update(n=_log(rng, 20_000, 10_000_000), dt=min(dt, 1e-5), precision="mixed")
        elif c["system"] == "membrane":
            c.update(n=_log(rng, 300, 1500) if precision == "fp64" else _log(rng, 500, 200_000), dt=1e-4)
        elif precision == "fp64" and c["angle"] == "exact":
            c.update(n=_log(rng, 300, 20_000 if dt > 1e-5 else 100_000))
        else:
            c.update(n=_log(rng, 300, 100_000))
        slow = c["precision"] == "fp64" and (c["angle"] == "exact" or c["system"] == "membrane")
        c["steps"] = 1 if kind == "exchange" or (slow and c["system"] == "membrane") else rng.randint(1, 4 if slow else 9)
        return c
    if kind == "pair_probs":
        dim = rng.choice([3, 3, 2])
        top = 1 << (25 if precision == "mixed" else (24 if dim == 3 else 14))
        return {"kind": kind, "n": _log(rng, 1000, top), "dt": dt if dim == 3 else 1e-4, "precision": precision, "dim": dim}
    if kind == "propagate":
        top = 500_001 if precision == "mixed" else 1000
        return {"kind": kind, "n": _log(rng, 60, top), "dt": min(dt, 1e-5), "precision": precision, "dim": 3}
    return {"kind": kind, "n": _log(rng, 1000, 1 << 20), "dt": min(dt, 1e-5), "precision": precision,
            "levels": rng.randint(1, 12)}


def _system(case, seed):
    name = case.get("system", "reversible" if case.get("dim", 3) == 3 else "membrane")
    n, dt = case["n"] if "system" in case else 100_000, case["dt"]
    if name == "reversible":
        s = W.reversible_3d(dt=dt, seed=seed, n_each=n, L=(n / PER_UM3) ** (1.0 / 3.0), equilibrium_start=True)
    elif name == "membrane":
        s = W.membrane_2d(seed=seed, n_each=n, L=math.sqrt(n / 2000.0), dt=dt, equilibrium_start=True)
    elif name == "ensemble":
        s = W.ensemble_3d(n_replicas=n)   # the replicas' sizes belong to the case, the draws to the seed
        s.seed = seed
        rule, kd = s.pairs[0], s.decays[0].kd
        for r in s.replicas:              # bound pairs x of mass action: ka (n - x)^2 / V = kd x
            m, h = r.n_init[0], 0.5 * kd * r.L ** 3 / rule.ka
            x = int(round(m + h - math.sqrt(h * (2.0 * m + h))))
            r.n_init = [m - x, m - x, x]
    else:
        s = W.network_3d(dt=dt, seed=seed, scale=n / 1e7)
    s.angle = case.get("angle", "exact")
    return s


def _host_buffers(sim, system):
    """Page-locked arrays for the state, with room for its growth during the passes, as a program that
    samples a trajectory keeps them."""
    cap = int(1.25 * sum(sum(r.n_init) for r in system.replica_list())) + 1024

    def pinned(shape, dtype):
        return torch.zeros(shape, dtype=dtype, pin_memory=True).numpy()

    out = {"x": pinned((cap, 3), torch.float64), "species": pinned(cap, torch.int32),
           "ids": pinned(cap, torch.int32).view(np.uint32), "next_id": pinned(sim.n_replicas, torch.int32).view(np.uint32)}
    if sim.n_replicas > 1:
        out["replica"] = pinned(cap, torch.int32)
    return out


def _separations(case, system, seed):
    """Start separations uniform in the cut-off shell and free end points, a quarter of them near
    contact: the candidate pairs of a step, as device tensors (r0 and r lengths, r0 as vectors)."""
    pr = system.pairs[0]
    dim, n = system.dim, case["n"]
    gen = torch.Generator(device="cuda").manual_seed(int(seed))

    def uniform(*shape):
        return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=gen)

    ell = math.sqrt(2.0 * (system.D[pr.s1] + system.D[pr.s2]) * system.dt)
    rc = pr.sigma + system.c_cut * ell
    r0 = (pr.sigma ** dim + uniform(n) * (rc ** dim - pr.sigma ** dim)) ** (1.0 / dim)
    v = torch.randn(n, 3, dtype=torch.float64, device="cuda", generator=gen)
    if dim == 2:
        v[:, 2] = 0.0
    v /= v.norm(dim=1, keepdim=True)
    step = torch.randn(n, 3, dtype=torch.float64, device="cuda", generator=gen)
    if dim == 2:
        step[:, 2] = 0.0
    k = n // 4
    r0[:k] = pr.sigma + 0.05 * ell * uniform(k)
    r = (r0[:, None] * v + ell * step).norm(dim=1)
    r[:k] = pr.sigma + 0.05 * ell * uniform(k)
    return r0, r, r0[:, None] * v, uniform


def _encountered(case, system, seed):
    """Encountered pairs: candidate pairs kept with their encounter probability (the closed form in 3D),
    the kept ones repeated up to the batch's size."""
    r0, r, vec, uniform = _separations(case, system, seed)
    pr = system.pairs[0]
    p, _ = _closed_forms(r0, r, pr, system.D[pr.s1] + system.D[pr.s2], system.dt)
    keep = (uniform(r0.numel()) < p).nonzero().flatten()
    at = keep.repeat(-(-case["n"] // max(1, keep.numel())))[:case["n"]]
    return r0[at].contiguous(), r[at].contiguous(), vec[at].contiguous(), uniform


def prepare(case, seed):
    system = _system(case, seed)
    sim = rd.Simulation(system, precision=case["precision"])
    state = {"case": case, "sim": sim}
    if case["kind"] in ("run", "exchange"):
        state["out"] = _host_buffers(sim, system)
        if case["kind"] == "exchange":
            state["now"] = sim.get_state(out=state["out"])
    elif case["kind"] == "pair_probs":
        state["r0"], state["r"], _, _ = _separations(case, system, seed)
    elif case["kind"] == "propagate":
        _, _, state["r0"], uniform = _encountered(case, system, seed)
        state["u"] = uniform(case["n"], 4)
    else:
        state["r0"], state["r"], _, _ = _encountered(case, system, seed)
        state["streams"] = torch.arange(case["n"], dtype=torch.int64, device="cuda") + (int(seed) << 24)
    return state


def run(state):
    case, sim = state["case"], state["sim"]
    if case["kind"] == "run":
        sim.run(case["steps"])
        return _whole(sim.get_state(out=state["out"]), state["out"])
    if case["kind"] == "exchange":
        now = state["now"]
        sim.set_state(now["x"], now["species"], now["ids"], None, now["next_id"], now["step"])
        sim.step()
        state["now"] = sim.get_state(out=state["out"])
        return _whole(state["now"], state["out"])
    if case["kind"] == "pair_probs":
        pe, pr = sim.pair_probs(state["r0"], state["r"])
        return {"p_enc": pe, "p_reac": pr}
    if case["kind"] == "propagate":
        return {"r": sim.propagate(state["r0"], state["u"])}
    return sim.first_passage(state["r0"], state["r"], state["streams"], case["levels"])


def _whole(st, out):
    """The caller's buffers (the first n entries are the state) and the counters."""
    whole = {k: (v.view(np.int32) if v.dtype == np.uint32 else v) for k, v in out.items()}
    return {**whole, "n": st["ids"].shape[0], "step": st["step"]}


def _particles(case):
    """Particles of a system case (the ensemble's sizes are log-uniform in 64..8192 of two species)."""
    if case["system"] == "ensemble":
        return 2100.0 * case["n"]
    return {"reversible": 1.25, "membrane": 1.2, "network": 1.0}[case["system"]] * case["n"]


def work(case):
    fp64 = case["precision"] == "fp64"
    if case["kind"] in ("run", "exchange"):
        n, rec = _particles(case), 36.0 if fp64 else 20.0        # position record and id
        # a step reads and writes every particle's record, and draws its displacement (one or two
        # Philox calls, two Box-Muller pairs); the caller's state is 32 bytes a particle
        to_host = 32.0 * n * (2 if case["kind"] == "exchange" else 1)
        flops = 200.0 * n
        if fp64 and case["angle"] == "exact":       # encounters per particle, each a partial-wave series
            flops += {"reversible": 9e-4, "membrane": 0.17}[case["system"]] * n * 3e6
        return {"bytes": 2.0 * rec * n * case["steps"] + to_host + rec * n, "flops": flops * case["steps"]}
    n = case["n"]
    if case["kind"] == "pair_probs":
        return {"bytes": 32.0 * n, "flops": (200.0 if case["dim"] == 3 or not fp64 else 2e5) * n}
    if case["kind"] == "propagate":
        return {"bytes": 80.0 * n, "flops": (400.0 if not fp64 else 5e6) * n}
    # one draw: four Philox calls, two Box-Muller pairs, two probabilities; about 1.5 draws a level,
    # a few more at the first
    return {"bytes": 48.0 * n, "flops": 500.0 * n * (5.0 + 1.5 * case["levels"])}


def _closed_forms(r0, r, rule, Drel, dt):
    """p_enc and p_reac of 3D pairs in 64 bits from the closed radial Green's functions (unit contact
    radius, tau = D dt / a^2)."""
    a = rule.sigma
    tau = Drel * dt / (a * a)
    s = math.sqrt(tau)
    R0, R = (r0 / a).clamp(min=1.0), (r / a)
    d0, d = R0 - 1.0, R.clamp(min=1.0) - 1.0
    p = torch.exp(-d * d0 / tau) * torch.expm1(-(d + d0 + 1.0) / tau) / torch.expm1(-(d + 1.0) * R0 / tau)
    p = torch.where(R <= 1.0, torch.ones_like(p), p)
    alpha = 1.0 + rule.ka / (4.0 * math.pi * a * Drel)
    z = (d + d0) / (2.0 * s)
    e = torch.special.erfcx(s + z)
    q = math.sqrt(math.pi) * s
    return p, (q * (alpha * torch.special.erfcx(alpha * s + z) - e) / (1.0 - q * e)).clamp(0.0, 1.0)


def exact(case, seed):
    """The closed forms of the 3D probabilities.  The other passes have no plain 64-bit value: a step, a
    propagated separation and a first-contact bin are random draws whose law is a series, a quadrature
    or a rejection loop per pair and whose accept-or-reject decisions a change of precision turns over."""
    if case["kind"] != "pair_probs" or case["dim"] != 3:
        return None
    system = _system(case, seed)
    r0, r, _, _ = _separations(case, system, seed)
    pr = system.pairs[0]
    p, q = _closed_forms(r0, r, pr, system.D[pr.s1] + system.D[pr.s2], system.dt)
    return {"p_enc": p, "p_reac": q}
