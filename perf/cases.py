"""Timed cases: what a program that uses this solver has it do, through the public calls.

A case is a dict of plain values.  ``op`` names the call:

* ``solve``     ``dgs_solve_ex`` on a square matrix that is in device memory, from the
                greedy start (the default), a random start or the last solution;
* ``rect``      ``dgs_solve_rect``: agents and jobs in unequal numbers;
* ``host``      ``dgs_solve_host``: the matrix in pinned host memory, both copies inside;
* ``batched``   ``dgs_solve_batched``: many instances of uneven size in one call;
* ``evaluate``  ``dgs_evaluate``: one difference evaluation of every agent and job.

``family`` is the kind of benefits: ``peer`` (peer assignment: positions in the unit
square, log-uniform capacities, integer noise), ``uniform`` (i.i.d. in [0, hi)) or
``geom`` (floored distances between random points in [0, 1000]^2).  All are int32, the
only type that the solver takes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1106_5694_gb300 import binding, inputs

PEER_POOL = 4  # batched: instances are leading blocks of this many peer matrices


def listed():
    return [
        # the smallest call: one small instance, where launches and host work count
        {"name": "solve_uniform_256", "op": "solve", "family": "uniform", "n": 256, "hi": 1000, "init": "greedy"},
        # an ordinary small peer assignment of odd size (its rows are not 16-byte aligned)
        {"name": "solve_peer_1021", "op": "solve", "family": "peer", "n": 1021, "init": "greedy"},
        # a peer assignment whose matrix stays in L2
        {"name": "solve_peer_4096", "op": "solve", "family": "peer", "n": 4096, "init": "greedy"},
        # the benchmark's instance: a large peer assignment
        {"name": "solve_peer_10000", "op": "solve", "family": "peer", "n": 10000, "init": "greedy"},
        # wide-range values without structure: thousands of sweeps
        {"name": "solve_uniform_10000", "op": "solve", "family": "uniform", "n": 10000, "hi": 1000000,
         "init": "greedy"},
        # the largest instance
        {"name": "solve_uniform_20000", "op": "solve", "family": "uniform", "n": 20000, "hi": 1000000,
         "init": "greedy"},
        # the paper's own workload: distances, random start, many exchanges per sweep
        {"name": "solve_geom_2048_random", "op": "solve", "family": "geom", "n": 2048, "init": "random"},
        # a periodic re-solve: a few peers changed, the last solution is the start
        {"name": "resolve_peer_3000", "op": "solve", "family": "peer", "n": 3000, "init": "warm"},
        # fewer agents than jobs (the rest stay free)
        {"name": "rect_peer_1500x2001", "op": "rect", "family": "peer", "n": 1500, "m": 2001},
        # the whole call from host memory
        {"name": "host_peer_10000", "op": "host", "family": "peer", "n": 10000},
        # a node that serves many groups of peers at once
        {"name": "batched_peer_1024", "op": "batched", "family": "peer", "count": 1024, "lo": 64, "hi_n": 4096,
         "sizes": 4},
        # the evaluation alone, of a given assignment
        {"name": "evaluate_peer_10000", "op": "evaluate", "family": "peer", "n": 10000},
    ]


def _size(rng, lo, hi):
    return int(min(hi, max(lo, math.floor(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "solve", "rect", "host", "batched", "evaluate"])
    if op == "solve":
        family, init = rng.choice([("peer", "greedy"), ("uniform", "greedy"), ("geom", "random"), ("peer", "warm")])
        top = {("peer", "greedy"): 20000, ("uniform", "greedy"): 16384, ("geom", "random"): 4096,
               ("peer", "warm"): 8192}[family, init]
        case = {"op": op, "family": family, "n": _size(rng, 64, top), "init": init}
        if family == "uniform":
            case["hi"] = rng.choice([1000, 1000000])
        return case
    if op == "rect":
        return {"op": op, "family": "peer", "n": _size(rng, 64, 6000), "m": _size(rng, 64, 6000)}
    if op == "host":
        return {"op": op, "family": "peer", "n": _size(rng, 64, 10000)}
    if op == "batched":
        return {"op": op, "family": "peer", "count": _size(rng, 16, 1024), "lo": 64,
                "hi_n": _size(rng, 512, 4096), "sizes": rng.randrange(1 << 20)}
    return {"op": op, "family": rng.choice(["peer", "uniform"]), "n": _size(rng, 64, 20000), "hi": 1000000}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _peer(n, m, g):
    """The distribution of ``inputs.peer_shaped``, drawn on the GPU."""
    def u(*shape):
        return torch.rand(*shape, generator=g, device="cuda")

    xy_a, xy_j = u(n, 2), u(m, 2)
    up, down = torch.exp(u(n) * math.log(100.0)), torch.exp(u(m) * math.log(100.0))
    out = torch.empty(n, m, dtype=torch.int32, device="cuda")
    for r0 in range(0, n, 2048):
        r1 = min(n, r0 + 2048)
        d = torch.sqrt((xy_a[r0:r1, None, 0] - xy_j[None, :, 0]) ** 2 + (xy_a[r0:r1, None, 1] - xy_j[None, :, 1]) ** 2)
        base = torch.floor(100.0 * torch.minimum(up[r0:r1, None], down[None, :]) * torch.exp(-4.0 * d))
        out[r0:r1] = base.to(torch.int32)
        out[r0:r1] += torch.randint(0, 16, (r1 - r0, m), generator=g, device="cuda", dtype=torch.int32)
    return out


def _geom(n, g):
    p = 1000.0 * torch.rand(n, 2, generator=g, device="cuda")
    out = torch.empty(n, n, dtype=torch.int32, device="cuda")
    for r0 in range(0, n, 2048):
        r1 = min(n, r0 + 2048)
        d = torch.sqrt((p[r0:r1, None, 0] - p[None, :, 0]) ** 2 + (p[r0:r1, None, 1] - p[None, :, 1]) ** 2)
        out[r0:r1] = torch.floor(d).to(torch.int32)
    return out


def _benefit(case, g):
    if case["family"] == "uniform":
        return torch.randint(0, case["hi"], (case["n"], case["n"]), generator=g, device="cuda", dtype=torch.int32)
    if case["family"] == "geom":
        return _geom(case["n"], g)
    return _peer(case["n"], case.get("m", case["n"]), g)


def prepare(case, seed):
    g = _generator(seed)
    op = case["op"]
    if op == "batched":
        pool = [_peer(case["hi_n"], case["hi_n"], g) for _ in range(PEER_POOL)]
        sizes = inputs.batched_sizes(case["count"], case["lo"], case["hi_n"], case["sizes"])
        sigma = torch.empty(int(sizes.sum()), dtype=torch.int32, device="cuda")  # every instance's result, end to end
        return {"op": op, "a": [pool[k % PEER_POOL][:n, :n].contiguous() for k, n in enumerate(sizes.tolist())],
                "sigma": sigma, "parts": list(sigma.split(sizes.tolist()))}
    a = _benefit(case, g)
    state = {"op": op, "a": a, "opts": {}}
    if op == "host":
        pinned = torch.empty(a.shape, dtype=torch.int32, pin_memory=True)
        pinned.copy_(a)
        return {"op": op, "a": pinned.numpy(), "pinned": pinned}
    if op == "evaluate":
        state["sigma"] = torch.randperm(case["n"], generator=g, device="cuda").to(torch.int32)
    elif op == "solve" and case["init"] == "random":
        state["opts"] = {"init": binding.DGS_INIT_RANDOM, "seed": int(seed)}
    elif op == "solve" and case["init"] == "warm":
        # the solution before one peer in a hundred was replaced by another
        n = case["n"]
        before = a.clone()
        k = max(1, n // 100)
        before[:k] = _peer(k, n, g)
        last = binding.dgs_solve(before)[1]
        state["opts"] = {"init": binding.DGS_INIT_USER, "init_sigma": last}
    return state


# ------------------------------------------------------------------ one pass
def _ok(status):
    if status != binding.DGS_OK:
        raise RuntimeError(binding.dgs_status_string(status))


def run(state):
    op, a = state["op"], state["a"]
    if op == "batched":
        status, _, objectives, _, _ = binding.dgs_solve_batched(a, state["parts"])
        _ok(status)
        return {"sigma": state["sigma"], "objective": np.array(objectives, dtype=np.int64)}
    if op == "evaluate":
        status, agent_gain, agent_job, job_gain, job_agent = binding.dgs_evaluate(a, state["sigma"])
        _ok(status)
        return {"agent_gain": agent_gain, "agent_job": agent_job, "job_gain": job_gain, "job_agent": job_agent}
    if op == "host":
        status, sigma, objective, stats = binding.dgs_solve_host(a)
    elif op == "rect":
        status, sigma, objective, stats = binding.dgs_solve_rect(a)
    else:
        status, sigma, objective, stats = binding.dgs_solve_ex(a, **state["opts"])
    _ok(status)
    return {"sigma": sigma, "objective": objective, "sweeps": stats["sweeps"]}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    """Bytes: every benefit read once, each output written once.  Operations: the gain
    a[i][k] + a[j][l] - a[i][l] - a[j][k] of every exchange of two agents once (three
    additions beside the shared sums), without which no result is known to be a local
    optimum."""
    if case["op"] == "batched":
        sizes = inputs.batched_sizes(case["count"], case["lo"], case["hi_n"], case["sizes"]).astype(np.int64)
        return {"bytes": int((4 * sizes * sizes + 4 * sizes + 8).sum()), "flops": int((3 * sizes * (sizes - 1) // 2).sum())}
    n = case["n"]
    m = case.get("m", n)
    s = max(n, m)
    out = 16 * n if case["op"] == "evaluate" else 4 * n + 12
    extra = 4 * n if case["op"] == "evaluate" or case.get("init") == "warm" else 0
    return {"bytes": 4 * n * m + out + extra, "flops": 3 * s * (s - 1) // 2}


def exact(case, seed):
    """The evaluation by its definition in 64-bit torch arithmetic: agent i on job s(i)
    gains G[i][k] = a[i][s(k)] + a[k][s(i)] - D[i] - D[k] by exchanging jobs with agent k;
    the best partner's lowest job (agent slots) and lowest agent (job slots).  A solve's
    result is what its sequence of exchanges ends at, which has no such closed form."""
    if case["op"] != "evaluate":
        return None
    state = prepare(case, seed)
    a, s = state["a"], state["sigma"].long()
    n = a.shape[0]
    diag = a[torch.arange(n, device="cuda"), s].long()
    out = {k: torch.zeros(n, dtype=torch.int64, device="cuda")
           for k in ("agent_gain", "agent_job", "job_gain", "job_agent")}
    agents = torch.arange(n, device="cuda")
    for r0 in range(0, n, 512):
        r1 = min(n, r0 + 512)
        gain = a[r0:r1][:, s].long() + a[:, s[r0:r1]].long().T - diag[r0:r1, None] - diag[None, :]
        best = gain.max(dim=1).values
        hit = gain == best[:, None]
        some = best > 0
        job = torch.where(hit, s[None, :], n).min(dim=1).values
        agent = torch.where(hit, agents[None, :], n).min(dim=1).values
        best = torch.where(some, best, 0)
        out["agent_gain"][r0:r1] = best
        out["agent_job"][r0:r1] = torch.where(some, job, -1)
        out["job_gain"][s[r0:r1]] = best
        out["job_agent"][s[r0:r1]] = torch.where(some, agent, -1)
    return out
