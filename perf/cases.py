"""Timed cases: the work a program has this library do, through the public Python binding.

A case is a dict of plain values; `prepare` builds the problem, the context (or batch, or
server) and the host buffers a program keeps, `run` is one pass through the entry points and
returns everything the pass computes: spin states, energies, int64 statistics, swap counts and
the rung permutation. All outputs are whole numbers.

Kinds:
  run     one context: pt_run(sweeps, per_swap), then the state and the statistics are read
  steps   one context driven by the caller's own loop of pt_sweep and pt_swap
  resume  one context restored from a checkpoint, run on, and checkpointed again
  batch   uneven independent requests in one persistent launch, results of each read back
  serve   a burst of requests through the continuous-batching server
"""
from __future__ import annotations

import math
import time

import numpy as np
import torch

from paper_1004_0023_gb300 import instances, pt


def listed():
    return [
        # an interactive loop on the smallest workload: a few sweeps, a swap pass, again, then a
        # look at the statistics. Launches and latency decide.
        {"name": "steps_n16", "kind": "steps", "graph": "regular", "n": 16, "degree": 3, "jmax": 2, "hmax": 1,
         "P": 32, "R": 16, "ladder": "linear", "sweeps": 100, "per_swap": 5},
        # the smallest workload run whole: 10^4 sweeps with a swap pass after each
        {"name": "run_n16", "kind": "run", "graph": "regular", "n": 16, "degree": 3, "jmax": 2, "hmax": 1,
         "P": 32, "R": 16, "ladder": "linear", "sweeps": 10000, "per_swap": 1},
        # the larger plain workload
        {"name": "run_n256", "kind": "run", "graph": "regular", "n": 256, "degree": 3, "jmax": 2, "hmax": 1,
         "P": 64, "R": 64, "ladder": "geometric", "sweeps": 2000, "per_swap": 1},
        # the lattice of K4,4 cells whose int8 chain is larger than a CTA's shared memory
        {"name": "run_lattice", "kind": "run", "graph": "chimera", "rows": 16, "cols": 16, "jmax": 4, "hmax": 0,
         "P": 128, "R": 96, "ladder": "geometric", "sweeps": 500, "per_swap": 1},
        # classical parallel tempering over temperatures (one copy per chain)
        {"name": "run_classical", "kind": "run", "graph": "regular", "n": 256, "degree": 3, "jmax": 2, "hmax": 1,
         "P": 1, "R": 64, "ladder": "temperature", "sweeps": 2000, "per_swap": 1},
        # a copy count that is no multiple of 8, an odd site count, a ragged ladder, rare swaps
        {"name": "run_ragged", "kind": "run", "graph": "sparse", "n": 97, "degree": 4, "jmax": 2, "hmax": 1,
         "P": 20, "R": 37, "ladder": "geometric", "sweeps": 1000, "per_swap": 5},
        # a denser graph than the lattices: degree 12
        {"name": "run_dense", "kind": "run", "graph": "sparse", "n": 64, "degree": 12, "jmax": 2, "hmax": 1,
         "P": 32, "R": 40, "ladder": "geometric", "sweeps": 1000, "per_swap": 1},
        # couplings of a wider integer range, swap pass after every second sweep
        {"name": "run_wide", "kind": "run", "graph": "sparse", "n": 300, "degree": 6, "jmax": 10, "hmax": 10,
         "P": 40, "R": 48, "ladder": "geometric", "sweeps": 1000, "per_swap": 2},
        # a job continued from its checkpoint: restore, run, checkpoint
        {"name": "resume_n512", "kind": "resume", "graph": "regular", "n": 512, "degree": 3, "jmax": 2, "hmax": 1,
         "P": 64, "R": 32, "ladder": "geometric", "sweeps": 300, "per_swap": 1},
        # the batched size mix: N 32..1024 on two graph families, P 32..128, R 16..128
        {"name": "batch_mix", "kind": "batch", "count": 128, "mix": 1, "n_lo": 32, "n_hi": 1024, "p_lo": 32,
         "p_hi": 128, "r_lo": 16, "r_hi": 128, "sweeps": 100, "per_swap": 1},
        # many small requests at once
        {"name": "batch_small", "kind": "batch", "count": 64, "mix": 2, "n_lo": 16, "n_hi": 64, "p_lo": 16,
         "p_hi": 64, "r_lo": 8, "r_hi": 32, "sweeps": 2000, "per_swap": 1},
        # a burst of requests that arrive together at the server
        {"name": "serve_burst", "kind": "serve", "count": 12, "mix": 3, "n_lo": 32, "n_hi": 512, "p_lo": 32,
         "p_hi": 128, "r_lo": 8, "r_hi": 32, "sweeps": 600, "per_swap": 1},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "steps", "resume", "batch", "serve"])
    if kind in ("batch", "serve"):
        n_hi = _log_int(rng, 48, 1024 if kind == "batch" else 512)
        r_hi = _log_int(rng, 10, 128 if kind == "batch" else 40)
        return {"kind": kind, "count": rng.randint(8, 96) if kind == "batch" else rng.randint(3, 14),
                "mix": rng.randint(10, 10 ** 6), "n_lo": max(8, n_hi // 16), "n_hi": n_hi,
                "p_lo": rng.choice([8, 16, 32]), "p_hi": rng.choice([32, 64, 128]), "r_lo": max(2, r_hi // 6),
                "r_hi": r_hi, "sweeps": rng.randint(20, 100), "per_swap": rng.choice([1, 1, 2, 5])}
    c = {"kind": kind}
    c["graph"] = rng.choice(["regular", "regular", "chimera", "sparse", "sparse"])
    if c["graph"] == "regular":
        c["n"], c["degree"] = 2 * _log_int(rng, 8, 512), 3
    elif c["graph"] == "chimera":
        c["rows"], c["cols"] = rng.randint(1, 16), rng.randint(1, 16)
    else:
        c["n"], c["degree"] = _log_int(rng, 16, 400), rng.choice([4, 5, 6, 7, 9, 12, 16])
        c["degree"] = min(c["degree"], c["n"] - 2)
    c["jmax"] = rng.choice([1, 2, 2, 4, 10 if c.get("degree", 6) <= 7 else 4])
    c["hmax"] = rng.choice([0, 1, 2])
    n = _sites(c)
    style = rng.random()
    if style < 0.12 and kind == "run" and n <= 1024:
        c["P"] = 1
    elif style < 0.35:
        c["P"] = 2 * rng.randint(1, 40)
    else:
        c["P"] = 8 * _log_int(rng, 1, 16)
    if c.get("degree", 6) > 7 or c["P"] % 8:
        while n * c["P"] > 65536:
            c["P"] -= 2
    c["R"] = _log_int(rng, 3, 100)
    c["ladder"] = "temperature" if c["P"] == 1 else rng.choice(["linear", "geometric"])
    c["per_swap"] = rng.choice([1, 1, 1, 2, 5, 10])
    slow = c.get("degree", 6) > 7 or c["P"] % 8 != 0
    budget = (2e8 if slow else 1.5e9) / (n * c["P"] * c["R"])
    c["sweeps"] = int(min(2000, max(20, budget)))
    if kind == "steps":
        c["per_swap"] = max(2, c["per_swap"])
        c["sweeps"] = min(c["sweeps"], 100) // c["per_swap"] * c["per_swap"]
    return c


def _sites(case):
    return 8 * case["rows"] * case["cols"] if case["graph"] == "chimera" else case["n"]


def _values(vmax, zero):
    return tuple(v for v in range(-vmax, vmax + 1) if v or zero)


def _sparse_graph(n, degree, rng):
    """Random simple graph with every degree at most `degree` and most sites at it."""
    a, b = np.triu_indices(n, 1)
    deg = [0] * n
    ei, ej = [], []
    for k in rng.permutation(a.size).tolist():
        i, j = int(a[k]), int(b[k])
        if deg[i] < degree and deg[j] < degree:
            deg[i] += 1
            deg[j] += 1
            ei.append(i)
            ej.append(j)
            if 2 * len(ei) >= n * degree - 1:
                break
    return np.asarray(ei, np.int32), np.asarray(ej, np.int32)


def _ladder(case):
    kind, R, P = case["ladder"], case["R"], case["P"]
    if kind == "temperature":
        return instances.gamma_ladder("geometric", 0.1, 3.0, R), np.zeros(R)
    if kind == "linear":
        return np.full(R, 0.05), instances.gamma_ladder("linear", 0.1, 3.0, R)
    return np.full(R, 0.02), instances.gamma_ladder("geometric", 0.05, 4.0, R)


def _problem(case, seed):
    rng = np.random.default_rng([seed, 77])
    if case["graph"] == "regular":
        ei, ej = instances.random_regular_graph(case["n"], case["degree"], rng)
    elif case["graph"] == "chimera":
        ei, ej = instances.chimera_graph(case["rows"], case["cols"])
    else:
        ei, ej = _sparse_graph(case["n"], case["degree"], rng)
    n = _sites(case)
    J = rng.choice(np.asarray(_values(case["jmax"], False), np.int32), ei.size)
    h = rng.choice(np.asarray(_values(case["hmax"], True), np.int32), n)
    T, gamma = _ladder(case)
    return instances.Problem(n, ei, ej, J, h, case["P"], T, gamma, 0x5EED0000 + seed, case["sweeps"],
                             case["per_swap"], case.get("name", ""))


def _mix_sizes(case):
    """(graph, n or (rows, cols), P, R) of every request: the case's own, whatever the seed."""
    rng = np.random.default_rng([case["mix"], case["count"]])
    ps = [p for p in (8, 16, 32, 64, 128) if case["p_lo"] <= p <= case["p_hi"]] or [case["p_lo"]]
    out = []
    for _ in range(case["count"]):
        n = int(rng.integers(case["n_lo"], case["n_hi"] + 1))
        P = ps[int(rng.integers(0, len(ps)))]
        R = int(rng.integers(case["r_lo"], case["r_hi"] + 1))
        if rng.integers(0, 2) == 0:
            out.append(("regular", n + n % 2, P, R))
        else:
            cells = max(1, n // 8)
            rows = max(1, math.isqrt(cells))
            out.append(("chimera", (rows, max(1, cells // rows)), P, R))
    return out


def _mix(case, seed):
    rng = np.random.default_rng([seed, 78])
    probs = []
    for k, (graph, size, P, R) in enumerate(_mix_sizes(case)):
        shape = {"n": size} if graph == "regular" else {"rows": size[0], "cols": size[1]}
        probs.append(instances.make_problem(graph, rng, P=P, R=R, n_sweeps=case["sweeps"],
                                            sweeps_per_swap=case["per_swap"], seed=0x5EED0000 + 1000 * seed + k,
                                            **shape))
    return probs


def _pinned(*shape):
    """Host memory that results are copied into, as a program that reads them often keeps it."""
    return torch.empty(shape, dtype=torch.int8, pin_memory=True).numpy()


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    kind = case["kind"]
    if kind == "batch":
        s.probs = _mix(case, seed)
        s.batch = pt.Batch(s.probs)
        sizes = [p.attempts_per_sweep for p in s.probs]
        s.flat = _pinned(sum(sizes))
        at = np.concatenate([[0], np.cumsum(sizes)])
        s.out = [s.flat[at[k]:at[k + 1]] for k in range(len(sizes))]
    elif kind == "serve":
        s.probs = _mix(case, seed)
        s.server = pt.Server(arena_bytes=1 << 30)
    else:
        s.prob = _problem(case, seed)
        s.ctx = pt.PT.from_problem(s.prob)
        s.out = _pinned(s.prob.R, s.prob.n, s.prob.P)
        if kind == "resume":
            # the checkpoint of an earlier job
            s.ctx.run(10 * case["per_swap"], case["per_swap"])
            s.saved = s.ctx.checkpoint()
    torch.cuda.synchronize()
    return s


_OBS = ("E", "M", "n_meas", "sum_E", "sum_E2", "sum_M", "sum_M2", "flip_acc", "swap_att", "swap_acc", "replica_at")


def _flat_obs(all_obs):
    return np.concatenate([np.asarray(o[k], np.int64) for o in all_obs for k in _OBS])


def run(state):
    case = state.case
    kind = case["kind"]
    if kind == "batch":
        state.batch.run()
        obs = [state.batch.obs(k) for k in range(len(state.probs))]
        for k, out in enumerate(state.out):
            state.batch.read_state(k, out)
        return {"state": state.flat, "obs": _flat_obs(obs)}
    if kind == "serve":
        srv = state.server
        ids = [srv.submit(p) for p in state.probs]
        got = {}
        while len(got) < len(ids):
            finished = srv.step()
            for rid in finished:
                got[rid] = srv.result(rid)
                srv.release(rid)
            if not finished:
                time.sleep(0.0002)
        return {"state": np.concatenate([got[i][0].reshape(-1) for i in ids]),
                "obs": _flat_obs([got[i][1] for i in ids])}
    ctx = state.ctx
    if kind == "steps":
        for _ in range(case["sweeps"] // case["per_swap"]):
            ctx.sweep(case["per_swap"])
            ctx.swap()
    else:
        if kind == "resume":
            ctx.restore(*state.saved)
        ctx.run(case["sweeps"], case["per_swap"])
    out = ctx.read_state(state.out)
    return dict(ctx.obs(), state=out)


def _shapes(case):
    """(sites, mean degree, P, R) of every problem of a case."""
    if case["kind"] in ("batch", "serve"):
        for graph, size, P, R in _mix_sizes(case):
            if graph == "regular":
                yield size, 3.0, P, R
            else:
                rows, cols = size
                yield 8 * rows * cols, 2.0 * (16 * rows * cols + 4 * (rows - 1) * cols + 4 * rows * (cols - 1)) / (
                    8 * rows * cols), P, R
    elif case["graph"] == "chimera":
        rows, cols = case["rows"], case["cols"]
        yield _sites(case), 2.0 * (16 * rows * cols + 4 * (rows - 1) * cols + 4 * rows * (cols - 1)) / (
            8 * rows * cols), case["P"], case["R"]
    else:
        yield case["n"], float(case["degree"]), case["P"], case["R"]


def work(case):
    """Bytes: each chain's spins in and out once, the couplings, and the statistics. Operations per
    spin-flip attempt: 2 d + 2 for the field of d neighbours and the site's own, 3 for the
    Trotter neighbours, 3 for the table entry, the comparison and the flip, and a quarter of a
    Philox4x32-10 call (10 rounds of 2 products and 4 exclusive-ors)."""
    nbytes = ops = 0.0
    for n, d, P, R in _shapes(case):
        attempts = float(n) * P * R * case["sweeps"]
        nbytes += 2.0 * n * P * R + 8.0 * n * (d + 1) + 8.0 * 11 * R
        ops += attempts * (2 * d + 2 + 3 + 3 + 15)
    return {"bytes": nbytes, "flops": ops}


def exact(case, seed):
    """Every output is a whole number and has to be equal; there is no rounded value to bound."""
    return None
