"""The measured cases: what a user has the T-count search do, through the
public calls of ``paper_1606_07413_gb300``.

kind "step"    Problem.walk_step: f of a list of states (the smallest calls).
kind "walk"    Problem.level_walk_static: fresh trails on every walk, then
               `steps` steps of each, with its distinguished points stored.
kind "search"  Problem.run_walks / wait up to a step budget: walk, re-walk of
               the merges and collection, launch after launch.
kind "exact"   Problem.run_walks / wait with exhaustive_first: a T-count
               settled by the exhaustive pass over its level.
kind "batch"   Batch: a group of targets admitted, walked for some rounds,
               polled and removed.

Sizes are those of the repository's workloads (n = 2, 3, 4; levels 3, 5, 7;
4096, 2^16 and 2^20 walks; theta 2^-1 .. 2^-12), and odd ones between them.

Which of two merging trails a table slot keeps depends on the order in which
the GPU's warps reach it, so the merge list, the merge counters and (where
several claws exist) the decomposition differ between two runs on the same
inputs; the outputs below are the ones the inputs determine.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_1606_07413_gb300 as Q
from paper_1606_07413_gb300 import workloads as W

LEN = {2: 32, 3: 48, 4: 64}  # state bits of the default parameters


def listed():
    return [
        # a handful of states of the smallest problem: launch latency
        dict(name="step_n2_k3", kind="step", n=2, t=3, k=3, count=4096),
        # f of a ragged list of 4-qubit states at an odd level
        dict(name="step_n4_k7", kind="step", n=4, t=7, k=7, count=50021),
        # the 2-qubit level walk at its configured size
        dict(name="walk_n2_k3", kind="walk", n=2, t=3, k=3, walks=4096, steps=512, dp_bits=6),
        # the 3-qubit level walk at its configured size, one default launch
        dict(name="walk_n3_k5", kind="walk", n=3, t=5, k=5, walks=1 << 16, steps=64, dp_bits=10),
        # the 4-qubit level walk at its configured size (the largest level)
        dict(name="walk_n4_k7", kind="walk", n=4, t=7, k=7, walks=1 << 20, steps=16, dp_bits=12),
        # the same at a large theta, as time-to-solution runs use it, an even
        # level and a number of walks that fills no group
        dict(name="walk_n4_k6_theta4", kind="walk", n=4, t=6, k=6, walks=100003, steps=24, dp_bits=2),
        # a target with so many rotations that C^ leaves int8
        dict(name="walk_n4_k7_wide", kind="walk", n=4, t=15, k=7, walks=1 << 15, steps=16, dp_bits=12),
        # whole searches with the default parameters up to a step budget
        dict(name="search_n3_t5", kind="search", n=3, t=5, budget=1 << 23),
        dict(name="search_n4_t6", kind="search", n=4, t=6, budget=1 << 26),
        # T-counts settled exactly: an odd level streams products without C^,
        # an even one probes with products that carry it
        dict(name="exact_n4_t5", kind="exact", n=4, t=5),
        dict(name="exact_n4_t6", kind="exact", n=4, t=6),
        # 3- and 4-qubit targets together, from admission to removal
        dict(name="batch_24", kind="batch", jobs=24, rounds=6),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, even over the logarithm."""
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["step", "walk", "walk", "walk", "search", "exact", "batch"])
    n = rng.choice([2, 3, 4])
    if kind == "step":
        k = rng.randint(2, 7)
        return dict(kind=kind, n=n, t=rng.randint(3, 7), k=k, count=_spread(rng, 257, 1 << 19))
    if kind == "walk":
        wide = n == 4 and rng.random() < 0.2
        k = rng.randint(4 if n > 2 else 2, 7)
        return dict(kind=kind, n=n, t=15 if wide else rng.randint(3, 9), k=k,
                    walks=_spread(rng, 1000, 1 << 15 if wide else 1 << 18), steps=_spread(rng, 8, 64 if n > 2 else 512),
                    dp_bits=rng.randint(1, 12))
    if kind == "search":
        n = rng.choice([3, 4])
        return dict(kind=kind, n=n, t=rng.randint(5, 6) if n == 4 else rng.randint(5, 7),
                    budget=_spread(rng, 1 << 22, 1 << 25))
    if kind == "exact":
        n, t = rng.choice([(2, 4), (2, 5), (2, 6), (3, 5), (3, 6), (3, 7), (4, 4), (4, 5)])
        return dict(kind=kind, n=n, t=t, salt=rng.randint(0, 999))
    return dict(kind=kind, jobs=rng.randint(5, 28), rounds=rng.randint(2, 8))


def _anticommute(n, p, q):
    m = (1 << n) - 1
    return (bin((p >> n) & (q & m)).count("1") + bin((p & m) & (q >> n)).count("1")) & 1


def _target(n, t, rng, late=None):
    """Gates of R(P_t) .. R(P_1) C0 with neighbouring rotations that do not
    commute, so that they come in one order only.  late: the place (1 .. t)
    whose rotation has one of the highest codes, the ones an exhaustive pass
    that counts its points by that place meets last."""
    top = 4 ** n
    while True:
        p = [int(v) for v in rng.integers(1, top, size=t)]
        if late:
            p[late - 1] = int(rng.integers(top - max(2, top // 24), top))
        if all(_anticommute(n, p[i], p[i + 1]) for i in range(t - 1)):
            break
    rot = np.asarray([(W.OP_RP, v, 0) for v in p], dtype=np.int32).reshape(-1, 3)
    return np.concatenate([W.clifford_word(rng, n), rot], axis=0)


def _problem(n, t, k_max, rng, late=None, **params):
    """A problem whose T-count bound from the denominator is t itself, as a
    target of t random rotations nearly always has it (the ladder then starts
    at level t), with trails of its own."""
    params = Q.default_params(n, seed=int(rng.integers(1, 1 << 62)), **params)
    for _ in range(16):
        prob = Q.Problem.from_circuit(n, _target(n, t, rng, late), k_max, params)
        if n == 2 or t > 9 or prob.sde == t:
            return prob
        prob.close()
    raise RuntimeError("no target of this T-count was drawn")


def prepare(case, seed):
    rng = np.random.Generator(np.random.PCG64([seed, case.get("n", 0), case.get("t", case.get("jobs", 0))]))
    kind, dev = case["kind"], torch.device("cuda")
    s = {"case": case}
    if kind == "step":
        n, k, count = case["n"], case["k"], case["count"]
        s["prob"] = _problem(n, case["t"], max(k, case["t"]), rng)
        s["chunk"] = int(rng.integers(1, 4 ** n)) if k & 1 else 0
        s["x"] = torch.from_numpy(W.seeded_states(count, LEN[n], seed).view(np.int64)).to(dev)
        s["y"] = torch.empty_like(s["x"])
        s["dp"] = torch.empty(count, dtype=torch.uint8, device=dev)
    elif kind == "walk":
        s["prob"] = _problem(case["n"], case["t"], 15, rng, table_log2=18, walks=case["walks"])
        s["walks"] = torch.zeros(case["walks"], 4, dtype=torch.int64, device=dev)
        s["merges"] = torch.zeros(1 << 20, 3, dtype=torch.int64, device=dev)
        s["counts"] = torch.zeros(8, dtype=torch.int64, device=dev)
    elif kind == "search":
        s["prob"] = _problem(case["n"], case["t"], case["t"], rng, stop_on_claw=0, exhaustive_log2=0)
    elif kind == "exact":
        # the place the pass counts by: the last rotation of its streamed side
        t = case["t"]
        late = t // 2 + 1 if t & 1 else t
        s["prob"] = _problem(case["n"], t, t, rng, late=late, exhaustive_first=1, exhaustive_log2=32)
    else:
        s["batch"] = Q.Batch(Q.default_batch_params(max_jobs=32))
        # levels that a few rounds do not settle, so that every job walks throughout
        s["probs"] = [_problem(n, t, t, rng) for n, t in
                      [(3 + int(rng.integers(0, 2)), 6 + int(rng.integers(0, 2))) for _ in range(case["jobs"])]]
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        s["prob"].walk_step(case["k"], s["chunk"], 1, s["x"], s["y"], s["dp"])
        return {"states": s["y"], "distinguished": s["dp"]}
    if kind == "walk":
        s["prob"].level_walk_static(case["k"], 1, case["dp_bits"], 1, s["walks"], case["steps"], s["merges"],
                                    s["counts"])
        # steps, W-side steps, distinguished points, abandoned trails
        return {"walks": s["walks"], "counts": s["counts"][:4]}
    if kind == "search":
        s["prob"].run_walks(step_budget=case["budget"])
        r = s["prob"].wait()
        return {f: r[f] for f in ("k", "sde", "version", "steps", "w_steps", "dps", "abandoned", "launches")}
    if kind == "exact":
        s["prob"].run_walks()
        r = s["prob"].wait()
        return {"paulis": np.asarray(r["paulis"], np.int64),
                **{f: r[f] for f in ("status", "k", "t_count", "sde", "certified_levels", "cert_points")}}
    batch = s["batch"]
    jobs = [batch.add(p) for p in s["probs"]]
    for _ in range(case["rounds"]):
        batch.round()
    rs = [batch.poll(j) for j in jobs]
    for j in jobs:
        batch.remove(j)
    return {f: np.asarray([r[f] for r in rs], np.int64) for f in ("k", "sde", "steps", "w_steps", "dps", "abandoned")}


def work(case):
    """Per W-side step (half of all) the contraction of 4^n - 1 weights, each
    of two parts, with 4^n - 1 columns; per step one multiply-add per weight
    for each rotation.  Bytes: states in and out (8 or 32 bytes each) and C^
    as bytes; a search or a pass keeps its work on the chip."""
    kind = case["kind"]
    if kind == "batch":
        steps, n, h, moved = case["jobs"] * case["rounds"] * 2048 * 64, 4, 3, case["jobs"] * 2048 * 64
    elif kind == "exact":
        n, h = case["n"], case["t"] // 2
        xi = 4 ** n - 1
        stored, streamed = xi ** h, xi ** (h + (case["t"] & 1))
        w_points = stored if case["t"] & 1 else streamed
        return {"bytes": 16.0 * stored + 8.0 * streamed,
                "flops": 4.0 * w_points * xi * xi + 4.0 * (stored + streamed) * xi * h}
    else:
        n = case["n"]
        h = case.get("k", case["t"]) // 2
        steps = {"step": case.get("count"), "walk": case.get("walks", 0) * case.get("steps", 0),
                 "search": case.get("budget")}[kind]
        moved = {"step": 17 * case.get("count", 0), "walk": 64 * case.get("walks", 0), "search": 0}[kind]
    d = 4 ** n - 1
    return {"bytes": float(moved + 2 * 4 ** (2 * n)), "flops": float(steps) * (2.0 * d * d + 4.0 * h * d)}


def exact(case, seed):
    """Every output is a whole number."""
    return None
