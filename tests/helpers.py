"""Shared helpers of the test-suite (fixture parsing, small random tasksets)."""
from __future__ import annotations

import os

import numpy as np

from paper_2406_05221_b200 import build
from paper_2406_05221_b200.taskgen import ARRAY_FIELDS, TasksetBatch

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")

POLICY = {"gcaps": 0, "rr": 1}
BUSY, LITERAL, BEST_EFFORT = 0x100, 0x200, 0x800
ALL_MODES = [0, BUSY, LITERAL, BUSY | LITERAL, 1, 1 | BUSY, 1 | LITERAL, 1 | BUSY | LITERAL]


def parse_vector_sets(name):
    """Reads a fixture of `taskset <name>` / `task ...` / `case ...` lines; returns a list of
    (taskset name, list of task dicts, list of cases), one entry per taskset of the file (a file
    without `taskset` lines holds one unnamed taskset)."""
    sets = []
    with open(os.path.join(GOLDEN, name)) as fh:
        for line in fh:
            line = line.split("#", 1)[0].strip()
            if not line:
                continue
            tok = line.split()
            if tok[0] == "taskset":
                sets.append((tok[1], [], []))
                continue
            if not sets:
                sets.append(("", [], []))
            _, tasks, cases = sets[-1]
            kv = dict(x.split("=", 1) for x in tok[2:])
            if tok[0] == "task":
                cseg = [int(x) for x in kv["cseg"].split(",") if x]
                gseg = [tuple(int(y) for y in x.split(":")) for x in kv["gseg"].split(",") if x]
                tasks.append(dict(T=int(kv["T"]), prio=int(kv["prio"]), core=int(kv["core"]),
                                  cseg=cseg, gseg=gseg))
            elif tok[0] == "case":
                flags = POLICY[kv["policy"]] | (BUSY if kv["busy"] == "1" else 0) | (
                    LITERAL if kv["literal"] == "1" else 0) | (
                    BEST_EFFORT if kv.get("be", "0") == "1" else 0)
                cases.append(dict(name=tok[1], policy=flags, L=int(kv["L"]), ovh=int(kv["ovh"]),
                                  expect=[int(x) for x in kv["expect"].split(",")]))
    return sets


def parse_vectors(name):
    """Reads a one-taskset fixture; returns (list of task dicts, list of cases)."""
    sets = parse_vector_sets(name)
    assert len(sets) == 1, name
    return sets[0][1], sets[0][2]


def random_tasksets(rng, count, max_tasks=6, max_cores=3, periods=(20, 30, 40, 60, 80, 120, 200),
                    max_gseg=3, wcet_hi=6, unique_prio=True):
    """Small random tasksets as lists of task dicts (rate-monotonic priorities)."""
    out = []
    for _ in range(count):
        n = int(rng.integers(1, max_tasks + 1))
        cores = int(rng.integers(1, max_cores + 1))
        ts = []
        for _i in range(n):
            T = int(rng.choice(periods))
            ng = int(rng.integers(0, max_gseg + 1))
            cs = [int(rng.integers(0, wcet_hi)) for _ in range(int(rng.integers(1, ng + 3)))]
            gs = [(int(rng.integers(0, 3)), int(rng.integers(0, wcet_hi))) for _ in range(ng)]
            ts.append(dict(T=T, D=int(rng.integers(max(1, T // 2), T + 1)), prio=0,
                           core=int(rng.integers(0, cores)), cseg=cs, gseg=gs))
        order = sorted(range(n), key=lambda i: (ts[i]["T"], i))
        for r, i in enumerate(order):
            ts[i]["prio"] = (n - r) if unique_prio else (n - r) // 2
        out.append(ts)
    return out


def batch_of(tasksets):
    return TasksetBatch.from_tasksets(tasksets)


def direct_most(several=False):
    """Batches of up to this many tasksets run without a plan; `several`: sweeps, several analyses and
    searches of GPU priorities."""
    return build.source_constant("kDirectSweepMost" if several else "kDirectMost")


def with_fillers(batch, several=False, middle=False):
    """`batch` and so many one-task tasksets behind it (or in its middle) that it runs with a plan and the
    kernels of the size bins."""
    few = batch_of([[dict(T=50, prio=1, core=0, cseg=[7])]] * 64)
    fillers = [few] * (max(0, direct_most(several) - batch.n_tasksets) // 64 + 1)
    half = batch.n_tasksets // 2 if middle else batch.n_tasksets
    return TasksetBatch.concat([batch.slice(0, half)] + fillers + [batch.slice(half, batch.n_tasksets)])


def repeated(batch, k):
    """The batch k times over."""
    offs = {f: np.concatenate([[0], np.tile(np.diff(getattr(batch, f)), k).cumsum()]) for f in ("task_off", "cseg_off", "gseg_off")}
    return TasksetBatch(**{f: offs[f] if f in offs else np.tile(getattr(batch, f), k) for f in ARRAY_FIELDS})


def left_by_tiles(workspace):
    """Tasksets that a call through tiles left to the launches behind it, from the header in its workspace.  (After
    a call with a plan these counters hold the tasksets of all size bins.)"""
    import torch
    return int(workspace[:256].view(torch.int32)[12:21].sum())


def both_ways(batch, several=False):
    """The batch as it is and, where that runs without a plan, with fillers behind it."""
    return [batch] if batch.n_tasksets > direct_most(several) else [batch, with_fillers(batch, several)]
