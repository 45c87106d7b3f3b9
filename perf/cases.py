"""The timed cases of this library: what its users have it do, from a handful of tasksets to a
million, through the public entry points of ``paper_2406_05221_b200.binding``.

A case names an operation (``op``), the generator stream its tasksets come from (``workload``,
``stream``: the ranges of ``taskgen.WORKLOADS``), how many tasksets it holds (``count``) and the
options of the call.  Device-resident inputs are made on the GPU by the integer-only generator
from the seed alone; a program that loops over calls keeps its output buffers and its workspace,
so ``prepare`` makes them once, except where ``fresh`` says that the call makes its own.  Where
the number of tasks of a batch varies from seed to seed the kept buffers are sized, as such a
program sizes them, for the most tasks the batch can hold.
All results are whole numbers, so every case is compared exactly.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2406_05221_b200 import binding, taskgen

DEVICE = "cuda:0"
ANALYSES = {"gcaps": binding.GCAPS_SUSPEND, "gcaps_busy": binding.GCAPS_BUSY,
            "rr": binding.RR_SUSPEND, "rr_busy": binding.RR_BUSY}


def listed():
    """Twelve calls that stand for how the library is used."""
    return [
        # an interactive query or an online admission test: a handful of tasksets of very
        # different sizes in one call
        _case("admission_37", "batch", "divergence", 0, 37, analysis="gcaps"),
        # the reference-sized batch (1,000 small tasksets): launches and latency, the call making
        # its own buffers
        _case("small_1000", "batch", "pr1", 0, 1_000, analysis="gcaps", fresh=True),
        # one point of a schedulability curve: 100,000 tasksets of 20 tasks, half of them
        # schedulable, so that the recurrence works
        _case("curve_point_100k", "batch", "sweep", 4, 100_000, analysis="gcaps"),
        # the large configuration under both policies (one call each): staging and early misses
        _case("large_gcaps_1m", "batch", "large", 0, 1_000_000, analysis="gcaps"),
        _case("large_rr_1m", "batch", "large", 0, 1_000_000, analysis="rr"),
        # 80-task tasksets that are all schedulable: every task of every taskset converges
        _case("converging_gcaps_200k", "batch", "large_light", 0, 200_000, analysis="gcaps"),
        # tasksets of 4 to 192 tasks side by side, busy-waiting lemmas, a ragged count
        _case("mixed_sizes_busy_700k", "batch", "divergence", 0, 700_001, analysis="gcaps_busy"),
        # the driver-model study: 25 (timeslice, overhead) pairs of one resident batch
        _case("driver_model_25_pairs", "sweep", "rr_model", 0, 200_000, analysis="rr", pairs=25),
        # every taskset under all four analyses in one pass (the comparison of the experiments)
        _case("four_analyses_100k", "multi", "sweep", 2, 100_001, analysis="all", pairs=1),
        # separate priorities for GPU segments, searched level by level
        _case("gpu_priorities_100k", "assign", "large", 0, 100_000, busy=False),
        # a Monte-Carlo experiment: the tasksets are made on the device and analysed at once
        _case("generate_analyse_250k", "generate", "large", 0, 250_000, analysis="gcaps"),
        # a batch that lives in page-locked host memory, both policies from one copy
        _case("host_batch_60k", "host", "large", 0, 60_000),
    ]


def _case(name, op, workload, stream, count, **options):
    return dict(name=name, op=op, workload=workload, stream=stream, count=count, **options)


def draw(rng):
    """One more case of the same operations, streams and ranges of sizes."""
    op = rng.choice(["batch"] * 5 + ["sweep", "multi", "assign", "generate", "host"])
    streams = ["pr1", "sweep", "large", "large_light", "rr_model"]
    if op not in ("assign", "generate"):  # (their result buffers are made by the call: whole sizes)
        streams.append("divergence")
    workload = rng.choice(streams)
    stream = rng.randrange(len(taskgen.WORKLOADS[workload].streams))
    tasks, csegs, gsegs = _mean_sizes(workload, stream)
    # at most what the largest listed case of the operation does, by tasks
    most = {"batch": 60e6, "sweep": 4.8e6, "multi": 8e6, "assign": 8e6, "generate": 20e6, "host": 4.8e6}[op]
    if workload == "large_light":
        most = min(most, 2e6)  # every task runs its recurrence
    count = max(1, int(math.exp(rng.uniform(math.log(8.0), math.log(most / tasks)))))
    c = dict(op=op, workload=workload, stream=stream, count=count)
    if op == "batch":
        c.update(analysis=rng.choice(list(ANALYSES)), fresh=workload != "divergence" and rng.random() < 0.3,
                 # priorities handed in with gaps, and tasks without a real-time priority
                 sparse=rng.random() < 0.15, best_effort=rng.random() < 0.15)
    elif op == "sweep":
        c.update(analysis=rng.choice(list(ANALYSES)), pairs=rng.randint(2, 25))
    elif op == "multi":
        c.update(analysis=rng.choice(["all", "suspend", "busy"]), pairs=rng.randint(1, 3))
    elif op == "assign":
        c.update(busy=rng.random() < 0.3)
    elif op == "generate":
        c.update(analysis=rng.choice(["gcaps", "rr"]))
    return c


def _mean_sizes(workload, stream):
    """Expected tasks, CPU segments and GPU segments of a taskset of the stream."""
    g = taskgen.WORKLOADS[workload].streams[stream]
    tasks = sum(g.cores) * sum(g.tasks_per_core) / 4.0
    gpu = round(g.gpu_frac * tasks) if g.gpu_mode == 0 else tasks
    gsegs = gpu * sum(g.gpu_segments) / 2.0
    return tasks, tasks + gsegs, gsegs


def _room(case):
    """The most tasks a batch of the case can hold."""
    g = taskgen.WORKLOADS[case["workload"]].streams[case["stream"]]
    return case["count"] * g.cores[1] * g.tasks_per_core[1]


def _analyses(case):
    a = case.get("analysis")
    return {"all": 15, "suspend": binding.GCAPS_SUSPEND | binding.RR_SUSPEND,
            "busy": binding.GCAPS_BUSY | binding.RR_BUSY}.get(a) or ANALYSES[a]


def _pairs(case, w):
    """The (timeslice, overhead) pairs of a sweep: the workload's own ones first."""
    if w.timeslices:
        both = [(L, o) for L in w.timeslices for o in w.overheads]
    else:
        both = [(L, max(1, w.overhead_us * k // 4)) for L in (256, 512, 1024, 2048, 4096) for k in range(1, 6)]
    step = max(1, len(both) // case["pairs"])
    both = both[::step][: case["pairs"]]
    return [L for L, _ in both], [o for _, o in both]


def _generator(case, seed):
    return dataclasses.replace(taskgen.WORKLOADS[case["workload"]].streams[case["stream"]],
                               seed=1 + seed % (1 << 62))


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


def prepare(case, seed):
    w = taskgen.WORKLOADS[case["workload"]]
    params, count, op = _generator(case, seed), case["count"], case["op"]
    s = {"case": case, "L": w.timeslice_us, "ovh": w.overhead_us}
    if op == "generate":
        s["params"], s["policy"] = params, binding.ANALYSIS_POLICY[_analyses(case)]
        return s
    ts = binding.generate_device(params, 0, count, device=DEVICE)
    if op == "host":
        arrays = {}
        for f in taskgen.ARRAY_FIELDS:
            arrays[f] = _pinned(ts.t[f].shape, torch.int64).copy_(ts.t[f]).numpy()
        s["arrays"] = arrays
        s["wcrt"] = [_pinned(_room(case), torch.int64).zero_().numpy() for _ in range(2)]
        s["sched"] = [_pinned(count, torch.uint8).zero_().numpy() for _ in range(2)]
        return s
    if case.get("sparse"):
        ts.t["priority"].mul_(3)
    flags = 0
    if case.get("best_effort"):  # the lowest priorities of every taskset become best-effort tasks
        ts.t["priority"].sub_(3 if case.get("sparse") else 2)
        flags = binding.BEST_EFFORT
    s["ts"] = ts
    s["kept"] = {}
    if not case.get("fresh"):
        s["kept"]["workspace"] = torch.empty(max(256, binding.workspace_bytes(count)), dtype=torch.uint8, device=DEVICE)
    if op == "assign":
        s["flags"] = binding.ASSIGN | (binding.BUSY if case["busy"] else 0)
        return s
    blocks = 1
    if op == "batch":
        s["policy"] = binding.ANALYSIS_POLICY[_analyses(case)] | flags
    elif op == "sweep":
        s["policy"] = binding.ANALYSIS_POLICY[_analyses(case)]
        s["Ls"], s["ovhs"] = _pairs(case, w)
        blocks = len(s["ovhs"])
    else:
        s["analyses"] = _analyses(case)
        s["Ls"], s["ovhs"] = _pairs(case, w)
        blocks = len(s["ovhs"]) * bin(s["analyses"]).count("1")
    if not case.get("fresh"):
        s["kept"]["out_wcrt"] = torch.zeros(blocks * _room(case), dtype=torch.int64, device=DEVICE)
        s["kept"]["out_sched"] = torch.zeros(blocks * count, dtype=torch.uint8, device=DEVICE)
    return s


def run(s):
    op = s["case"]["op"]
    if op == "batch":
        return binding.rta_batch(s["ts"], s["policy"], s["L"], s["ovh"], **s["kept"])
    if op == "sweep":
        return binding.rta_sweep(s["ts"], s["policy"], s["Ls"], s["ovhs"], **s["kept"])
    if op == "multi":
        return binding.rta_multi(s["ts"], s["analyses"], s["Ls"], s["ovhs"], **s["kept"])
    if op == "assign":
        return binding.rta_gpu_priority(s["ts"], s["flags"], s["ovh"], **s["kept"])
    if op == "generate":
        ts = binding.generate_device(s["params"], 0, s["case"]["count"], device=DEVICE)
        wcrt, sched = binding.rta_batch(ts, s["policy"], s["L"], s["ovh"])
        # the tasksets' per-task arrays with the results (the number of segments is random, so
        # arrays of segments have no fixed length; every segment is in the results' sums)
        return [wcrt, sched] + [ts.t[f] for f in taskgen.ARRAY_FIELDS if f[:4] not in ("cseg", "gseg") or f[-3:] == "off"]
    return binding.rta_batch_host_multi(s["arrays"], [binding.POLICY_GCAPS, binding.POLICY_RR], s["L"], s["ovh"],
                                        s["wcrt"], s["sched"])


def work(case):
    """Bytes: every input array read once, every result written once.  Operations: one addition
    per segment value and the constant part of Eq. 1 per task and analysis (16 operations); the
    sweeps of the recurrence depend on the drawn tasksets and are not counted."""
    tasks, csegs, gsegs = _mean_sizes(case["workload"], case["stream"])
    count, op = case["count"], case["op"]
    inputs = 8.0 * (6 * tasks + 3 + csegs + 2 * gsegs)
    result = 8.0 * tasks + 1
    k = {"batch": 1, "sweep": case.get("pairs", 1), "multi": case.get("pairs", 1), "assign": 1, "generate": 1, "host": 2}[op]
    if op == "multi":
        k *= bin(_analyses(case)).count("1")
    if op == "assign":
        result += 8.0 * tasks  # the level found beside the bound
    if op == "generate":  # written, then read and analysed once
        return {"bytes": count * (2 * inputs + result), "flops": count * (2 * csegs + 4 * gsegs + 32 * tasks)}
    return {"bytes": count * (inputs + k * result), "flops": count * (csegs + 2 * gsegs + 16 * tasks * max(1, k))}


def tolerance(case):
    return "exact"
