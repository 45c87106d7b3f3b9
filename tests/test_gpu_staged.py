"""Analysis of larger tasksets out of stages in shared memory against the oracle, where it can go
wrong: sizes at the edges of the bins, arrays that start on odd elements, slices at the very ends of
their arrays, tasksets too large for a stage, values beyond the 32-bit path, offsets out of range,
undecided tasksets that are kept or left to the second launch, priorities with gaps and best-effort
tasks."""
import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding, taskgen
from paper_2406_05221_b200.taskgen import ARRAY_FIELDS, TasksetBatch
from tests.helpers import ALL_MODES, BEST_EFFORT, batch_of, direct_most

pytestmark = pytest.mark.gpu

FILLERS = direct_most()   # with these a batch is more than the path without a plan takes


def taskset(rng, n, load, segs, gaps=False):
    ts = []
    for i in range(n):
        T = int(rng.integers(1000, 1_000_000))
        eta = int(rng.integers(0, segs + 1))
        w = max(1, int(T * load / n / (2 * eta + 1)))
        ts.append(dict(T=T, D=int(rng.integers(T // 2, T + 1)), prio=0, core=int(rng.integers(0, 8)),
                       cseg=[int(rng.integers(0, w + 1)) for _ in range(eta + 1)],
                       gseg=[(int(rng.integers(0, w // 4 + 1)), int(rng.integers(0, w + 1))) for _ in range(eta)]))
    order = sorted(range(n), key=lambda i: ts[i]["T"])
    for r, i in enumerate(order):
        ts[i]["prio"] = (n - r) * (3 if gaps else 1) - (2 if gaps else 0)
    return ts


def check(tasksets, policies, shift=0, L=1024, ovh=20, fillers=FILLERS, spoil=None):
    """Parity on `tasksets` at the two ends of a batch whose middle is one-task tasksets, after
    `spoil(batch)` has changed it."""
    torch = pytest.importorskip("torch")
    half = len(tasksets) // 2
    few = batch_of([[dict(T=50, prio=1, core=0, cseg=[7])]] * 64)
    middle = TasksetBatch.concat([few] * (fillers // 64 + 1))
    batch = TasksetBatch.concat([batch_of(tasksets[:half]), middle, batch_of(tasksets[half:])])
    if spoil:
        spoil(batch)
    t = {}
    for f in ARRAY_FIELDS:   # the arrays start `shift` elements into an allocation of exactly their size
        room = torch.empty(getattr(batch, f).shape[0] + shift, dtype=torch.int64, device="cuda")
        t[f] = room[shift:]
        t[f].copy_(torch.from_numpy(getattr(batch, f)))
    ts = binding.DeviceTasksets(t)
    for policy in policies:
        wcrt, sched = binding.rta_batch(ts, policy, L, ovh)
        torch.cuda.synchronize()
        ref, ref_s, _ = rta.analyse(batch, policy, L, ovh)
        assert np.array_equal(wcrt.cpu().numpy(), ref), hex(policy)
        assert np.array_equal(sched.cpu().numpy(), ref_s), hex(policy)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [33, 64, 65, 80, 96, 97, 128, 129, 192, 193, 256])
def test_sizes_and_alignment(n, shift):
    rng = np.random.default_rng(1000 * shift + n)
    tasksets = [taskset(rng, n - (k % 2), load, 4) for k, load in enumerate([0.05, 0.5, 2.0, 8.0] * 3)]
    check(tasksets, [0, binding.BUSY, 1, 1 | binding.BUSY], shift)


@pytest.mark.parametrize("segs", [0, 12, 40, 70])
def test_segments_beyond_a_stage(segs):
    """No segments at all; so many that some or all tasksets do not fit a stage (or the 32-bit path)."""
    rng = np.random.default_rng(segs)
    tasksets = [taskset(rng, n, 1.0, segs if k % 3 else 1) for k, n in enumerate([40, 70, 90, 100, 150, 230] * 3)]
    check(tasksets, ALL_MODES)


def test_gaps_ties_best_effort_and_bad_values():
    rng = np.random.default_rng(5)
    tasksets = []
    for k in range(48):
        n = int(rng.integers(33, 120))
        ts = taskset(rng, n, float(rng.choice([0.1, 1.0])), 3, gaps=k % 2 == 0)
        if k % 4 == 1:
            for tk in ts[: n // 2]:
                tk["prio"] = 5
        if k % 6 == 2:
            ts[n // 2]["T"] = ts[n // 2]["D"] = 1 << 30      # beyond the 32-bit path
        if k % 6 == 3:
            ts[n - 1]["D"] = ts[n - 1]["T"] + 1              # outside the domain
        if k % 6 == 4:
            ts[0]["cseg"] = [(1 << 26) - 1] * 40             # a sum that overflows 32 bits
        if k % 6 == 5:
            ts[3]["prio"] = 1 << 40
        tasksets.append(ts)
    for policy in (0, 1, binding.BUSY | BEST_EFFORT, 1 | BEST_EFFORT):
        check(tasksets, [policy])


@pytest.mark.parametrize("every", [1, 2, 7])
def test_deferred_tasksets(every):
    """Long runs of tasksets that converge beyond the first ranks, alone or among others that do not."""
    rng = np.random.default_rng(every)
    kinds = [taskset(rng, n, load, 2) for n in (40, 80, 130, 200, 250) for load in (0.02, 6.0)]
    tasksets = [kinds[2 * (k % 5) + (0 if k % every == 0 else 1)] for k in range(4200)]
    check(tasksets, [0, 1], fillers=8400)


@pytest.mark.parametrize("kind", ["cseg", "gseg"])
@pytest.mark.parametrize("where", ["below", "beyond"])
def test_constant_offsets_out_of_range(kind, where):
    """Tasksets without segments of one kind whose offsets of that kind are all the same value outside
    the array: no segment is read for them, every step between two offsets is 0, and they are
    INVALID all the same.  The segments of the other kind make them miss within the first ranks."""
    rng = np.random.default_rng(3)
    tasksets = []
    for n in (33, 64, 80, 96, 120, 128, 180, 192, 200, 256) * 2:
        ts = taskset(rng, n, 60.0, 2)
        for tk in ts:
            if kind == "gseg":
                tk["gseg"] = []
            else:
                tk["cseg"], tk["gseg"] = [], tk["gseg"] or [(1, 5)]
        tasksets += [ts, taskset(rng, n, 60.0, 2)]   # (the second: its own first offset is in front of it)

    def spoil(batch):
        off, total = getattr(batch, kind + "_off"), getattr(batch, kind + "_off")[-1]
        large = np.nonzero(np.diff(batch.task_off) > 32)[0]
        for t in large[::2]:
            a, b = batch.task_off[t], batch.task_off[t + 1]
            off[a:b + 1] = -3 if where == "below" else total + 5
    check(tasksets, [0, binding.BUSY, 1, 1 | binding.BUSY], spoil=spoil)


@pytest.mark.parametrize("tasks_per_core,segs,overhead", [(16, (1, 5), 50), (16, (3, 8), 50), (16, (3, 8), 2), (12, (3, 8), 5), (8, (3, 8), 5)])
def test_stages_of_large_tasksets(tasks_per_core, segs, overhead):
    """A batch of tasksets of one size with many segments, so that a stage takes up to a quarter of an SM's
    shared memory; some miss among the first ranks, some later."""
    torch = pytest.importorskip("torch")
    params = taskgen.GenParams(seed=15, cores=(16, 16), tasks_per_core=(tasks_per_core, tasks_per_core), util_per_core=(0.02, 0.8),
                               period_us=(1e3, 1e6), gpu_frac=0.8, gpu_segments=segs, gpu_ratio=(0.2, 0.6))
    count = direct_most() + 37
    ts = binding.generate_device(params, 0, count)
    batch = TasksetBatch(**{f: ts.t[f].cpu().numpy() for f in ARRAY_FIELDS})
    sample = np.sort(np.random.default_rng(2).choice(count, 500, replace=False))
    part, n = batch.select(sample), 16 * tasks_per_core
    for policy in (0, binding.BUSY, 1, 1 | binding.BUSY):
        wcrt, sched = binding.rta_batch(ts, policy, 1024, overhead)
        torch.cuda.synchronize()
        ref, ref_s, _ = rta.analyse(part, policy, 1024, overhead)
        assert np.array_equal(wcrt.cpu().numpy().reshape(count, n)[sample].reshape(-1), ref), hex(policy)
        assert np.array_equal(sched.cpu().numpy()[sample], ref_s), hex(policy)
