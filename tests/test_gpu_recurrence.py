"""The recurrence in single precision and its continuation in integers against the oracle, where they
can go wrong: periods on both sides of the single-precision limit in every place of the priority
order, deadlines that long climbs reach, tasks without any demand, tasksets that end on a block of
lanes.  Results are whole numbers, compared exactly."""
import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding, taskgen
from tests.helpers import ALL_MODES, batch_of, both_ways

pytestmark = pytest.mark.gpu

NARROW_LIMIT = 2_796_200   # kNarrowLimit of csrc/rta_recurrence.cuh


def check(tasksets, policies, L=1024, ovh=3):
    torch = pytest.importorskip("torch")
    batch = batch_of(tasksets)
    n, k = batch.n_tasks, batch.n_tasksets
    # (with fillers: the groups of 8 and 16 lanes, the stages and the second launch; without: a warp each)
    one = [binding.DeviceTasksets.from_host(b) for b in both_ways(batch)]
    several = [binding.DeviceTasksets.from_host(b) for b in both_ways(batch, several=True)]
    for policy in policies:
        analysis = {0: 1, binding.BUSY: 2, 1: 4, 1 | binding.BUSY: 8}[policy & 0x101]
        ref, ref_s, _ = rta.analyse(batch, policy, L, ovh)
        for ts in one:
            wcrt, sched = binding.rta_batch(ts, policy, L, ovh)
            torch.cuda.synchronize()
            assert np.array_equal(wcrt.cpu().numpy()[:n], ref), hex(policy)
            assert np.array_equal(sched.cpu().numpy()[:k], ref_s), hex(policy)
        ref2, ref2_s, _ = rta.analyse(batch, policy, L + 1, 0)
        for ts in several:
            many, many_s = binding.rta_multi(ts, analysis, [L, L + 1], [ovh, 0], flags=policy & binding.LITERAL)
            torch.cuda.synchronize()
            assert np.array_equal(many[0, 0].cpu().numpy()[:n], ref), hex(policy)
            assert np.array_equal(many[1, 0].cpu().numpy()[:n], ref2), hex(policy)
            assert np.array_equal(many_s[1, 0].cpu().numpy()[:k], ref2_s), hex(policy)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 16, 24, 25, 31, 32, 33, 64, 65, 80, 96, 97, 128, 129, 192, 255, 256])
def test_periods_around_the_limit(n):
    rng = np.random.default_rng(n)
    tasksets = []
    for k in range(24):
        ts = []
        for i in range(n):
            # none, some or all periods at or beyond the limit; the others well below or just below
            far = rng.random() < (0.0, 0.05, 0.5, 1.0)[k % 4]
            T = int(rng.integers(NARROW_LIMIT, 1 << 26)) if far else int(rng.choice(
                [rng.integers(2000, 90000), rng.integers(1 << 20, NARROW_LIMIT), NARROW_LIMIT - 1]))
            budget = max(4, int(T * rng.uniform(0.0, 1.2) / n))
            uses = rng.random() < 0.6
            ts.append(dict(T=T, D=int(rng.integers(T - T // 4, T + 1)), prio=0, core=int(rng.integers(0, 4)),
                           cseg=[int(rng.integers(0, budget))],
                           gseg=[(int(rng.integers(0, budget // 4)), int(rng.integers(0, budget // 2)))] if uses else []))
        order = rng.permutation(n) if k % 3 == 0 else sorted(range(n), key=lambda i: ts[i]["T"])
        for r, i in enumerate(order):
            ts[i]["prio"] = n - r
        tasksets.append(ts)
    check(tasksets, ALL_MODES)


@pytest.mark.parametrize("lanes", [1, 9, 40])
def test_long_climbs(lanes):
    """A core filled to the brim: the iterates climb by 2 per sweep, into the deadline or into the
    sweep limit (2^20 sweeps), at deadlines on both sides of what 2^20 sweeps reach."""
    sets = []
    for D in ((1 << 20) - 1, 1 << 20, (1 << 20) + 1, 2_000_000, (1 << 21) - 1, 1 << 21, (1 << 21) + 1, (1 << 21) + 2,
              (1 << 21) + 3, (1 << 21) + 5, NARROW_LIMIT - 1, NARROW_LIMIT, NARROW_LIMIT + 5):
        ts = [dict(T=2, prio=900, core=0, cseg=[2]), dict(T=D, prio=1, core=0, cseg=[1])]
        ts += [dict(T=100, prio=500 - i, core=1 + i, cseg=[3]) for i in range(lanes - 1)]
        sets.append(ts)
    check(sets, [0, binding.BUSY, 1], ovh=0)


@pytest.mark.parametrize("n", [3, 20, 80])
def test_tasks_without_demand(n):
    """A task of demand 0 has the bound 0 whatever is above it (its first iterate is a fixed point)."""
    tasksets = []
    for z in range(0, n, max(1, n // 7)):
        ts = [dict(T=1000 + i, prio=n - i, core=i % 2, cseg=[0] if i >= z else [2],
                   gseg=[(0, 0)] if i % 5 == 0 else []) for i in range(n)]
        tasksets.append(ts)
    for ovh in (0, 1):
        check(tasksets, ALL_MODES, ovh=ovh)


@pytest.mark.parametrize("count", [1, 2, 3, 4, 5, 8193, 12288, 12289])
def test_groups_of_a_warp(count):
    """Tasksets that share a warp end at different ranks and sweeps (one that declines the 32-bit
    path among them)."""
    torch = pytest.importorskip("torch")
    for name, stream in (("sweep", 5), ("pr1", 0), ("rr_model", 0)):
        batch = taskgen.WORKLOADS[name].generate(0, count, stream=stream)
        batch.period[batch.task_off[:-1][::5]] += 1 << 33
        ts = binding.DeviceTasksets.from_host(batch)
        for policy in (0, binding.BUSY, 1, 1 | binding.BUSY):
            wcrt, sched = binding.rta_batch(ts, policy, 512, 25)
            torch.cuda.synchronize()
            ref, ref_s, _ = rta.analyse(batch, policy, 512, 25)
            assert np.array_equal(wcrt.cpu().numpy(), ref), (name, hex(policy))
            assert np.array_equal(sched.cpu().numpy(), ref_s), (name, hex(policy))
