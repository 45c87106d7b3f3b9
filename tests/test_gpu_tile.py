"""Tasksets of up to 24 tasks in tiles, a lane or a few per taskset: sizes around the edges of the stage, what a walk
keeps in registers and what it loops over, and what tiles leave to the kernels behind them, against the oracle.  The
header in the workspace tells that a call took tiles, and how many tasksets these left; all of them where it took the size bins
because the batch was a mixture."""
import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding
from paper_2406_05221_b200.taskgen import TasksetBatch
from tests.helpers import BEST_EFFORT, BUSY, LITERAL, batch_of, direct_most, left_by_tiles, repeated

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L, OVH = 300, 1
LAST_T = 2_796_199   # the longest period that single precision takes (kNarrowLimit)


def taskset(rng, n, cores, segs, util=0.4, hi=100_000, step=1):
    ts = []
    for i in range(n):
        T = int(rng.integers(1000, hi))
        g = int(rng.integers(0, segs + 1))
        w = max(1, int(util * T / (n * (2 * g + 1))))
        ts.append(dict(T=T, D=int(rng.integers(T // 2, T + 1)), prio=0, core=int(rng.integers(0, cores)),
                       cseg=[int(rng.integers(0, w + 1)) for _ in range(g + 1)],
                       gseg=[(int(rng.integers(0, w + 1)), int(rng.integers(0, w + 1))) for _ in range(g)]))
    for r, i in enumerate(sorted(range(n), key=lambda i: ts[i]["T"])):
        ts[i]["prio"] = step * (n - r)
    return ts


def taken_ones(rng, n):
    """Tasksets that a tile takes, each another way."""
    few = taskset(rng, n, 3, 3)
    ties = [dict(t, prio=t["prio"] // 2) for t in few]
    zero = [dict(t, cseg=[0], gseg=[]) for t in few]
    same = [dict(t, T=5000, D=5000, core=0, prio=n - i) for i, t in enumerate(few)]
    edge = [dict(t, T=LAST_T, D=LAST_T) for t in few]
    own = [dict(t, core=i % 16, gseg=[(1, 1)]) for i, t in enumerate(few)]
    return [few, taskset(rng, n, 1, 2, util=0.6), taskset(rng, n, 2, 9), ties, zero, same, edge, own, taskset(rng, n, 4, 3, step=5),
            taskset(rng, n, 15, 3, util=0.2), taskset(rng, n, 4, 3, util=2.0), taskset(rng, n, 4, 62, hi=2_000_000)]


def left_ones(rng, n):
    """Tasksets that a tile leaves to the launches behind it."""
    wide, many_cores, big = taskset(rng, n, 3, 2), taskset(rng, n, 16, 2), taskset(rng, n, 2, 1)
    wide[0].update(T=LAST_T + 1, D=LAST_T + 1)
    many_cores[-1]["core"] = 16                   # one core more than tiles know
    big[n // 2]["cseg"] = [1 << 27]               # beyond the 32-bit path
    bad, high, many = taskset(rng, n, 3, 3), taskset(rng, n, 3, 3), taskset(rng, n, 3, 1)
    bad[0]["core"] = -1
    high[0]["prio"] = 1 << 33
    many[-1]["cseg"] = [1] * 64
    left = [wide, many_cores, big, bad, high, many]
    if n >= 7:  # 4,585 sweeps of the seventh task: more than a tile makes
        left.append([dict(T=250 << i, prio=n - i, core=0, cseg=[125 if i < 5 else 249]) for i in range(6)] +
                    [dict(T=2_790_000, prio=n - 6, core=0, cseg=[325])] +
                    [dict(T=2_000_000, prio=n - 7 - i, core=1 + i % 14, cseg=[1]) for i in range(n - 7)])
    return left


def some(n, outliers=()):
    """Tasksets of n tasks on average, and which of them a tile leaves.  Light ones lie between the others: a tile
    whose first four are left is left as a whole."""
    rng = np.random.default_rng(1000 * n)
    odd, left = taken_ones(rng, n), left_ones(rng, n)
    few = [(t, False) for t in odd] + [(t, True) for t in left]
    few = [x for k, odd in enumerate(few) for x in (odd, (taskset(rng, n, 4 + k % 3, 1 + k % 3), False))]
    extra = [(taskset(rng, s, 4, 2), s > n) for s in outliers]
    surplus = sum(len(t) - n for t, _ in extra)
    while surplus > 0:  # (smaller ones, so that the mean stays n)
        extra.append((taskset(rng, max(1, n - surplus), 4, 2), False))
        surplus -= n - len(extra[-1][0])
    few += [few[2 * k + 1] for k in range(16)] * len(extra)
    for k, x in enumerate(extra):
        few.insert(3 * k + 2, x)
    return batch_of([t for t, _ in few]), np.array([x for _, x in few])


def times(few, at_least):
    return at_least // few.n_tasksets + 1


def through_tiles(batch, left, call):
    """The results of call(tasksets, workspace), which leaves `left` tasksets behind its tiles (and more if the few tasksets
    of the last tile have crowded cores)."""
    dev = binding.DeviceTasksets.from_host(batch)
    ws = torch.zeros(binding.workspace_bytes(batch.n_tasksets), dtype=torch.uint8, device="cuda")
    w, s = call(dev, ws)
    assert left <= left_by_tiles(ws) < left + 32
    return None if w is None else w.cpu().numpy(), s.cpu().numpy()


def check_one(few, left, policies):
    n = few.n_tasks // few.n_tasksets
    k = times(few, max(direct_most(), 1750 * n))
    batch = repeated(few, k)
    for policy in policies:
        # (with the printed jitters of CPU-only tasks the one with many sweeps misses after a few)
        leaves = left.sum() - (1 if n >= 7 and policy == 1 | LITERAL else 0)
        w, s = through_tiles(batch, leaves * k, lambda dev, ws: binding.rta_batch(dev, policy, L, OVH, workspace=ws))
        want_w, want_s, _ = rta.analyse(few, policy, L, OVH)
        assert np.array_equal(s, np.tile(want_s, k)), (n, hex(policy))
        assert np.array_equal(w, np.tile(want_w, k)), (n, hex(policy))


def check_several(few, left, analyses, pairs, at_least=0):
    n = few.n_tasks // few.n_tasksets
    k = times(few, max(at_least, 25_000 if n > 12 and analyses < 4 else direct_most(several=True)))
    batch = repeated(few, k)
    if analyses & 12:  # a tile of several analyses has room for half as many GPU segments again as there are on average
        segments = few.gseg_off[few.task_off[1:]] - few.gseg_off[few.task_off[:-1]]
        left = left | (segments > min(255, int(1.5 * few.n_gsegs / few.n_tasksets) + 8 | 1))
    Ls, ovhs = [L, L, 1, 40_000, 77][:pairs], [OVH, 0, 1, 20, 5][:pairs]
    policies = [p for bit, p in binding.ANALYSIS_POLICY.items() if analyses & bit]
    want_w, want_s = rta.analyse_multi(few, policies, Ls, ovhs)
    for want in (True, False):
        w, s = through_tiles(batch, left.sum() * k,
                             lambda dev, ws: binding.rta_multi(dev, analyses, Ls, ovhs, workspace=ws, want_wcrt=want))
        assert np.array_equal(s, np.tile(want_s, k)), (n, analyses, pairs)
        assert not want or np.array_equal(w, np.tile(want_w, k)), (n, analyses, pairs)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 16, 17, 20, 24])
def test_one_analysis(n):
    few, left = some(n)
    check_one(few, left, (0, BUSY, LITERAL, 1, 1 | BUSY, 1 | LITERAL, 1 | BUSY | LITERAL))
    few.priority[:] -= n - 7 if n >= 7 else n // 2   # (the one with many sweeps needs seven real-time tasks)
    check_one(few, left, (BEST_EFFORT, BUSY | BEST_EFFORT, 1 | BEST_EFFORT, 1 | BUSY | BEST_EFFORT))


@pytest.mark.parametrize("n", [1, 8, 17, 20, 24])
@pytest.mark.parametrize("analyses,pairs", [(15, 1), (3, 2), (4, 5), (10, 3), (1, 4), (12, 1), (15, 5)])
def test_several_analyses(n, analyses, pairs):
    check_several(*some(n), analyses, pairs)


# (GCAPS by bins and RR in tiles; both in tiles, one after the other, with four lanes per taskset and with two)
@pytest.mark.parametrize("n,pairs,count", [(24, 3, 14_000), (16, 3, 17_000), (24, 3, 17_000), (24, 1, 50_000)])
def test_analyses_of_both_policies_apart(n, pairs, count):
    check_several(*some(n), 15, pairs, count)


@pytest.mark.parametrize("n", [4, 8, 20])
def test_a_few_larger_and_smaller_ones(n):
    few, left = some(n, outliers=(25, 33, 97, 200, 256))
    check_one(few, left, (0, BUSY, 1, 1 | BUSY))
    check_several(few, left, 15, 1)
    check_several(few, left, 4, 3)


@pytest.mark.parametrize("n", [2, 8, 20])
def test_malformed_offsets(n):
    few, _ = some(n)
    batch = repeated(few, times(few, max(direct_most(), 1750 * n)))
    rng = np.random.default_rng(n)
    broken = np.sort(rng.choice(batch.n_tasksets // 2, 200, replace=False)) * 2   # (no two side by side)
    for kind, t in enumerate(broken):
        first = int(batch.task_off[t]) + 1   # offsets of the second task: the first's end
        off = batch.cseg_off if kind & 1 else batch.gseg_off
        off[first] += (-1 << 40, 1 << 40, -1 - off[first], 100_000, -100_000)[kind // 2 % 5]
    last = int(broken[-1])
    inside = np.ones(batch.n_tasks, bool)   # (results of a taskset without a range have no place)
    inside[int(batch.task_off[last]):int(batch.task_off[last + 2])] = False
    batch.task_off[last + 1] = 1 << 50      # nor has the next one a range
    dev = binding.DeviceTasksets.from_host(batch)
    for policy in (0, 1, 1 | BUSY):
        ws = torch.zeros(binding.workspace_bytes(batch.n_tasksets), dtype=torch.uint8, device="cuda")
        w, s = binding.rta_batch(dev, policy, L, OVH, workspace=ws)
        want_w, want_s, _ = rta.analyse(batch, policy, L, OVH)
        assert left_by_tiles(ws) < batch.n_tasksets / 2
        s, w = s.cpu().numpy(), w.cpu().numpy()
        assert np.array_equal(s, want_s) and (want_s[broken] == binding.SCHED_INVALID).all(), hex(policy)
        assert np.array_equal(w[inside], want_w[inside]), hex(policy)


def a_mixture():
    rng = np.random.default_rng(77)
    sizes = [25, 32, 33, 64, 65, 96, 97, 128, 129, 192, 193, 256] + [1 + k % 24 for k in range(130)]
    sizes += [1 + (-sum(sizes) - 1) % (len(sizes) + 1)]
    assert sum(sizes) % len(sizes) == 0 and sum(sizes) // len(sizes) <= 24
    ts = [taskset(rng, s, 1 + k % 6, 1 + k % 4, step=1 + k % 2) for k, s in enumerate(sizes)]
    for k in range(5, len(ts), 9):
        ts[k] = left_ones(rng, len(ts[k]))[k % 6]
    order = rng.permutation(len(ts))
    return batch_of([ts[k] for k in order])


@pytest.mark.parametrize("count", [13_000, 42_000])
def test_mixtures_take_the_size_bins(count):
    few = a_mixture()
    k = times(few, count)
    batch = repeated(few, k)
    for policy in (0, BUSY, 1, 1 | BUSY, 1 | BEST_EFFORT):
        w, s = through_tiles(batch, batch.n_tasksets, lambda dev, ws: binding.rta_batch(dev, policy, L, OVH, workspace=ws))
        want_w, want_s, _ = rta.analyse(few, policy, L, OVH)
        assert np.array_equal(s, np.tile(want_s, k)) and np.array_equal(w, np.tile(want_w, k)), hex(policy)
    for analyses, pairs in ((15, 1), (4, 3), (15, 2)):
        policies = [p for bit, p in binding.ANALYSIS_POLICY.items() if analyses & bit]
        want_w, want_s = rta.analyse_multi(few, policies, [L, 1][:pairs] + [77] * (pairs - 2), [OVH, 0, 4][:pairs])
        w, s = through_tiles(batch, batch.n_tasksets, lambda dev, ws: binding.rta_multi(
            dev, analyses, [L, 1][:pairs] + [77] * (pairs - 2), [OVH, 0, 4][:pairs], workspace=ws))
        assert np.array_equal(s, np.tile(want_s, k)) and np.array_equal(w, np.tile(want_w, k)), (analyses, pairs)


@pytest.mark.parametrize("n", [8, 20])
def test_a_stretch_that_tiles_leave(n):
    rng = np.random.default_rng(5)
    light, wide = [taskset(rng, n, 4, 2) for _ in range(10)], [left_ones(rng, n)[0] for _ in range(10)]
    few, k, stretch = batch_of(light + wide), 2 * 1750 * 20 // 10, 200
    front = repeated(few.slice(10, 20), stretch)
    batch = TasksetBatch.concat([front, repeated(few.slice(0, 10), k)])
    dev = binding.DeviceTasksets.from_host(batch)
    for policy in (0, 1):
        ws = torch.zeros(binding.workspace_bytes(batch.n_tasksets), dtype=torch.uint8, device="cuda")
        w, s = binding.rta_batch(dev, policy, L, OVH, workspace=ws)
        assert front.n_tasksets <= left_by_tiles(ws) < front.n_tasksets + 32   # (the tile on the border)
        want_w, want_s, _ = rta.analyse(batch.slice(0, front.n_tasksets + 10), policy, L, OVH)
        want_w = np.concatenate([want_w, np.tile(want_w[-10 * n:], k - 1)])
        want_s = np.concatenate([want_s, np.tile(want_s[-10:], k - 1)])
        assert np.array_equal(s.cpu().numpy(), want_s) and np.array_equal(w.cpu().numpy(), want_w), policy


@pytest.mark.parametrize("n,what", [(8, "long"), (20, "long"), (24, "cores"), (12, "crowded"), (16, "crowded")])
def test_batches_that_are_none_for_tiles(n, what):
    rng = np.random.default_rng(6)
    ts = [taskset(rng, n, 1 if what == "crowded" and k < 55 else 4, 2) for k in range(60)]
    for t in ts[:55]:
        if what == "long":
            t[n - 1].update(T=1 << 40, D=1 << 40)
        if what == "cores":
            t[0]["core"] = 16
    few = batch_of([ts[k] for k in rng.permutation(60)])
    k = times(few, 60_000)   # (more than one tile per warp)
    batch = repeated(few, k)
    for policy in (0, BUSY, 1, 1 | BUSY):
        w, s = through_tiles(batch, batch.n_tasksets, lambda dev, ws: binding.rta_batch(dev, policy, L, OVH, workspace=ws))
        want_w, want_s, _ = rta.analyse(few, policy, L, OVH)
        assert np.array_equal(s, np.tile(want_s, k)) and np.array_equal(w, np.tile(want_w, k)), hex(policy)
