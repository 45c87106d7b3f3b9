"""Tasksets of up to 32 tasks in tiles, a lane or a few per taskset: sizes around the edges of the stage, what a walk
keeps in registers and what it loops over, and what tiles leave to the kernels behind them, against the oracle."""
import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding
from tests.helpers import BEST_EFFORT, BUSY, batch_of, direct_most

pytestmark = pytest.mark.gpu


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


def odd_ones(rng, n):
    """Tasksets that a tile takes another way, or not at all."""
    few, one_core = taskset(rng, n, 3, 3), taskset(rng, n, 1, 2, util=0.6)
    wide, many_cores, big = taskset(rng, n, 3, 2), taskset(rng, n, 16, 2), taskset(rng, n, 2, 1)
    wide[0].update(T=2_796_200, D=2_796_200)      # the first period beyond single precision
    many_cores[-1]["core"] = 16                   # one core more than tiles know
    big[n // 2]["cseg"] = [1 << 27]               # beyond the 32-bit path
    slow = [dict(T=1000, prio=2, core=0, cseg=[999]),  # 14,000 sweeps
            dict(T=2_500_000, prio=1, core=0, cseg=[2000])]
    ties = [dict(t, prio=t["prio"] // 2) for t in few]
    zero = [dict(t, cseg=[0], gseg=[]) for t in few]
    bad = [dict(t, core=-1) if k == 0 else t for k, t in enumerate(few)]
    return [few, one_core, taskset(rng, n, 2, 9), wide, many_cores, big, slow, ties, zero, bad,
            taskset(rng, n, 4, 3, step=5), taskset(rng, n, 15, 3, util=0.2)]


def a_batch(n, count):
    rng = np.random.default_rng(1000 * n + count)
    kinds = odd_ones(rng, n) + [taskset(rng, n, c, s) for c in (1, 2, 4) for s in (1, 3) for _ in range(6)]
    return batch_of([kinds[(7 * k) % len(kinds)] if k % 5 else kinds[12 + k % 36] for k in range(count)])


def same(got, want, what):
    w, s = (x.cpu().numpy() for x in got)
    assert np.array_equal(s.reshape(-1), want[1].reshape(-1)), what
    assert np.array_equal(w.reshape(-1), want[0].reshape(-1)), what


@pytest.mark.parametrize("n", [1, 7, 8, 9, 16, 17, 20, 24, 25, 32])
def test_one_analysis(n):
    batch = a_batch(n, direct_most() + 37)
    dev = binding.DeviceTasksets.from_host(batch)
    for policy in (0, BUSY, 1, 1 | BUSY):
        same(binding.rta_batch(dev, policy, 300, 3), rta.analyse(batch, policy, 300, 3), (n, hex(policy)))
    batch.priority[:] -= 3 * (n // 4)
    dev = binding.DeviceTasksets.from_host(batch)
    for policy in (BEST_EFFORT, 1 | BEST_EFFORT):
        same(binding.rta_batch(dev, policy, 300, 3), rta.analyse(batch, policy, 300, 3), (n, hex(policy)))


@pytest.mark.parametrize("n", [1, 8, 17, 24, 32])
@pytest.mark.parametrize("analyses,pairs", [(15, 1), (3, 2), (4, 5), (10, 3), (1, 1), (8, 1)])
def test_several_analyses(n, analyses, pairs):
    batch = a_batch(n, direct_most(several=True) + 61)
    dev = binding.DeviceTasksets.from_host(batch)
    Ls, ovhs = [300, 300, 1, 40_000, 77][:pairs], [3, 0, 1, 20, 5][:pairs]
    policies = [p for bit, p in binding.ANALYSIS_POLICY.items() if analyses & bit]
    want = rta.analyse_multi(batch, policies, Ls, ovhs)
    same(binding.rta_multi(dev, analyses, Ls, ovhs), want, (n, analyses, pairs))
    sched = binding.rta_multi(dev, analyses, Ls, ovhs, want_wcrt=False)[1]
    assert np.array_equal(sched.cpu().numpy().reshape(-1), want[1].reshape(-1))
