"""Batches that run without a plan, around the sizes where the launches change and where the pairs of a
sweep are shared out among blocks, every size class in one batch, against the oracles."""
import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding, taskgen
from tests.helpers import batch_of

pytestmark = pytest.mark.gpu


def mixed(count):
    """Tasksets of `divergence` (4 to 192 tasks) with empty, broken and 64-bit ones among them."""
    b = taskgen.WORKLOADS["divergence"].generate(11, count)
    if count > 30:
        b.period[b.task_off[7]] += 1 << 33
        b.deadline[b.task_off[11]] = 0
        b.gseg_off[b.task_off[19] + 1] = -3
        b = taskgen.TasksetBatch.concat([b, batch_of([[]]), batch_of([[dict(T=9, prio=1, core=0, cseg=[2])] * 1])])
    return b


@pytest.mark.parametrize("count", [1, 2, 40, 500, 1183, 2369, 4096, 4097])
def test_sweeps_and_searches_without_a_plan(count):
    torch = pytest.importorskip("torch")
    batch = mixed(count)
    ts = binding.DeviceTasksets.from_host(batch)
    Ls, ovhs = [512, 512, 64, 4096, 1, 1000, 7], [50, 0, 200, 3, 10, 100, 1]
    for analyses in (1, 8, 15) if count < 2000 else (4, 10):
        w, s = binding.rta_multi(ts, analyses, Ls, ovhs)
        torch.cuda.synchronize()
        policies = [p for bit, p in binding.ANALYSIS_POLICY.items() if analyses & bit]
        wr, sr = rta.analyse_multi(batch, policies, Ls, ovhs)
        assert np.array_equal(w.cpu().numpy(), wr), analyses
        assert np.array_equal(s.cpu().numpy(), sr), analyses
    for flags in (binding.ASSIGN, binding.ASSIGN | binding.BUSY):
        w, s, g = binding.rta_gpu_priority(ts, flags, 20)
        torch.cuda.synchronize()
        wr, sr, gr = rta.analyse_gpu_priority(batch, flags, 20)
        assert np.array_equal(w.cpu().numpy(), wr) and np.array_equal(s.cpu().numpy(), sr)
        assert np.array_equal(g.cpu().numpy(), gr)


@pytest.mark.parametrize("count", [1, 40, 12287, 12290])
def test_one_analysis_without_a_plan(count):
    torch = pytest.importorskip("torch")
    batch = mixed(count)
    ts = binding.DeviceTasksets.from_host(batch)
    for policy in (0, binding.BUSY, 1, 1 | binding.BUSY):
        w, s = binding.rta_batch(ts, policy, 512, 25)
        torch.cuda.synchronize()
        wr, sr, _ = rta.analyse(batch, policy, 512, 25)
        assert np.array_equal(w.cpu().numpy(), wr), hex(policy)
        assert np.array_equal(s.cpu().numpy(), sr), hex(policy)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 32, 33, 63, 65, 94, 97, 127, 130, 191, 194, 255, 256])
def test_ranks_of_any_priorities(n):
    """Priorities that are no dense numbering: ties, gaps, the ends of 32 bits."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    kinds = ([7], [1, 2], [-(1 << 31), (1 << 31) - 1, 0], list(range(-3, 40)), [int(x) for x in rng.integers(-(1 << 31), 1 << 31, 500)])
    sets = [[dict(T=10_000 + i, prio=int(rng.choice(kind)), core=i % 3, cseg=[int(rng.integers(0, 30000 // n + 1))], gseg=[(1, 2)] * (i % 2))
             for i in range(n)] for kind in kinds for _ in range(2)]
    batch = batch_of(sets)
    ts = binding.DeviceTasksets.from_host(batch)
    for policy in (0, 1 | binding.BUSY):
        w, s = binding.rta_batch(ts, policy, 512, 2)
        torch.cuda.synchronize()
        wr, sr, _ = rta.analyse(batch, policy, 512, 2)
        assert np.array_equal(w.cpu().numpy(), wr), hex(policy)
        assert np.array_equal(s.cpu().numpy(), sr), hex(policy)
    w, s, g = binding.rta_gpu_priority(ts, binding.ASSIGN, 2)
    torch.cuda.synchronize()
    for got, want in zip((w, s, g), rta.analyse_gpu_priority(batch, binding.ASSIGN, 2)):
        assert np.array_equal(got.cpu().numpy(), want)
