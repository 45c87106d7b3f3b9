"""The sums of a task's segments, from none to as many as the 32-bit path takes and
beyond, below and above its 2^26 and where 32-bit sums would wrap, against the oracle."""
import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding
from tests.helpers import batch_of, direct_most, left_by_tiles, repeated

pytestmark = pytest.mark.gpu

BIG = 1 << 26


def _taskset(rng, n, odd):
    """Light tasks with 0 .. 5 segments of a kind, and one (odd: its segments) in their middle."""
    ts = []
    for i in range(n):
        T = int(rng.integers(100_000, 2_000_000))
        w = T // (8 * n)
        c, g = int(rng.integers(0, 6)), int(rng.integers(0, 6))
        ts.append(dict(T=T, D=T, core=i % 16, cseg=[int(rng.integers(0, w + 1)) for _ in range(c)],
                       gseg=[(int(rng.integers(0, w + 1)), int(rng.integers(0, w + 1))) for _ in range(g)]))
    ts[n // 2].update(odd)
    for r, i in enumerate(sorted(range(n), key=lambda i: ts[i]["T"])):
        ts[i]["prio"] = n - r
    return ts


ODD = [dict(), dict(cseg=[3] * 63, gseg=[(1, 2)] * 63), dict(cseg=[3] * 64), dict(gseg=[(1, 2)] * 64),
       dict(cseg=[BIG - 1]), dict(cseg=[BIG]), dict(cseg=[1 << 32]), dict(gseg=[(0, 1 << 33)]), dict(gseg=[(1 << 34, 0)]),
       dict(cseg=[BIG // 32] * 33), dict(gseg=[(0, BIG // 32)] * 33), dict(cseg=[BIG // 2], gseg=[(BIG // 2, 1)]),
       dict(T=BIG - 1, D=BIG - 1, cseg=[BIG // 8] * 2, gseg=[(BIG // 8, 1)]),
       # (the most that pure GPU parts add up to: 63 values below 2^26 stay below 2^32)
       dict(gseg=[(0, BIG - 1)] * 63),
       # sums that are small again modulo 2^32: 0, 100, 4, 2^26 - 65, 500
       dict(cseg=[BIG - 1] * 60, gseg=[(BIG - 1, 0)] * 4 + [(64, 0)]), dict(cseg=[BIG - 1] * 63, gseg=[(BIG - 1, 1), (164, 1)]),
       dict(cseg=[66_076_420] * 33, gseg=[(66_076_420, 0)] * 32), dict(cseg=[BIG - 1] * 2 + [0] * 61, gseg=[(BIG - 1, 0)] * 63),
       dict(cseg=[BIG - 1] * 63, gseg=[(BIG - 1, 0), (64, 0), (500, 0)])]


@pytest.mark.parametrize("n", ["1 to 8", 33, 64, 65, 96, 97, 128, 129, 160, 161, 250])
def test_segment_sums(n):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(35)
    few = batch_of([_taskset(rng, 1 + k % 8 if n == "1 to 8" else n, odd) for k, odd in enumerate(ODD)])
    k = direct_most() // len(ODD) + 1
    for batch, times in ((few, 1), (repeated(few, k), k)):  # one launch, and the kernels behind a plan
        dev = binding.DeviceTasksets.from_host(batch)
        for policy in (0, 1, binding.BUSY, 1 | binding.BUSY):
            wcrt, sched = binding.rta_batch(dev, policy, 256, 2)
            torch.cuda.synchronize()
            ref, ref_s, _ = rta.analyse(few, policy, 256, 2)
            assert np.array_equal(wcrt.cpu().numpy(), np.tile(ref, times)), (times, policy)
            assert np.array_equal(sched.cpu().numpy(), np.tile(ref_s, times)), (times, policy)


@pytest.mark.parametrize("n", [1, 8, 20])
def test_segment_sums_in_tiles(n):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(36)
    light = [_taskset(rng, n, {}) for _ in ODD]
    few = batch_of([ts for k, odd in enumerate(ODD) for ts in (light[k], _taskset(rng, n, odd))])
    k = 1750 * 20 // few.n_tasksets + 1
    batch = repeated(few, k)
    dev = binding.DeviceTasksets.from_host(batch)
    workspace = torch.zeros(binding.workspace_bytes(batch.n_tasksets), dtype=torch.uint8, device="cuda")
    for policy in (0, 1, binding.BUSY, 1 | binding.BUSY):
        wcrt, sched = binding.rta_batch(dev, policy, 256, 2, workspace=workspace)
        assert left_by_tiles(workspace) <= len(ODD) * k
        ref, ref_s, _ = rta.analyse(few, policy, 256, 2)
        assert np.array_equal(wcrt.cpu().numpy(), np.tile(ref, k)), policy
        assert np.array_equal(sched.cpu().numpy(), np.tile(ref_s, k)), policy
    for analyses, Ls, ovhs in ((15, [256], [2]), (15, [256, 1000], [2, 7]), (4, [256, 300, 1000], [2, 2, 7]), (3, [1, 1, 1], [2, 0, 7])):
        wcrt, sched = binding.rta_multi(dev, analyses, Ls, ovhs, workspace=workspace)
        assert left_by_tiles(workspace) <= len(ODD) * k
        policies = [p for bit, p in binding.ANALYSIS_POLICY.items() if analyses & bit]
        ref, ref_s = rta.analyse_multi(few, policies, Ls, ovhs)[:2]
        assert np.array_equal(wcrt.cpu().numpy(), np.tile(ref, (1, 1, k))), analyses
        assert np.array_equal(sched.cpu().numpy(), np.tile(ref_s, (1, 1, k))), analyses
