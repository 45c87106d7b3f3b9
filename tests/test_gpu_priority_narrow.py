"""The search in single precision against its oracle where it can go wrong: sizes at the edges of the
lane groups, one core and one core per task, periods around the single-precision limit, tasks without
demand, and both waiting modes with and without the printed form."""
import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding
from tests.helpers import BUSY, LITERAL, batch_of, both_ways

pytestmark = pytest.mark.gpu

NARROW_LIMIT = 2_796_200   # kNarrowLimit of csrc/rta_recurrence.cuh


@pytest.mark.parametrize("cores", [1, 5, 300])
@pytest.mark.parametrize("n", [1, 8, 9, 16, 24, 25, 32, 33, 64, 80, 96, 97, 128, 129, 192, 193, 256])
def test_search_matches_oracle(n, cores):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(7 * n + cores)
    tasksets = []
    for k in range(14):
        ts = []
        for i in range(n):
            T = int(rng.integers(1000, 100_000)) if k % 7 else int(rng.integers(NARROW_LIMIT - 40, NARROW_LIMIT + (0 if k == 0 else 3)))
            w = int(T * (0.02, 0.3, 1.0, 4.0)[k % 4] / n)
            uses = rng.random() < 0.6
            ts.append(dict(T=T, D=int(rng.integers(T // 2, T + 1)), prio=0, core=int(rng.integers(0, cores)) if cores < 300 else i,
                           cseg=[int(rng.integers(0, w + 1))],
                           gseg=[(int(rng.integers(0, w // 4 + 1)), int(rng.integers(0, w + 1)))] if uses else []))
        if k % 5 == 4:
            ts[0]["cseg"], ts[0]["gseg"] = [0], [(0, 0)]
        order = sorted(range(n), key=lambda i: ts[i]["T"])
        for r, i in enumerate(order):
            ts[i]["prio"] = n - r if k % 3 else 2 * (n - r)
        tasksets.append(ts)
    batch = batch_of(tasksets)
    nt, ns = batch.n_tasks, batch.n_tasksets
    devs = [binding.DeviceTasksets.from_host(b) for b in both_ways(batch, several=True)]
    for flags in (0, BUSY, LITERAL, BUSY | LITERAL):
        for eps in (0, 5):
            wr, sr, gr = rta.analyse_gpu_priority(batch, flags | binding.ASSIGN, eps)
            for dev in devs:   # a warp each, then the lane groups of the size bins
                w, s, g = binding.rta_gpu_priority(dev, flags | binding.ASSIGN, eps)
                torch.cuda.synchronize()
                assert np.array_equal(w.cpu().numpy()[:nt], wr), (flags, eps)
                assert np.array_equal(g.cpu().numpy()[:nt], gr), (flags, eps)
                assert np.array_equal(s.cpu().numpy()[:ns], sr), (flags, eps)
