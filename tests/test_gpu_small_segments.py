"""Small tasksets with as many segments as a group's prefix arrays take, and more: the 32-bit path up to
its capacity and the 64-bit path behind it, side by side in a warp, against the oracle."""
import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding
from tests.helpers import ALL_MODES, batch_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 8, 15, 16, 24, 32])
@pytest.mark.parametrize("count", [40, 12300])
def test_segment_counts_around_the_capacity(n, count):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n)
    kinds = []
    for segs in range(4, 13):      # CPU segments per task: capacity is 8 per task and a bit
        ts = []
        for i in range(n):
            T = int(rng.integers(1000, 100_000))
            w = max(1, T // (6 * n * segs))
            ts.append(dict(T=T, D=T, prio=0, core=i % 3, cseg=[int(rng.integers(0, w + 1)) for _ in range(segs)],
                           gseg=[(int(rng.integers(0, w + 1)), int(rng.integers(0, w + 1))) for _ in range(segs - 1)]))
        for r, i in enumerate(sorted(range(n), key=lambda i: ts[i]["T"])):
            ts[i]["prio"] = n - r
        kinds.append(ts)
    batch = batch_of([kinds[(7 * k) % len(kinds)] for k in range(count)])
    dev = binding.DeviceTasksets.from_host(batch)
    for policy in ALL_MODES if count < 100 else (0, 1):
        wcrt, sched = binding.rta_batch(dev, policy, 256, 2)
        torch.cuda.synchronize()
        ref, ref_s, _ = rta.analyse(batch, policy, 256, 2)
        assert np.array_equal(wcrt.cpu().numpy(), ref), hex(policy)
        assert np.array_equal(sched.cpu().numpy(), ref_s), hex(policy)
