"""The segment split of the on-device generator against its oracle at the ends of what a warp handles at
once: 0 to 16 GPU segments per task, tasksets around multiples of 32 tasks, demands from the least that
holds its segments to 2^30 us."""
import numpy as np
import pytest

from oracle.igen_oracle import reference_taskset
from paper_2406_05221_b200 import binding, taskgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("segs", [(0, 0), (0, 1), (1, 1), (0, 16), (16, 16)])
@pytest.mark.parametrize("tasks", [1, 31, 32, 33, 64, 65, 256])
def test_split_matches_the_oracle(tasks, segs):
    torch = pytest.importorskip("torch")
    for util, period in (((0.9, 0.99), (1e9, 1.07e9)), ((0.001, 0.01), (1000, 30000))):
        params = taskgen.GenParams(seed=tasks, cores=(1, 1), tasks_per_core=(tasks, tasks), util_per_core=util,
                                   period_us=period, gpu_mode=1, gpu_segments=segs, gpu_ratio=(0.0, 0.99))
        ts = binding.generate_device(params, 5, 9)
        torch.cuda.synchronize()
        p = params.int_params()
        want = taskgen.TasksetBatch.from_tasksets([reference_taskset(p, 5 + t) for t in range(9)])
        for f in taskgen.ARRAY_FIELDS:
            assert np.array_equal(ts.t[f].cpu().numpy(), getattr(want, f)), f
