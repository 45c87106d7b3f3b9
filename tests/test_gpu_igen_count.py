"""The per-task part of the on-device generator against its oracle where the warp's way differs from the
step-by-step definition: few and many cores, cores without tasks, the limit of 256 tasks, every share
of GPU-using tasks, harmonic periods, periods beyond 2^24, worst fit on up to 64 cores; and on both sides
of the number of small tasksets from which a thread takes each."""
import numpy as np
import pytest

from oracle.igen_oracle import reference_taskset
from paper_2406_05221_b200 import binding, taskgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wfd", [False, True])
@pytest.mark.parametrize("cores,per_core,gpu_frac,harmonic,period", [
    ((1, 1), (0, 1), 1.0, 0.0, (1000, 1e6)), ((1, 2), (1, 33), 0.5, 0.5, (100, 1e7)),
    ((33, 64), (0, 3), 0.9, 0.0, (1e4, 1e6)), ((20, 40), (7, 9), 0.0, 1.0, (50, 1e5)),
    ((64, 64), (4, 5), 1.0, 0.3, (1e3, 1.07e9)), ((2, 3), (100, 120), 0.77, 0.5, (2, 40)),
    # periods that are alike, in few buckets by their leading bits or in one
    ((7, 8), (9, 11), 0.8, 0.0, (1e5, 100_500)), ((16, 16), (16, 16), 0.5, 0.0, (1e5, 1e5)), ((5, 5), (17, 17), 0.5, 1.0, (16_776_000, 16_777_215))])
def test_tasks_match_the_oracle(cores, per_core, gpu_frac, harmonic, period, wfd):
    torch = pytest.importorskip("torch")
    for count in (1, 37):
        params = taskgen.GenParams(seed=9, stream=2, cores=cores, tasks_per_core=per_core, util_per_core=(0.05, 0.9),
                                   period_us=period, gpu_frac=gpu_frac, harmonic_frac=harmonic, wfd=wfd)
        ts = binding.generate_device(params, 100, count)
        torch.cuda.synchronize()
        p = params.int_params()
        want = taskgen.TasksetBatch.from_tasksets([reference_taskset(p, 100 + t) for t in range(count)])
        for f in taskgen.ARRAY_FIELDS:
            assert np.array_equal(ts.t[f].cpu().numpy(), getattr(want, f)), f


@pytest.mark.parametrize("wfd", [False, True])
@pytest.mark.parametrize("cores,per_core,gpu_mode", [((1, 1), (0, 1), 0), ((1, 2), (0, 2), 1), ((2, 3), (1, 3), 0), ((3, 3), (4, 5), 0),
                                                     ((4, 4), (8, 8), 0)])
def test_many_small_tasksets(cores, per_core, gpu_mode, wfd):
    torch = pytest.importorskip("torch")
    params = taskgen.GenParams(seed=4, stream=1, cores=cores, tasks_per_core=per_core, util_per_core=(0.05, 0.9), period_us=(100, 1e7),
                               gpu_mode=gpu_mode, gpu_frac=0.6, gpu_segments=(0, 5), harmonic_frac=0.3, wfd=wfd)
    n = cores[1] * per_core[1]
    for count in (160 * n * n - 1, 160 * n * n, 160 * n * n + 130):   # thread_per_taskset of csrc/gcaps_igen.cu (up to 48 tasks)
        ts = binding.generate_device(params, 1000, count)
        torch.cuda.synchronize()
        want = taskgen.generate(params, 1000, count, integer=True)   # (the host's run of the definition)
        for f in taskgen.ARRAY_FIELDS:
            assert np.array_equal(ts.t[f].cpu().numpy(), getattr(want, f)), (f, count)
