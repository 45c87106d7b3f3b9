"""Host-buffer calls that span several chunks of staging: results equal those of one device call, with
malformed tasksets on a chunk's edge judged on their own."""
import numpy as np
import pytest

from paper_2406_05221_b200 import binding, taskgen

pytestmark = pytest.mark.gpu

CHUNK_TASKS = 1 << 18   # the least chunk_tasks of gcaps_rta_batch_host_multi (csrc/gcaps_rta.cu)


@pytest.mark.parametrize("workload,tasks", [("large", CHUNK_TASKS - 64), ("large", CHUNK_TASKS + 80), ("pr1", 5 * CHUNK_TASKS),
                                            ("divergence", 4 * CHUNK_TASKS + 123)])
def test_chunked_call_equals_device_call(workload, tasks):
    torch = pytest.importorskip("torch")
    w = taskgen.WORKLOADS[workload]
    per = {"large": 80, "pr1": 8, "divergence": 63}[workload]
    batch = w.generate(0, max(1, tasks // per))
    arrays = {f: getattr(batch, f) for f in taskgen.ARRAY_FIELDS}
    first_of_second = int(np.searchsorted(batch.task_off, CHUNK_TASKS, side="right")) - 1
    for broken in (None, first_of_second - 1, first_of_second):
        if broken is not None and broken < batch.n_tasksets:
            k = int(batch.task_off[broken])
            if batch.task_off[broken + 1] - k > 1:
                arrays["gseg_off"] = batch.gseg_off.copy()
                arrays["gseg_off"][k + 1] = -1   # (the neighbours' own offsets stay as they are)
        wcrt, sched = binding.rta_batch_host_multi(arrays, [binding.POLICY_GCAPS, binding.POLICY_RR], w.timeslice_us, w.overhead_us)
        ts = binding.DeviceTasksets({f: torch.from_numpy(arrays[f]).cuda() for f in taskgen.ARRAY_FIELDS})
        for q, policy in enumerate((binding.POLICY_GCAPS, binding.POLICY_RR)):
            dw, ds = binding.rta_batch(ts, policy, w.timeslice_us, w.overhead_us)
            assert np.array_equal(wcrt[q], dw.cpu().numpy()), (broken, policy)
            assert np.array_equal(sched[q], ds.cpu().numpy()), (broken, policy)
        arrays["gseg_off"] = batch.gseg_off
    binding.release_host()
