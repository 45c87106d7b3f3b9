"""The binding hands device pointers to kernels, so tensors that do not live on a CUDA device are refused
before anything is enqueued.  No GPU: the library is a stand-in that counts its calls."""
import pytest

from paper_2406_05221_b200 import binding, taskgen

CALLS = {
    "rta_batch": lambda ts: binding.rta_batch(ts, 0),
    "rta_sweep": lambda ts: binding.rta_sweep(ts, 1, [512], [3]),
    "rta_multi": lambda ts: binding.rta_multi(ts, 15),
    "rta_batch_static": lambda ts: binding.rta_batch_static(ts, 0),
    "rta_gpu_priority": lambda ts: binding.rta_gpu_priority(ts, binding.ASSIGN),
    "rta_plan": lambda ts: binding.rta_plan(ts, ts.t["period"]),
    "rta_validate": lambda ts: binding.rta_validate(ts),
    "generate_device": lambda ts: binding.generate_device(taskgen.WORKLOADS["pr1"].streams[0], 0, 1, device="cpu"),
}


class CountingLibrary:
    def __init__(self):
        self.enqueued = []

    def __getattr__(self, name):
        def call(*args):
            if not name.endswith("_bytes"):
                self.enqueued.append(name)
            return 0
        return call


@pytest.mark.parametrize("name", sorted(CALLS))
def test_host_tensors_are_refused(monkeypatch, name):
    torch = pytest.importorskip("torch")
    lib = CountingLibrary()
    monkeypatch.setattr(binding, "load_library", lambda path=None: lib)
    monkeypatch.setattr(binding, "_raw_stream", lambda device: 0)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    batch = taskgen.WORKLOADS["pr1"].generate(0, 2)
    ts = binding.DeviceTasksets({f: torch.from_numpy(getattr(batch, f)) for f in taskgen.ARRAY_FIELDS})
    with pytest.raises(ValueError):
        CALLS[name](ts)
    assert lib.enqueued == []
