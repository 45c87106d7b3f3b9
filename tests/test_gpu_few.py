"""Batches that need no workspace: the call without one, up to its limit and beyond."""
import ctypes

import numpy as np
import pytest

from oracle import rta
from paper_2406_05221_b200 import binding, build, taskgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 1000, binding.FEW_MAX_TASKSETS, binding.FEW_MAX_TASKSETS + 1])
def test_without_a_workspace(count):
    torch = pytest.importorskip("torch")
    assert binding.FEW_MAX_TASKSETS == build.source_constant("kDirectMost")
    batch = taskgen.WORKLOADS["pr1"].generate(0, count)
    ts = binding.DeviceTasksets.from_host(batch)
    for policy in (0, 1 | binding.BUSY):
        w, s = binding.rta_batch(ts, policy, 1024, 50)
        torch.cuda.synchronize()
        wr, sr, _ = rta.analyse(batch, policy, 1024, 50)
        assert np.array_equal(w.cpu().numpy(), wr) and np.array_equal(s.cpu().numpy(), sr)
    lib = binding.load_library()
    rc = lib.gcaps_rta_batch_few(ctypes.byref(ts.c), count, 0, 1024, 50, w.data_ptr(), s.data_ptr(), None)
    torch.cuda.synchronize()
    assert rc == (binding.OK if count <= binding.FEW_MAX_TASKSETS else binding.ERR_TOO_LARGE)
    assert lib.gcaps_rta_batch_few(ctypes.byref(ts.c), 1, 7, 1024, 50, None, None, None) == binding.ERR_INVALID_ARG
