"""What the on-device generator does another way than the definition: 2^y from looked-up factors (for every fraction, on the
CPU), and a thread per taskset where there are many small ones (both sides of the line)."""
import os
import subprocess

import numpy as np
import pytest

from paper_2406_05221_b200 import binding, taskgen


def test_powers_from_factors(tmp_path):
    exe = str(tmp_path / "exp2_host")
    subprocess.check_call(["gcc", "-O2", "-fopenmp", "-o", exe, os.path.join(os.path.dirname(__file__), "exp2_host.c")])
    assert int(subprocess.check_output([exe])) == 0


@pytest.mark.gpu
@pytest.mark.parametrize("cores,per_core", [((1, 2), (1, 2)), ((3, 4), (2, 3)), ((6, 6), (8, 8)), ((7, 7), (7, 7))])
def test_both_sides_of_a_thread_per_taskset(cores, per_core):
    torch = pytest.importorskip("torch")
    params = taskgen.GenParams(seed=6, stream=3, cores=cores, tasks_per_core=per_core, util_per_core=(0.05, 0.9), period_us=(100, 1e7),
                               gpu_frac=0.6, gpu_segments=(1, 4), harmonic_frac=0.3)
    n = cores[1] * per_core[1]
    for count in {160 * n * n - 1, 160 * n * n} if n < 40 else {160 * n * n}:  # (49 tasks: warps at every count)
        ts = binding.generate_device(params, 500, count)
        torch.cuda.synchronize()
        want = taskgen.generate(params, 500, count, integer=True)
        for f in taskgen.ARRAY_FIELDS:
            assert np.array_equal(ts.t[f].cpu().numpy(), getattr(want, f)), (f, count)
