"""The order of work of the staged kernels (csrc/staged_walk.h) on the host: whatever can be staged and
decided, and wherever a wait for copies gives up, every taskset is decided once or left to the second
launch once, the count that the second launch is told is right, and the stage is not touched after a
wait that gave up."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("walk") / "staged_walk_host")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-o", exe, os.path.join(HERE, "staged_walk_host.cpp")])
    return exe


@pytest.mark.parametrize("stages", [1, 0])
@pytest.mark.parametrize("give_up", [0, 0.002, 0.1, 1])
@pytest.mark.parametrize("decided", [1, 0.9, 0.3, 0])
def test_every_taskset_is_decided_or_left_once(program, decided, give_up, stages):
    for seed, (count, chunk, warps, stageable) in enumerate(
            [(1, 8, 3, 1), (7, 8, 1, 1), (9, 1, 4, 0.8), (400, 4, 40, 1), (3000, 8, 6, 0.95), (6001, 8, 50, 1), (900, 8, 2, 0)]):
        done = subprocess.run([program] + [str(x) for x in (count, chunk, warps, decided, stageable, give_up, stages, seed)],
                              capture_output=True, text=True, timeout=120)
        assert done.returncode == 0, (count, chunk, warps, stageable, done.stdout[:500])
