"""Which tiles a warp looks at (csrc/tile_patience.h), on the host: seven are passed by behind one that had to be left, and then
one is looked at again, whatever came before."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("patience") / "tile_patience_host")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-o", exe, os.path.join(HERE, "tile_patience_host.cpp")])
    return exe


@pytest.mark.parametrize("row,looks", [
    ("." * 30, "l" * 30),
    ("x" + "." * 24, "l" + "-" * 7 + "l" * 17),
    ("x" * 9 + "." * 24, "l" + "-" * 7 + "l" + "-" * 7 + "l" * 17),
    ("x" * 25, ("l" + "-" * 7) * 3 + "l"),
    ("..x......x.....", "l" * 3 + "-" * 7 + "l" * 5),
])
def test_a_warp_looks_again(program, row, looks):
    assert subprocess.check_output([program, row], text=True) == looks
