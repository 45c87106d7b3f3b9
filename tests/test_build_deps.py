"""The library counts as stale after an edit of any file that its sources include."""
import os
import re

import pytest

from paper_2406_05221_b200 import build


def included_files():
    """Every file that the CUDA sources include by a quoted path, directly or through another one."""
    found, todo = set(), list(build.CUDA_SRCS)
    while todo:
        path = todo.pop()
        for name in re.findall(r'^\s*#\s*include\s+"([^"]+)"', open(path).read(), flags=re.M):
            dep = os.path.normpath(os.path.join(os.path.dirname(path), name))
            if dep not in found:
                found.add(dep)
                todo.append(dep)
    return sorted(found)


def test_the_sources_are_those_of_the_folder():
    folder = os.path.dirname(build.CUDA_SRC)
    assert sorted(build.CUDA_SRCS) == sorted(os.path.join(folder, f) for f in os.listdir(folder) if f.endswith(".cu"))


@pytest.mark.parametrize("dep", included_files(), ids=os.path.basename)
def test_an_edited_header_makes_the_library_stale(monkeypatch, dep):
    monkeypatch.setattr(os.path, "exists", lambda path: True)
    monkeypatch.setattr(os.path, "getmtime", lambda path: {build.CUDA_LIB: 2.0, dep: 3.0}.get(os.path.normpath(path), 1.0))
    assert build.cuda_lib_is_stale()
