"""What bench.py states beside its times: the DRAM bytes of a capture count only for the source they were
taken from, and the number of kernels follows the library's rules."""
import re

import bench
from paper_2406_05221_b200 import build
from tests.test_build_deps import included_files


def test_the_digest_covers_every_header_of_the_kernel():
    # (igen.h belongs to the generator, gcaps_rta.h is the interface)
    wanted = {build.CUDA_SRC} | {p for p in included_files() if not p.endswith(("igen.h", "gcaps_rta.h"))}
    assert set(bench.kernel_sources()) == wanted


def test_traffic_is_reported_for_the_captured_source_only(monkeypatch):
    monkeypatch.setattr(bench, "kernel_source_digest", lambda: bench.CAPTURED_TRAFFIC["source_sha256"])
    assert bench.captured_traffic("large", "gcaps", 1000) > 9000 * 1000
    assert bench.captured_traffic("divergence", "gcaps", 1000) is None
    monkeypatch.setattr(bench, "kernel_source_digest", lambda: "another")
    assert bench.captured_traffic("large", "gcaps", 1000) is None


def test_launches_follow_the_dispatch():
    one, several = build.source_constant("kDirectMost"), build.source_constant("kDirectSweepMost")
    assert [bench.kernel_launches(n) for n in (1, one, one + 1, 10 ** 6)] == [1, 1, 11, 11]
    small = build.source_constant("kPlanSmall")
    assert [bench.kernel_launches(n, "several") for n in (several, several + 1, small, small + 1)] == [1, 7, 7, 9]
    assert [bench.kernel_launches(n, "search") for n in (several, several + 1, small, small + 1)] == [1, 8, 8, 10]
    text = open(build.CUDA_SRC).read()
    body = text[text.index("cudaError_t launch_all_bins("):]
    body = body[:body.index("\n}\n")]
    assert len(re.findall(r"e = launch_(?:persistent|big|deferred)\W", body)) == 8
