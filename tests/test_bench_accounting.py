"""What bench.py states beside its times: the DRAM bytes of a capture count only for the source they were
taken from."""
import bench
from paper_2406_05221_b200 import build
from tests.test_build_deps import included_files


def test_the_digest_covers_every_header_of_the_kernel():
    wanted = {build.CUDA_SRC} | {p for p in included_files() if p.endswith(".cuh")}
    assert set(bench.kernel_sources()) == wanted


def test_traffic_is_reported_for_the_captured_source_only(monkeypatch):
    monkeypatch.setattr(bench, "kernel_source_digest", lambda: bench.CAPTURED_TRAFFIC["source_sha256"])
    assert bench.captured_traffic("large", "gcaps", 1000) > 9000 * 1000
    assert bench.captured_traffic("divergence", "gcaps", 1000) is None
    monkeypatch.setattr(bench, "kernel_source_digest", lambda: "another")
    assert bench.captured_traffic("large", "gcaps", 1000) is None

