"""bench.py reports captured DRAM bytes only while every source they depend on is the
captured one: the kernels, the layout they stream and the rules that shape a launch."""
import os
import shutil

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join("paper_1905_06234_gb300", "csrc")
SOURCES = ["spmv_tc.cu", "tile_build.cu", "tile_layout.cuh", "launch_rules.cuh", "tc_ptx.cuh", "life_internal.cuh"]


@pytest.fixture
def bench(tmp_path, monkeypatch):
    import bench
    os.makedirs(tmp_path / CSRC)
    for name in SOURCES:
        shutil.copy(os.path.join(ROOT, CSRC, name), tmp_path / CSRC / name)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setitem(bench.TRAFFIC_CAPTURE, "sha256", bench.traffic_digest())
    return bench


def test_reported_for_the_captured_sources(bench):
    cap = bench.TRAFFIC_CAPTURE
    for path, kinds in cap["bytes"].items():
        for kind, n in kinds.items():
            assert bench.kernel_traffic(path, kind, cap["nnz"]) == n
            assert bench.kernel_traffic(path, kind, 2 * cap["nnz"]) == 2 * n
    assert bench.kernel_traffic("fp32-simt", "dsc", cap["nnz"]) is None


@pytest.mark.parametrize("name", SOURCES)
def test_null_after_a_change(bench, tmp_path, name):
    with open(tmp_path / CSRC / name, "a") as fh:
        fh.write("\n")
    assert bench.kernel_traffic("bf16-tc", "dsc", 1) is None
    os.remove(tmp_path / CSRC / name)
    assert bench.kernel_traffic("bf16-tc", "dsc", 1) is None
