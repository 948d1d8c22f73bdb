"""bench.py reports recorded DRAM traffic only for the sources it was measured on (CPU)."""
import os
import shutil

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_1305_4196_gb300", "csrc")


@pytest.mark.parametrize("name", ["k_force.cu", "full_task.cuh", "tile.cuh", "fixpt.cuh", "mdgb_internal.cuh"])
def test_a_change_to_any_source_of_the_force_kernel_shows(tmp_path, name):
    csrc = tmp_path / "csrc"
    shutil.copytree(CSRC, csrc)
    assert bench.force_source_sha256(str(csrc)) == bench.force_source_sha256()
    with open(csrc / name, "a") as f:
        f.write("// changed\n")
    assert bench.force_source_sha256(str(csrc)) != bench.force_source_sha256()


def test_other_sources_do_not(tmp_path):
    csrc = tmp_path / "csrc"
    shutil.copytree(CSRC, csrc)
    with open(csrc / "k_grad.cu", "a") as f:
        f.write("// changed\n")
    assert bench.force_source_sha256(str(csrc)) == bench.force_source_sha256()


def test_stale_traffic_is_dropped(monkeypatch):
    monkeypatch.setattr(bench, "force_source_sha256", lambda *a: "0" * 64)
    assert bench.measured_force_traffic(1 << 20, True) is None
