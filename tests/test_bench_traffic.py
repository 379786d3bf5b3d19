"""Which sources a recorded DRAM traffic belongs to (CPU only)."""
import os
import shutil
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


@pytest.mark.parametrize("header,changed", [
    ("fft_radix.cuh", {"spec_mul", "fft_r2c", "fft_c2r"}),
    ("fine_levels.cuh", {"synth", "synth_l1", "analysis", "analysis_l1"}),
    ("common.cuh", set(bench.FAMILY_SOURCE)),
    ("grid_kernels.cu", {"degrid", "grid", "fold"}),
])
def test_a_changed_header_changes_its_families(tmp_path, monkeypatch, header, changed):
    csrc = tmp_path / "paper_2406_18356_gb300" / "csrc"
    shutil.copytree(os.path.join(ROOT, "paper_2406_18356_gb300", "csrc"), csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = {f: bench.kernel_source_digest(f) for f in bench.FAMILY_SOURCE}
    with open(csrc / header, "a") as f:
        f.write("// another line\n")
    after = {f: bench.kernel_source_digest(f) for f in bench.FAMILY_SOURCE}
    assert {f for f in before if before[f] != after[f]} == changed
