"""What bench.py counts as moved: the grid cells in use, and which sources a
recorded DRAM traffic belongs to (CPU only)."""
import os
import shutil
import sys
import types

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


class _Plan:
    """counts, layout and reach of a plan whose longest baseline is N / 3 cells"""

    def partition_counts(self, chan=0):
        return {"L": 3000, "H": 5000, "LH": 100, "ALL": 7900}

    def partition_layout(self, part, chan=0):
        return {"L": 7, "H": 11}[part], 22 * 22, 8

    def grid_extent(self):
        return 687


@pytest.mark.parametrize("fam,rest", [("degrid", 4000 * 28), ("grid", 4000 * 20),
                                      ("fold", 9 * 22 * 22 * 8)])
def test_only_grid_cells_in_use_count(fam, rest):
    cells = 1375 ** 2 * 8   # +-687 of 1024 on either side, complex FP32
    assert bench.family_bytes(fam, 1024, 8, 4, 4, _Plan(), 687) == rest + cells
    assert bench.family_bytes(fam, 1024, 8, 4, 4, _Plan(), 1024) == rest + 2048 ** 2 * 8
    # 1 ms a span
    r = bench.roofline_of({fam: (2, 2.0)}, types.SimpleNamespace(npix=1024), _Plan(),
                          types.SimpleNamespace(precision="fp32"))
    assert r["algorithmic_bytes_per_launch"] == rest + cells
