"""bench.py's record of the near field's DRAM bytes holds for the code it was captured on alone (CPU)."""

import os
import shutil

import pytest

import bench

#: (file, text, what it becomes): the kernel, the order of the points that it reads, and the items' sizes
CHANGES = [
    ("near_fwd.cuh", "kRows = R == 1", "kRows = R == 2"),
    ("near_warp.cuh", "constexpr int kListCap = 256", "constexpr int kListCap = 128"),
    ("internal.h", "constexpr int kOrderRun = 2048", "constexpr int kOrderRun = 1024"),
    ("internal.h", "strips * (strips + 1) < pieces", "strips * strips < pieces"),
    ("kernels_bin.cu", "key[t] = ((unsigned long long)strip << 48)", "key[t] = ((unsigned long long)strip << 47)"),
    ("sort_shared.cuh", "(a > b)", "(a >= b)"),
    ("femnfft.cu", "per_cell < 25.0 ? 8", "per_cell < 24.0 ? 8"),
    ("femnfft.cu", "*cap = near_item_lanes(", "*cap = 2 * near_item_lanes("),
    ("femnfft.cu", "std::min({count, cap, max_item})", "std::min({count, cap})"),
]


@pytest.mark.parametrize("name,text,other", CHANGES)
def test_changed_item_layouts_change_the_key(tmp_path, monkeypatch, name, text, other):
    csrc = tmp_path / "paper_0807_2387_gb300" / "csrc"
    shutil.copytree(os.path.join(bench.ROOT, "paper_0807_2387_gb300", "csrc"), csrc)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    before = bench.near_source_sha()
    code = (csrc / name).read_text()
    assert code.count(text) == 1
    (csrc / name).write_text(code.replace(text, other))
    assert bench.near_source_sha() != before
