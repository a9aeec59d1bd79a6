"""The bench reports a share of the issue rate only where ncu counted that very
launch on the current sources and an SM clock was sampled."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_count_of_other_sources_is_not_used(tmp_path, monkeypatch):
    (tmp_path / "profiles").mkdir()
    (tmp_path / "profiles" / "rollout_paper_scale.json").write_text(
        json.dumps({"kernel_sources_hash": "aa", "warp_instructions": 1000, "dram_bytes_per_launch": 5}))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.load_profile("bb") is None
    assert bench.load_profile("aa", "multi_speed") is None
    assert bench.load_profile("aa")["dram_bytes_per_launch"] == 5


def test_issue_rates():
    prof = {"warp_instructions": 8_000_000}
    assert bench.issue_rates(None, 1e-4, 152, 2070.0) == (None, None)
    assert bench.issue_rates(prof, 1e-4, 152, None) == (None, None)
    got, most = bench.issue_rates(prof, 1e-4, 100, 2000.0)
    assert got == pytest.approx(8e10) and most == pytest.approx(4 * 100 * 2e9)
