"""bench.py quotes DRAM bytes per launch only where they were taken on the present sources of the stage's
kernels: the unit itself and every header that it includes.
"""
import json
import os
import re
import shutil

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_1905_00182_gb300", "csrc")


def _included(name, seen=None):
    """the unit and the headers of its folder that it includes, directly or not"""
    seen = set() if seen is None else seen
    if name not in seen and os.path.exists(os.path.join(CSRC, name)):
        seen.add(name)
        with open(os.path.join(CSRC, name)) as f:
            for h in re.findall(r'#include "([^"/]+)"', f.read()):
                _included(h, seen)
    return seen


@pytest.mark.parametrize("precision,unit", [("fp32", "stage_fp32.cu"), ("fp64", "stage_fp64_fast.cu")])
def test_any_changed_source_voids_the_figures(precision, unit, tmp_path, monkeypatch):
    names = _included(unit)
    assert set(bench.STAGE_SOURCES[precision]) == names
    copy = tmp_path / "paper_1905_00182_gb300" / "csrc"
    shutil.copytree(CSRC, copy)
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    rec = {f"{precision}:pad": {"source_sha": bench.source_sha(precision), "bytes_per_launch_full": 7.0}}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(rec))
    assert bench.ncu_traffic("pad", precision) == 7.0
    for name in names:
        text = (copy / name).read_text()
        (copy / name).write_text(text + "// changed\n")
        assert bench.ncu_traffic("pad", precision) is None, name
        (copy / name).write_text(text)
    assert bench.ncu_traffic("pad", precision) == 7.0
