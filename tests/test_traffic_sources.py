"""The hash that keeps a recorded DRAM traffic figure covers what decides a step's traffic: the
step units with everything they include, and capi.cu, whose rules choose the form of a run's
steps (a 256^3 step moves 497 MB where the mixed derivatives are rebuilt, 1124 MB where not)."""
import os
import re

import pytest

import bench

CSRC = os.path.join(bench.ROOT, "paper_0905_3409_gb300", "csrc")


def _included(name, seen):
    if name in seen:
        return
    seen.add(name)
    with open(os.path.join(CSRC, name)) as f:
        for inc in re.findall(r'#include "([^"/]+)"', f.read()):
            if os.path.exists(os.path.join(CSRC, inc)):
                _included(inc, seen)


@pytest.mark.parametrize("dim", [2, 3])
def test_sources_are_complete(dim):
    need = set()
    for unit in os.listdir(CSRC):
        if unit.startswith(f"step{dim}d") and unit.endswith(".cu"):
            _included(unit, need)
    listed = bench.KERNEL_SOURCES[dim]
    assert need | {"capi.cu"} <= set(listed), sorted((need | {"capi.cu"}) - set(listed))
    assert len(set(listed)) == len(listed)


def test_every_form_of_a_run_changes_the_hash(tmp_path, monkeypatch):
    before = bench.kernel_source_hash(3)
    copy = tmp_path / "paper_0905_3409_gb300" / "csrc"
    copy.mkdir(parents=True)
    for fn in bench.KERNEL_SOURCES[3]:
        with open(os.path.join(CSRC, fn), "rb") as f:
            text = f.read()
        (copy / fn).write_bytes(text)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.kernel_source_hash(3) == before
    rule = copy / "capi.cu"
    rule.write_bytes(rule.read_bytes().replace(b"> 1.05", b"> 1.5"))
    assert bench.kernel_source_hash(3) != before
