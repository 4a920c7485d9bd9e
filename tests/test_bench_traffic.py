"""The captured traffic of the step is tied to every source its kernel is compiled from."""
import os
import re

import bench
from paper_2106_01557_gb300 import build


def _includes(name, seen):
    if name not in seen:
        seen.add(name)
        with open(os.path.join(build.CSRC, name)) as f:
            for inc in re.findall(r'#include "([^"]+)"', f.read()):
                _includes(inc, seen)
    return seen


def test_step_sources_are_the_kernels_include_closure():
    assert sorted(bench.STEP_SOURCES) == sorted(_includes("lbm_march.cu", set()))


def test_a_changed_source_makes_the_traffic_null(monkeypatch):
    monkeypatch.setitem(bench.STEP_TRAFFIC, "sources_sha256", "0" * 64)
    assert bench.step_traffic() is None
