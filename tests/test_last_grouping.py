"""Which sort grouped the pairs: pss_get_last_grouping, and the benchmark's description of it (a
segment-local pass may count the distinct locations, so the collision rate does not tell)."""
import os
import re

import pytest

import bench
from paper_2207_10731_gb300 import binding, workloads as wl
from tests import gpu_util as gu
from tests.test_bench_host import _parse

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_values_match_the_header():
    src = open(os.path.join(ROOT, "include", "pss.h")).read()
    vals = {k: int(v) for k, v in re.findall(r"\bPSS_GROUPED_([A-Z]+)\s*=\s*(\d+)", src)}
    assert sorted(vals) == ["COUNTING", "LOCAL", "NONE", "RADIX"]
    for name, value in vals.items():
        assert getattr(binding, f"GROUPED_{name}") == value


@pytest.mark.parametrize("grouping,rate,says", [
    (binding.GROUPED_LOCAL, 0.5, "segment-local"), (binding.GROUPED_LOCAL, -1.0, "segment-local"),
    (binding.GROUPED_COUNTING, 0.5, "counting sort"), (binding.GROUPED_RADIX, 0.5, "radix sort")])
def test_description_follows_the_sort_that_ran(grouping, rate, says):
    class H:
        def info(self):
            return dict(last_path=binding.PATH_SORTED, last_collision_rate=rate, R=1 << 20)

        def last_grouping(self):
            return grouping
    d = bench._sort_desc(H(), binding, _parse([]))
    assert d["sort"].startswith(says)
    assert d.get("collision_rate") == (rate if rate >= 0 else None)


@pytest.mark.gpu
@pytest.mark.parametrize("name,B,opts,want", [
    ("tb", 65536, {}, binding.GROUPED_LOCAL),              # counted: a rate is reported
    ("tb", 2048, {}, binding.GROUPED_LOCAL),
    ("tb", 2048, {binding.OPT_SORT_SCOPE: binding.SORT_GLOBAL}, binding.GROUPED_COUNTING),
    ("tb", 2048, {binding.OPT_DETERMINISTIC: 1}, binding.GROUPED_RADIX),
    ("kaggle", 2048, {}, binding.GROUPED_NONE)])
def test_last_grouping(name, B, opts, want):
    w = wl.make_workload(name, B=B)
    h, _ = gu.make_pair(w)
    for k, v in opts.items():
        h.set_option(k, v)
    assert h.last_grouping() == binding.GROUPED_NONE
    h.forward(gu.cuda(w.indices), gu.cuda(w.offsets), B)
    h.backward_update(gu.cuda(w.grad_out), w.lr)
    assert h.last_grouping() == want
    h.close()
