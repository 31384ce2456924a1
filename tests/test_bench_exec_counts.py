"""The roofline's counts of what the rule kernel executes (bench.py RULE_EXEC_*):
they cover the benchmark's families -- a family without them drops the roofline
from the line -- and the fingerprints they are tied to cover every header that
the counted kernels are compiled from."""
import os
import re

import bench


def test_executed_counts_cover_the_benchmark_families():
    from paper_2511_01573_gb300 import genz_inputs as G
    for fam in G.GENZ_D8_FAMILIES:
        assert bench.RULE_EXEC_FP64_INST_D8[fam] > 0
        assert bench.RULE_EXEC_FP64_FLOPS_D8[fam] > 0
        # FP64 instructions are among all of them
        assert bench.RULE_EXEC_INST_D8[fam] > bench.RULE_EXEC_FP64_INST_D8[fam]


def _headers(name, seen):
    if name not in seen:
        seen.add(name)
        path = os.path.join(bench.ROOT, "paper_2511_01573_gb300", "csrc", name)
        with open(path) as f:
            for h in re.findall(r'#include "(\w+\.cuh)"', f.read()):
                _headers(h, seen)
    return seen


def test_fingerprints_cover_the_included_headers():
    assert _headers("gm_rule.cuh", set()) == set(bench.RULE_COUNTS_SOURCES)
    # gm_rule_mixed.cuh takes the launch helpers of the FP64 kernel; what it
    # evaluates a region with is gm_region32.cuh
    mixed = _headers("gm_region32.cuh", set()) | {"gm_rule_mixed.cuh"}
    assert mixed == set(bench.MIXED_COUNTS_SOURCES)
