"""The sources a DRAM-traffic figure is keyed by are those that define the family's kernels (CPU)."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

KERNELS = {"k_cross_query": ["k_cross_query"], "k_join": ["k_join_tc", "k_join_sparse"], "k_prune": ["k_prune_bytes", "k_prune"]}


@pytest.mark.parametrize("family", sorted(KERNELS))
def test_a_family_is_keyed_by_the_files_of_its_kernels(family):
    import bench
    csrc = os.path.join(ROOT, "paper_2603_21710_gb300", "csrc")
    text = "".join(open(os.path.join(csrc, f)).read() for f in bench.TRAFFIC_SOURCES[family])
    for k in KERNELS[family]:
        assert re.search(r"__global__[^;{]*\b%s\(" % k, text), k
    # and by what those files include of the device code
    for inc in re.findall(r'#include "(k_[a-z]+\.cuh|tc_[a-z0-9]+\.cuh)"', text):
        assert inc in bench.TRAFFIC_SOURCES[family], inc
