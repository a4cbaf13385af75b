"""The committed profile summaries of the weak-pair kernels match the sources
they were taken from (else bench.py reports their traffic as null)."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("kernel,workload", [("pair_step_grp_weak", "bh16384"),
                                             ("pair_step_weak", "plummer2048")])
def test_weak_profile_summaries_match_the_current_kernel_sources(kernel, workload):
    with open(os.path.join(ROOT, "profiles", f"{kernel}_{workload}.md")) as fh:
        taken = re.search(r"- sources_sha256_16: `(\w+)`", fh.read()).group(1)
    assert taken == bench._kernel_sources_hash(kernel)
