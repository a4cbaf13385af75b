"""bench.py's count of the library's kernel launches against the library's own
dispatch (tests/test_dispatch_host.py), and the iteration counts that it
reports."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_1402_3325_gb300 import sakura as sk  # noqa: E402
from test_dispatch_host import Run, fake_library  # noqa: E402,F401


@pytest.mark.parametrize("n", [9, 500, 700, 1000, 2999, 4100, 14000])
@pytest.mark.parametrize("form,rule,guess,pairs", [
    ("fp64", "hyp", "fp32", "symmetric"), ("fp64", "hyp", "standard", "symmetric"),
    ("df64", "hyp", "fp32", "symmetric"), ("mixed", "hyp", "fp32", "symmetric"),
    ("mixed", "literal", "fp32", "symmetric"), ("mixed", "literal", "standard", "symmetric"),
    ("fp64", "hyp", "fp32", "ordered")])
def test_launches_are_those_of_the_dispatch(fake_library, n, form, rule, guess, pairs):  # noqa: F811
    opts = bench._form_options(sk, form, pairs, rule)
    small = n <= sk.SMALL_MAX_N and form in ("fp64", "df64") and pairs == "symmetric"
    for per_call in (1, 4):
        with Run(fake_library, guess=bench._guess_code(sk, guess), **opts) as r:
            count = sum(len(r.evolve(n, 2.0 ** -8, 2, per_call)) for _ in range(8 // per_call))
        assert bench._launches(sk, n, form, pairs, rule, guess, 8, per_call, small) == count


@pytest.mark.parametrize("guess,counted", [("fp32", True), ("standard", False)])
def test_iteration_counts_are_the_timed_kernels_or_none(guess, counted):
    m = {"kepler_evals_per_solve": 1.0, "carried_share": 1.0, "iteration_lane_efficiency": 1.0,
         "fp32_pair_share": 0.0, "solves_per_pair": 0.5, "row_groups": True,
         "pair_kernel_ms": 5.0, "ms_per_step": 5.1, "fp64_evals_per_fp64_pair": 1.0}
    roof = bench._roofline("bh16384", "fp64", "symmetric", guess, 16384, False, m)
    for key in ("kepler_evals_per_solve", "carried_share", "iteration_lane_efficiency"):
        assert (roof[key] is not None) == counted
