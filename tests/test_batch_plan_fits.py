"""Which bodies the batched solver accepts a CG plan for, checked on the CPU.

The coarse matrix is inverted in shared memory where the edge slice will lie,
below the body's plan record: a plan may be taken only if that scratch and the
slice both end before it.  A fan's hub has every rim vertex in its halo, which
leaves little room behind the vectors; such bodies run matrix-free."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2102_05791_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("plan") / "batch_plan_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC, os.path.join(HERE, "batch_plan_check.cpp"),
                    os.path.join(CSRC, "cg_plan.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("n,n_cta,threads,taken", [
    (3, 1, 128, True), (900, 1, 256, True), (4000, 8, 256, True), (9000, 16, 128, True),
    (15200, 16, 128, False), (15900, 16, 128, False)])
def test_scratch_and_slice_end_before_the_plan_record(checker, n, n_cta, threads, taken):
    fits, scratch, slice_end, limit = map(int, subprocess.run([checker, str(n), str(n_cta), str(threads)], check=True,
                                                              capture_output=True, text=True).stdout.split())
    if limit:  # else no plan could be built at all
        assert (scratch <= limit and slice_end <= limit) == taken
    assert bool(fits) == taken
