"""When the persistent CG solver may be launched, from what the device reports (on the CPU).

Its CTAs wait for one another, so all must be on the device at once: a device
that cannot form the cluster, or with fewer places than the grid has CTAs,
must get the per-iteration kernels instead of a failing launch."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2102_05791_gb300", "csrc")

SRC = """
#include <cstdio>
#include <cstdlib>
#include "cg_plan.h"
int main(int, char **v)
{
    printf("%d", softsim::pcg_resident(atoi(v[1]), atoi(v[2]), atoi(v[3]), atoi(v[4]), atoi(v[5])) ? 1 : 0);
}
"""


@pytest.fixture(scope="module")
def resident(tmp_path_factory):
    d = tmp_path_factory.mktemp("resident")
    (d / "r.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "r.cpp"), "-o", str(d / "r")], check=True)
    return lambda *a: subprocess.run([str(d / "r"), *map(str, a)], check=True, capture_output=True, text=True).stdout == "1"


@pytest.mark.parametrize("cluster,n_cta,clusters,per_sm,sms,may", [
    (1, 16, 8, 0, 152, True), (1, 16, 1, 0, 152, True), (1, 16, 0, 1, 152, False),   # no room for one cluster
    (0, 152, 0, 1, 152, True), (0, 152, 0, 1, 148, False), (0, 64, 0, 1, 40, False),  # fewer SMs than CTAs
    (0, 1, 0, 1, 1, True), (0, 1, 0, 0, 152, False), (0, 300, 0, 2, 152, True)])
def test_launch_only_what_is_resident(resident, cluster, n_cta, clusters, per_sm, sms, may):
    assert resident(cluster, n_cta, clusters, per_sm, sms) == may
