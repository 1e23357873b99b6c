"""Which meshes the persistent CG solver takes, known from their size alone (on the CPU).

x and r of a slot stay in a thread's registers, 8 slots of 480 threads (FP64: 4)
on each SM at most; a larger mesh must be refused before any table of its plan
is built, which takes seconds there."""
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
    const softsim::PcgSizes z = softsim::pcg_sizes(atoi(v[1]), atoi(v[2]), atoll(v[3]), atoi(v[4]));
    printf("%d %d %d %d %d", z.n_cta, z.n_agg, z.cluster ? 1 : 0, z.rows ? 1 : 0, z.fits ? 1 : 0);
}
"""


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    d = tmp_path_factory.mktemp("sizes")
    (d / "s.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC, str(d / "s.cpp"),
                    os.path.join(CSRC, "cg_plan.cpp"), "-o", str(d / "s")], check=True)
    return lambda *a: [int(x) for x in subprocess.run([str(d / "s"), *map(str, a)], check=True, capture_output=True,
                                                      text=True).stdout.split()]


@pytest.mark.parametrize("dim,elt,nv,fits", [
    (3, 4, 1, True), (3, 4, 545025, True), (3, 4, 583680, True), (3, 4, 583681, False), (3, 4, 1056321, False),
    (3, 4, 2 ** 30, False), (3, 8, 291840, True), (3, 8, 291841, False), (2, 4, 583680, True), (2, 4, 583681, False),
    (2, 8, 291840, True), (2, 8, 291841, False)])
def test_capacity(sizes, dim, elt, nv, fits):
    assert sizes(dim, elt, nv, 152)[4] == fits


@pytest.mark.parametrize("elt", [4, 8])
@pytest.mark.parametrize("dim", [2, 3])
def test_every_size_below_it_has_a_layout(sizes, dim, elt):
    """Parts, aggregates and coarse unknowns within the solver's limits; one CTA and clusters by rows."""
    nv = 1
    while nv <= (583680 if elt == 4 else 291840):
        n_cta, n_agg, cluster, rows, fits = sizes(dim, elt, nv, 152)
        assert fits and 1 <= n_cta <= min(152, nv) and n_agg * (6 if dim == 3 else 3) <= 192
        assert cluster == (1 < n_cta <= 16) and (rows or n_cta > 16)
        nv = nv + max(1, nv // 5)
