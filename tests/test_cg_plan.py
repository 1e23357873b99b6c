"""The persistent CG solver's plan (parts, edge layouts, coarse items), checked on the CPU.

cg_plan_check.cpp builds the plan of one grid mesh and checks its invariants;
here over one CTA, a cluster and a grid, aligned and uneven sizes, both edge
layouts, both precisions, and vertices in grid order and in random order."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2102_05791_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("plan") / "cg_plan_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC, os.path.join(HERE, "cg_plan_check.cpp"),
                    os.path.join(CSRC, "cg_plan.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("rows", [0, 1])
@pytest.mark.parametrize("shuffle", [0, 1])
@pytest.mark.parametrize("dim,nx,ny,nz,n_cta,n_agg", [
    (2, 1, 1, 0, 1, 1), (2, 16, 8, 0, 1, 8), (2, 19, 7, 0, 5, 8), (2, 64, 32, 0, 16, 64), (2, 10, 2, 0, 2, 1), (2, 9, 4, 0, 4, 2), (2, 120, 61, 0, 75, 25),
    (3, 1, 1, 1, 1, 1), (3, 3, 4, 5, 2, 6), (3, 13, 9, 8, 16, 32), (3, 25, 13, 12, 31, 31), (3, 33, 17, 15, 150, 30)])
def test_plan_invariants(checker, dim, nx, ny, nz, n_cta, n_agg, shuffle, rows):
    for elt in (4, 8):
        r = subprocess.run([checker, *[str(a) for a in (dim, nx, ny, nz, n_cta, n_agg, shuffle, rows, elt)]],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stdout


def test_rows_beyond_shared_memory_go_to_the_second_chunk(checker):
    """Parts whose rows do not fit in shared memory (about 560 vertices in 3D FP32)."""
    r = subprocess.run([checker, "3", "40", "20", "20", "16", "32", "0", "1", "8"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
