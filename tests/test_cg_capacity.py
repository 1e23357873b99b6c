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
def program(tmp_path_factory):
    """Builds a program on the plan's source; returns what runs it."""
    d = tmp_path_factory.mktemp("plan")
    cxx = ["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC]
    subprocess.run([*cxx, "-c", os.path.join(CSRC, "cg_plan.cpp"), "-o", str(d / "cg_plan.o")], check=True)

    def build(name, src):
        if not (d / name).exists():
            (d / f"{name}.cpp").write_text(src)
            subprocess.run([*cxx, str(d / f"{name}.cpp"), str(d / "cg_plan.o"), "-o", str(d / name)], check=True)
        return lambda *a: subprocess.run([str(d / name), *map(str, a)], capture_output=True, text=True)

    return build


@pytest.fixture(scope="module")
def sizes(program):
    run = program("sizes", SRC)
    return lambda *a: [int(x) for x in run(*a).stdout.split()]


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


VARIANT = """
#include <cstdio>
#include <cstdlib>
#include "cg_plan.h"
int main(int, char **v)
{
    const int dim = atoi(v[1]), elt = atoi(v[2]);
    const long long top = elt == 4 ? 583680 : 291840;
    bool used[2][2][9] = {};
    for (long long nv = 1; nv <= top; nv += 1 + nv / 997) {
        const softsim::PcgSizes z = softsim::pcg_sizes(dim, elt, nv, 152);
        const bool grid = z.n_cta > 16;
        long long per = (nv + z.n_cta - 1) / z.n_cta, a = z.n_agg > z.n_cta ? z.n_agg / z.n_cta : 1;
        const int slots = (int)(a * (((per + a - 1) / a + 31) / 32 * 32));
        for (int threads : {softsim::kPcgThreads, softsim::kPcgStreamThreads}) {
            if (z.rows && threads != softsim::kPcgThreads) continue;
            if (slots > softsim::pcg_max_vpt(elt, z.rows) * threads) continue;
            const int need = (slots + threads - 1) / threads, got = softsim::pcg_variant(dim, elt, z.rows, grid, need);
            if (got < need) return printf("%lld vertices, %d slots: none", nv, slots), 1;
            used[z.rows][grid][got] = true;
        }
    }
    for (int r = 0; r < 2; ++r)
        for (int g = 0; g < 2; ++g)
            for (int k = 1; k < 9; ++k)
                if (used[r][g][k]) printf("%s%s%d ", r ? "rows" : "colours", g ? "-grid-" : "-", k);
    return 0;
}
"""


@pytest.mark.parametrize("dim,elt,variants", [
    (2, 4, "colours-grid-4 colours-grid-8 rows-1 rows-4 rows-grid-1 rows-grid-4"),
    (2, 8, "rows-1 rows-grid-1 rows-grid-4"),
    (3, 4, "colours-grid-2 colours-grid-4 colours-grid-8 rows-1 rows-grid-1 rows-grid-4"),
    (3, 8, "colours-grid-2 colours-grid-4 rows-1 rows-grid-1 rows-grid-4")])
def test_every_size_has_a_kernel_and_every_kernel_a_size(program, dim, elt, variants):
    r = program("variants", VARIANT)(dim, elt)
    assert r.returncode == 0 and r.stdout.split() == variants.split(), r.stdout


CHUNKS = """
#include <cstdio>
#include <cstdlib>
#include "cg_plan.h"
using namespace softsim;
int main(int, char **v)
{
    const int n = atoi(v[1]), elt = atoi(v[2]), N = n + 1;
    std::vector<double> X;
    std::vector<int32_t> T, perm;
    for (int i = 0; i < N * N * N; ++i) X.insert(X.end(), {double(i % N), double(i / N % N), double(i / N / N)});
    const int hex[6][4] = {{0, 1, 3, 7}, {0, 1, 5, 7}, {0, 2, 3, 7}, {0, 2, 6, 7}, {0, 4, 5, 7}, {0, 4, 6, 7}};
    for (int c = 0; c < n * n * n; ++c)
        for (auto &h : hex)
            for (int o : h) T.push_back(c % n + (o & 1) + N * (c / n % n + (o >> 1 & 1) + N * (c / n / n + (o >> 2))));
    for (int i = 0; i < (int)T.size() / 4; ++i) perm.push_back(i);
    CgPlan P;
    std::string err;
    if (!build_cg_plan(3, N * N * N, (int64_t)perm.size(), X.data(), T.data(), perm.data(), (int64_t)perm.size(), 16, 32,
                       true, elt, false, P, err))
        return 1;
    int rest = 0;
    for (int c = 0; c < P.n_cta; ++c) rest += P.chunk_ent[P.chunk_ptr[c] + 2] - P.chunk_ent[P.chunk_ptr[c] + 1];
    printf("%d", rest);
}
"""


@pytest.mark.parametrize("n,elt,beyond", [(8, 4, False), (22, 4, True), (8, 8, False), (18, 8, True)])
def test_rows_beyond_shared_memory_fill_the_second_chunk(program, n, elt, beyond):
    """16 CTAs: 46 and 761 vertices each in FP32, 46 and 429 in FP64 (76 bytes an entry, 14 a vertex, 214 KB)."""
    r = program("chunks", CHUNKS)(n, elt)
    assert r.returncode == 0 and (int(r.stdout) > 0) == beyond
