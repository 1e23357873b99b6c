"""The CG plan's construction with one host allocation failing, each in turn (on the CPU).

It runs behind C entries and on several threads: a failed allocation, a thread's
own start included, must end in a plan or in an exception that the entry
catches, never in an abort."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2102_05791_gb300", "csrc")

SRC = """
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include "cg_plan.h"
using namespace softsim;
static std::atomic<long> left(-1), seen(0);
void *operator new(size_t n)
{
    seen++;
    if (left.load() >= 0 && left.fetch_sub(1) == 0) throw std::bad_alloc();
    if (void *p = malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }
int main()
{
    const int n = 28, N = n + 1;
    std::vector<double> X;
    std::vector<int32_t> T, perm;
    for (int i = 0; i < N * N * N; ++i) X.insert(X.end(), {double(i % N), double(i / N % N), double(i / N / N)});
    const int hex[6][4] = {{0, 1, 3, 7}, {0, 1, 5, 7}, {0, 2, 3, 7}, {0, 2, 6, 7}, {0, 4, 5, 7}, {0, 4, 6, 7}};
    for (int c = 0; c < n * n * n; ++c)
        for (auto &h : hex)
            for (int o : h) T.push_back(c % n + (o & 1) + N * (c / n % n + (o >> 1 & 1) + N * (c / n / n + (o >> 2))));
    for (int i = 0; i < (int)T.size() / 4; ++i) perm.push_back(i);
    auto build = [&]() {
        CgPlan P;
        std::string err;
        return build_cg_plan(3, N * N * N, (int64_t)perm.size(), X.data(), T.data(), perm.data(), (int64_t)perm.size(), 64,
                             32, true, 4, true, P, err);
    };
    seen = 0;
    if (!build()) return 1;
    const long total = seen;
    int caught = 0, built = 0;
    for (long k = 0; k < total; k += k < 120 ? 1 : total / 60 + 1) {
        left = k;
        try {
            if (!build()) return 2;
            ++built;
        } catch (const std::bad_alloc &) {
            ++caught;
        }
        left = -1;
    }
    printf("%ld allocations: %d caught, %d built all the same", total, caught, built);
    return caught > 0 ? 0 : 3;
}
"""


def test_every_allocation_may_fail(tmp_path):
    (tmp_path / "m.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "m.cpp"),
                    os.path.join(CSRC, "cg_plan.cpp"), "-o", str(tmp_path / "m")], check=True)
    r = subprocess.run([str(tmp_path / "m")], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout, r.stderr)
