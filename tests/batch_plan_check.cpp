// Plan of a batched body whose topology is a fan: n triangles around one hub
// vertex, cut over n_cta CTAs (arguments n n_cta threads).  Prints whether the
// batched solver takes the plan, and the bytes of shared memory that the
// coarse inverse's scratch and the rows' first chunk end at, and their limit.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <numeric>

#include "cg_plan.h"

using namespace softsim;

int main(int argc, char **argv)
{
    if (argc != 4) return 2;
    const int n = atoi(argv[1]), n_cta = atoi(argv[2]), threads = atoi(argv[3]);
    std::vector<double> X = {0.0, 0.0};
    std::vector<int32_t> T, perm(n);
    for (int i = 0; i < n; ++i) {
        const double t = 2.0 * std::acos(-1.0) * i / n;
        X.push_back(std::cos(t));
        X.push_back(std::sin(t));
        T.insert(T.end(), {0, 1 + i, 1 + (i + 1) % n});
    }
    std::iota(perm.begin(), perm.end(), 0);
    CgPlan P;
    std::string err;
    if (!build_cg_plan(2, n + 1, n, X.data(), T.data(), perm.data(), n, n_cta, 2 * n_cta, true, 4, false, P, err)) {
        printf("0 0 0 0\n");
        return 0;
    }
    const size_t N = (size_t)P.n_agg * P.n_modes;
    const PcgSmem L(2, 4, P.ns, P.max_halo, P.max_items, (int)N, P.n_meta, 0);
    printf("%d %zu %zu %d\n", batch_plan_fits(P, threads) ? 1 : 0, L.ring + 4 * (N * N + 3 * N),
           L.ring + (size_t)P.max_entries * (4 + 4 * 4), kBatchPlanAt);
    return 0;
}
