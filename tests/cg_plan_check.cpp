// Checks the plan of the persistent CG solver (paper_2102_05791_gb300/csrc/
// cg_plan.cpp) on one grid mesh: arguments dim nx ny nz n_cta n_agg shuffle
// rows elt.  Every contribution, edge, slot and coarse item must be covered
// exactly once, no two entries of a colour may add to one vertex, local ids
// must be in range, and the product formed from the stored entries must equal
// the one formed from the elements.  Exits 0 when all holds.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "cg_plan.h"

using namespace softsim;

#define REQ(c)                                             \
    do {                                                   \
        if (!(c)) {                                        \
            printf("line %d: %s\n", __LINE__, #c);         \
            exit(1);                                       \
        }                                                  \
    } while (0)

int main(int argc, char **argv)
{
    REQ(argc == 10);
    const int dim = atoi(argv[1]), nx = atoi(argv[2]), ny = atoi(argv[3]), nz = atoi(argv[4]);
    const bool shuffle = atoi(argv[7]), rows = atoi(argv[8]);
    const int NX = nx + 1, NY = ny + 1, NZ = dim == 3 ? nz + 1 : 1, nc = dim + 1, np = nc * (nc - 1) / 2;
    std::vector<double> X;
    std::vector<int32_t> T;
    for (int k = 0; k < NZ; ++k)
        for (int j = 0; j < NY; ++j)
            for (int i = 0; i < NX; ++i) {
                X.push_back(i);
                X.push_back(j);
                if (dim == 3) X.push_back(k);
            }
    const int hex[6][4] = {{0, 1, 3, 7}, {0, 1, 5, 7}, {0, 2, 3, 7}, {0, 2, 6, 7}, {0, 4, 5, 7}, {0, 4, 6, 7}};
    const int quad[2][3] = {{0, 1, 3}, {0, 3, 2}};
    for (int k = 0; k < (dim == 3 ? nz : 1); ++k)
        for (int j = 0; j < ny; ++j)
            for (int i = 0; i < nx; ++i)
                for (int e = 0; e < (dim == 3 ? 6 : 2); ++e)
                    for (int c = 0; c < nc; ++c) {
                        const int o = dim == 3 ? hex[e][c] : quad[e][c];
                        T.push_back(i + (o & 1) + NX * (j + (o >> 1 & 1) + NY * (k + (o >> 2))));
                    }
    const int64_t nv = (int64_t)X.size() / dim, ne = (int64_t)T.size() / nc;
    std::mt19937 rng(3);
    if (shuffle) {
        std::vector<int> to(nv);
        for (int i = 0; i < nv; ++i) to[i] = i;
        std::shuffle(to.begin(), to.end(), rng);
        const std::vector<double> Y = X;
        for (int i = 0; i < nv; ++i)
            for (int c = 0; c < dim; ++c) X[to[i] * dim + c] = Y[i * dim + c];
        for (int32_t &t : T) t = to[t];
    }
    std::vector<int32_t> perm;  // with padding, as the tiles have it
    for (int i = 0; i < ne; ++i) {
        perm.push_back(i);
        if (i % 37 == 5) perm.push_back(-1);
    }
    CgPlan P;
    std::string err;
    const int want = atoi(argv[5]);
    REQ(build_cg_plan(dim, nv, ne, X.data(), T.data(), perm.data(), (int64_t)perm.size(), want, atoi(argv[6]), rows,
                      atoi(argv[9]), want > 16, P, err));
    const int G = P.n_cta;
    std::vector<int> slot(nv, -1);
    for (int s = 0; s < (int)P.slot_gid.size(); ++s)
        if (P.slot_gid[s] >= 0) {
            REQ(slot[P.slot_gid[s]] < 0 && s % P.ns < P.nslot[s / P.ns]);
            slot[P.slot_gid[s]] = s;
        }
    for (int s : slot) REQ(s >= 0);

    // contributions: each once, to the right edge and side
    std::vector<double> con(P.n_contrib, 0.0), blk(P.n_edges, 0.0), p(nv), y(nv, 0.0), z(nv, 0.0);
    std::vector<char> seen(P.n_contrib, 0);
    std::uniform_real_distribution<double> uni(-1.0, 1.0);
    for (double &v : p) v = uni(rng);
    for (size_t e = 0; e < perm.size(); ++e) {
        int q = 0;
        for (int a = 0; a < nc; ++a)
            for (int b = a + 1; b < nc; ++b, ++q) {
                const uint32_t w = P.cpos[e * np + q], k = w & ~kCgTransposed;
                if (perm[e] < 0) {
                    REQ(w == kCgPadEntry);
                    continue;
                }
                const int i = T[(int64_t)perm[e] * nc + a], j = T[(int64_t)perm[e] * nc + b];
                REQ(k < P.n_contrib && !seen[k]);
                seen[k] = 1;
                REQ(((w & kCgTransposed) != 0) == (slot[i] > slot[j]));
                const int ed = (int)(std::upper_bound(P.edge_ptr.begin(), P.edge_ptr.end(), (int)k) - P.edge_ptr.begin()) - 1;
                REQ(P.edge_lo[ed] == std::min(slot[i], slot[j]) && P.edge_hi[ed] == std::max(slot[i], slot[j]));
                con[k] = uni(rng);
                y[i] += con[k] * (p[j] - p[i]);
                y[j] += con[k] * (p[i] - p[j]);
            }
    }
    for (char c : seen) REQ(c);
    for (int64_t e = 0; e < P.n_edges; ++e) {
        REQ(P.edge_ptr[e] < P.edge_ptr[e + 1]);
        for (int q = P.edge_ptr[e]; q < P.edge_ptr[e + 1]; ++q) blk[e] += con[q];
    }

    // entries
    for (int c = 0; c < G; ++c) {
        const int ns = P.nslot[c], h0 = P.halo_ptr[c], nh = P.halo_ptr[c + 1] - h0, k0 = P.chunk_ptr[c];
        REQ(ns % 32 == 0 && ns <= P.ns && nh <= P.max_halo);
        auto gid = [&](int local) { return P.slot_gid[local < ns ? c * P.ns + local : P.halo_slot[h0 + local - ns]]; };
        auto check = [&](int e, int i, int j) {
            REQ(i < ns && j < ns + nh && gid(i) >= 0 && gid(j) >= 0);
            const int ed = P.ent_edge[e] & ~kCgTransposed, lo = P.slot_gid[P.edge_lo[ed]], hi = P.slot_gid[P.edge_hi[ed]];
            REQ(P.ent_edge[e] & kCgTransposed ? gid(i) == hi && gid(j) == lo : gid(i) == lo && gid(j) == hi);
            z[gid(i)] += blk[ed] * (p[gid(j)] - p[gid(i)]);
        };
        if (rows) {
            REQ(P.chunk_ptr[c + 1] - k0 == 2);
            REQ(P.chunk_ent[k0 + 1] - P.chunk_ent[k0] <= P.max_entries);
            const int n_vw = ns * P.tpr / 32;
            REQ(2 * (n_vw + 1) <= P.n_meta);
            for (int part = 0; part < 2; ++part)
                for (int vw = 0; vw < n_vw; ++vw) {
                    const uint32_t *at = &P.row_step[(size_t)c * P.n_meta + part * (n_vw + 1) + vw];
                    for (uint32_t s = at[0]; s < at[1]; ++s)
                        for (int l = 0; l < 32; ++l) {
                            const int e = P.chunk_ent[k0 + part] + (int)s * 32 + l;
                            REQ(e < P.chunk_ent[k0 + part + 1]);
                            const int i = P.ent_idx[e] & 0xffff, j = P.ent_idx[e] >> 16;
                            REQ(i == (vw * 32 + l) / P.tpr);
                            if (P.ent_edge[e] == kCgPadEntry)
                                REQ(i == j);
                            else
                                check(e, i, j);
                        }
                }
        } else {
            REQ(P.chunk_ptr[c + 1] - k0 <= P.max_chunks);
            REQ(P.chunk_ent[P.chunk_ptr[c + 1]] - P.chunk_ent[k0] <= P.max_entries);
            std::vector<char> used(ns, 0);
            for (int k = k0; k < P.chunk_ptr[c + 1]; ++k) {
                const int n = (int)(P.chunk_n[k] & ~kCgLastOfColour);
                REQ(n == P.chunk_ent[k + 1] - P.chunk_ent[k] && n % 4 == 0 && n <= kCgChunk);
                for (int e = P.chunk_ent[k]; e < P.chunk_ent[k + 1]; ++e) {
                    if (P.ent_idx[e] == kCgPadEntry) {
                        REQ(P.ent_edge[e] == kCgPadEntry);
                        continue;
                    }
                    const int i = P.ent_idx[e] & 0xffff, j = P.ent_idx[e] >> 16;
                    check(e, i, j);
                    REQ(!used[i]);
                    used[i] = 1;
                    if (j < ns) {  // two-sided
                        REQ(!used[j]);
                        used[j] = 1;
                        z[gid(j)] += blk[P.ent_edge[e] & ~kCgTransposed] * (p[gid(i)] - p[gid(j)]);
                    }
                }
                if (P.chunk_n[k] & kCgLastOfColour) std::fill(used.begin(), used.end(), 0);
            }
        }
        const int a0 = P.item_agg[P.item_ptr[c]], ni = P.item_ptr[c + 1] - P.item_ptr[c];
        REQ(ni <= P.max_items);
        for (int q = 0; q < ni; ++q) REQ(P.item_agg[P.item_ptr[c] + q] == a0 + q);
        for (int g = 0; g < ns / 32; ++g) {
            const int a = P.grp_agg[c * P.ns / 32 + g];
            REQ(a >= a0 && a < a0 + ni);
        }
    }
    for (int i = 0; i < nv; ++i) REQ(std::fabs(y[i] - z[i]) < 1e-11);

    // aggregates and the items of the coarse matrix
    for (int a = 0; a < P.n_agg; ++a) {
        REQ(P.agg_item[a] < P.agg_item[a + 1]);
        REQ(want > 16 || P.agg_item[a + 1] - P.agg_item[a] == 1);  // a cluster does not sum items
        for (int q = P.agg_item[a]; q < P.agg_item[a + 1]; ++q) REQ(P.item_agg[q] == a);
    }
    std::vector<int> slots(P.slot_gid.size(), 0), edges(P.n_edges, 0);
    for (size_t t = 0; t < P.ctgt_i.size(); ++t)
        for (int q = P.ctgt_ptr[t]; q < P.ctgt_ptr[t + 1]; ++q)
            for (int s = P.citem_begin[q]; s < P.citem_end[q]; ++s) {
                const int kind = P.citem_kind[q];
                if (kind == CK_VERT) {
                    slots[s] += 1;
                    REQ(P.grp_agg[s / 32] == P.ctgt_i[t] && P.ctgt_i[t] == P.ctgt_j[t]);
                    continue;
                }
                const int e = P.seg_edge[s], I = P.grp_agg[P.edge_lo[e] / 32], J = P.grp_agg[P.edge_hi[e] / 32];
                if (kind == CK_INNER) REQ(I == J);
                if (kind == CK_INNER || kind == CK_CROSS) {
                    edges[e] += 1;
                    REQ(I == P.ctgt_i[t] && J == P.ctgt_j[t]);
                }
                if (kind == CK_LO) REQ(I == P.ctgt_i[t] && I != J);
                if (kind == CK_HI) REQ(J == P.ctgt_i[t] && I != J);
            }
    for (int n : slots) REQ(n == 1);
    for (int n : edges) REQ(n == 1);
    return 0;
}
