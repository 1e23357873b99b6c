// Plan of the persistent CG solver (see cg_plan.h).
#include "cg_plan.h"

#include <algorithm>
#include <array>
#include <cmath>
#include <numeric>

#include "host_parallel.h"

namespace softsim {

// Recursive coordinate bisection: orders ids so that unit k, of weight
// w[k + 1] - w[k], is ids[cut[first + k]] .. ids[cut[first + k + 1]) with its
// share of the n ids; the longest axis is cut at the quantile of half the units.
static void bisect(int dim, const double *X, int32_t *ids, int64_t n, const int *w, int n_units, int64_t base,
                   int64_t *cut, int depth)
{
    if (n_units == 1) {
        cut[0] = base;
        return;
    }
    double lo[3], hi[3];
    for (int c = 0; c < dim; ++c) lo[c] = INFINITY, hi[c] = -INFINITY;
    for (int64_t i = 0; i < n; ++i)
        for (int c = 0; c < dim; ++c) {
            const double v = X[(int64_t)ids[i] * dim + c];
            lo[c] = std::min(lo[c], v);
            hi[c] = std::max(hi[c], v);
        }
    int ax = 0;
    for (int c = 1; c < dim; ++c)
        if (hi[c] - lo[c] > hi[ax] - lo[ax]) ax = c;
    const int left = n_units / 2;
    const int64_t m = n * (w[left] - w[0]) / (w[n_units] - w[0]);
    std::nth_element(ids, ids + m, ids + n, [&](int32_t a, int32_t b) {
        const double xa = X[(int64_t)a * dim + ax], xb = X[(int64_t)b * dim + ax];
        return xa != xb ? xa < xb : a < b;
    });
    std::thread t;
    if (depth > 0 && n > 20000) {
        try {
            t = std::thread([&]() { bisect(dim, X, ids, m, w, left, base, cut, depth - 1); });
        } catch (...) {  // no thread, or no memory to start one: this thread does both halves
        }
    }
    const bool both = !t.joinable();
    if (both) bisect(dim, X, ids, m, w, left, base, cut, 0);
    bisect(dim, X, ids + m, n - m, w + left, n_units - left, base + m, cut + left, both ? 0 : depth - 1);
    if (!both) t.join();
}

// Position along a Morton curve through the box lo .. lo + ext (10 bits an axis).
static uint32_t morton(int dim, const double *x, const double *lo, double inv)
{
    uint32_t q[3] = {0, 0, 0}, code = 0;
    for (int c = 0; c < dim; ++c) q[c] = (uint32_t)std::min(1023.0, std::max(0.0, (x[c] - lo[c]) * inv));
    for (int b = 9; b >= 0; --b)
        for (int c = dim - 1; c >= 0; --c) code = code << 1 | (q[c] >> b & 1);
    return code;
}

// Orders a colour's entries so that in each group of 32 (a warp) the targets
// lie in distinct shared-memory banks and, as far as a short search finds
// them, the sources too.
template <typename E>
static void bank_groups(E *e, int n)
{
    std::vector<E> by[32];
    for (int q = 0; q < n; ++q) by[e[q].tgt & 31].push_back(e[q]);
    size_t at[32] = {0};
    for (int out = 0; out < n;) {
        uint32_t used = 0;
        const int end = std::min(n, out + 32);
        for (int round = 0; out < end; ++round) {
            bool any = false;
            for (int t = 0; t < 32 && out < end; ++t) {
                if (at[t] >= by[t].size()) continue;
                size_t pick = at[t];
                const size_t lim = std::min(by[t].size(), at[t] + 24);
                while (pick < lim && (used >> (by[t][pick].src & 31) & 1u)) ++pick;
                if (pick == lim) {
                    if (round == 0) continue;
                    pick = at[t];
                }
                used |= 1u << (by[t][pick].src & 31);
                e[out++] = by[t][pick];
                std::swap(by[t][pick], by[t][at[t]]);
                ++at[t];
                any = true;
            }
            if (!any && round > 0) break;
        }
    }
}

namespace {
struct CtaBuild {
    std::vector<int32_t> halo;                    // global slots
    std::vector<uint32_t> idx, edge;              // entries in chunk order, padded
    std::vector<int32_t> n_chunk;                 // padded entries per chunk
    std::vector<uint32_t> chunk_n;
    std::vector<int> steps;                       // rows: steps of each 32 threads, idx and edge in that order
    std::vector<uint32_t> step;                   // rows: first step of each 32 threads in either chunk
    bool ok = true;
};
}  // namespace

int aggregates_per_part(int64_t v, int most, int threads)
{
    int best = 1;
    int64_t best_slots = INT64_MAX;
    for (int a = std::max(1, most); a >= 1; --a) {
        const int64_t slots = a * (((v + a - 1) / a + 31) / 32 * 32);
        if (slots <= threads || slots * 5 <= v * 6) return a;
        if (slots < best_slots) {
            best_slots = slots;
            best = a;
        }
    }
    return best;
}

// Parts (CTAs), aggregates and storage of the persistent CG solver for a mesh
// of nv vertices.  The lines lie where both sides measured alike (microseconds
// an iteration on GB300): one cluster exchanges in about 1 us, a grid in about
// 2 us, so a cluster's 16 CTAs serve as long as their rows stay in shared
// memory (3D FP32: 4.7 us at 1,260 vertices; 7.9 on a grid of 64 at 9,537, where
// 16 CTAs need 18; 2D: 7.2 at 20,000).  FP64 arithmetic is scarce, so FP64
// spreads over more CTAs earlier (16.0 us on 64 CTAs against 18.8 on 16 at 2,640
// vertices).  More aggregates save iterations but cost a larger inverse (192
// coarse unknowns: 0.12 ms, 96: 0.02 ms), which small meshes do not win back.
// Rows beat colours until the part's rows no longer stay in L2 (3D FP32: 23.4
// against 22.9 us at 122,000 vertices, 42.8 against 30.9 at 180,000).  (Figures of
// the solver with plain FP32 dots; compensated it takes 4.2 us at 1,260 vertices,
// 7.4 at 9,537, FP64 13.5 on 64 CTAs.)
PcgSizes pcg_sizes(int dim, int elt, int64_t nv, int n_sm)
{
    const bool f32 = elt == 4;
    const int nm = dim == 3 ? 6 : 3;
    const int64_t per_cta = dim == 3 ? (f32 ? 270 : 100) : (f32 ? 1300 : 256);  // the most a cluster's CTA takes
    int64_t g, a = std::max<int64_t>(1, std::min<int64_t>((nv <= 4096 ? kCgMaxCoarse / 2 : kCgMaxCoarse) / nm, nv / 18));
    if (nv <= 16 * per_cta) {
        g = f32 && nv <= 160 ? 1 : std::min<int64_t>(16, (nv + 31) / 32);
        a = std::min(a, 16 * g);
    } else {
        g = std::min<int64_t>(n_sm, std::max<int64_t>(kCgMaxCoarse / nm, nv / (dim == 3 ? (f32 ? 150 : 40) : 256)));
        a = std::min(a, g);
    }
    const int64_t per = (nv + g - 1) / g;
    if (a > g) a = g * aggregates_per_part(per, (int)(a / g), 512);
    const bool rows = per <= (dim == 3 ? (f32 ? 750 : 600) : 2000);
    return {(int)g, (int)a, g > 1 && g <= 16, rows, per <= (int64_t)pcg_max_vpt(elt, rows) * kPcgStreamThreads};
}

bool batch_plan_fits(const CgPlan &P, int threads)
{
    const size_t N = (size_t)P.n_agg * P.n_modes, esz = 4 + (size_t)P.dim * P.dim * sizeof(float);
    const PcgSmem L(P.dim, sizeof(float), P.ns, P.max_halo, P.max_items, (int)N, P.n_meta, 0);
    return P.ns <= kBatchVpt * threads && P.max_items <= 16 && N <= (size_t)kCgMaxCoarse &&
           L.ring + sizeof(float) * (N * N + 3 * N) <= (size_t)kBatchPlanAt &&
           L.ring + (size_t)P.max_entries * esz <= (size_t)kBatchPlanAt;
}

bool build_cg_plan(int dim, int64_t nv, int64_t ne, const double *X, const int32_t *T, const int32_t *perm,
                   int64_t ne_int, int n_cta, int n_agg, bool rows, int elt, bool on_grid, CgPlan &P, std::string &err)
{
    P = CgPlan();
    P.dim = dim;
    P.n_cta = n_cta;
    P.n_modes = dim == 3 ? 6 : 3;
    const int nc = dim + 1, np = nc * (nc - 1) / 2;
    // a cluster's CTAs write their items into each other's shared memory instead
    // of summing them: every aggregate lies in one CTA there
    if (!on_grid) n_agg = std::max(n_agg, n_cta);
    const int per = n_agg >= n_cta ? n_agg / n_cta : 1;  // aggregates per CTA
    n_agg = n_agg >= n_cta ? per * n_cta : n_agg;
    P.n_agg = n_agg;
    const int n_parts = n_cta * per;
    if (nv < n_parts || n_agg < 1) {
        err = "fewer vertices than parts";
        return false;
    }
    if (ne > INT32_MAX / nc) {  // the incidences are counted in 32 bits
        err = "too many elements";
        return false;
    }

    // --- parts and slots
    std::vector<int32_t> ids(nv);
    std::iota(ids.begin(), ids.end(), 0);
    std::vector<int64_t> cut(n_parts + 1, 0);
    {
        // the coarser level first (aggregates of one or more CTAs, or CTAs of one or
        // more aggregates), so that both are compact
        const int n_top = per > 1 ? n_cta : n_agg;
        std::vector<int> w(n_top + 1), one(n_parts + 1);
        for (int k = 0; k <= n_top; ++k) w[k] = (int)((int64_t)k * n_parts / n_top);
        std::iota(one.begin(), one.end(), 0);
        std::vector<int64_t> top(n_top + 1, nv);
        bisect(dim, X, ids.data(), nv, w.data(), n_top, 0, top.data(), 4);
        parallel_for(nv, n_top, 1, [&](int64_t k) {
            bisect(dim, X, ids.data() + top[k], top[k + 1] - top[k], one.data() + w[k], w[k + 1] - w[k], top[k],
                   cut.data() + w[k], 0);
        });
        cut[n_parts] = nv;
    }
    double lo[3], hi[3];
    for (int c = 0; c < dim; ++c) lo[c] = INFINITY, hi[c] = -INFINITY;
    for (int64_t i = 0; i < nv; ++i)
        for (int c = 0; c < dim; ++c) {
            lo[c] = std::min(lo[c], X[i * dim + c]);
            hi[c] = std::max(hi[c], X[i * dim + c]);
        }
    double ext = 0.0, vol = 1.0;
    for (int c = 0; c < dim; ++c) {
        ext = std::max(ext, hi[c] - lo[c]);
        vol *= std::max(hi[c] - lo[c], 1e-300);
    }
    P.length = std::pow(vol / n_agg, 1.0 / dim);
    if (!(P.length > 0.0) || !std::isfinite(P.length) || !(ext > 0.0)) {
        err = "degenerate extent";
        return false;
    }
    std::vector<uint32_t> code(nv);
    parallel_for(nv, nv, 4096, [&](int64_t v) { code[v] = morton(dim, X + v * dim, lo, 1023.0 / ext); });
    parallel_for(nv, n_parts, 1, [&](int64_t p) {
        std::sort(ids.begin() + cut[p], ids.begin() + cut[p + 1], [&](int32_t a, int32_t b) {
            return code[a] != code[b] ? code[a] < code[b] : a < b;
        });
    });
    P.nslot.resize(n_cta);
    auto up32 = [](int64_t v) { return (int)((v + 31) / 32 * 32); };
    for (int c = 0; c < n_cta; ++c) {
        int s = 0;
        for (int a = 0; a < per; ++a) s += up32(cut[c * per + a + 1] - cut[c * per + a]);
        P.nslot[c] = s;
        P.ns = std::max(P.ns, s);
    }
    const int ns = P.ns;
    if (ns > 32767) {
        err = "too many vertices per CTA";
        return false;
    }
    P.slot_gid.assign((size_t)n_cta * ns, -1);
    P.grp_agg.assign((size_t)n_cta * ns / 32, 0);
    P.agg_ref.assign(n_agg, -1);
    std::vector<int32_t> slot_of(nv);
    P.item_ptr.push_back(0);
    for (int c = 0; c < n_cta; ++c) {
        int s = 0;
        int last_agg = (c + 1) * per - 1;
        if (per == 1) {  // the aggregate k whose parts k n_cta / n_agg .. hold part c
            last_agg = (int)((int64_t)c * n_agg / n_cta);
            while ((int64_t)(last_agg + 1) * n_cta / n_agg <= c) ++last_agg;
        }
        for (int g = 0; g < ns / 32; ++g) P.grp_agg[(size_t)c * ns / 32 + g] = last_agg;
        for (int a = 0; a < per; ++a) {
            const int part = c * per + a, agg = per > 1 ? part : last_agg;
            P.item_agg.push_back(agg);
            for (int64_t k = cut[part]; k < cut[part + 1]; ++k) {
                const int32_t slot = c * ns + s + (int32_t)(k - cut[part]);
                P.slot_gid[slot] = ids[k];
                slot_of[ids[k]] = slot;
                P.grp_agg[slot / 32] = agg;
                if (P.agg_ref[agg] < 0) P.agg_ref[agg] = ids[k];
            }
            s += up32(cut[part + 1] - cut[part]);
        }
        P.item_ptr.push_back((int32_t)P.item_agg.size());
        P.max_items = std::max(P.max_items, per);
    }
    P.agg_item.assign(n_agg + 1, 0);
    for (int32_t a : P.item_agg) P.agg_item[a + 1] += 1;
    for (int a = 0; a < n_agg; ++a) {
        if (P.agg_item[a + 1] == 0 || P.agg_ref[a] < 0) {
            err = "empty aggregate";
            return false;
        }
        P.agg_item[a + 1] += P.agg_item[a];
    }

    // --- edges: of every vertex, its neighbours in later slots
    std::vector<int32_t> vptr(nv + 1, 0);
    for (int64_t i = 0; i < ne * nc; ++i) vptr[T[i] + 1] += 1;
    for (int64_t v = 0; v < nv; ++v) vptr[v + 1] += vptr[v];
    std::vector<int32_t> velem((size_t)ne * nc);
    {
        std::vector<int32_t> fill(vptr.begin(), vptr.end() - 1);
        for (int64_t e = 0; e < ne; ++e)
            for (int k = 0; k < nc; ++k) velem[fill[T[e * nc + k]]++] = (int32_t)e;
    }
    // edges in slot order of their lower end: neighbours with their counts, offsets, then the tables
    std::vector<int32_t> ecount(nv, 0), ccount(nv, 0);  // edges and contributions that start at a vertex
    std::vector<int32_t> nbr((size_t)ne * nc * dim), ncnt((size_t)ne * nc * dim);  // vertex v's from vptr[v] * dim
    parallel_for(nv, nv, 1024, [&](int64_t v) {
        int32_t *nb = nbr.data() + (size_t)vptr[v] * dim, *cn = ncnt.data() + (size_t)vptr[v] * dim;
        const int32_t sv = slot_of[v];
        int n = 0, m = 0;
        for (int32_t q = vptr[v]; q < vptr[v + 1]; ++q) {
            const int32_t *t = T + (int64_t)velem[q] * nc;
            for (int k = 0; k < nc; ++k)
                if (slot_of[t[k]] > sv) nb[n++] = slot_of[t[k]];
        }
        ccount[v] = n;
        std::sort(nb, nb + n);
        for (int q = 0; q < n; ++q) {
            if (m == 0 || nb[q] != nb[m - 1]) {
                nb[m] = nb[q];
                cn[m++] = 0;
            }
            cn[m - 1] += 1;
        }
        ecount[v] = m;
    });
    std::vector<int32_t> eoff(nv), coff(nv);
    {
        int64_t en = 0, cn = 0;
        for (size_t s = 0; s < P.slot_gid.size(); ++s) {
            const int32_t v = P.slot_gid[s];
            if (v < 0) continue;
            eoff[v] = (int32_t)en;
            coff[v] = (int32_t)cn;
            en += ecount[v];
            cn += ccount[v];
        }
        if (cn > (int64_t)kCgTransposed - 2 || cn > INT32_MAX) {
            err = "too many edge contributions";
            return false;
        }
        P.n_edges = en;
        P.n_contrib = cn;
    }
    P.edge_lo.resize(P.n_edges);
    P.edge_hi.resize(P.n_edges);
    P.edge_ptr.resize(P.n_edges + 1);
    P.edge_ptr[P.n_edges] = (int32_t)P.n_contrib;
    std::vector<int32_t> inv(ne, -1);  // caller order -> tile order
    for (int64_t i = 0; i < ne_int; ++i)
        if (perm[i] >= 0) inv[perm[i]] = (int32_t)i;
    P.cpos.assign((size_t)ne_int * np, kCgPadEntry);
    parallel_for(nv, nv, 1024, [&](int64_t v) {
        const int32_t *nb = nbr.data() + (size_t)vptr[v] * dim;
        int32_t *cnt = ncnt.data() + (size_t)vptr[v] * dim;
        const int32_t sv = slot_of[v], m = ecount[v];
        int32_t at = coff[v];
        for (int32_t q = 0; q < m; ++q) {
            const int32_t e = eoff[v] + q;
            P.edge_lo[e] = sv;
            P.edge_hi[e] = nb[q];
            P.edge_ptr[e] = at;
            const int32_t c = cnt[q];
            cnt[q] = at;
            at += c;
        }
        for (int32_t q = vptr[v]; q < vptr[v + 1]; ++q) {
            const int32_t el = velem[q];
            const int32_t *t = T + (int64_t)el * nc;
            int pair = 0;
            for (int a = 0; a < nc; ++a)
                for (int b = a + 1; b < nc; ++b, ++pair) {
                    const int32_t sa = slot_of[t[a]], sb = slot_of[t[b]];
                    if (std::min(sa, sb) != sv) continue;
                    const size_t k = std::lower_bound(nb, nb + m, std::max(sa, sb)) - nb;
                    P.cpos[(size_t)inv[el] * np + pair] = (uint32_t)cnt[k]++ | (sa < sb ? 0u : kCgTransposed);
                }
        }
    });

    // --- entries of every CTA: its own edges, and the edges of others that end in it
    std::vector<int32_t> first_edge(n_cta + 1, 0);  // edges by the CTA of their lower end
    for (int64_t e = 0; e < P.n_edges; ++e) first_edge[P.edge_lo[e] / ns + 1] += 1;
    for (int c = 0; c < n_cta; ++c) first_edge[c + 1] += first_edge[c];
    std::vector<int32_t> in_ptr(n_cta + 1, 0), in_edge;
    for (int64_t e = 0; e < P.n_edges; ++e)
        if (P.edge_hi[e] / ns != P.edge_lo[e] / ns) in_ptr[P.edge_hi[e] / ns + 1] += 1;
    for (int c = 0; c < n_cta; ++c) in_ptr[c + 1] += in_ptr[c];
    in_edge.resize(in_ptr[n_cta]);
    {
        std::vector<int32_t> fill(in_ptr.begin(), in_ptr.end() - 1);
        for (int64_t e = 0; e < P.n_edges; ++e)
            if (P.edge_hi[e] / ns != P.edge_lo[e] / ns) in_edge[fill[P.edge_hi[e] / ns]++] = (int32_t)e;
    }
    if (rows)
        for (P.tpr = 8; P.tpr > 1 && P.tpr * ns > 512;) P.tpr >>= 1;
    std::vector<CtaBuild> cb(n_cta);
    parallel_for(nv, n_cta, 1, [&](int64_t c) {
        CtaBuild &B = cb[c];
        const int32_t s0 = (int32_t)c * ns;
        struct Ent {
            int32_t tgt, src;
            uint32_t edge;
            int colour;
        };
        std::vector<Ent> ent;
        ent.reserve(first_edge[c + 1] - first_edge[c] + in_ptr[c + 1] - in_ptr[c]);
        for (int32_t e = first_edge[c]; e < first_edge[c + 1]; ++e) ent.push_back({P.edge_lo[e], P.edge_hi[e], (uint32_t)e, 0});
        for (int32_t q = in_ptr[c]; q < in_ptr[c + 1]; ++q) {
            const int32_t e = in_edge[q];
            ent.push_back({P.edge_hi[e], P.edge_lo[e], (uint32_t)e | kCgTransposed, 0});
        }
        for (const Ent &t : ent)
            if (t.src / ns != c) B.halo.push_back(t.src);
        std::sort(B.halo.begin(), B.halo.end());
        B.halo.erase(std::unique(B.halo.begin(), B.halo.end()), B.halo.end());
        if (P.nslot[c] + (int64_t)B.halo.size() > 65534) {
            B.ok = false;
            return;
        }
        if (rows) {
            // every row's entries, in edge order; padding points at the row itself
            struct Src {
                int32_t j;
                uint32_t edge;
            };
            const int n_row = P.nslot[c];
            std::vector<int32_t> ptr(n_row + 1, 0), src(ent.size());
            for (size_t q = 0; q < ent.size(); ++q) {
                const Ent &t = ent[q];
                const bool two = t.src / ns == c;
                src[q] = two ? t.src - s0
                             : n_row + (int32_t)(std::lower_bound(B.halo.begin(), B.halo.end(), t.src) - B.halo.begin());
                ptr[t.tgt - s0 + 1] += 1;
                if (two) ptr[src[q] + 1] += 1;
            }
            for (int r = 0; r < n_row; ++r) ptr[r + 1] += ptr[r];
            std::vector<Src> row(ptr[n_row]);
            std::vector<int32_t> end(ptr.begin(), ptr.end() - 1);  // fill position, then the row's last entry left
            for (size_t q = 0; q < ent.size(); ++q) {
                const int32_t i = ent[q].tgt - s0;
                row[end[i]++] = {src[q], ent[q].edge};
                if (src[q] < n_row) row[end[src[q]]++] = {i, ent[q].edge ^ kCgTransposed};
            }
            const int tpr = P.tpr, per_warp = 32 / tpr;
            for (int r0 = 0; r0 < n_row; r0 += per_warp) {
                int steps = 0;
                for (int r = r0; r < r0 + per_warp; ++r) steps = std::max(steps, (ptr[r + 1] - ptr[r] + tpr - 1) / tpr);
                for (int s = 0; s < steps; ++s) {
                    uint32_t banks = 0;
                    for (int l = 0; l < 32; ++l) {
                        // an entry left of the row whose source lies in a bank not used in this step
                        const int r = r0 + l / tpr;
                        int q = ptr[r];
                        while (q < end[r] && (banks >> (row[q].j & 31) & 1u)) ++q;
                        if (q == end[r]) q = ptr[r];
                        if (end[r] == ptr[r]) {
                            B.idx.push_back((uint32_t)r | (uint32_t)r << 16);
                            B.edge.push_back(kCgPadEntry);
                        } else {
                            banks |= 1u << (row[q].j & 31);
                            B.idx.push_back((uint32_t)r | (uint32_t)row[q].j << 16);
                            B.edge.push_back(row[q].edge);
                            row[q] = row[--end[r]];
                        }
                    }
                }
                B.steps.push_back(steps);
            }
            return;
        }
        // greedy colouring: the smallest colour free at both ends (128 colours)
        std::vector<std::array<uint64_t, 2>> used(P.nslot[c], std::array<uint64_t, 2>{0, 0});
        int n_col = 0;
        std::vector<int32_t> count(128, 0);
        for (Ent &t : ent) {
            const bool two = t.src / ns == c;
            t.tgt -= s0;
            t.src = two ? t.src - s0
                        : P.nslot[c] + (int32_t)(std::lower_bound(B.halo.begin(), B.halo.end(), t.src) - B.halo.begin());
            uint64_t m0 = used[t.tgt][0], m1 = used[t.tgt][1];
            if (two) m0 |= used[t.src][0], m1 |= used[t.src][1];
            int k = ~m0 ? __builtin_ctzll(~m0) : (~m1 ? 64 + __builtin_ctzll(~m1) : -1);
            if (k < 0) {
                B.ok = false;
                return;
            }
            used[t.tgt][k >> 6] |= 1ull << (k & 63);
            if (two) used[t.src][k >> 6] |= 1ull << (k & 63);
            t.colour = k;
            count[k] += 1;
            n_col = std::max(n_col, k + 1);
        }
        std::vector<int32_t> at(n_col + 1, 0);
        for (int k = 0; k < n_col; ++k) at[k + 1] = at[k] + count[k];
        std::vector<Ent> sorted(ent.size());
        {
            std::vector<int32_t> fill(at.begin(), at.end() - 1);
            for (const Ent &t : ent) sorted[fill[t.colour]++] = t;
        }
        for (int k = 0; k < n_col; ++k) {
            bank_groups(sorted.data() + at[k], at[k + 1] - at[k]);
            for (int32_t b = at[k]; b < at[k + 1]; b += kCgChunk) {
                const int n = std::min(kCgChunk, at[k + 1] - b), n4 = (n + 3) / 4 * 4;
                for (int q = 0; q < n4; ++q) {
                    const bool pad = q >= n;
                    B.idx.push_back(pad ? kCgPadEntry : (uint32_t)sorted[b + q].tgt | (uint32_t)sorted[b + q].src << 16);
                    B.edge.push_back(pad ? kCgPadEntry : sorted[b + q].edge);
                }
                B.n_chunk.push_back(n4);
                B.chunk_n.push_back((uint32_t)n4 | (b + kCgChunk >= at[k + 1] ? kCgLastOfColour : 0u));
            }
        }
    });
    if (rows) {
        // the steps that fit in shared memory, the same number for every 32 threads
        int max_steps = 0, max_vw = 0;
        for (const CtaBuild &B : cb) {
            P.max_halo = std::max(P.max_halo, (int)B.halo.size());
            max_vw = std::max(max_vw, (int)B.steps.size());
            for (int s : B.steps) max_steps = std::max(max_steps, s);
        }
        P.n_meta = 2 * (max_vw + 1);
        const PcgSmem L(dim, elt, ns, P.max_halo, P.max_items, n_agg * P.n_modes, P.n_meta, on_grid ? n_cta : 0);
        const size_t room = kPcgSmem - kPcgStatic, esz = 4 + (size_t)dim * dim * elt;
        const int keep = L.ring >= room ? 0 : (int)std::min<size_t>(max_steps, (room - L.ring) / (esz * 32 * max_vw));
        if (keep == 0) {
            err = "a CTA's vectors do not fit in shared memory";
            return false;
        }
        parallel_for(nv, n_cta, 1, [&](int64_t c) {
            CtaBuild &B = cb[c];
            std::vector<uint32_t> idx, edge;
            for (int part = 0; part < 2; ++part) {
                const size_t n0 = idx.size();
                size_t at = 0;
                for (int steps : B.steps) {
                    B.step.push_back((uint32_t)((idx.size() - n0) / 32));
                    const size_t b = at + (size_t)(part ? std::min(keep, steps) : 0) * 32;
                    const size_t e = at + (size_t)(part ? steps : std::min(keep, steps)) * 32;
                    idx.insert(idx.end(), B.idx.begin() + b, B.idx.begin() + e);
                    edge.insert(edge.end(), B.edge.begin() + b, B.edge.begin() + e);
                    at += (size_t)steps * 32;
                }
                B.step.push_back((uint32_t)((idx.size() - n0) / 32));
                B.n_chunk.push_back((int32_t)(idx.size() - n0));
                B.chunk_n.push_back((uint32_t)(idx.size() - n0));
            }
            B.idx.swap(idx);
            B.edge.swap(edge);
        });
    }
    P.halo_ptr.push_back(0);
    P.chunk_ptr.push_back(0);
    P.chunk_ent.push_back(0);
    for (int c = 0; c < n_cta; ++c) {
        const CtaBuild &B = cb[c];
        if (!B.ok) {
            err = "a CTA's part does not fit the edge layout";
            return false;
        }
        P.halo_slot.insert(P.halo_slot.end(), B.halo.begin(), B.halo.end());
        P.halo_ptr.push_back((int32_t)P.halo_slot.size());
        for (size_t k = 0; k < B.n_chunk.size(); ++k) {
            P.chunk_ent.push_back(P.chunk_ent.back() + B.n_chunk[k]);
            P.chunk_n.push_back(B.chunk_n[k]);
        }
        P.chunk_ptr.push_back((int32_t)P.chunk_n.size());
        P.ent_idx.insert(P.ent_idx.end(), B.idx.begin(), B.idx.end());
        P.ent_edge.insert(P.ent_edge.end(), B.edge.begin(), B.edge.end());
        P.max_halo = std::max(P.max_halo, (int)B.halo.size());
        P.max_entries = std::max(P.max_entries, rows ? B.n_chunk[0] : (int)B.idx.size());
        P.max_chunks = std::max(P.max_chunks, (int)B.n_chunk.size());
    }
    if (rows) {
        for (int c = 0; c < n_cta; ++c) {
            P.row_step.insert(P.row_step.end(), cb[c].step.begin(), cb[c].step.end());
            P.row_step.resize((size_t)(c + 1) * P.n_meta, 0);
        }
    } else {
        P.n_meta = P.max_chunks;
    }

    // --- coarse matrix: edges by aggregate pair, cut into items of bounded size
    auto agg_of = [&](int32_t slot) { return P.grp_agg[slot / 32]; };
    std::vector<int32_t> key_ptr((size_t)n_agg * n_agg + 1, 0);
    for (int64_t e = 0; e < P.n_edges; ++e) key_ptr[(size_t)agg_of(P.edge_lo[e]) * n_agg + agg_of(P.edge_hi[e]) + 1] += 1;
    for (size_t k = 0; k < (size_t)n_agg * n_agg; ++k) key_ptr[k + 1] += key_ptr[k];
    P.seg_edge.resize(P.n_edges);
    {
        std::vector<int32_t> fill(key_ptr.begin(), key_ptr.end() - 1);
        for (int64_t e = 0; e < P.n_edges; ++e)
            P.seg_edge[fill[(size_t)agg_of(P.edge_lo[e]) * n_agg + agg_of(P.edge_hi[e])]++] = (int32_t)e;
    }
    std::vector<std::vector<std::array<int32_t, 3>>> diag(n_agg);
    auto add = [&](std::vector<std::array<int32_t, 3>> &to, int kind, int b, int e) {
        for (int q = b; q < e; q += kCgCoarseItem) to.push_back({kind, q, std::min(e, q + kCgCoarseItem)});
    };
    std::vector<std::pair<std::pair<int, int>, std::vector<std::array<int32_t, 3>>>> cross;
    for (int i = 0; i < n_agg; ++i)
        for (int j = i; j < n_agg; ++j) {
            const int b = key_ptr[(size_t)i * n_agg + j], e = key_ptr[(size_t)i * n_agg + j + 1];
            if (b == e) continue;
            if (i == j) {
                add(diag[i], CK_INNER, b, e);
            } else {
                add(diag[i], CK_LO, b, e);
                add(diag[j], CK_HI, b, e);
                cross.push_back({{i, j}, {}});
                add(cross.back().second, CK_CROSS, b, e);
            }
        }
    for (size_t g = 0; g < P.grp_agg.size();) {  // runs of groups of one aggregate
        size_t g1 = g;
        while (g1 < P.grp_agg.size() && P.grp_agg[g1] == P.grp_agg[g]) ++g1;
        add(diag[P.grp_agg[g]], CK_VERT, (int)g * 32, (int)g1 * 32);
        g = g1;
    }
    P.ctgt_ptr.push_back(0);
    auto put = [&](int i, int j, const std::vector<std::array<int32_t, 3>> &items) {
        for (const auto &t : items) {
            P.citem_kind.push_back(t[0]);
            P.citem_begin.push_back(t[1]);
            P.citem_end.push_back(t[2]);
        }
        P.ctgt_i.push_back(i);
        P.ctgt_j.push_back(j);
        P.ctgt_ptr.push_back((int32_t)P.citem_kind.size());
    };
    for (int i = 0; i < n_agg; ++i) put(i, i, diag[i]);
    for (const auto &c : cross) put(c.first.first, c.first.second, c.second);
    return true;
}

}  // namespace softsim
