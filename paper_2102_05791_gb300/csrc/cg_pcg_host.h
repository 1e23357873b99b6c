// Host side of a persistent CG plan: its sizes, and the placement of its
// tables and work buffers in one device allocation each (of one mesh, or of
// all meshes of a batch).
#pragma once

#include <cstring>

#include "cg_pcg.h"

namespace softsim {

inline void pcg_sizes_of(const CgPlan &P, bool cluster, bool has_diag, PcgDev &pd)
{
    pd.n_cta = P.n_cta;
    pd.n_agg = P.n_agg;
    pd.n_modes = P.n_modes;
    pd.n_coarse = P.n_agg * P.n_modes;
    pd.ns = P.ns;
    pd.max_halo = P.max_halo;
    pd.max_entries = P.max_entries;
    pd.max_chunks = P.max_chunks;
    pd.tpr = P.tpr;
    pd.n_meta = P.n_meta;
    pd.max_items = P.max_items;
    pd.n_items = (int)P.item_agg.size();
    pd.cluster = cluster ? 1 : 0;
    pd.has_diag = has_diag ? 1 : 0;
    pd.n_edges = P.n_edges;
    pd.n_contrib = P.n_contrib;
    pd.n_entries = (int64_t)P.ent_idx.size();
    pd.n_chunks = (int64_t)P.chunk_n.size();
    pd.inv_len = (float)(1.0 / P.length);
    pd.n_citems = (int)P.citem_kind.size();
    pd.n_ctgts = (int)P.ctgt_i.size();
}

// Places the plan's tables from byte `at` on and returns the end; with host and
// dev it also copies them to host and sets pd's pointers into dev (else it only
// measures).
inline size_t pcg_place_tables(const CgPlan &P, PcgDev &pd, unsigned char *host, unsigned char *dev, size_t at)
{
    auto put = [&](const auto &v, auto **dst) {
        const size_t bytes = v.size() * sizeof(v[0]);
        if (host) {
            if (bytes) memcpy(host + at, v.data(), bytes);
            *dst = reinterpret_cast<decltype(&v[0])>(dev + at);
        }
        at += (bytes + 255) / 256 * 256;
    };
    put(P.slot_gid, &pd.slot_gid);
    put(P.grp_agg, &pd.grp_agg);
    put(P.nslot, &pd.nslot);
    put(P.halo_ptr, &pd.halo_ptr);
    put(P.halo_slot, &pd.halo_slot);
    put(P.item_ptr, &pd.item_ptr);
    put(P.item_agg, &pd.item_agg);
    put(P.agg_item, &pd.agg_item);
    put(P.agg_ref, &pd.agg_ref);
    put(P.chunk_ptr, &pd.chunk_ptr);
    put(P.chunk_ent, &pd.chunk_ent);
    put(P.chunk_n, &pd.chunk_n);
    put(P.row_step, &pd.row_step);
    put(P.ent_idx, &pd.ent_idx);
    put(P.ent_edge, &pd.ent_edge);
    put(P.cpos, &pd.cpos);
    put(P.edge_lo, &pd.edge_lo);
    put(P.edge_hi, &pd.edge_hi);
    put(P.edge_ptr, &pd.edge_ptr);
    put(P.seg_edge, &pd.seg_edge);
    put(P.citem_kind, &pd.citem_kind);
    put(P.citem_begin, &pd.citem_begin);
    put(P.citem_end, &pd.citem_end);
    put(P.ctgt_ptr, &pd.ctgt_ptr);
    put(P.ctgt_i, &pd.ctgt_i);
    put(P.ctgt_j, &pd.ctgt_j);
    return at;
}

// The same for the work buffers of a solve in precision T.
template <typename T>
size_t pcg_place_buffers(const CgPlan &P, PcgDev &pd, unsigned char *dev, size_t at)
{
    const size_t dd = (size_t)P.dim * P.dim, slots = (size_t)P.n_cta * P.ns, N = pd.n_coarse;
    auto put = [&](size_t bytes, auto **dst) {
        if (dev) {
            void *p = dev + at;
            memcpy(dst, &p, sizeof(p));
        }
        at += (bytes + 255) / 256 * 256;
    };
    put(sizeof(T) * dd * P.n_contrib, &pd.contrib);
    put(sizeof(T) * dd * P.n_edges, &pd.blk);
    put((4 + sizeof(T) * dd) * P.ent_idx.size(), &pd.slices);
    put(sizeof(float4) * slots, &pd.pos4);
    put(sizeof(T) * 2 * slots, &pd.diag2);
    put(sizeof(T) * (P.dim == 3 ? 6 : 3) * slots, &pd.dinv);
    put(sizeof(T) * 4 * slots, &pd.zr);
    put(sizeof(float) * 36 * pd.n_citems, &pd.cpart);
    put(sizeof(float) * N * N, &pd.E);
    put(sizeof(float) * N * N, &pd.Einv);
    put(8 * 2 * kPcgWords * P.n_cta, &pd.words);
    return at;
}

}  // namespace softsim
