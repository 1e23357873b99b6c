// Host-side plan of the persistent CG solver (cg_pcg_kernel.cuh): how a mesh's
// vertices, edges and coarse aggregates are spread over the CTAs of one
// launch.  Plain C++, no CUDA.
//
// The operator of a CG solve is constant, so the solver applies it from the
// assembled off-diagonal blocks A_ij (one dim x dim block per mesh edge)
// instead of re-evaluating the elements:
//   (A p)_i = sum_j A_ij (p_j - p_i) + diagonal vertex terms,
// exact because the elastic energy does not change under translations.
//
// Vertices are cut into n_cta compact parts by recursive coordinate
// bisection; a part's vertices are the CTA's slots (local ids 0 .. nslot-1,
// in groups of 32 that belong to one aggregate each; a group's unused slots
// have gid -1), the vertices of other parts that its edges touch are its
// halo (local ids nslot ..).  An edge inside a part is stored once (two-sided:
// it adds to both ends), an edge between two parts once in each (one-sided:
// it adds to the part's own end).  A part's edges are coloured so that no
// two of one colour add to the same vertex: the vertex sums then need no
// atomics and have one fixed order.  A colour's edges are cut into chunks of
// at most kCgChunk entries, padded to a multiple of 4; in memory a chunk is
// [n] index words (target | source << 16, kCgPadEntry for padding) followed by
// dim*dim arrays of [n] values, so that one bulk copy moves it.
//
// Parts of few vertices are stored by rows instead, each edge inside a part
// twice: tpr threads share a row and take its entries in turn, and the
// entries of 32 threads lie together, step by step (padding entries have a
// zero block and the row itself as source), so a pass reads shared memory
// without conflicts and needs no barrier.  A part is then two chunks: the
// first steps of all rows, which stay in shared memory, and the rest.  Entries
// are ordered so that a warp's sources mostly lie in distinct banks.
//
// Aggregates (coarse space: the rigid motions of each) are unions of
// contiguous slot ranges in part order: one or several per part on small
// meshes (always on a cluster), several parts per aggregate on large ones.
#pragma once

#include <cstdint>
#include <string>
#include <vector>

namespace softsim {

constexpr int kCgChunk = 480;
constexpr uint32_t kCgPadEntry = 0xffffffffu;
constexpr uint32_t kCgLastOfColour = 0x80000000u;
constexpr uint32_t kCgTransposed = 0x80000000u;
constexpr int kPcgMaxStages = 8;
constexpr int kPcgThreads = 512;          // threads of a CTA at most (128 registers each)
constexpr int kPcgStreamThreads = kPcgThreads - 32;  // beside the producer warp of a streamed slice
constexpr int kPcgSmem = 226 * 1024;     // shared memory of one CTA, static part included
constexpr int kPcgStatic = 12 * 1024;     // room for the kernels' static part when a slice is sized
// Words of a CTA in a grid's exchange: items from 0, two words a dot from kPcgDots; in
// memory a 128-byte line (80 bytes, sharing lines: 0.2 to 1.1 us an iteration more), in
// shared memory rows that spread over the banks.
constexpr int kPcgWords = 16, kPcgRow = 18, kPcgDots = 6;
constexpr int kCgMaxCoarse = 192;  // coarse unknowns (cg_assemble.cu inverts the coarse matrix in one CTA's registers)
constexpr int kCgCoarseItem = 1024;  // edges or slots per partial sum of the coarse matrix

// Partial sum of one block of the coarse matrix: which entries it covers and how they enter
enum CoarseKind { CK_INNER = 0, CK_CROSS = 1, CK_LO = 2, CK_HI = 3, CK_VERT = 4 };

// Shared-memory plan of the solver (byte offsets; the edge slice or ring starts at ring).
struct PcgSmem {
    size_t p, y, e, s, t, meta, halo, word, ring;
#ifdef __CUDACC__
    __host__ __device__
#endif
    PcgSmem(int dim, size_t elt, int ns, int max_halo, int items, int n_coarse, int n_meta, int grid_ctas)
    {
        p = 2 * kPcgMaxStages * 8;  // mbarriers first
        y = p + (size_t)(ns + max_halo) * dim * elt;
        e = y + (size_t)ns * dim * elt;
        e = (e + 15) / 16 * 16;
        s = e + (size_t)items * (dim == 3 ? 6 : 3) * n_coarse * 4;
        t = s + (size_t)n_coarse * 8;  // two buffers
        meta = t + (size_t)n_coarse * 4;
        halo = meta + (size_t)n_meta * 4;
        word = (halo + (size_t)max_halo * 4 + 7) / 8 * 8;
        ring = (word + (size_t)grid_ctas * kPcgRow * 4 + 127) / 128 * 128;
    }
};

// Whether a launch of n_cta CTAs that wait for one another may be made: one
// cluster when the device can hold at least one of its kind, else a grid of at
// most the CTAs that fit on its SMs together.
inline bool pcg_resident(bool cluster, int n_cta, int max_clusters, int per_sm, int sms)
{
    return cluster ? max_clusters >= 1 : n_cta <= (int64_t)per_sm * sms;
}

struct CgPlan {
    int dim = 0, n_cta = 0, n_agg = 0, n_modes = 0;
    int ns = 0;                        // slots per CTA (maximum over CTAs, a multiple of 32)
    int tpr = 0;                       // threads per row, 0: stored by colours
    int n_meta = 0;                    // words per CTA of row_step, or the largest chunk count
    std::vector<uint32_t> row_step;    // [n_cta][n_meta] first step of each 32 threads (+ 1 end), in either chunk (rows)
    int max_halo = 0, max_entries = 0, max_chunks = 0, max_items = 0;
    std::vector<int32_t> slot_gid;     // [n_cta * ns] vertex of a slot, -1: unused
    std::vector<int32_t> grp_agg;      // [n_cta * ns / 32] aggregate of a group of slots
    std::vector<int32_t> nslot;        // [n_cta]
    std::vector<int32_t> halo_ptr, halo_slot;   // [n_cta + 1], global slot (cta * ns + local) of a halo vertex
    std::vector<int32_t> item_ptr, item_agg;    // [n_cta + 1], aggregates of a CTA (restriction items)
    std::vector<int32_t> agg_item;     // [n_agg + 1] items of an aggregate (contiguous)
    std::vector<int32_t> agg_ref;      // [n_agg] a vertex of the aggregate (origin of its rotations)
    std::vector<int32_t> chunk_ptr;    // [n_cta + 1]
    std::vector<int32_t> chunk_ent;    // [n_chunks + 1] first entry of a chunk
    std::vector<uint32_t> chunk_n;     // [n_chunks] entries | kCgLastOfColour
    std::vector<uint32_t> ent_idx;     // [n_entries] target | source << 16
    std::vector<uint32_t> ent_edge;    // [n_entries] edge | kCgTransposed (kCgPadEntry: padding)
    int64_t n_edges = 0, n_contrib = 0;
    std::vector<int32_t> edge_lo, edge_hi;  // [n_edges] global slots, lo < hi; the block is A_lo,hi
    std::vector<int32_t> edge_ptr;     // [n_edges + 1] its element contributions
    std::vector<uint32_t> cpos;        // [ne_int][npair] contribution of an element's corner pair | kCgTransposed
    // coarse matrix: items sorted by target block (I, J), I <= J
    std::vector<int32_t> seg_edge;     // [n_edges] edges sorted by aggregate pair
    std::vector<int32_t> citem_kind, citem_begin, citem_end;
    std::vector<int32_t> ctgt_ptr, ctgt_i, ctgt_j;
    double length = 1.0;               // scale of the rotation modes
};

// Aggregates per CTA, at most `most`, for parts of v vertices: the slots of an
// aggregate are padded to a multiple of 32, so the largest number is taken that
// keeps to `threads` slots (one a thread) or wastes less than a fifth of the
// slots, else the least wasteful.
int aggregates_per_part(int64_t v, int most, int threads);

// Slots of a thread at most: x and r of a slot stay in its registers.
inline int pcg_max_vpt(int elt, bool rows) { return elt == 8 || rows ? 4 : 8; }

// Slots a thread of the kernel variant that serves `need` of them, 0 if there is
// none.  One CTA and clusters store by rows and, but for 2D FP32, never have more
// slots than threads; parts stored by colours have more than 600 vertices in 3D and
// more than 2,000 in 2D, which FP64 does not reach (pcg_sizes).
inline int pcg_variant(int dim, int elt, bool rows, bool grid, int need)
{
    const int few = rows ? 1 : dim == 3 ? 2 : 4;
    const int most = rows ? (grid || (dim == 2 && elt == 4) ? 4 : 1) : !grid || (dim == 2 && elt == 8) ? 0 : pcg_max_vpt(elt, false);
    if (need > most) return 0;
    if (need <= few) return few;
    return need <= 4 ? 4 : 8;
}

// Parts (CTAs), aggregates and storage of the persistent solver for a mesh of nv
// vertices; fits: a CTA's threads can hold its vertices (a part is streamed at
// the limit, by kPcgStreamThreads threads).
struct PcgSizes {
    int n_cta, n_agg;
    bool cluster, rows, fits;
};
PcgSizes pcg_sizes(int dim, int elt, int64_t nv, int n_sm);

// The batched solver: dynamic shared memory of the plan's layout (the body's
// plan record lies behind it), and vertices of a body per thread at most.
constexpr int kBatchPlanAt = kPcgSmem - kPcgStatic;
constexpr int kBatchVpt = 8;

// Whether a body's plan (FP32, by rows) fits the batched kernel with that many
// threads: its slots, its aggregates, and below the plan record the edge slice
// and, in the same place, the scratch the coarse matrix is inverted in.
bool batch_plan_fits(const CgPlan &P, int threads);

// rows: store the parts by rows; elt: bytes of a value of the solver; on_grid: the
// CTAs are not one cluster.  perm: tile order -> caller order (-1 padding), ne_int entries; max_entries of any CTA
// and halo sizes are left to the caller to check against shared memory.  Returns false
// (with a reason) for meshes the layout cannot hold.
bool build_cg_plan(int dim, int64_t nv, int64_t ne, const double *X, const int32_t *T, const int32_t *perm,
                   int64_t ne_int, int n_cta, int n_agg, bool rows, int elt, bool on_grid, CgPlan &out, std::string &err);

}  // namespace softsim
