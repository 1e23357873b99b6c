// Device side of the persistent CG solver's plan (cg_plan.h) and its launchers.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "cg_plan.h"
#include "internal.h"

namespace softsim {

struct PcgDev {
    int n_cta = 0, n_agg = 0, n_modes = 0, n_coarse = 0;  // n_coarse = n_agg * n_modes
    int ns = 0, max_halo = 0, max_entries = 0, max_chunks = 0, max_items = 0, n_items = 0;
    int threads = 0;                 // consumer threads per CTA
    int vpt = 0;                     // slots per thread: 1, 2, 4 or 8
    int has_diag = 0;                // inertia, friction or contact: the vertex diagonal is not zero
    int tpr = 0;                     // threads per row of a slice stored by rows, 0: by colours
    int n_meta = 0;                  // words of a CTA's chunk sizes or row step offsets
    int stages = 0;                  // ring stages of a streamed edge slice, 0: the slice stays in shared memory
    int cluster = 0;                 // the grid is one thread-block cluster
    int64_t n_edges = 0, n_contrib = 0, n_entries = 0, n_chunks = 0;
    float inv_len = 1.0f;
    const int32_t *slot_gid = nullptr, *grp_agg = nullptr, *nslot = nullptr, *halo_ptr = nullptr, *halo_slot = nullptr,
                  *item_ptr = nullptr, *item_agg = nullptr, *agg_item = nullptr, *agg_ref = nullptr,
                  *chunk_ptr = nullptr, *chunk_ent = nullptr;
    const uint32_t *row_step = nullptr, *chunk_n = nullptr, *ent_idx = nullptr, *ent_edge = nullptr, *cpos = nullptr;
    const int32_t *edge_lo = nullptr, *edge_hi = nullptr, *edge_ptr = nullptr, *seg_edge = nullptr,
                  *citem_kind = nullptr, *citem_begin = nullptr, *citem_end = nullptr, *ctgt_ptr = nullptr,
                  *ctgt_i = nullptr, *ctgt_j = nullptr;
    int n_citems = 0, n_ctgts = 0;
    // per-solve data (T: the CG precision)
    void *contrib = nullptr;         // [n_contrib][D*D] element contributions to the edge blocks
    void *blk = nullptr;             // [D*D][n_edges] edge blocks
    unsigned char *slices = nullptr; // the CTAs' edge slices, chunk by chunk
    float4 *pos4 = nullptr;          // [n_cta*ns] rotation arm of a slot (scaled), aggregate | pinned << 30
    void *diag2 = nullptr;           // [n_cta*ns][2] vertex diagonal: horizontal axes, y
    void *dinv = nullptr;            // [6 or 3][n_cta*ns] inverse diagonal blocks
    void *zr = nullptr;              // [n_cta*ns][4 or 2] published z
    float *cpart = nullptr;          // [n_citems][36]
    float *E = nullptr, *Einv = nullptr;  // [n_coarse][n_coarse]
    unsigned long long *words = nullptr;          // [2][n_cta][kPcgWords] (value, tag) words of a grid's exchanges
};

// The edge blocks at displacement u, the vertex terms and the rotation arms (every CG solve's
// operator); with coarse also the coarse matrix and its inverse.  u64: the same displacement.
template <typename T>
void launch_pcg_assemble(const Ctx &c, const PcgDev &pd, const Phys &ph, const T *u, const double *u64, bool coarse,
                         cudaStream_t s);

// Shared memory of the solver and whether the slice is streamed: fills threads, vpt and stages;
// false when a CTA's vectors do not fit, or the device cannot hold all CTAs at once.
template <typename T>
bool pcg_configure(const Ctx &c, PcgDev &pd);

// Solves A d = sign * b (b in FP64, pinned entries ignored; d zero there) to |r| <= rtol |b| in one launch;
// sc->gn2 holds |b|^2; results in sc as from the per-iteration kernels.
template <typename T>
cudaError_t launch_pcg(const Ctx &c, const PcgDev &pd, const double *b, double sign, T *d, double rtol, int max_iter,
                       cudaStream_t s);

}  // namespace softsim
