// Preconditioned conjugate gradients of a whole solve in ONE launch, on the
// assembled edge blocks of its operator (layout: cg_plan.h; assembly:
// cg_assemble.cu).
//
// Operator.  A CG solve applies one constant operator many times.  Applying
// it from edge blocks moves 36 bytes and ~40 flops per mesh edge (3D FP32)
// where re-evaluating the elements moves 72 bytes and ~450 flops per tet,
// and there are about as many edges as tets: 4.1 M stored blocks (163 MB)
// against 246 MB per application on a 3.1 M-tet body.  The difference form
// A_ij (p_j - p_i) keeps the rounding error of smooth fields as small as the
// elements' edge differences do.
//
// Preconditioner.  z = D^-1 r + Z E^-1 Z^T r: inverse diagonal blocks plus a
// Galerkin coarse correction over the rigid motions of 16-64 aggregates
// (additive two-level Schwarz), symmetric positive definite and fixed during
// a solve (its coarse part in FP32 on FP64 handles too).  It cuts the iterations 2.5
// to 7 times (the more the larger the mesh; 1.2 times at 256 triangles).
//
// Each CTA owns one part of the vertices.  Its x and r stay in registers, p
// (with the halo's copy) and A p in shared memory.  Its edge slice is stored by
// rows and stays in shared memory for the whole solve as far as it fits (the
// last steps of the rows are read from L2), or, for large parts, by colours,
// each edge once, streamed every iteration by a producer warp through a ring of
// bulk copies that runs ahead across the barriers.  Two exchanges between the
// CTAs an iteration:
//   1. p = z + beta p at own and halo vertices (z as published); A p; p.Ap and
//      Z^T A p; exchange;
//   2. alpha; x, r; the coarse values of the CTA's own aggregates for the new
//      residual from E^-1 (Z^T r - alpha Z^T A p), so z is whole before the
//      exchange; z (published); r.r, r.z, the new Z^T r; exchange; beta and the
//      convergence test.
// The dots are formed from the vectors themselves, compensated pairs in FP32 and
// FP64 else, through threads, warps and CTAs up to the quotients alpha and
// beta: the first step length is within 7e-8 of its value in 64 bits (FP32's own
// rounding; 1.2e-7 to 2.2e-7 with plain FP32 sums), on FP64 handles within 4e-16
// (5e-8 with the coarse share of r.z from the FP32 restriction).
// An exchange is barrier and data in one: on a grid every CTA stores its sums
// as (value, tag) words and polls the words of all CTAs; in a cluster it pushes
// them into the other CTAs' shared memory before the hardware barrier.  Every
// CTA then forms the same sums in the same order.
// The right-hand side is scaled to unit norm, so FP32 neither under- nor
// overflows.  Every wait is bounded and reported through kerr.
#pragma once

#include <algorithm>
#include <cstdint>

#include "cg_pcg_device.cuh"

namespace softsim {

// ROWS: the slices are stored by rows (see cg_plan.h), else by colours.  GRID: a
// cooperative grid, else one CTA or one cluster.
template <typename T, int D, int VPT, bool ROWS, bool GRID>
__global__ void __launch_bounds__(512, 1)
    k_pcg(PcgDev pd, const double *__restrict__ b, double sign, T *__restrict__ dout, double rtol, int max_iter,
          int polls, DevScalars *sc)
{
    constexpr size_t esz = 4 + D * D * sizeof(T);
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int sbad, sstop;
    const int cta = blockIdx.x, nthr = pd.threads, tid = threadIdx.x, lane = tid & 31;
    constexpr bool grid = GRID;
    Slice sl = pcg_slice<D, T, ROWS>(pd, cta, grid, smem, polls, &sbad);
    const unsigned char *gsl = sl.rest - sl.n_ent * esz;  // this CTA's slice in global memory
    if (tid == 0) {
        for (int k = 0; k < (sl.stages ? sl.stages : 1); ++k) {
            mbar_init(sl.full + k, 1);
            mbar_init(sl.empty + k, nthr >> 5);
        }
        sbad = 0;
        sstop = 0;
    }
    pcg_tables<D, T, ROWS>(pd, cta, grid, smem);
    __syncthreads();
    if (tid >= nthr) {  // producer warp of a streamed slice
        if (lane == 0) {
            volatile int *stop = &sstop;
            const uint64_t pol = l2_evict_first_policy();
            const uint32_t S = (uint32_t)sl.stages;
            uint32_t q = 0;
            int c = 0;
            size_t off = 0;
            for (;; ++q) {
                const uint32_t st = q % S;
                bool go = true;
                if (q >= S) {
                    int i = 0;
                    while (!mbar_try_wait(sl.empty + st, ((q / S) - 1u) & 1u))
                        if (*stop || ++i > (1 << 26)) {
                            go = false;
                            break;
                        }
                }
                if (!go || *stop) break;
                const uint32_t n = sl.meta[c] & ~kCgLastOfColour, bytes = (uint32_t)(n * esz);
                mbar_arrive_expect_tx(sl.full + st, bytes);
                bulk_g2s_stream(sl.base + (size_t)st * sl.stage_bytes, gsl + off, bytes, sl.full + st, pol);
                off += bytes;
                if (++c == sl.n_chunks) c = 0, off = 0;
            }
            // the copies still in flight land before the CTA exits
            for (uint32_t k = q > S ? q - S : 0; k < q; ++k) mbar_wait_bounded(sl.full + k % S, (k / S) & 1u);
        }
        return;
    }
    if (!sl.stages) {  // the slice stays in shared memory
        const uint32_t bytes = (uint32_t)(sl.n_ent * esz);
        if (tid == 0) {
            mbar_arrive_expect_tx(sl.full, bytes);
            for (uint32_t o = 0; o < bytes; o += 65536)
                bulk_g2s(sl.base + o, gsl + o, bytes - o < 65536 ? bytes - o : 65536, sl.full);
        }
        if (!mbar_wait_bounded(sl.full, 0, polls)) sbad = 1;
        csync(nthr);
        const int bad = sbad;
        int any = bad;
        if (!GRID && pd.cluster) {  // the CTAs of a cluster leave together or not at all
            cluster_sync();
            for (int k = 0; k < pd.n_cta; ++k) any |= ld_dsmem_s32(&sbad, (uint32_t)k);
            cluster_sync();
        }
        if (any) {
            if (tid == 0) {
                if (bad) mbar_wait_bounded(sl.full, 0);  // let the copies in flight land
                atomicOr(&sc->kerr, 1);
            }
            return;
        }
    }
    const PcgResult res =
        pcg_run<T, D, VPT, ROWS, GRID>(pd, sl, cta, smem, b, sign, sc->gn2, dout, rtol, max_iter, true);
    if (sl.stages) {
        csync(nthr);
        if (tid == 0) *(volatile int *)&sstop = 1;
    }
    if (!GRID && pd.cluster) cluster_sync();  // no CTA leaves while another may still write to it
    if (res.fail && tid == 0) atomicOr(&sc->kerr, sbad ? 1 : 2);
    if (cta == 0 && tid == 0) {
        sc->iter = res.iter;
        sc->negcurv = res.neg;
        sc->rr = res.rr;
        sc->done = 1;
    }
}

// ---------------------------------------------------------------- host side

template <typename T, int D>
static void *pcg_kernel(const PcgDev &pd)
{
    constexpr bool F32 = sizeof(T) == 4;
    const bool grid = pd.n_cta > 1 && !pd.cluster;
    if (pd.tpr) {
        if (pd.vpt == 1) return grid ? (void *)k_pcg<T, D, 1, true, true> : (void *)k_pcg<T, D, 1, true, false>;
        if (grid) return (void *)k_pcg<T, D, 4, true, true>;
        if constexpr (F32 && D == 2) return (void *)k_pcg<T, D, 4, true, false>;
    } else {
        if constexpr (D == 3)
            if (pd.vpt == 2) return (void *)k_pcg<T, D, 2, false, true>;
        if constexpr (F32 || D == 3)
            if (pd.vpt == 4) return (void *)k_pcg<T, D, 4, false, true>;
        if constexpr (F32)
            if (pd.vpt == 8) return (void *)k_pcg<T, D, 8, false, true>;
    }
    return nullptr;
}

// The launch of a configured plan, in place; at[1] is filled in too.
template <typename T>
static cudaLaunchConfig_t pcg_launch_config(int dim, const PcgDev &pd, cudaLaunchAttribute *at, cudaStream_t s)
{
    const size_t esz = 4 + dim * dim * sizeof(T);
    const bool on_grid = pd.n_cta > 1 && !pd.cluster;
    const PcgSmem L(dim, sizeof(T), pd.ns, pd.max_halo, pd.max_items, pd.n_coarse, pd.n_meta, on_grid ? pd.n_cta : 0);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pd.n_cta);
    cfg.blockDim = dim3(pd.threads + (pd.stages ? 32 : 0));
    cfg.dynamicSmemBytes = L.ring + (pd.stages ? (size_t)pd.stages * kCgChunk * esz : (size_t)pd.max_entries * esz);
    cfg.stream = s;
    cfg.attrs = at;
    if (pd.cluster) {  // one cluster: every CTA co-scheduled by construction
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = pd.n_cta;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.numAttrs = 1;
    } else if (on_grid) {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cfg.numAttrs = 1;
    }
    return cfg;
}

// Whether the device can hold all CTAs of the configured launch at once.
template <typename T>
static bool resident(int dim, const PcgDev &pd, const void *k)
{
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = pcg_launch_config<T>(dim, pd, at, nullptr);
    int clusters = 0, per_sm = 0, dev = 0, sms = 0;
    cudaError_t e;
    if (pd.cluster) {
        e = cudaOccupancyMaxActiveClusters(&clusters, k, &cfg);
    } else {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, (int)cfg.blockDim.x, cfg.dynamicSmemBytes);
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    return e == cudaSuccess && pcg_resident(pd.cluster != 0, pd.n_cta, clusters, per_sm, sms);
}

template <typename T, int D>
static bool configure(const Ctx &c, PcgDev &pd)
{
    const size_t esz = 4 + D * D * sizeof(T);
    const bool on_grid = pd.n_cta > 1 && !pd.cluster;
    const PcgSmem base(D, sizeof(T), pd.ns, pd.max_halo, pd.max_items, pd.n_coarse, pd.n_meta, on_grid ? pd.n_cta : 0);
    if (pd.max_items > (on_grid ? 1 : kMaxWarps) || pd.n_cta > 32 * kMaxWarps) return false;
    const bool rows = pd.tpr > 0;
    for (int streamed = 0; streamed < (rows ? 1 : 2); ++streamed) {
        // a producer warp takes one warp's place
        pd.threads = streamed ? kPcgStreamThreads
                     : rows   ? std::min(kPcgThreads, std::max(128, pd.ns * pd.tpr))
                     : kPcgThreads;
        const int need = (pd.ns + pd.threads - 1) / pd.threads;
        pd.vpt = pcg_variant(D, sizeof(T), rows, on_grid, need);
        if (!pd.vpt) return false;
        void *k = pcg_kernel<T, D>(pd);
        cudaFuncAttributes at;
        if (!k || cudaFuncGetAttributes(&at, k) != cudaSuccess) break;
        // every handle sets the same limit: attributes belong to the function, not to a handle
        const size_t limit = kPcgSmem - at.sharedSizeBytes;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit) != cudaSuccess ||
            (pd.cluster && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess))
            break;
        if (!streamed) {
            pd.stages = 0;
            if (base.ring + (size_t)pd.max_entries * esz > limit) {
                if (pd.cluster) return false;
                continue;
            }
        } else {
            if (base.ring + 3 * kCgChunk * esz > limit) return false;
            pd.stages = (int)((limit - base.ring) / (kCgChunk * esz));
            if (pd.stages > kPcgMaxStages) pd.stages = kPcgMaxStages;
        }
        if (resident<T>(D, pd, k)) return true;
        break;
    }
    cudaGetLastError();
    return false;
}

template <typename T>
bool pcg_configure(const Ctx &c, PcgDev &pd)
{
    return c.dim == 2 ? configure<T, 2>(c, pd) : configure<T, 3>(c, pd);
}

template <typename T>
cudaError_t launch_pcg(const Ctx &c, const PcgDev &pd, const double *b, double sign, T *d, double rtol, int max_iter,
                       cudaStream_t s)
{
    void *k = c.dim == 2 ? pcg_kernel<T, 2>(pd) : pcg_kernel<T, 3>(pd);
    int polls = c.td.wait_polls;
    DevScalars *sc = c.sc;
    void *args[] = {(void *)&pd, (void *)&b, &sign, &d, &rtol, &max_iter, &polls, &sc};
    cudaLaunchAttribute at[1];
    const cudaLaunchConfig_t cfg = pcg_launch_config<T>(c.dim, pd, at, s);
    if (pd.n_cta > 1 && !pd.cluster) {
        const cudaError_t e = cudaMemsetAsync(pd.words, 0, (size_t)16 * kPcgWords * pd.n_cta, s);
        if (e != cudaSuccess) return e;
    }
    c.n_launch += 1;
    return cudaLaunchKernelExC(&cfg, k, args);
}

}  // namespace softsim
