// Assembly of the operator of a CG solve: one dim x dim block per mesh edge,
// the vertex diagonal, and the coarse matrix of the preconditioner with its
// inverse (see cg_plan.h for the layout, cg_pcg_kernel.cuh for the solver).
//
// The block of an element's corners a, b is, with g_a the gradient of corner
// a's shape function, c_a = cof(F) g_a, gamma_a = g_a . f and q = F f
// (Eq. matrix-free-dfdx applied to dF = v g_b^T),
//   K_ab = W [ (mu g_a.g_b + c1 gamma_a gamma_b) I + c' c_a c_b^T
//              + c [F (g_b x g_a)]_x + c2 gamma_a gamma_b q q^T ],
// with c(J), c'(J) as in the HVP kernels and c1, c2 the muscle's stiffness.
#include <cstdint>

#include "cg_blocks.cuh"
#include "pdl.cuh"

namespace softsim {

// ---------------------------------------------------------------- edge blocks

// One thread per element: its corner pairs' blocks to their contribution
// slots.  Bound by the writes of 36-byte (3D FP32) blocks to scattered slots: a
// warp's 32 blocks go through shared memory, so that neighbouring lanes write
// neighbouring words of a slot (4 slots an instruction instead of 32): 3.1
// million tets 1,091 -> 412 us.  gridDim.y CTAs share a tile's elements, so that
// small meshes fill the SMs (5,616 tets: 15.5 -> 6.5 us).
template <typename T, int D, bool SPRING>
__global__ void __launch_bounds__(256) k_asm_elem(TileDev td, const T *__restrict__ erec, const T *__restrict__ act,
                                                  Phys ph, const T *__restrict__ u, const uint32_t *__restrict__ cpos,
                                                  T *__restrict__ contrib)
{
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int NF = hvp_fields(D, SPRING), RS = rec_stride(NF), NP = (D + 1) * D / 2, DD = D * D;
    const int lane = threadIdx.x & 31, wrp = threadIdx.x >> 5;
    T *su = reinterpret_cast<T *>(smem);
    T *stage = su + (size_t)td.max_tv * D + (size_t)wrp * 32 * DD;  // this warp's blocks (3D)
    const int t = blockIdx.x;
    const int es = td.tile_elem[t], ne_t = td.tile_elem[t + 1] - es;
    const int vs = td.tile_vert[t], nlv = td.tile_vert[t + 1] - vs;
    for (int k = threadIdx.x; k < nlv; k += blockDim.x) {
        const int64_t gid = td.lv_gid[vs + k];
#pragma unroll
        for (int c = 0; c < D; ++c) su[k * D + c] = u[gid * D + c];
    }
    __syncthreads();
    pdl_trigger();
    const T mu = pick<T>(ph.mu, ph.mu_f), lam = pick<T>(ph.lam, ph.lam_f);
    const T sel = pick<T>(ph.s_el, ph.s_el_f), kk = pick<T>(ph.k, ph.k_f);
    for (int l0 = (blockIdx.y * (blockDim.x >> 5) + wrp) * 32; l0 < ne_t; l0 += gridDim.y * blockDim.x) {
        const int64_t e = es + min(l0 + lane, ne_t - 1);
        const bool on = l0 + lane < ne_t && td.perm[e] >= 0;  // else past the end, or padding
        int lid[D + 1];
        unpack<D>(td.conn[e], lid);
        T rv[RS], B[D][D], Du[D][D], gv[D], f[D];
        load_pairs<T, RS>(erec + e * RS, rv);
        uint32_t w[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) w[q] = on ? cpos[e * NP + q] : kCgPadEntry;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            gv[i] = rv[FI<D>::G + i];
            f[i] = SPRING ? rv[FI<D>::F + i] : T(0);
#pragma unroll
            for (int j = 0; j < D; ++j) B[i][j] = rv[FI<D>::B + i * D + j];
        }
        edges<T, D>(su, lid, Du);
        elem_blocks<T, D>(B, gv, f, rv[FI<D>::W] * sel, act[e], Du, SPRING, ph.log_mode, mu, lam, kk,
                          [&](int pair, const T K[D][D]) {
                              if constexpr (D == 2) {
                                  if (on) store_block<T, D>(contrib, w[pair], K);
                              } else {
                                  const bool tr = (w[pair] & kCgTransposed) != 0;
#pragma unroll
                                  for (int i = 0; i < D; ++i)
#pragma unroll
                                      for (int j = 0; j < D; ++j) stage[lane * DD + i * D + j] = tr ? K[j][i] : K[i][j];
                                  __syncwarp();
#pragma unroll
                                  for (int q = 0; q < DD; ++q) {
                                      const int k = lane + 32 * q, src = k / DD;
                                      const uint32_t ws = __shfl_sync(0xffffffffu, w[pair], src);
                                      if (ws != kCgPadEntry)
                                          contrib[(int64_t)(ws & ~kCgTransposed) * DD + (k - src * DD)] = stage[k];
                                  }
                                  __syncwarp();
                              }
                          });
    }
}

// One thread per edge: the sum of its contributions (contiguous, in element order).
template <typename T, int D>
__global__ void __launch_bounds__(256) k_asm_edge(int64_t n_edges, const int32_t *__restrict__ edge_ptr,
                                                  const T *__restrict__ contrib, T *__restrict__ blk)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int q0 = e < n_edges ? edge_ptr[e] : 0, q1 = e < n_edges ? edge_ptr[e + 1] : 0;
    pdl_trigger();
    pdl_wait();
    if (e >= n_edges) return;
    T acc[D * D];
#pragma unroll
    for (int k = 0; k < D * D; ++k) acc[k] = T(0);
    for (int q = q0; q < q1; ++q)
#pragma unroll
        for (int k = 0; k < D * D; ++k) acc[k] += contrib[(int64_t)q * (D * D) + k];
#pragma unroll
    for (int k = 0; k < D * D; ++k) blk[k * n_edges + e] = acc[k];
}

// Index words and blocks in the solver's order; grid (chunks, blocks per chunk).
template <typename T, int D>
__global__ void __launch_bounds__(256) k_asm_slice(int64_t n_edges, const int32_t *__restrict__ chunk_ent,
                                                   const uint32_t *__restrict__ ent_idx,
                                                   const uint32_t *__restrict__ ent_edge, const T *__restrict__ blk,
                                                   unsigned char *__restrict__ slices)
{
    const int e0 = chunk_ent[blockIdx.x], n = chunk_ent[blockIdx.x + 1] - e0;
    unsigned char *base = slices + (size_t)e0 * (4 + D * D * sizeof(T));
    uint32_t *idx = reinterpret_cast<uint32_t *>(base);
    T *val = reinterpret_cast<T *>(base + (size_t)n * 4);
    pdl_trigger();
    pdl_wait();
    for (int k = blockIdx.y * blockDim.x + threadIdx.x; k < n; k += gridDim.y * blockDim.x) {
        const uint32_t w = ent_edge[e0 + k];
        idx[k] = ent_idx[e0 + k];
        const int64_t e = w & ~kCgTransposed;
        const bool pad = w == kCgPadEntry, tr = (w & kCgTransposed) != 0;
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j)
                val[(i * D + j) * n + k] = pad ? T(0) : blk[(tr ? j * D + i : i * D + j) * n_edges + e];
    }
}

// ---------------------------------------------------------------- vertex data

template <typename T, int D>
__global__ void __launch_bounds__(256) k_asm_slots(PcgDev pd, VertDev vd, Phys ph, const double *__restrict__ u)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (k < pd.n_cta * pd.ns) slot_data<T, D>(k, pd, vd, ph, u);
}

// ---------------------------------------------------------------- coarse matrix

// One block per item: its partial sum of a coarse block, in a fixed order.
template <typename T, int D>
__global__ void __launch_bounds__(128) k_coarse_item(PcgDev pd)
{
    constexpr int NM = D == 3 ? 6 : 3;
    const int kind = pd.citem_kind[blockIdx.x], b = pd.citem_begin[blockIdx.x], e = pd.citem_end[blockIdx.x];
    float acc[NM * NM];
#pragma unroll
    for (int k = 0; k < NM * NM; ++k) acc[k] = 0.0f;
    for (int q = b + threadIdx.x; q < e; q += blockDim.x) coarse_add<T, D>(pd, kind, q, acc);
    __shared__ float red[4][NM * NM];
#pragma unroll
    for (int k = 0; k < NM * NM; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_down_sync(0xffffffffu, acc[k], o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = acc[k];
    }
    __syncthreads();
    for (int k = threadIdx.x; k < NM * NM; k += blockDim.x)
        pd.cpart[(int64_t)blockIdx.x * (NM * NM) + k] = (red[0][k] + red[1][k]) + (red[2][k] + red[3][k]);
}

// One block per coarse block (I, J): the sum of its items, and its transpose.
template <int D>
__global__ void __launch_bounds__(64) k_coarse_sum(PcgDev pd)
{
    constexpr int NM = D == 3 ? 6 : 3;
    const int k = threadIdx.x, N = pd.n_coarse;
    if (k >= NM * NM) return;
    const int I = pd.ctgt_i[blockIdx.x], J = pd.ctgt_j[blockIdx.x], m = k / NM, n = k % NM;
    float s = 0.0f, st = 0.0f;
    for (int q = pd.ctgt_ptr[blockIdx.x]; q < pd.ctgt_ptr[blockIdx.x + 1]; ++q) {
        s += pd.cpart[(int64_t)q * (NM * NM) + k];
        st += pd.cpart[(int64_t)q * (NM * NM) + n * NM + m];
    }
    if (I == J) s = 0.5f * (s + st);
    pd.E[(size_t)(I * NM + m) * N + J * NM + n] = s;
    pd.E[(size_t)(J * NM + n) * N + I * NM + m] = s;
}

// Inverse of the coarse matrix (symmetric, scaled to unit diagonal) by
// Gauss-Jordan elimination in place, in the registers of one CTA: thread
// (ty, tx) of a 32 x 32 grid holds the entries (ty + 32 i, tx + 32 j), i, j <
// BS.  A step broadcasts its pivot row through shared memory (one barrier a
// step, two buffers); the pivot column is the row with its sign changed at the
// indices already eliminated.  A mode whose pivot is not clearly positive (a
// pinned or degenerate aggregate, an indefinite state) is left out: its row
// and column of the inverse are zero.  Bound by instruction issue (N^3 FMAs on
// one SM).
template <int BS>
__global__ void __launch_bounds__(1024) k_coarse_invert(int N, const float *__restrict__ E, float *__restrict__ Einv)
{
    __shared__ float row[2][32 * BS], scale[32 * BS];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int k = threadIdx.x; k < 32 * BS; k += 1024) {
        const float d = k < N ? E[(size_t)k * N + k] : 1.0f;
        scale[k] = d > 0.0f ? rsqrtf(d) : 0.0f;
    }
    __syncthreads();
    float a[BS][BS];
#pragma unroll
    for (int i = 0; i < BS; ++i)
#pragma unroll
        for (int j = 0; j < BS; ++j) {
            const int r = ty + 32 * i, c = tx + 32 * j;
            a[i][j] = (r < N && c < N) ? E[(size_t)r * N + c] * scale[r] * scale[c] : 0.0f;
        }
#pragma unroll
    for (int kq = 0; kq < BS; ++kq)
        for (int kr = 0; kr < 32 && kq * 32 + kr < N; ++kr) {
            const int b = kr & 1;
            if (ty == kr)
#pragma unroll
                for (int j = 0; j < BS; ++j) row[b][tx + 32 * j] = a[kq][j];
            __syncthreads();
            const float p = row[b][kq * 32 + kr];
            const float ip = p > 1e-5f ? __frcp_rn(p) : 0.0f;
            float rk[BS], ck[BS];
#pragma unroll
            for (int j = 0; j < BS; ++j) {
                rk[j] = row[b][tx + 32 * j] * ip;
                const float c = row[b][ty + 32 * j];
                ck[j] = j < kq || (j == kq && ty < kr) ? c : -c;  // minus the column entry
            }
            if (tx == kr) {
                rk[kq] = ip;
#pragma unroll
                for (int i = 0; i < BS; ++i) a[i][kq] = 0.0f;
            }
#pragma unroll
            for (int i = 0; i < BS; ++i)
#pragma unroll
                for (int j = 0; j < BS; ++j) a[i][j] = fmaf(ck[i], rk[j], a[i][j]);
            if (ty == kr)
#pragma unroll
                for (int j = 0; j < BS; ++j) a[kq][j] = rk[j];
        }
#pragma unroll
    for (int i = 0; i < BS; ++i)
#pragma unroll
        for (int j = 0; j < BS; ++j) {
            const int r = ty + 32 * i, c = tx + 32 * j;
            if (r < N && c < N) Einv[(size_t)r * N + c] = a[i][j] * scale[r] * scale[c];
        }
}

// ---------------------------------------------------------------- launchers

template <typename T, int D>
static void assemble(const Ctx &c, const PcgDev &pd, const Phys &ph, const T *u, const double *u64, bool coarse,
                     cudaStream_t s)
{
    const T *er = sizeof(T) == 4 ? reinterpret_cast<const T *>(c.rec32) : reinterpret_cast<const T *>(c.rec64);
    const T *ac = sizeof(T) == 4 ? reinterpret_cast<const T *>(c.a32) : reinterpret_cast<const T *>(c.a64);
    const size_t sm = ((size_t)c.td.max_tv * D + (D == 3 ? (size_t)c.threads * D * D : 0)) * sizeof(T);
    const dim3 ge(c.td.n_tiles, c.asm_split);
    T *contrib = static_cast<T *>(pd.contrib), *blk = static_cast<T *>(pd.blk);
    if (c.muscle)
        k_asm_elem<T, D, true><<<ge, c.threads, sm, s>>>(c.td, er, ac, ph, u, pd.cpos, contrib);
    else
        k_asm_elem<T, D, false><<<ge, c.threads, sm, s>>>(c.td, er, ac, ph, u, pd.cpos, contrib);
    launch_k(true, k_asm_edge<T, D>, dim3((unsigned)((pd.n_edges + 255) / 256)), dim3(256), 0, s, pd.n_edges,
             pd.edge_ptr, (const T *)contrib, blk);
    const dim3 gs((unsigned)pd.n_chunks, pd.tpr ? (unsigned)((pd.max_entries + 255) / 256) : 1u);
    launch_k(true, k_asm_slice<T, D>, gs, dim3(256), 0, s, pd.n_edges, pd.chunk_ent, pd.ent_idx, pd.ent_edge,
             (const T *)blk, pd.slices);
    const int n = pd.n_cta * pd.ns;
    launch_k(true, k_asm_slots<T, D>, dim3((n + 255) / 256), dim3(256), 0, s, pd, c.vd, ph, u64);
    c.n_launch += 4;
    if (!coarse) return;
    cudaMemsetAsync(pd.E, 0, sizeof(float) * pd.n_coarse * pd.n_coarse, s);
    k_coarse_item<T, D><<<pd.n_citems, 128, 0, s>>>(pd);
    k_coarse_sum<D><<<pd.n_ctgts, 64, 0, s>>>(pd);
    const int N = pd.n_coarse;
    if (N <= 32)
        k_coarse_invert<1><<<1, 1024, 0, s>>>(N, pd.E, pd.Einv);
    else if (N <= 64)
        k_coarse_invert<2><<<1, 1024, 0, s>>>(N, pd.E, pd.Einv);
    else if (N <= 96)
        k_coarse_invert<3><<<1, 1024, 0, s>>>(N, pd.E, pd.Einv);
    else if (N <= 128)
        k_coarse_invert<4><<<1, 1024, 0, s>>>(N, pd.E, pd.Einv);
    else
        k_coarse_invert<6><<<1, 1024, 0, s>>>(N, pd.E, pd.Einv);
    c.n_launch += 3;
}

template <typename T>
void launch_pcg_assemble(const Ctx &c, const PcgDev &pd, const Phys &ph, const T *u, const double *u64, bool coarse,
                         cudaStream_t s)
{
    c.dim == 2 ? assemble<T, 2>(c, pd, ph, u, u64, coarse, s) : assemble<T, 3>(c, pd, ph, u, u64, coarse, s);
}

template void launch_pcg_assemble<float>(const Ctx &, const PcgDev &, const Phys &, const float *, const double *, bool,
                                         cudaStream_t);
template void launch_pcg_assemble<double>(const Ctx &, const PcgDev &, const Phys &, const double *, const double *,
                                          bool, cudaStream_t);

}  // namespace softsim
