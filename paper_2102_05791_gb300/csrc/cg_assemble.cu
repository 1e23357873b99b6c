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

#include "cg_pcg.h"
#include "elem_math.cuh"

namespace softsim {

// ---------------------------------------------------------------- edge blocks

// One thread per element: its corner pairs' blocks to their contribution
// slots.  Bound by the scattered 36-byte (FP32) writes.
template <typename T, int D, bool SPRING>
__global__ void __launch_bounds__(256) k_asm_elem(TileDev td, const T *__restrict__ erec, Phys ph,
                                                  const T *__restrict__ u, const uint32_t *__restrict__ cpos,
                                                  T *__restrict__ contrib)
{
    extern __shared__ __align__(16) unsigned char smem[];
    T *su = reinterpret_cast<T *>(smem);
    constexpr int NF = hvp_fields(D, SPRING), RS = rec_stride(NF), NP = (D + 1) * D / 2;
    const int t = blockIdx.x;
    const int es = td.tile_elem[t], ne_t = td.tile_elem[t + 1] - es;
    const int vs = td.tile_vert[t], nlv = td.tile_vert[t + 1] - vs;
    for (int k = threadIdx.x; k < nlv; k += blockDim.x) {
        const int64_t gid = td.lv_gid[vs + k];
#pragma unroll
        for (int c = 0; c < D; ++c) su[k * D + c] = u[gid * D + c];
    }
    __syncthreads();
    const T mu = pick<T>(ph.mu, ph.mu_f), lam = pick<T>(ph.lam, ph.lam_f);
    const T sel = pick<T>(ph.s_el, ph.s_el_f), kk = pick<T>(ph.k, ph.k_f);
    for (int le = threadIdx.x; le < ne_t; le += blockDim.x) {
        const int64_t e = es + le;
        if (td.perm[e] < 0) continue;  // padding
        int lid[D + 1];
        unpack<D>(td.conn[e], lid);
        T rv[RS], B[D][D], Du[D][D], F[D][D], C[D][D];
        load_pairs<T, RS>(erec + e * RS, rv);
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) B[i][j] = rv[FI<D>::B + i * D + j];
        edges<T, D>(su, lid, Du);
        mul<T, D>(Du, B, F, true);
        cof<T, D>(F, C);
        const T J = detF<T, D>(F, C);
        T l, cc, cp;
        log_terms<T>(ph.log_mode, mu, lam, J, l, cc, cp);
        const T W = rv[FI<D>::W] * sel, aval = rv[NF];
        T c1 = kk * aval, c2 = T(0), q[D];
        if constexpr (SPRING) {
            T s2 = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                T s = rv[FI<D>::F + i];
#pragma unroll
                for (int k = 0; k < D; ++k) s += Du[i][k] * rv[FI<D>::G + k];
                q[i] = s;
                s2 += s * s;
            }
            spring_terms<T>(true, kk, aval, sqrt(s2), c1, c2);
        }
        T g[D + 1][D], cg[D + 1][D], gam[D + 1];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            T s = T(0);
#pragma unroll
            for (int k = 0; k < D; ++k) {
                g[k + 1][i] = B[k][i];
                s += B[k][i];
            }
            g[0][i] = -s;
        }
        gam[0] = T(0);
#pragma unroll
        for (int k = 0; k < D; ++k) {
            gam[k + 1] = rv[FI<D>::G + k];
            gam[0] -= gam[k + 1];
        }
#pragma unroll
        for (int k = 0; k <= D; ++k)
#pragma unroll
            for (int i = 0; i < D; ++i) {
                T s = T(0);
#pragma unroll
                for (int m = 0; m < D; ++m) s += C[i][m] * g[k][m];
                cg[k][i] = s;
            }
        const T muW = mu * W, cpW = cp * W, ccW = cc * W;
        int pair = 0;
#pragma unroll
        for (int a = 0; a <= D; ++a)
#pragma unroll
            for (int b = a + 1; b <= D; ++b, ++pair) {
                const uint32_t w = cpos[e * NP + pair];
                T K[D][D];
                T gg = T(0);
#pragma unroll
                for (int i = 0; i < D; ++i) gg += g[a][i] * g[b][i];
                const T d = muW * gg + c1 * W * gam[a] * gam[b];
#pragma unroll
                for (int i = 0; i < D; ++i)
#pragma unroll
                    for (int j = 0; j < D; ++j) K[i][j] = cpW * cg[a][i] * cg[b][j] + (i == j ? d : T(0));
                if constexpr (D == 3) {
                    T n[3], wv[3];
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        const int p = (i + 1) % 3, r = (i + 2) % 3;
                        n[i] = g[b][p] * g[a][r] - g[b][r] * g[a][p];  // g_b x g_a
                    }
#pragma unroll
                    for (int i = 0; i < 3; ++i)
                        wv[i] = ccW * (F[i][0] * n[0] + F[i][1] * n[1] + F[i][2] * n[2]);
                    K[0][1] -= wv[2];
                    K[0][2] += wv[1];
                    K[1][0] += wv[2];
                    K[1][2] -= wv[0];
                    K[2][0] -= wv[1];
                    K[2][1] += wv[0];
                } else {
                    const T s = ccW * (g[b][1] * g[a][0] - g[b][0] * g[a][1]);
                    K[0][1] += s;
                    K[1][0] -= s;
                }
                if constexpr (SPRING) {
                    const T m = c2 * W * gam[a] * gam[b];
#pragma unroll
                    for (int i = 0; i < D; ++i)
#pragma unroll
                        for (int j = 0; j < D; ++j) K[i][j] += m * q[i] * q[j];
                }
                T *out = contrib + (int64_t)(w & ~kCgTransposed) * (D * D);
                const bool tr = (w & kCgTransposed) != 0;
#pragma unroll
                for (int i = 0; i < D; ++i)
#pragma unroll
                    for (int j = 0; j < D; ++j) out[i * D + j] = tr ? K[j][i] : K[i][j];
            }
    }
}

// One thread per edge: the sum of its contributions (contiguous, in element order).
template <typename T, int D>
__global__ void __launch_bounds__(256) k_asm_edge(int64_t n_edges, const int32_t *__restrict__ edge_ptr,
                                                  const T *__restrict__ contrib, T *__restrict__ blk)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n_edges) return;
    T acc[D * D];
#pragma unroll
    for (int k = 0; k < D * D; ++k) acc[k] = T(0);
    for (int q = edge_ptr[e]; q < edge_ptr[e + 1]; ++q)
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

// Per slot: the arm of the rigid rotations about the aggregate's reference
// vertex in the current shape, and the vertex diagonal (inertia + friction,
// contact curvature), formed in FP64 as in the HVP kernels.
template <typename T, int D>
__global__ void __launch_bounds__(256) k_asm_slots(int n, const int32_t *__restrict__ slot_gid,
                                                   const int32_t *__restrict__ grp_agg,
                                                   const int32_t *__restrict__ agg_ref, float inv_len, VertDev vd,
                                                   Phys ph, const double *__restrict__ u, float4 *__restrict__ pos4,
                                                   T *__restrict__ diag2)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int64_t v = slot_gid[k];
    const int agg = grp_agg[k >> 5];
    float4 o = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(agg | 1 << 30));
    T dh = T(0), dy = T(0);
    if (v >= 0) {
        const int64_t r = agg_ref[agg];
        o.x = (float)(vd.X[v * D] + u[v * D] - vd.X[r * D] - u[r * D]) * inv_len;
        o.y = (float)(vd.X[v * D + 1] + u[v * D + 1] - vd.X[r * D + 1] - u[r * D + 1]) * inv_len;
        if (D == 3) o.z = (float)(vd.X[v * D + 2] + u[v * D + 2] - vd.X[r * D + 2] - u[r * D + 2]) * inv_len;
        o.w = __int_as_float(agg | (vd.fixed[v] ? 1 << 30 : 0));
        double h = 0.0, y = 0.0;
        if (ph.dyn) {
            const double m = vd.mass[v];
            h = ph.fw ? m + ph.fw[v] : m;
            y = m;
        }
        if (ph.contact) {
            const double yy = vd.X[v * D + 1] + u[v * D + 1];
            const double pen = yy < 0.0 ? -yy : 0.0;
            if (pen > 0.0) y += ph.s_el * (ph.cpow * (ph.cpow - 1) * ph.kc * (ph.cpow == 2 ? 1.0 : pen));
        }
        dh = T(h);
        dy = T(y);
    }
    pos4[k] = o;
    diag2[2 * k] = dh;
    diag2[2 * k + 1] = dy;
}

// ---------------------------------------------------------------- coarse matrix

// Mode n of the rigid motions at arm R: translations, then rotations (one in 2D).
template <int D>
__device__ __forceinline__ void rigid_mode(int n, float4 R, float out[D])
{
    if constexpr (D == 3) {
        const float x = R.x, y = R.y, z = R.z;
        out[0] = n == 0 ? 1.0f : n == 4 ? z : n == 5 ? -y : 0.0f;
        out[1] = n == 1 ? 1.0f : n == 3 ? -z : n == 5 ? x : 0.0f;
        out[2] = n == 2 ? 1.0f : n == 3 ? y : n == 4 ? -x : 0.0f;
    } else {
        out[0] = n == 0 ? 1.0f : n == 2 ? -R.y : 0.0f;
        out[1] = n == 1 ? 1.0f : n == 2 ? R.x : 0.0f;
    }
}

// acc[m] += Z_m . f for the modes of arm R
template <int D>
__device__ __forceinline__ void restrict_add(float4 R, const float f[D], float s, float *acc, int stride)
{
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c * stride] += s * f[c];
    if constexpr (D == 3) {
        acc[3 * stride] += s * (R.y * f[2] - R.z * f[1]);
        acc[4 * stride] += s * (R.z * f[0] - R.x * f[2]);
        acc[5 * stride] += s * (R.x * f[1] - R.y * f[0]);
    } else {
        acc[2 * stride] += s * (R.x * f[1] - R.y * f[0]);
    }
}

// One block per item: its partial sum of a coarse block, in a fixed order.
template <typename T, int D>
__global__ void __launch_bounds__(128) k_coarse_item(PcgDev pd, const T *__restrict__ blk, const T *__restrict__ diag2)
{
    constexpr int NM = D == 3 ? 6 : 3;
    const int kind = pd.citem_kind[blockIdx.x], b = pd.citem_begin[blockIdx.x], e = pd.citem_end[blockIdx.x];
    float acc[NM * NM];
#pragma unroll
    for (int k = 0; k < NM * NM; ++k) acc[k] = 0.0f;
    for (int q = b + threadIdx.x; q < e; q += blockDim.x) {
        if (kind == CK_VERT) {
            const float4 R = pd.pos4[q];
            if (__float_as_int(R.w) >> 30) continue;
            const float dh = (float)diag2[2 * q], dy = (float)diag2[2 * q + 1];
#pragma unroll
            for (int n = 0; n < NM; ++n) {
                float z[D];
                rigid_mode<D>(n, R, z);
#pragma unroll
                for (int c = 0; c < D; ++c) z[c] *= c == 1 ? dy : dh;
                restrict_add<D>(R, z, 1.0f, acc + n, NM);
            }
            continue;
        }
        const int ed = pd.seg_edge[q];
        const float4 Ri = pd.pos4[pd.edge_lo[ed]], Rj = pd.pos4[pd.edge_hi[ed]];
        const float fi = (__float_as_int(Ri.w) >> 30) ? 0.0f : 1.0f, fj = (__float_as_int(Rj.w) >> 30) ? 0.0f : 1.0f;
        float M[D][D];
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) M[i][j] = (float)blk[(i * D + j) * pd.n_edges + ed];
        const bool lo = kind == CK_LO, hi = kind == CK_HI, inner = kind == CK_INNER;
#pragma unroll
        for (int n = 0; n < NM; ++n) {
            float zi[D], zj[D], f[D], g[D];
            rigid_mode<D>(n, Ri, zi);
            rigid_mode<D>(n, Rj, zj);
#pragma unroll
            for (int c = 0; c < D; ++c) zi[c] *= fi, zj[c] *= fj;
            // f = M (z_j - z_i) at lo, g = -M^T (z_j - z_i) at hi; a cross edge's blocks take one of the terms
            float dl[D], dh[D];
#pragma unroll
            for (int c = 0; c < D; ++c) {
                dl[c] = inner ? zj[c] - zi[c] : lo ? -zi[c] : hi ? 0.0f : zj[c];
                dh[c] = inner ? zi[c] - zj[c] : hi ? -zj[c] : 0.0f;
            }
#pragma unroll
            for (int i = 0; i < D; ++i) {
                f[i] = g[i] = 0.0f;
#pragma unroll
                for (int j = 0; j < D; ++j) {
                    f[i] += M[i][j] * dl[j];
                    g[i] += M[j][i] * dh[j];
                }
            }
            restrict_add<D>(Ri, f, fi, acc + n, NM);
            restrict_add<D>(Rj, g, fj, acc + n, NM);
        }
    }
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
    const size_t sm = (size_t)c.td.max_tv * D * sizeof(T);
    T *contrib = static_cast<T *>(pd.contrib), *blk = static_cast<T *>(pd.blk);
    if (c.muscle)
        k_asm_elem<T, D, true><<<c.td.n_tiles, c.threads, sm, s>>>(c.td, er, ph, u, pd.cpos, contrib);
    else
        k_asm_elem<T, D, false><<<c.td.n_tiles, c.threads, sm, s>>>(c.td, er, ph, u, pd.cpos, contrib);
    k_asm_edge<T, D><<<(unsigned)((pd.n_edges + 255) / 256), 256, 0, s>>>(pd.n_edges, pd.edge_ptr, contrib, blk);
    const dim3 gs((unsigned)pd.n_chunks, pd.tpr ? (unsigned)((pd.max_entries + 255) / 256) : 1u);
    k_asm_slice<T, D><<<gs, 256, 0, s>>>(pd.n_edges, pd.chunk_ent, pd.ent_idx, pd.ent_edge, blk,
                                                           pd.slices);
    const int n = pd.n_cta * pd.ns;
    k_asm_slots<T, D><<<(n + 255) / 256, 256, 0, s>>>(n, pd.slot_gid, pd.grp_agg, pd.agg_ref, pd.inv_len, c.vd, ph,
                                                      u64, pd.pos4, static_cast<T *>(pd.diag2));
    c.n_launch += 4;
    if (!coarse) return;
    cudaMemsetAsync(pd.E, 0, sizeof(float) * pd.n_coarse * pd.n_coarse, s);
    k_coarse_item<T, D><<<pd.n_citems, 128, 0, s>>>(pd, blk, static_cast<const T *>(pd.diag2));
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
