// Device functions of the assembly shared by the kernels of one mesh
// (cg_assemble.cu) and the batched solver (batched_kernel.cuh): an element's
// edge blocks, a slot's vertex data, and the terms of the coarse matrix.
#pragma once

#include <cstdint>

#include "cg_pcg.h"
#include "elem_math.cuh"

namespace softsim {

// A pair's block K into its contribution slot (w: slot | kCgTransposed).
template <typename T, int D>
__device__ __forceinline__ void store_block(T *contrib, uint32_t w, const T K[D][D])
{
    T *out = contrib + (int64_t)(w & ~kCgTransposed) * (D * D);
    const bool tr = (w & kCgTransposed) != 0;
    if constexpr (sizeof(T) == 4 && D == 2) {
        *reinterpret_cast<float4 *>(out) = make_float4(K[0][0], tr ? K[1][0] : K[0][1], tr ? K[0][1] : K[1][0], K[1][1]);
        return;
    }
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
        for (int j = 0; j < D; ++j) out[i * D + j] = tr ? K[j][i] : K[i][j];
}

// Blocks of the element's corner pairs (2D: 3, 3D: 6), each to emit(pair, K); W
// is scaled, f is used by the spring muscle only.
template <typename T, int D, typename Emit>
__device__ __forceinline__ void elem_blocks(const T B[D][D], const T gv[D], const T f[D], T W, T aval, const T Du[D][D],
                                            bool spring, int log_mode, T mu, T lam, T kk, Emit emit)
{
    T F[D][D], C[D][D];
    mul<T, D>(Du, B, F, true);
    cof<T, D>(F, C);
    const T J = detF<T, D>(F, C);
    T l, cc, cp;
    log_terms<T>(log_mode, mu, lam, J, l, cc, cp);
    T c1 = kk * aval, c2 = T(0), q[D];
    if (spring) {
        T s2 = T(0);
#pragma unroll
        for (int i = 0; i < D; ++i) {
            T s = f[i];
#pragma unroll
            for (int k = 0; k < D; ++k) s += Du[i][k] * gv[k];
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
        gam[k + 1] = gv[k];
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
            if (spring) {
                const T m = c2 * W * gam[a] * gam[b];
#pragma unroll
                for (int i = 0; i < D; ++i)
#pragma unroll
                    for (int j = 0; j < D; ++j) K[i][j] += m * q[i] * q[j];
            }
            emit(pair, K);
        }
}

// Slot k: the arm of the rigid rotations about the aggregate's reference
// vertex in the current shape, and the vertex diagonal (inertia + friction,
// contact curvature), formed in FP64 as in the HVP kernels.
template <typename T, int D>
__device__ __forceinline__ void slot_data(int k, const PcgDev &pd, const VertDev &vd, const Phys &ph, const double *u)
{
    const float inv_len = pd.inv_len;
    T *diag2 = static_cast<T *>(pd.diag2);
    const int64_t v = pd.slot_gid[k];
    const int agg = pd.grp_agg[k >> 5];
    float4 o = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(agg | 1 << 30));
    T dh = T(0), dy = T(0);
    if (v >= 0) {
        const int64_t r = pd.agg_ref[agg];
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
    pd.pos4[k] = o;
    diag2[2 * k] = dh;
    diag2[2 * k + 1] = dy;
}

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

// Adds entry q of a coarse item (a slot, or an edge of pd.seg_edge) to the block acc.
template <typename T, int D>
__device__ __forceinline__ void coarse_add(const PcgDev &pd, int kind, int q, float *acc)
{
    constexpr int NM = D == 3 ? 6 : 3;
    const T *blk = static_cast<const T *>(pd.blk), *diag2 = static_cast<const T *>(pd.diag2);
    if (kind == CK_VERT) {
        const float4 R = pd.pos4[q];
        if (__float_as_int(R.w) >> 30) return;
        const float dh = (float)diag2[2 * q], dy = (float)diag2[2 * q + 1];
#pragma unroll
        for (int n = 0; n < NM; ++n) {
            float z[D];
            rigid_mode<D>(n, R, z);
#pragma unroll
            for (int c = 0; c < D; ++c) z[c] *= c == 1 ? dy : dh;
            restrict_add<D>(R, z, 1.0f, acc + n, NM);
        }
        return;
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

}  // namespace softsim
