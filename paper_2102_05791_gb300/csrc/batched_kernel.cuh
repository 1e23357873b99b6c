// Batched persistent solver, device side (see batched.cu): a team of CTAs -- one
// CTA, or one thread-block cluster -- runs a mesh's whole rollout and its
// backward pass.
//
// What bounds it: the chain of CG iterations of the largest mesh, and the FP64
// passes (GB300's FP64 rate is 1/64 of FP32).  A CG solve therefore runs on the
// assembled edge blocks with the two-level preconditioner of cg_pcg_device.cuh,
// the blocks kept in the team's shared memory: an iteration takes about 4.3 us
// plus 6.4 ns per vertex on one CTA (24 us at 2,100 triangles when every
// iteration gathered elements and corners through L2), and there are half as
// many.  256 bodies of 200 to 8,000 triangles, 4 steps and back: 225 -> 60 ms;
// 12 such bodies, 6 steps, on clusters: 230 -> 23 ms.
// Spills cost much here (226 KB of shared memory leave the L1 28 KB): per-slot
// addresses are looked up in the plan where they are used.  All passes are
// spread over the team's threads; between them the team synchronises (block or
// cluster barrier) and sums in a fixed order, so a result depends on the team's
// size and thread count only, not on which team takes the mesh.
#pragma once

#include <cstdint>

#include "cg_blocks.cuh"
#include "cg_pcg_device.cuh"
#include "elem_math.cuh"
#include "internal.h"
#include "softsim.h"

namespace softsim {

struct BatchDev {
    int M = 0, dim = 0;
    const int64_t *voff = nullptr, *eoff = nullptr;  // [M+1]
    const int32_t *order = nullptr;                  // [M] processing order
    const double *X = nullptr, *mass = nullptr;      // [V][d], [V]
    const uint8_t *fixed = nullptr;                  // [V]
    const int32_t *conn = nullptr;                   // [E][d+1] mesh-local vertex ids
    const int64_t *vinc_ptr = nullptr;               // [V+1]
    const int32_t *vinc = nullptr;                   // [E*(d+1)] mesh-local corner ids (elem*(d+1)+corner)
    const float *e32 = nullptr;                      // SoA fields over E
    const double *e64 = nullptr;
    int64_t estride = 0;
    const double *mu = nullptr, *lam = nullptr;      // [M]
    double k = 0, grav = 0, kc = 0, dt = 0;
    double kf = 0, feps = 0;  // ground friction k_f and its height; kf == 0: off
    float k_f = 0, dt2_f = 0;  // FP32 copies of k and dt^2
    int cpow = 3, log_mode = 0, muscle = 0;
    double newton_rtol = 1e-8, adj_rtol = 1e-6;
    int max_newton = 100, max_cg = 500, max_adj_cg = 2000, max_ls = 30;
    // workspace [V][d]
    double *u = nullptr, *uhat = nullptr, *g = nullptr, *w64 = nullptr, *r64 = nullptr, *Hx = nullptr,
           *lacc = nullptr, *xbar = nullptr, *vbar = nullptr;
    double *fw = nullptr, *u0 = nullptr;  // friction: [V] 2 k_f ReLU(eps - y0), [V][d] x0 - X (kf > 0 only)
    float *u32 = nullptr, *d = nullptr, *r = nullptr, *p = nullptr, *Ap = nullptr;
    // FP32 HVP inputs fixed during one CG solve (no FP64 arithmetic or
    // conversion inside the CG loop; GB300's FP64 rate is 1/64 of FP32):
    float *a32 = nullptr;   // [E] the step's activations
    float *dg32 = nullptr;  // [V][2] vertex diagonal: horizontal (m + fw), vertical (m + h^2 contact'')
    float *c32 = nullptr;   // corners [E*(d+1)][d]
    double *c64 = nullptr;
    const PcgDev *pcg = nullptr;  // [M] plan of each mesh's CG solves (n_cta = 0: the mesh does not fit it)
    int team = 1, n_big = 0;      // the first n_big meshes of the order go to teams of `team` CTAs, the others to one CTA each
    int *counter = nullptr;       // [2] meshes taken so far, of the large and of the others
    int *mstat = nullptr;   // [M][4]: status, newton iters, cg iters fwd, cg iters adj
    double *mgrad = nullptr;  // [M][3]: dL/dmu, dL/dlambda, dL/dk of each mesh over the rollout
};

struct Mesh {
    int64_t v0, e0;
    int nv, ne;
    double mu, lam;
    float mu_f, lam_f;
    bool planned;         // its CG solves have a plan (else they run matrix-free)
};

namespace {

// Dynamic shared memory: the plan's layout (PcgSmem), then the mesh's PcgDev.
// Referred to by name everywhere, so that it is addressed as shared memory also
// in functions that are not inlined.
extern __shared__ __align__(128) unsigned char batch_smem[];
__device__ __forceinline__ const PcgDev &plan() { return *reinterpret_cast<const PcgDev *>(batch_smem + kBatchPlanAt); }

// The CTAs that share a mesh: barrier, fixed-order sums, and the thread's share of a loop.
struct Team {
    int rank, size, tid, stride;
    double *red;          // [33] block sums
    double (*slot)[16];   // [2][16] the CTAs' sums, two buffers in turn
    int par;
    __device__ __forceinline__ void sync() const
    {
        if (size == 1)
            __syncthreads();
        else
            cluster_sync();
    }
    // Sum of every thread's v, the same in every thread (also a barrier).
    __device__ double sum(double v)
    {
        v = warp_sum(v);
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
        __syncthreads();
        if (lane == 0) red[w] = v;
        __syncthreads();
        if (w == 0) {
            double t = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
            t = warp_sum(t);
            if (size == 1) {
                if (lane == 0) red[32] = t;
            } else {
                t = __shfl_sync(0xffffffffu, t, 0);
                if (lane < size) st_dsmem(&slot[par][rank], (uint32_t)lane, t);
            }
        }
        if (size == 1) {
            __syncthreads();
            return red[32];
        }
        cluster_sync();
        double t = 0.0;
        for (int k = 0; k < size; ++k) t += slot[par][k];
        par ^= 1;
        return t;
    }
};

template <typename T, int D>
__device__ __forceinline__ void load_elem(const T *ed, int64_t stride, int64_t e, T B[D][D], T gv[D], T &W, T f[D])
{
#pragma unroll
    for (int i = 0; i < D; ++i)
#pragma unroll
        for (int j = 0; j < D; ++j) B[i][j] = ed[(FI<D>::B + i * D + j) * stride + e];
#pragma unroll
    for (int i = 0; i < D; ++i) {
        gv[i] = ed[(FI<D>::G + i) * stride + e];
        f[i] = ed[(FI<D>::F + i) * stride + e];
    }
    W = ed[FI<D>::W * stride + e];
}

// Edge matrix of a vertex field for element e of mesh m (field indexed globally).
template <typename T, typename S, int D>
__device__ __forceinline__ void edge_of(const S *x, const Mesh &m, const int lid[D + 1], T E[D][D])
{
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const T x0 = T(x[(m.v0 + lid[0]) * D + i]);
#pragma unroll
        for (int k = 0; k < D; ++k) E[i][k] = T(x[(m.v0 + lid[k + 1]) * D + i]) - x0;
    }
}

template <int D>
__device__ __forceinline__ void elem_ids(const BatchDev &b, int64_t e, int lid[D + 1])
{
#pragma unroll
    for (int k = 0; k <= D; ++k) lid[k] = b.conn[e * (D + 1) + k];
}

// Sum of the corners of mesh m touching local vertex lv (fixed order).
template <typename T, int D>
__device__ __forceinline__ void corner_sum(const BatchDev &b, const Mesh &m, const T *c, int lv, T acc[D])
{
#pragma unroll
    for (int q = 0; q < D; ++q) acc[q] = T(0);
    const int64_t v = m.v0 + lv;
    for (int64_t s = b.vinc_ptr[v]; s < b.vinc_ptr[v + 1]; ++s) {
        const int64_t base = (m.e0 * (D + 1) + b.vinc[s]) * D;
#pragma unroll
        for (int q = 0; q < D; ++q) acc[q] += c[base + q];
    }
}

template <typename T, int D>
__device__ __forceinline__ void put_corners(T *c, int64_t e, const T G[D][D])
{
#pragma unroll
    for (int i = 0; i < D; ++i) {
        T s = T(0);
#pragma unroll
        for (int j = 0; j < D; ++j) {
            c[(e * (D + 1) + j + 1) * D + i] = G[i][j];
            s += G[i][j];
        }
        c[(e * (D + 1)) * D + i] = -s;
    }
}

__device__ __forceinline__ double contact_d1(double y, double kc, int p)
{
    const double pen = y < 0.0 ? -y : 0.0;
    return pen > 0.0 ? -p * kc * (p == 2 ? pen : pen * pen) : 0.0;
}
__device__ __forceinline__ double contact_d2(double y, double kc, int p)
{
    const double pen = y < 0.0 ? -y : 0.0;
    return pen > 0.0 ? p * (p - 1) * kc * (p == 2 ? 1.0 : pen) : 0.0;
}

// ---------------------------------------------------------------- passes (team-wide)

// Muscle energy density from |F f|^2: contractile (k/2) a |F f|^2 or the
// active spring (k/2)(|F f|/a - 1)^2.
__device__ __forceinline__ double muscle_psi(const BatchDev &b, double a, double Ff2)
{
    if (!b.muscle) return 0.5 * b.k * a * Ff2;
    const double r = sqrt(Ff2) / a - 1.0;
    return 0.5 * b.k * r * r;
}

// FP64 gradient of the incremental potential at u; returns |g|^2 over free entries.
template <int D>
__device__ __noinline__ double grad_pass(const BatchDev &b, const Mesh &m, Team &tm, const double *a_t)
{
    const double s_el = b.dt * b.dt;
    for (int le = tm.tid; le < m.ne; le += tm.stride) {
        const int64_t e = m.e0 + le;
        int lid[D + 1];
        elem_ids<D>(b, e, lid);
        double B[D][D], gv[D], W, f[D], Du[D][D], F[D][D], C[D][D];
        load_elem<double, D>(b.e64, b.estride, e, B, gv, W, f);
        edge_of<double, double, D>(b.u, m, lid, Du);
        mul<double, D>(Du, B, F, true);
        cof<double, D>(F, C);
        const double J = detF<double, D>(F, C);
        double l, cc, cp;
        log_terms<double>(b.log_mode, m.mu, m.lam, J, l, cc, cp);
        double Ff[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < D; ++q) s += F[i][q] * f[q];
            Ff[i] = s;
        }
        double ka = b.k * a_t[e];  // dpsi_m/dq = ka q
        if (b.muscle) {
            double s2 = 0.0, c2;
#pragma unroll
            for (int i = 0; i < D; ++i) s2 += Ff[i] * Ff[i];
            spring_terms<double>(W != 0.0, b.k, a_t[e], sqrt(s2), ka, c2);
        }
        double G[D][D];
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) {
                double s = 0.0;
#pragma unroll
                for (int q = 0; q < D; ++q) s += (m.mu * F[i][q] + cc * C[i][q]) * B[j][q];
                G[i][j] = s_el * W * (s + ka * Ff[i] * gv[j]);
            }
        put_corners<double, D>(b.c64, e, G);
    }
    tm.sync();
    double g2 = 0.0;
    for (int lv = tm.tid; lv < m.nv; lv += tm.stride) {
        const int64_t v = m.v0 + lv;
        double acc[D];
        corner_sum<double, D>(b, m, b.c64, lv, acc);
        const double mass = b.mass[v];
        const double y = b.X[v * D + 1] + b.u[v * D + 1];
        acc[1] += s_el * (mass * b.grav + contact_d1(y, b.kc, b.cpow));
#pragma unroll
        for (int q = 0; q < D; ++q) acc[q] += mass * (b.u[v * D + q] - b.uhat[v * D + q]);
        if (b.fw) {
            const double fv = b.fw[v];
#pragma unroll
            for (int q = 0; q < D; ++q)
                if (q != 1) acc[q] += fv * (b.u[v * D + q] - b.u0[v * D + q]);
        }
        const bool fx = b.fixed[v] != 0;
#pragma unroll
        for (int q = 0; q < D; ++q) {
            const double o = fx ? 0.0 : acc[q];
            b.g[v * D + q] = o;
            g2 += o * o;
        }
    }
    return tm.sum(g2);
}

// FP64 incremental potential at u + t dir (dir may be null); returns E and the
// sum of |terms| through S.
template <int D>
__device__ __noinline__ double energy_pass(const BatchDev &b, const Mesh &m, Team &tm, const double *a_t, const double *dir, double t,
                              double *S)
{
    const double s_el = b.dt * b.dt;
    double E = 0.0, A = 0.0;
    for (int le = tm.tid; le < m.ne; le += tm.stride) {
        const int64_t e = m.e0 + le;
        int lid[D + 1];
        elem_ids<D>(b, e, lid);
        double B[D][D], gv[D], W, f[D], Du[D][D], Dd[D][D], F[D][D], C[D][D];
        load_elem<double, D>(b.e64, b.estride, e, B, gv, W, f);
        edge_of<double, double, D>(b.u, m, lid, Du);
        if (dir) {
            edge_of<double, double, D>(dir, m, lid, Dd);
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int q = 0; q < D; ++q) Du[i][q] += t * Dd[i][q];
        }
        mul<double, D>(Du, B, F, true);
        cof<double, D>(F, C);
        const double J = detF<double, D>(F, C);
        double I1 = 0.0, Ff2 = 0.0;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            double ff = 0.0;
#pragma unroll
            for (int q = 0; q < D; ++q) {
                I1 += F[i][q] * F[i][q];
                ff += F[i][q] * f[q];
            }
            Ff2 += ff * ff;
        }
        double l;
        if (b.log_mode == 0)
            l = J > 0.0 ? log(J) : 0.0;
        else
            l = (J - 1.0) - 0.5 * (J - 1.0) * (J - 1.0);
        double w = s_el * W *
                   (0.5 * m.mu * (I1 - D) - m.mu * l + 0.5 * m.lam * l * l + muscle_psi(b, a_t[e], Ff2));
        if (b.log_mode == 0 && J <= 0.0) w = INFINITY;  // a NaN J (non-finite input) stays NaN
        E += w;
        A += fabs(w);
    }
    for (int lv = tm.tid; lv < m.nv; lv += tm.stride) {
        const int64_t v = m.v0 + lv;
        const double mass = b.mass[v];
        double in = 0.0, yv = 0.0;
#pragma unroll
        for (int q = 0; q < D; ++q) {
            const double uq = b.u[v * D + q] + (dir ? t * dir[v * D + q] : 0.0);
            const double rq = uq - b.uhat[v * D + q];
            in += 0.5 * mass * rq * rq;
            if (q == 1) yv = b.X[v * D + 1] + uq;
            else if (b.fw) {
                const double rf = uq - b.u0[v * D + q];
                in += 0.5 * b.fw[v] * rf * rf;
            }
        }
        const double pen = yv < 0.0 ? -yv : 0.0;
        const double w = s_el * (mass * b.grav * yv + b.kc * (b.cpow == 2 ? pen * pen : pen * pen * pen));
        E += w + in;
        A += fabs(w) + in;
    }
    const double Et = tm.sum(E);
    *S = tm.sum(A);
    return Et;
}

// y = (M + h^2 H(u)) v with pinned rows/columns dropped; returns v.y (FP64
// sum, of FP32 terms per thread for T = float).
template <typename T, int D>
__device__ __noinline__ double hvp_pass(const BatchDev &b, const Mesh &m, Team &tm, const double *a_t, const T *us, const T *v, T *y, T *c,
                           const T *ed)
{
    constexpr bool F32 = sizeof(T) == 4;
    const T s_el = pick<T>(b.dt * b.dt, b.dt2_f);
    const T mu = pick<T>(m.mu, m.mu_f), lam = pick<T>(m.lam, m.lam_f);
    const T kk = pick<T>(b.k, b.k_f);
    for (int le = tm.tid; le < m.ne; le += tm.stride) {
        const int64_t e = m.e0 + le;
        int lid[D + 1];
        elem_ids<D>(b, e, lid);
        const T ae = F32 ? T(b.a32[e]) : T(a_t[e]);
        T B[D][D], gv[D], W, f[D], Du[D][D], Dv[D][D], F[D][D], dF[D][D], C[D][D], dC[D][D];
        load_elem<T, D>(ed, b.estride, e, B, gv, W, f);
        edge_of<T, T, D>(us, m, lid, Du);
        T vv[D + 1][D];
#pragma unroll
        for (int k = 0; k <= D; ++k) {
            const int64_t gvid = m.v0 + lid[k];
            const bool fx = b.fixed[gvid] != 0;
#pragma unroll
            for (int q = 0; q < D; ++q) vv[k][q] = fx ? T(0) : v[gvid * D + q];
        }
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int k = 0; k < D; ++k) Dv[i][k] = vv[k + 1][i] - vv[0][i];
        mul<T, D>(Du, B, F, true);
        mul<T, D>(Dv, B, dF, false);
        cof<T, D>(F, C);
        dcof<T, D>(F, dF, dC);
        const T J = detF<T, D>(F, C);
        T dJ = T(0);
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) dJ += C[i][j] * dF[i][j];
        T l, cc, cp;
        log_terms<T>(b.log_mode, mu, lam, J, l, cc, cp);
        const T ka = F32 ? kk * ae : T(b.k * a_t[e]);
        T dvg[D];  // (d2psi_m/dq2) dq with dq = Dv g
#pragma unroll
        for (int i = 0; i < D; ++i) {
            T s = T(0);
#pragma unroll
            for (int k = 0; k < D; ++k) s += Dv[i][k] * gv[k];
            dvg[i] = s;
        }
        if (b.muscle) {  // spring, q = F f = f + Du g
            T q[D], s2 = T(0), qdq = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                T s = f[i];
#pragma unroll
                for (int k = 0; k < D; ++k) s += Du[i][k] * gv[k];
                q[i] = s;
                s2 += s * s;
                qdq += s * dvg[i];
            }
            T c1, c2;
            spring_terms<T>(W != T(0), kk, ae, sqrt(s2), c1, c2);
#pragma unroll
            for (int i = 0; i < D; ++i) dvg[i] = c1 * dvg[i] + c2 * qdq * q[i];
        } else {
#pragma unroll
            for (int i = 0; i < D; ++i) dvg[i] *= ka;
        }
        T G[D][D];
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) {
                T s = T(0);
#pragma unroll
                for (int k = 0; k < D; ++k) s += (mu * dF[i][k] + cp * dJ * C[i][k] + cc * dC[i][k]) * B[j][k];
                G[i][j] = s_el * W * (s + dvg[i] * gv[j]);
            }
        put_corners<T, D>(c, e, G);
    }
    tm.sync();
    T dot = T(0);
    for (int lv = tm.tid; lv < m.nv; lv += tm.stride) {
        const int64_t vg = m.v0 + lv;
        T acc[D];
        corner_sum<T, D>(b, m, c, lv, acc);
        const bool fx = b.fixed[vg] != 0;
        T dh, dy;  // diagonal: horizontal axes (inertia + friction), y (inertia + contact)
        if constexpr (F32) {
            dh = b.dg32[2 * vg];
            dy = b.dg32[2 * vg + 1];
        } else {
            const double mass = b.mass[vg];
            const double yy = b.X[vg * D + 1] + us[vg * D + 1];
            dh = b.fw ? mass + b.fw[vg] : mass;  // friction stiffens the horizontal axes
            dy = mass + b.dt * b.dt * contact_d2(yy, b.kc, b.cpow);
        }
        T vv[D];
#pragma unroll
        for (int q = 0; q < D; ++q) vv[q] = fx ? T(0) : v[vg * D + q];
#pragma unroll
        for (int q = 0; q < D; ++q) {
            const T o = fx ? T(0) : acc[q] + (q == 1 ? dy : dh) * vv[q];
            y[vg * D + q] = o;
            dot += vv[q] * o;
        }
    }
    if constexpr (F32)
        return tm.sum((double)dot);
    else
        return tm.sum(dot);
}

// CG on (M + h^2 H) d = rhs (FP64 rhs, FP32 vectors), matrix-free, for meshes
// whose parts do not fit the team's shared memory; returns iterations.
template <int D>
__device__ __noinline__ int cg_matrix_free(const BatchDev &b, const Mesh &m, Team &tm, const double *a_t, const double *rhs, double rtol, int max_it)
{
    const int64_t o = m.v0 * D, n = (int64_t)m.nv * D;
    float rr32 = 0.0f;
    for (int64_t i = tm.tid; i < n; i += tm.stride) {
        const float ri = (float)rhs[o + i];
        b.r[o + i] = ri;
        b.p[o + i] = ri;
        b.d[o + i] = 0.0f;
        rr32 += ri * ri;
    }
    double rr = tm.sum((double)rr32);
    const double tol2 = rtol * rtol * rr;
    int k = 0;
    for (; k < max_it; ++k) {
        if (!(rr > tol2)) break;
        const double pAp = hvp_pass<float, D>(b, m, tm, a_t, b.u32, b.p, b.Ap, b.c32, b.e32);
        if (!(pAp > 0.0)) {
            if (k == 0)
                for (int64_t i = tm.tid; i < n; i += tm.stride) b.d[o + i] = b.p[o + i];
            tm.sync();
            break;
        }
        const float alpha = (float)(rr / pAp);
        float rn32 = 0.0f;
        for (int64_t i = tm.tid; i < n; i += tm.stride) {
            b.d[o + i] += alpha * b.p[o + i];
            const float ri = b.r[o + i] - alpha * b.Ap[o + i];
            b.r[o + i] = ri;
            rn32 += ri * ri;
        }
        const double rn = tm.sum((double)rn32);
        const float beta = (float)(rn / rr);
        rr = rn;
        for (int64_t i = tm.tid; i < n; i += tm.stride) b.p[o + i] = b.r[o + i] + beta * b.p[o + i];
        tm.sync();
    }
    return k;
}

// The edge blocks, vertex data and (with coarse) coarse inverse of
// M + h^2 H at the current u, into the team's slices.
template <int D>
__device__ __noinline__ void assemble(const BatchDev &b, const Mesh &m, Team &tm, bool coarse)
{
    constexpr int NP = (D + 1) * D / 2, DD = D * D, NM = D == 3 ? 6 : 3;
    const PcgDev &pd = plan();
    float *contrib = static_cast<float *>(pd.contrib), *blk = static_cast<float *>(pd.blk);
    const int lane = threadIdx.x & 31, wrp = threadIdx.x >> 5, nw = blockDim.x >> 5, N = pd.n_coarse;
    for (int le = tm.tid; le < m.ne; le += tm.stride) {
        const int64_t e = m.e0 + le;
        int lid[D + 1];
        elem_ids<D>(b, e, lid);
        float B[D][D], gv[D], W, f[D], Du[D][D];
        load_elem<float, D>(b.e32, b.estride, e, B, gv, W, f);
        edge_of<float, float, D>(b.u32, m, lid, Du);
        elem_blocks<float, D>(B, gv, f, W * b.dt2_f, b.a32[e], Du, b.muscle != 0, b.log_mode, m.mu_f, m.lam_f, b.k_f,
                              [&](int pair, const float K[D][D]) {
                                  store_block<float, D>(contrib, pd.cpos[(int64_t)le * NP + pair], K);
                              });
    }
    {
        VertDev vd;
        vd.nv = m.nv;
        vd.X = b.X + m.v0 * D;
        vd.mass = b.mass + m.v0;
        vd.fixed = b.fixed + m.v0;
        Phys ph;
        ph.kc = b.kc;
        ph.cpow = b.cpow;
        ph.dyn = 1;
        ph.s_el = b.dt * b.dt;
        ph.contact = b.kc > 0.0;
        ph.fw = b.fw ? b.fw + m.v0 : nullptr;
        for (int k = tm.tid; k < pd.n_cta * pd.ns; k += tm.stride) slot_data<float, D>(k, pd, vd, ph, b.u + m.v0 * D);
    }
    if (coarse)
        for (int k = tm.tid; k < N * N; k += tm.stride) pd.E[k] = 0.0f;
    tm.sync();
    for (int e = tm.tid; e < (int)pd.n_edges; e += tm.stride) {
        float acc[DD];
#pragma unroll
        for (int k = 0; k < DD; ++k) acc[k] = 0.0f;
        for (int q = pd.edge_ptr[e]; q < pd.edge_ptr[e + 1]; ++q)
#pragma unroll
            for (int k = 0; k < DD; ++k) acc[k] += contrib[(int64_t)q * DD + k];
#pragma unroll
        for (int k = 0; k < DD; ++k) blk[k * pd.n_edges + e] = acc[k];
    }
    tm.sync();
    const PcgSmem L(D, sizeof(float), pd.ns, pd.max_halo, pd.max_items, N, pd.n_meta, 0);
    if (coarse) {
        for (int i = tm.rank * nw + wrp; i < pd.n_citems; i += tm.size * nw) {  // a warp per partial sum
            float acc[NM * NM];
#pragma unroll
            for (int k = 0; k < NM * NM; ++k) acc[k] = 0.0f;
            for (int q = pd.citem_begin[i] + lane; q < pd.citem_end[i]; q += 32)
                coarse_add<float, D>(pd, pd.citem_kind[i], q, acc);
#pragma unroll
            for (int k = 0; k < NM * NM; ++k) {
                const float v = warp_all(acc[k]);
                if (lane == 0) pd.cpart[(int64_t)i * (NM * NM) + k] = v;
            }
        }
        tm.sync();
        for (int w = tm.tid; w < pd.n_ctgts * NM * NM; w += tm.stride) {
            const int t = w / (NM * NM), k = w - t * (NM * NM), r = k / NM, c = k % NM;
            const int I = pd.ctgt_i[t], J = pd.ctgt_j[t];
            float s = 0.0f, st = 0.0f;
            for (int q = pd.ctgt_ptr[t]; q < pd.ctgt_ptr[t + 1]; ++q) {
                s += pd.cpart[(int64_t)q * (NM * NM) + k];
                st += pd.cpart[(int64_t)q * (NM * NM) + c * NM + r];
            }
            if (I == J) s = 0.5f * (s + st);
            pd.E[(size_t)(I * NM + r) * N + J * NM + c] = s;
            pd.E[(size_t)(J * NM + c) * N + I * NM + r] = s;
        }
        tm.sync();
        if (tm.rank == 0) {
            // Gauss-Jordan in shared memory (batch_plan_fits has its size), scaled to unit diagonal (as k_coarse_invert)
            float *A = reinterpret_cast<float *>(batch_smem + L.ring), *scale = A + N * N, *row = scale + N, *col = row + N;
            for (int k = threadIdx.x; k < N; k += blockDim.x) {
                const float d = pd.E[(size_t)k * N + k];
                scale[k] = d > 0.0f ? rsqrtf(d) : 0.0f;
            }
            __syncthreads();
            for (int r = wrp; r < N; r += nw)
                for (int c = lane; c < N; c += 32) A[r * N + c] = pd.E[(size_t)r * N + c] * scale[r] * scale[c];
            for (int k = 0; k < N; ++k) {
                __syncthreads();
                for (int q = threadIdx.x; q < N; q += blockDim.x) {
                    row[q] = A[k * N + q];
                    col[q] = A[q * N + k];
                }
                __syncthreads();
                const float p = row[k], ip = p > 1e-5f ? __frcp_rn(p) : 0.0f;
                for (int r = wrp; r < N; r += nw)
                    for (int c = lane; c < N; c += 32) {
                        const float rk = c == k ? ip : row[c] * ip;
                        A[r * N + c] = r == k ? rk : fmaf(-col[r], rk, c == k ? 0.0f : A[r * N + c]);
                    }
            }
            __syncthreads();
            for (int r = wrp; r < N; r += nw)
                for (int c = lane; c < N; c += 32) pd.Einv[(size_t)r * N + c] = A[r * N + c] * scale[r] * scale[c];
        }
        tm.sync();
    }
    // this CTA's slice: the first steps of its rows to shared memory, the rest beside the plan
    const int c0 = pd.chunk_ptr[tm.rank];
    for (int part = 0; part < 2; ++part) {
        const int e0 = pd.chunk_ent[c0 + part], n = pd.chunk_ent[c0 + part + 1] - e0;
        unsigned char *base = part ? pd.slices + (size_t)e0 * (4 + DD * sizeof(float)) : batch_smem + L.ring;
        uint32_t *idx = reinterpret_cast<uint32_t *>(base);
        float *val = reinterpret_cast<float *>(base + (size_t)n * 4);
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const uint32_t w = pd.ent_edge[e0 + k];
            const int64_t e = w & ~kCgTransposed;
            const bool pad = w == kCgPadEntry, tr = (w & kCgTransposed) != 0;
            idx[k] = pd.ent_idx[e0 + k];
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j)
                    val[(i * D + j) * n + k] = pad ? 0.0f : blk[(tr ? j * D + i : i * D + j) * pd.n_edges + e];
        }
    }
    tm.sync();
}

template <int D, int VPT>
__device__ __noinline__ int cg_assembled(const double *rhs, double rhs2, float *d, double rtol, int max_it, int rank,
                                         bool new_coarse)
{
    __shared__ int never_bad;  // the slice is in place: no copy to wait for
    if (threadIdx.x == 0) never_bad = 0;
    Slice sl = pcg_slice<D, float, true>(plan(), rank, false, batch_smem, 0, &never_bad);
    return pcg_run<float, D, VPT, true, false>(plan(), sl, rank, batch_smem, rhs, 1.0, rhs2, d, rtol, max_it,
                                               new_coarse).iter;
}

// CG on (M + h^2 H) d = rhs (|rhs|^2 = rhs2) with the assembled operator, or
// matrix-free; returns iterations.
template <int D>
__device__ int cg_solve(const BatchDev &b, const Mesh &m, Team &tm, const double *a_t, const double *rhs, double rhs2,
                        double rtol, int max_it, bool new_coarse)
{
    if (!m.planned) return cg_matrix_free<D>(b, m, tm, a_t, rhs, rtol, max_it);
    const int bt = blockDim.x;
    const double *r = rhs + m.v0 * D;
    float *d = b.d + m.v0 * D;
    // the same branch in every CTA of the team: by the largest part
    const int vpt = (plan().ns + bt - 1) / bt;
    const int it = vpt <= 1   ? cg_assembled<D, 1>(r, rhs2, d, rtol, max_it, tm.rank, new_coarse)
                   : vpt <= 4 ? cg_assembled<D, 4>(r, rhs2, d, rtol, max_it, tm.rank, new_coarse)
                              : cg_assembled<D, kBatchVpt>(r, rhs2, d, rtol, max_it, tm.rank, new_coarse);
    tm.sync();
    return it;
}

// FP32 state and vertex diagonals of mesh m for the CG solves at the current
// u (the caller synchronises before the next pass reads them).
template <int D>
__device__ void set_fp32_state(const BatchDev &b, const Mesh &m, Team &tm)
{
    const int64_t o = m.v0 * D, n = (int64_t)m.nv * D;
    for (int64_t i = tm.tid; i < n; i += tm.stride) b.u32[o + i] = (float)b.u[o + i];
    for (int lv = tm.tid; lv < m.nv; lv += tm.stride) {
        const int64_t v = m.v0 + lv;
        const double mass = b.mass[v];
        const double yy = b.X[v * D + 1] + b.u[v * D + 1];
        b.dg32[2 * v] = (float)(b.fw ? mass + b.fw[v] : mass);
        b.dg32[2 * v + 1] = (float)(mass + b.dt * b.dt * contact_d2(yy, b.kc, b.cpow));
    }
}

// FP32 activations of mesh m for this step.
__device__ void set_a32(const BatchDev &b, const Mesh &m, Team &tm, const double *a_t)
{
    for (int le = tm.tid; le < m.ne; le += tm.stride) b.a32[m.e0 + le] = (float)a_t[m.e0 + le];
}

// Friction data of a step of mesh m started at x0: u0 = x0 - X and
// fw = 2 k_f ReLU(eps - y0) per vertex.
template <int D>
__device__ void friction_prep(const BatchDev &b, const Mesh &m, Team &tm, const double *x0)
{
    for (int lv = tm.tid; lv < m.nv; lv += tm.stride) {
        const int64_t v = m.v0 + lv;
#pragma unroll
        for (int q = 0; q < D; ++q) b.u0[v * D + q] = x0[v * D + q] - b.X[v * D + q];
        const double r = b.feps - x0[v * D + 1];
        b.fw[v] = r > 0.0 ? 2.0 * b.kf * r : 0.0;
    }
}

// Backward-Euler step of mesh m: x1 = argmin of the incremental potential,
// started from x0; returns the step's status and adds iteration counts.
template <int D>
__device__ int step_forward(const BatchDev &b, const Mesh &m, Team &tm, const double *x0, const double *v0, const double *a_t,
                            double *x1, double *v1, int *newton_it, int *cg_it)
{
    const int64_t o = m.v0 * D, n = (int64_t)m.nv * D;
    for (int64_t i = tm.tid; i < n; i += tm.stride) {
        b.u[o + i] = b.fixed[m.v0 + i / D] ? 0.0 : x0[o + i] - b.X[o + i];
        b.uhat[o + i] = x0[o + i] + b.dt * v0[o + i] - b.X[o + i];
    }
    if (b.fw) friction_prep<D>(b, m, tm, x0);
    set_a32(b, m, tm, a_t);
    tm.sync();
    double S0;
    double gn = sqrt(grad_pass<D>(b, m, tm, a_t));
    double E = energy_pass<D>(b, m, tm, a_t, nullptr, 0.0, &S0);
    const double g0 = gn;
    int status = SIM_ENOTCONVERGED;
    const double eps = 2.220446049250313e-16;
    for (int it = 0;; ++it) {
        if (gn <= b.newton_rtol * g0) {
            status = SIM_OK;
            break;
        }
        if (it >= b.max_newton || !isfinite(gn) || !isfinite(E)) {
            status = (!isfinite(gn) || !isfinite(E)) ? SIM_ENAN : SIM_ENOTCONVERGED;
            break;
        }
        ++*newton_it;
        set_fp32_state<D>(b, m, tm);
        for (int64_t i = tm.tid; i < n; i += tm.stride) b.w64[o + i] = -b.g[o + i];
        tm.sync();
        if (m.planned) assemble<D>(b, m, tm, it == 0);  // the coarse operator of the first step serves the whole solve
        const double eta = fmin(0.5, sqrt(gn / g0));
        *cg_it += cg_solve<D>(b, m, tm, a_t, b.w64, gn * gn, eta, b.max_cg, it == 0);
        double gd = 0.0;
        for (int64_t i = tm.tid; i < n; i += tm.stride) gd += b.g[o + i] * (double)b.d[o + i];
        gd = tm.sum(gd);
        if (!(gd < 0.0)) {
            for (int64_t i = tm.tid; i < n; i += tm.stride) b.d[o + i] = (float)(-b.g[o + i]);
            gd = -gn * gn;
        }
        for (int64_t i = tm.tid; i < n; i += tm.stride) b.r64[o + i] = (double)b.d[o + i];
        tm.sync();
        bool ok = false;
        double t = 1.0, Et = INFINITY, St = 0.0;
        for (int ls = 0; ls < b.max_ls; ++ls) {
            Et = energy_pass<D>(b, m, tm, a_t, b.r64, t, &St);
            if (isfinite(Et) && Et <= E + 1e-4 * t * gd + 64.0 * eps * fmax(S0, St)) {
                ok = true;
                break;
            }
            t *= 0.5;
        }
        if (!ok) {
            status = SIM_ELINESEARCH;
            break;
        }
        for (int64_t i = tm.tid; i < n; i += tm.stride) b.u[o + i] += t * b.r64[o + i];
        tm.sync();
        E = Et;
        S0 = St;
        gn = sqrt(grad_pass<D>(b, m, tm, a_t));
    }
    for (int64_t i = tm.tid; i < n; i += tm.stride) {
        const double xi = b.X[o + i] + b.u[o + i];
        x1[o + i] = xi;
        v1[o + i] = (xi - x0[o + i]) / b.dt;
    }
    tm.sync();
    return status;
}

// Backward of one step at its converged state x1: lambda = (M + h^2 H)^-1
// (xbar + vbar/h) with FP64 refinement, then xbar <- M lambda - vbar/h,
// vbar <- h M lambda, abar_t = -h^2 lambda^T d2E/dx da.
template <int D>
__device__ int step_backward(const BatchDev &b, const Mesh &m, Team &tm, const double *x0, const double *x1, const double *a_t,
                             double *abar_t, int *cg_it, double mat[3])
{
    const int64_t o = m.v0 * D, n = (int64_t)m.nv * D;
    const double h = b.dt;
    if (b.fw) friction_prep<D>(b, m, tm, x0);
    double bn = 0.0;
    set_a32(b, m, tm, a_t);
    for (int64_t i = tm.tid; i < n; i += tm.stride) {
        b.u[o + i] = x1[o + i] - b.X[o + i];
        const double bi = b.fixed[m.v0 + i / D] ? 0.0 : b.xbar[o + i] + b.vbar[o + i] / h;
        b.w64[o + i] = bi;
        b.r64[o + i] = bi;
        b.lacc[o + i] = 0.0;
        bn += bi * bi;
    }
    bn = sqrt(tm.sum(bn));
    set_fp32_state<D>(b, m, tm);
    tm.sync();
    if (m.planned && isfinite(bn)) assemble<D>(b, m, tm, true);
    double rn = bn;
    int status = SIM_ENOTCONVERGED;
    int budget = b.max_adj_cg;
    for (int pass = 0; pass < 12 && isfinite(bn); ++pass) {
        if (rn <= b.adj_rtol * bn || !(rn > 0.0)) {
            status = SIM_OK;
            break;
        }
        if (budget <= 0) break;
        const double rtol = fmax(fmax(b.adj_rtol, 1e-4), 0.5 * b.adj_rtol * bn / rn);
        const int it = cg_solve<D>(b, m, tm, a_t, b.r64, rn * rn, rtol, budget, pass == 0);
        *cg_it += it;
        budget -= it > 0 ? it : 1;
        for (int64_t i = tm.tid; i < n; i += tm.stride) b.lacc[o + i] += (double)b.d[o + i];
        tm.sync();
        hvp_pass<double, D>(b, m, tm, a_t, b.u, b.lacc, b.Hx, b.c64, b.e64);
        double r2 = 0.0;
        for (int64_t i = tm.tid; i < n; i += tm.stride) {
            const double ri = b.w64[o + i] - b.Hx[o + i];
            b.r64[o + i] = ri;
            r2 += ri * ri;
        }
        const double rnew = sqrt(tm.sum(r2));
        if (!isfinite(rnew)) {
            status = SIM_ENAN;
            break;
        }
        if (rnew >= rn) {
            rn = rnew;
            break;
        }
        rn = rnew;
    }
    if (rn <= b.adj_rtol * bn) status = SIM_OK;
    if (!isfinite(bn)) status = SIM_ENAN;  // non-finite right-hand side
    // xbar0 = M lambda - vbar1/h, vbar0 = h M lambda; with friction, plus
    // fw lambda_h on the horizontal axes and 2 k_f [y0 < eps] lambda_h . (x1 - x0)_h on y
    for (int lv = tm.tid; lv < m.nv; lv += tm.stride) {
        const int64_t v = m.v0 + lv;
        const bool fx = b.fixed[v] != 0;
        const double fv = b.fw ? b.fw[v] : 0.0;
        double ysum = 0.0;
#pragma unroll
        for (int q = 0; q < D; ++q) {
            const int64_t i = v * D + q;
            const double l = b.lacc[i];
            const double ml = b.mass[v] * l;
            const double vb = b.vbar[i];
            double xb = ml - vb / h;
            if (q != 1 && fv > 0.0) {
                xb += fv * l;
                ysum += l * (x1[i] - x0[i]);
            }
            b.xbar[i] = fx ? 0.0 : xb;
            b.vbar[i] = fx ? 0.0 : h * ml;
        }
        if (fv > 0.0 && !fx) b.xbar[v * D + 1] += 2.0 * b.kf * ysum;
    }
    // parameter VJP at x1, and this step's material VJPs summed over the mesh:
    // -h^2 W (dP/dtheta) : dF(lambda), dP/dmu = F - l' cof F, dP/dlambda = l l' cof F
    double tmu = 0.0, tlam = 0.0, tk = 0.0;
    for (int le = tm.tid; le < m.ne; le += tm.stride) {
        const int64_t e = m.e0 + le;
        int lid[D + 1];
        elem_ids<D>(b, e, lid);
        double B[D][D], gv[D], W, f[D], Du[D][D], Dl[D][D], F[D][D], dF[D][D], C[D][D];
        load_elem<double, D>(b.e64, b.estride, e, B, gv, W, f);
        edge_of<double, double, D>(b.u, m, lid, Du);
        edge_of<double, double, D>(b.lacc, m, lid, Dl);
        mul<double, D>(Du, B, F, true);
        mul<double, D>(Dl, B, dF, false);
        cof<double, D>(F, C);
        const double J = detF<double, D>(F, C);
        double FdF = 0.0, CdF = 0.0;
#pragma unroll
        for (int i = 0; i < D; ++i)
#pragma unroll
            for (int j = 0; j < D; ++j) {
                FdF += F[i][j] * dF[i][j];
                CdF += C[i][j] * dF[i][j];
            }
        double l, lp;
        if (b.log_mode == 0) {
            l = log(J);
            lp = 1.0 / J;
        } else {
            l = (J - 1.0) - 0.5 * (J - 1.0) * (J - 1.0);
            lp = 2.0 - J;
        }
        const double sW = -h * h * W;
        tmu += sW * (FdF - lp * CdF);
        tlam += sW * l * lp * CdF;
        double dot = 0.0, s2 = 0.0;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            double Ff = 0.0, dFf = 0.0;
#pragma unroll
            for (int q = 0; q < D; ++q) {
                Ff += F[i][q] * f[q];
                dFf += Dl[i][q] * gv[q];
            }
            dot += Ff * dFf;
            s2 += Ff * Ff;
        }
        double kq = b.k;                  // d2psi_m/dq da = kq q
        double ck = a_t[e];               // d2psi_m/dq dk = ck q
        if (b.muscle) {
            const double s = sqrt(s2), ia = 1.0 / a_t[e];
            kq = b.k * (ia * ia - 2.0 * s * ia * ia * ia) / s;
            ck = (s * ia - 1.0) * ia / s;
        }
        abar_t[e] = -h * h * W * kq * dot;
        tk += sW * ck * dot;
    }
    mat[0] += tm.sum(tmu);
    mat[1] += tm.sum(tlam);
    mat[2] += tm.sum(tk);
    tm.sync();
    return status;
}

}  // namespace

// BT threads per CTA (128, 256 or 512), one CTA per SM; b.team CTAs (one
// cluster) per mesh.
template <int D, int BT>
__global__ void __launch_bounds__(BT, 1)
    k_batch_rollout(BatchDev b, int n_steps, const double *__restrict__ a_seq, double *xs, double *vs,
                    const double *__restrict__ xbarT, const double *__restrict__ vbarT, double *__restrict__ abar_seq,
                    int64_t V, int64_t E)
{
    __shared__ double red[33], slot[2][16];
    __shared__ float sm_mesh;  // a mesh number's bits
    Team tm;
    tm.red = red;
    tm.slot = slot;
    tm.par = 0;
    auto form = [&](int size, int rank) {
        tm.size = size;
        tm.rank = rank;
        tm.tid = rank * BT + threadIdx.x;
        tm.stride = size * BT;
    };
    form(b.team, b.team > 1 ? (int)cluster_rank() : 0);
    bool big = b.team > 1;
    tm.sync();
    for (;;) {
        if (tm.tid == 0) {
            const float s = __int_as_float(atomicAdd(b.counter + (big ? 0 : 1), 1) + (big ? 0 : b.n_big));
            if (tm.size == 1)
                sm_mesh = s;
            else
                for (int k = 0; k < tm.size; ++k) st_dsmem(&sm_mesh, (uint32_t)k, s);
        }
        tm.sync();
        const int next = __float_as_int(sm_mesh);
        tm.sync();
        if (big && next >= b.n_big) {  // the large meshes are taken: every CTA for itself from here on
            big = false;
            form(1, 0);
            continue;
        }
        if (next >= b.M) break;
        const int mi = b.order[next];
        Mesh m;
        m.v0 = b.voff[mi];
        m.e0 = b.eoff[mi];
        m.nv = (int)(b.voff[mi + 1] - m.v0);
        m.ne = (int)(b.eoff[mi + 1] - m.e0);
        m.mu = b.mu[mi];
        m.lam = b.lam[mi];
        m.mu_f = (float)m.mu;
        m.lam_f = (float)m.lam;
        for (int k = threadIdx.x; k < (int)(sizeof(PcgDev) / 4); k += BT)
            reinterpret_cast<uint32_t *>(batch_smem + kBatchPlanAt)[k] = reinterpret_cast<const uint32_t *>(b.pcg + mi)[k];
        __syncthreads();
        m.planned = plan().n_cta > 0;
        if (m.planned) pcg_tables<D, float, true>(plan(), tm.rank, false, batch_smem);
        __syncthreads();
        int status = SIM_OK, newton_it = 0, cg_f = 0, cg_a = 0;
        const size_t VD = (size_t)V * D;
        for (int t = 0; t < n_steps; ++t) {
            const int st = step_forward<D>(b, m, tm, xs + t * VD, vs + t * VD, a_seq + (size_t)t * E,
                                                xs + (t + 1) * VD, vs + (t + 1) * VD, &newton_it, &cg_f);
            if (st != SIM_OK) status = st;
        }
        const int64_t o = m.v0 * D, n = (int64_t)m.nv * D;
        for (int64_t i = tm.tid; i < n; i += tm.stride) {
            b.xbar[o + i] = xbarT[o + i];
            b.vbar[o + i] = vbarT[o + i];
        }
        tm.sync();
        double mat[3] = {0.0, 0.0, 0.0};
        for (int t = n_steps - 1; t >= 0; --t) {
            const int st = step_backward<D>(b, m, tm, xs + t * VD, xs + (t + 1) * VD, a_seq + (size_t)t * E,
                                                 abar_seq + (size_t)t * E, &cg_a, mat);
            if (st != SIM_OK && status == SIM_OK) status = st;
        }
        if (tm.tid == 0) {
            b.mgrad[3 * mi + 0] = mat[0];
            b.mgrad[3 * mi + 1] = mat[1];
            b.mgrad[3 * mi + 2] = mat[2];
            b.mstat[4 * mi + 0] = status;
            b.mstat[4 * mi + 1] = newton_it;
            b.mstat[4 * mi + 2] = cg_f;
            b.mstat[4 * mi + 3] = cg_a;
        }
        tm.sync();
    }
}

using BatchKernel = void (*)(BatchDev, int, const double *, double *, double *, const double *, const double *,
                             double *, int64_t, int64_t);
BatchKernel batch_kernel_2d(int threads);
BatchKernel batch_kernel_3d(int threads);

}  // namespace softsim
