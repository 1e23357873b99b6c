// Element kernels: energy, gradient, Hessian-vector product and parameter
// VJP of the neo-Hookean + muscle energy on triangle (D = 2) and tet (D = 3)
// meshes.
//
// Model (Sec. 2, Eq. neohookean-psi; 3D form with I1 - 3):
//   F = Ds Dm^-1 = I + Du Dm^-1 (Du: edge matrix of the displacement u = x - X,
//   which keeps F accurate in FP32), J = det F,
//   Psi = mu/2 (|F|^2 - D) - mu l(J) + lambda/2 l(J)^2,
//   l = log (exact) or q(J) = (J-1) - (J-1)^2/2 (quadratic stand-in),
//   muscle Psi_m = k/2 a |F f|^2 (contractile) or k/2 (|F f|/a - 1)^2 (active
//   spring, Eq. active-spring-potential).
// Writing P_el = mu F + c(J) cof(F) with c = (lambda l - mu) l', the
// differential is dP = mu dF + c'(J) (cof F : dF) cof F + c(J) dcof(F)[dF].
// The element force matrix is G = W dPsi/dF Dm^-T; column j goes to vertex
// j+1 and minus the column sum to vertex 0 (f = -grad E, Eq. f-as-grad; the
// HVP is the paper's Eq. matrix-free-dfdx written out analytically).
//
// Each CTA processes one tile: it stages the tile's vertex values in shared
// memory, evaluates its elements (one thread per element, coalesced SoA
// loads), writes the per-corner results to shared memory, and then one
// thread per tile vertex adds that vertex's corners in a fixed order.
// Vertices shared with other tiles go through halo slots and a finalize
// kernel, so every sum has one fixed order: no float atomics.
#include <cstdio>

#include "internal.h"
#include "reduce.cuh"
#include "tma.cuh"
#include "elem_math.cuh"
#include "grid_sync.cuh"
#include "pdl.cuh"
#include "tile_device.cuh"

namespace softsim {

// Per-vertex potential terms: gravity m g y and ground penalty kc max(0,-y)^p.
__device__ __forceinline__ double pen_pow(double pen, int p) { return p == 2 ? pen * pen : pen * pen * pen; }

// Gradient of one vertex's gravity, contact, inertia and friction added to
// acc; with EN their energy to e[0] and its absolute value to e[1].
template <int D, bool EN>
__device__ __forceinline__ void add_vertex_terms(const VertDev &vd, const Phys &ph, int64_t gid, const double *u,
                                                 const double *__restrict__ uhat, double acc[D], double *e)
{
    const double m = vd.mass[gid];
    const double y = vd.X[gid * D + 1] + u[1];
    const double pen = y < 0.0 ? -y : 0.0;
    const double dcon = pen > 0.0 ? -ph.cpow * ph.kc * (ph.cpow == 2 ? pen : pen * pen) : 0.0;
    acc[1] += ph.s_el * (m * ph.grav + dcon);
    double w = 0.0, in = 0.0;
    if (EN) w = ph.s_el * (m * ph.grav * y + (pen > 0.0 ? ph.kc * pen_pow(pen, ph.cpow) : 0.0));
    if (EN) e[1] += fabs(w);
    if (ph.dyn) {
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const double r = u[c] - uhat[gid * D + c];
            acc[c] += m * r;
            if (EN) in += 0.5 * m * r * r;
        }
        if (ph.fw) {
            const double f = ph.fw[gid];
#pragma unroll
            for (int c = 0; c < D; ++c) {
                if (c == 1) continue;
                const double r = u[c] - ph.u0[gid * D + c];
                acc[c] += f * r;
                if (EN) in += 0.5 * f * r * r;
            }
        }
    }
    if (EN) {
        e[0] += w + in;
        e[1] += in;
    }
}

// ---------------------------------------------------------------- energy

// One launch evaluates the energy at u + t_j dir for n_trials step lengths,
// sharing the element loads; FP64 throughout.
template <int D>
__global__ void __launch_bounds__(256) k_tile_energy(TileDev td, ElemDev<double> ed, VertDev vd, Phys ph,
                                                     const double *__restrict__ u, const double *__restrict__ dir,
                                                     const double *__restrict__ uhat, const double *__restrict__ a,
                                                     TrialT tr, double *__restrict__ partials,
                                                     DevScalars *__restrict__ sc)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double *su = reinterpret_cast<double *>(smem);
    double *sd = su + td.max_tv * D;
    const int t = blockIdx.x;
    const int es = td.tile_elem[t], ne_t = td.tile_elem[t + 1] - es;
    const int vs = td.tile_vert[t], nlv = td.tile_vert[t + 1] - vs;
    const int nt = tr.n;
    for (int k = threadIdx.x; k < nlv; k += blockDim.x) {
        const int64_t gid = td.lv_gid[vs + k];
#pragma unroll
        for (int c = 0; c < D; ++c) {
            su[k * D + c] = u[gid * D + c];
            sd[k * D + c] = dir ? dir[gid * D + c] : 0.0;
        }
    }
    __syncthreads();
    double Eacc[kMaxTrials], Sacc[kMaxTrials];
#pragma unroll
    for (int j = 0; j < kMaxTrials; ++j) Eacc[j] = Sacc[j] = 0.0;
    double minJ = INFINITY;
    const double mu = ph.mu, lam = ph.lam;
    for (int le = threadIdx.x; le < ne_t; le += blockDim.x) {
        const int64_t e = es + le;
        int lid[D + 1];
        unpack<D>(td.conn[e], lid);
        double B[D][D], Du[D][D], Dd[D][D], Z0[D][D], Zd[D][D];
        load_B<double, D>(ed, e, B);
        edges<double, D>(su, lid, Du);
        edges<double, D>(sd, lid, Dd);
        mul<double, D>(Du, B, Z0, true);
        mul<double, D>(Dd, B, Zd, false);
        const double W = __ldg(ed.field(FI<D>::W) + e);
        double f[D];
#pragma unroll
        for (int i = 0; i < D; ++i) f[i] = __ldg(ed.field(FI<D>::F + i) + e);
        const double ka = ph.k * a[e];
#pragma unroll
        for (int j = 0; j < kMaxTrials; ++j) {
            if (j >= nt) break;
            const double tj = tr.t[j];
            double F[D][D], C[D][D];
#pragma unroll
            for (int r = 0; r < D; ++r)
#pragma unroll
                for (int q = 0; q < D; ++q) F[r][q] = Z0[r][q] + tj * Zd[r][q];
            cof<double, D>(F, C);
            const double J = detF<double, D>(F, C);
            if (j == 0) minJ = fmin(minJ, J);
            double I1 = 0.0, Ff2 = 0.0;
#pragma unroll
            for (int r = 0; r < D; ++r) {
                double ff = 0.0;
#pragma unroll
                for (int q = 0; q < D; ++q) {
                    I1 += F[r][q] * F[r][q];
                    ff += F[r][q] * f[q];
                }
                Ff2 += ff * ff;
            }
            double l;
            if (ph.log_mode == 0) {
                l = J > 0.0 ? log(J) : 0.0;
            } else {
                const double jm = J - 1.0;
                l = jm - 0.5 * jm * jm;
            }
            double musc = 0.5 * ka * Ff2;
            if (ph.muscle) {
                const double r = sqrt(Ff2) / a[e] - 1.0;
                musc = W != 0.0 ? 0.5 * ph.k * r * r : 0.0;
            }
            double w = ph.s_el * W * (0.5 * mu * (I1 - D) - mu * l + 0.5 * lam * l * l + musc);
            if (ph.log_mode == 0 && J <= 0.0) w = INFINITY;  // a NaN J (non-finite input) stays NaN
            Eacc[j] += w;
            Sacc[j] += fabs(w);
        }
    }
    // per-vertex terms, added by each vertex's owner tile
    for (int k = threadIdx.x; k < nlv; k += blockDim.x) {
        const int code = td.lv_code[vs + k];
        if (code == LV_PAD || (code >= 0 && !(code & 1))) continue;  // padding, or not the owner
        const int64_t gid = td.lv_gid[vs + k];
        const double m = vd.mass[gid];
        const double X1 = vd.X[gid * D + 1];
#pragma unroll
        for (int j = 0; j < kMaxTrials; ++j) {
            if (j >= nt) break;
            const double tj = tr.t[j];
            const double y = X1 + su[k * D + 1] + tj * sd[k * D + 1];
            const double pen = y < 0.0 ? -y : 0.0;
            double w = ph.s_el * (m * ph.grav * y + ph.kc * pen_pow(pen, ph.cpow));
            double s = fabs(w);
            if (ph.dyn) {
                double in = 0.0;
#pragma unroll
                for (int c = 0; c < D; ++c) {
                    const double r = su[k * D + c] + tj * sd[k * D + c] - uhat[gid * D + c];
                    in += 0.5 * m * r * r;
                }
                if (ph.fw) {
                    const double f = ph.fw[gid];
#pragma unroll
                    for (int c = 0; c < D; ++c) {
                        if (c == 1) continue;
                        const double r = su[k * D + c] + tj * sd[k * D + c] - ph.u0[gid * D + c];
                        in += 0.5 * f * r * r;
                    }
                }
                w += in;
                s += in;
            }
            Eacc[j] += w;
            Sacc[j] += s;
        }
    }
    const int nb = gridDim.x;
    for (int j = 0; j < nt; ++j) {
        double e = block_sum(Eacc[j]);
        double s = block_sum(Sacc[j]);
        if (threadIdx.x == 0) {
            partials[(size_t)j * nb + t] = e;
            partials[(size_t)(kMaxTrials + j) * nb + t] = s;
        }
    }
    double mj = block_min(minJ);
    if (threadIdx.x == 0) partials[(size_t)(2 * kMaxTrials) * nb + t] = mj;
    if (last_block(&sc->ticket[TK_ENERGY], nb)) {
        for (int j = 0; j < nt; ++j) {
            double e = sum_partials(partials + (size_t)j * nb, nb);
            double s = sum_partials(partials + (size_t)(kMaxTrials + j) * nb, nb);
            if (threadIdx.x == 0) {
                sc->E[j] = e;
                sc->S[j] = s;
            }
        }
        double m = min_partials(partials + (size_t)(2 * kMaxTrials) * nb, nb);
        if (threadIdx.x == 0) sc->minJ = m;
    }
}

// ---------------------------------------------------------------- gradient

// Block sums of v[0..N) and minimum of mn, one tree for all; valid in thread 0.
template <int N>
__device__ __forceinline__ void block_sums_min(double (&v)[N], double &mn)
{
    __shared__ double red[N + 1][32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
        mn = fmin(mn, __shfl_down_sync(0xffffffffu, mn, o));
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < N; ++q) red[q][w] = v[q];
        red[N][w] = mn;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
#pragma unroll
            for (int q = 0; q < N; ++q) v[q] += red[q][k];
            mn = fmin(mn, red[N][k]);
        }
    }
}

// Gradient of one tile and, with EN, its energy terms (energy, sum of their
// absolute values, smallest J), FP64.
//
// What bounds it: the FP64 pipe (1/64 of the FP32 rate), about 230 operations a
// tet.  Energy and gradient share the gathers, F, cof F, J and the logarithm,
// so one pass gives both (393,216 tets: 352 us the call with a gradient and an
// energy kernel of 167 + 143 us, 225 us with this one).  A mesh with fewer tiles than SMs splits each tile's elements
// over a cluster of `split` CTAs: an element sends each corner's force to the
// CTA that sums the corner's vertex (distributed shared memory), so the sums
// keep their order.
template <int D, bool EN>
__global__ void __launch_bounds__(256) k_tile_grad(TileDev td, ElemDev<double> ed, VertDev vd, Phys ph,
                                                   const double *__restrict__ u, const double *__restrict__ uhat,
                                                   const double *__restrict__ a, double *__restrict__ g,
                                                   double *__restrict__ hp, double *__restrict__ partials, int split)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double *su = reinterpret_cast<double *>(smem);
    double *scr = su + td.max_tv * D;
    const int t = blockIdx.x / split, rank = blockIdx.x % split;
    const int es = td.tile_elem[t], ne_t = td.tile_elem[t + 1] - es;
    const int vs = td.tile_vert[t], nlv = td.tile_vert[t + 1] - vs;
    // this CTA's share of the tile's elements and of its vertices
    const int ech = (ne_t + split - 1) / split, vch = (nlv + split - 1) / split;
    const int e0 = rank * ech, e1 = min(ne_t, e0 + ech), k0 = rank * vch, k1 = min(nlv, k0 + vch);
    pdl_wait();  // everything above is static
    for (int k = threadIdx.x; k < nlv; k += blockDim.x) {
        const int64_t gid = td.lv_gid[vs + k];
#pragma unroll
        for (int c = 0; c < D; ++c) su[k * D + c] = u[gid * D + c];
    }
    if (split > 1)
        cluster_sync();  // every CTA of the cluster runs: its shared memory may be written
    else
        __syncthreads();
    const double mu = ph.mu, lam = ph.lam;
    double acc_e[3] = {0.0, 0.0, 0.0}, minJ = INFINITY;  // E, sum |terms|, |g|^2
    for (int le = e0 + threadIdx.x; le < e1; le += blockDim.x) {
        const int64_t e = es + le;
        int lid[D + 1];
        unpack<D>(td.conn[e], lid);
        double B[D][D], Du[D][D], F[D][D], C[D][D];
        load_B<double, D>(ed, e, B);
        edges<double, D>(su, lid, Du);
        mul<double, D>(Du, B, F, true);
        cof<double, D>(F, C);
        const double J = detF<double, D>(F, C);
        double l, cc, cp;
        log_terms<double>(ph.log_mode, mu, lam, J, l, cc, cp);
        const double W0 = __ldg(ed.field(FI<D>::W) + e);
        const double W = W0 * ph.s_el;
        double f[D], gv[D], Ff[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            f[i] = __ldg(ed.field(FI<D>::F + i) + e);
            gv[i] = __ldg(ed.field(FI<D>::G + i) + e);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < D; ++q) s += F[i][q] * f[q];
            Ff[i] = s;
        }
        const double av = a[e];
        double ka = ph.k * av;  // dpsi_m/dq = ka q
        double s2 = 0.0;
        if (EN || ph.muscle) {
#pragma unroll
            for (int i = 0; i < D; ++i) s2 += Ff[i] * Ff[i];
        }
        if constexpr (EN) {
            double I1 = 0.0;
#pragma unroll
            for (int i = 0; i < D; ++i)
#pragma unroll
                for (int j = 0; j < D; ++j) I1 += F[i][j] * F[i][j];
            if (ph.log_mode == 0 && !(J > 0.0)) l = 0.0;
            double musc = 0.5 * ka * s2;
            if (ph.muscle) {
                const double r = sqrt(s2) / av - 1.0;
                musc = W0 != 0.0 ? 0.5 * ph.k * r * r : 0.0;
            }
            double w = W * (0.5 * mu * (I1 - D) - mu * l + 0.5 * lam * l * l + musc);
            if (ph.log_mode == 0 && J <= 0.0) w = INFINITY;  // a NaN J (non-finite input) stays NaN
            acc_e[0] += w;
            acc_e[1] += fabs(w);
            minJ = fmin(minJ, J);
        }
        if (ph.muscle) {
            double c2;
            spring_terms<double>(W != 0.0, ph.k, av, sqrt(s2), ka, c2);
        }
        const double muW = mu * W, ccW = cc * W, kaW = ka * W;
#pragma unroll
        for (int i = 0; i < D; ++i) Ff[i] *= kaW;
        double G[D][D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
#pragma unroll
            for (int k = 0; k < D; ++k) F[i][k] = muW * F[i][k] + ccW * C[i][k];
#pragma unroll
            for (int j = 0; j < D; ++j) {
                double s = Ff[i] * gv[j];
#pragma unroll
                for (int k = 0; k < D; ++k) s += F[i][k] * B[j][k];
                G[i][j] = s;
            }
        }
        double *rec = scr + (int64_t)le * td.rs + corner_base(le);
        if (split == 1)
            store_corners<double, D>(rec, G);
        else
            send_corners<D>(rec, G, lid, vch);
    }
    if (split > 1)
        cluster_sync();
    else
        __syncthreads();
    pdl_trigger();  // the finalize kernel may be scheduled
    double gn2 = 0.0;
    const uint16_t *tinc = td.inc + (int64_t)es * (D + 1);
    for (int k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
        const int code = td.lv_code[vs + k];
        if (code == LV_PAD) continue;
        double acc[D];
        gather_corners<double, D>(tinc, td.lv_inc[vs + k], scr, acc);
        const int64_t gid = td.lv_gid[vs + k];
        if (code == LV_INTERIOR) {
            add_vertex_terms<D, EN>(vd, ph, gid, su + k * D, uhat, acc, acc_e);
            const bool fx = vd.fixed[gid] != 0;
#pragma unroll
            for (int c = 0; c < D; ++c) {
                const double o = fx ? 0.0 : acc[c];
                g[gid * D + c] = o;
                gn2 += o * o;
            }
        } else {
#pragma unroll
            for (int c = 0; c < D; ++c) hp[(int64_t)(code >> 1) * D + c] = acc[c];
        }
    }
    if constexpr (EN) {
        acc_e[2] = gn2;
        block_sums_min<3>(acc_e, minJ);
        if (threadIdx.x == 0) {
            double *p = partials + 4 * (size_t)blockIdx.x;
            p[0] = acc_e[0];
            p[1] = acc_e[1];
            p[2] = acc_e[2];
            p[3] = minJ;
        }
    } else {
        const double s = block_sum(gn2);
        if (threadIdx.x == 0) partials[blockIdx.x] = s;
    }
}

// Completes the gradient at halo vertices (their tiles' partial sums in tile
// order plus the vertex terms); the last block sums the partials of both
// kernels: [n_part] of the tile kernel, then one entry per block.
template <int D, bool EN>
__global__ void __launch_bounds__(256) k_fin_grad(TileDev td, VertDev vd, Phys ph, const double *__restrict__ u,
                                                  const double *__restrict__ uhat, const double *__restrict__ hp,
                                                  double *__restrict__ g, double *__restrict__ partials, int n_part,
                                                  DevScalars *__restrict__ sc)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = i < td.n_fin;
    const int64_t gid = in ? td.fin_gid[i] : 0;
    const int p0 = in ? td.fin_ptr[i] : 0, p1 = in ? td.fin_ptr[i + 1] : 0;
    const bool fx = in && vd.fixed[gid] != 0;
    pdl_wait();  // everything above is static
    double gn2 = 0.0, acc_e[3] = {0.0, 0.0, 0.0}, minJ = INFINITY;
    if (in) {
        double acc[D], uv[D];
#pragma unroll
        for (int c = 0; c < D; ++c) acc[c] = 0.0, uv[c] = u[gid * D + c];
        for (int s = p0; s < p1; ++s)
#pragma unroll
            for (int c = 0; c < D; ++c) acc[c] += hp[(int64_t)s * D + c];
        add_vertex_terms<D, EN>(vd, ph, gid, uv, uhat, acc, acc_e);
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const double o = fx ? 0.0 : acc[c];
            g[gid * D + c] = o;
            gn2 += o * o;
        }
    }
    if constexpr (EN) {
        acc_e[2] = gn2;
        block_sums_min<3>(acc_e, minJ);
        if (threadIdx.x == 0) {
            double *p = partials + 4 * (size_t)(n_part + blockIdx.x);
            p[0] = acc_e[0];
            p[1] = acc_e[1];
            p[2] = acc_e[2];
            p[3] = minJ;
        }
        if (last_block(&sc->ticket[TK_GRAD], gridDim.x)) {
            const double2 *p = reinterpret_cast<const double2 *>(partials);
            double v[3] = {0.0, 0.0, 0.0}, mj = INFINITY;
            const int n = n_part + gridDim.x;
#pragma unroll 4
            for (int k = threadIdx.x; k < n; k += blockDim.x) {
                const double2 q0 = __ldcg(p + 2 * k), q1 = __ldcg(p + 2 * k + 1);
                v[0] += q0.x;
                v[1] += q0.y;
                v[2] += q1.x;
                mj = fmin(mj, q1.y);
            }
            block_sums_min<3>(v, mj);
            if (threadIdx.x == 0) {
                sc->E[0] = v[0];
                sc->S[0] = v[1];
                sc->gn2 = v[2];
                sc->minJ = mj;
            }
        }
    } else {
        const double s = block_sum(gn2);
        if (threadIdx.x == 0) partials[n_part + blockIdx.x] = s;
        if (last_block(&sc->ticket[TK_GRAD], gridDim.x)) {
            const double tot = sum_partials(partials, n_part + gridDim.x);
            if (threadIdx.x == 0) sc->gn2 = tot;
        }
    }
}

// ---------------------------------------------------------------- HVP

// Shared-memory plan of the HVP tile kernel (offsets in bytes, all 16-byte
// aligned because max_te is a multiple of 8, max_tv of 4 and rs even).
template <typename T, int D>
struct HvpSmem {
    size_t e, rec, conn, inc, gid, code, linc, uv, total;
    __host__ __device__ HvpSmem(int max_te, int max_tv, int rs)
    {
        e = 16;  // two mbarriers
        rec = e;  // [max_te][rs] element records
        conn = rec + (size_t)rs * max_te * sizeof(T);
        inc = conn + (size_t)max_te * 4;
        gid = inc + (size_t)max_te * (D + 1) * 2;
        code = gid + (size_t)max_tv * 4;
        linc = code + (size_t)max_tv * 4;
        uv = linc + (size_t)max_tv * 4;  // [max_tv][2D]: u then v of each local vertex
        total = uv + (size_t)max_tv * 2 * D * sizeof(T);
    }
};

// HVP of one tile per CTA.  Thread 0 pulls the tile's element records
// (fields and activation), connectivity, incidence lists and local-vertex
// tables into shared memory with bulk copies on two mbarriers; the tile's
// vertex values are then gathered, each thread evaluates dP(dF) for its
// elements from their records (pair loads), the element's corner forces
// overwrite its own record in place (slots corner_base(le) .. +(D+1)*D <= RS),
// and one thread
// per local vertex adds its corners in fixed order.
// SPRING selects the active-spring muscle at compile time, so the
// contractile kernel carries none of its code or its extra fields.
// MODE: HVP_STATE reads the displacement u and the activations in tile order;
// HVP_CG also forms p.Ap and, launched hundreds of times on the same
// activations, has them in the records (launch_record_activation; a load of
// its own cost it 62.0 against 59.8 us at 3.1 million tets); HVP_CALLER takes positions x and activations as
// the caller has them (u = x - X rounded to T while staging), which saves a
// small mesh one launch.  A thread fetches its elements' activations before the
// wait for the records and puts them into its records (not HVP_CG).
enum HvpMode { HVP_STATE, HVP_CG, HVP_CALLER };

template <typename T, int D, int MODE, int MINB, int MTE, bool SPRING>
__global__ void __launch_bounds__(256, MINB) k_tile_hvp(TileDev td, const T *__restrict__ erec, VertDev vd,
                                                  Phys ph, const T *__restrict__ u, const double *__restrict__ x,
                                                  const void *__restrict__ act, const T *__restrict__ v,
                                                  T *__restrict__ y, T *__restrict__ hp,
                                                  double *__restrict__ partials, DevScalars *__restrict__ sc)
{
    constexpr bool CG = MODE == HVP_CG;
    extern __shared__ __align__(128) unsigned char smem[];
    // MTE != 0: the tile capacity is a compile-time constant, so every
    // record and corner offset below folds into an immediate
    constexpr int NF = hvp_fields(D, SPRING);
    constexpr int RS = rec_stride(NF);  // record: NF fields, the activation at slot NF, padding
    const HvpSmem<T, D> L(MTE ? MTE : td.max_te, td.max_tv, RS);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem);  // [0]: vertex tables, [1]: element data
    T *sRec = reinterpret_cast<T *>(smem + L.rec);
    // vertex table: [gid, code, lv_inc] per local vertex (stride 3 words:
    // a warp's lanes read distinct banks)
    const int32_t *sLv = reinterpret_cast<const int32_t *>(smem + L.gid);
    T *suv = reinterpret_cast<T *>(smem + L.uv);  // per local vertex: u (D values), then v (D values)
    const int t = blockIdx.x;
    // a tile's ranges: from its index for equal tiles (no dependent load before
    // the bulk copies can be issued), else from the offset tables
    const int es = td.uni_te ? t * td.uni_te : td.tile_elem[t];
    const int ne_t = td.uni_te ? td.uni_te : td.tile_elem[t + 1] - es;
    const int vs = td.uni_tv ? t * td.uni_tv : td.tile_vert[t];
    const int nlv = td.uni_tv ? td.uni_tv : td.tile_vert[t + 1] - vs;
    // the tile's connectivity and incidence block arrive as one blob: conn
    // [ne_t] then inc [ne_t (D+1)] (both 16-byte multiples)
    const uint32_t *sConn = reinterpret_cast<const uint32_t *>(smem + L.conn);
    const uint16_t *sInc = reinterpret_cast<const uint16_t *>(smem + L.conn + (size_t)ne_t * 4);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        // vertex table first: the vertex gather below overlaps the element copy
        mbar_arrive_expect_tx(bar, 12u * nlv);
        bulk_g2s(smem + L.gid, td.lv3 + (int64_t)vs * 3, 12u * nlv, bar);
        const uint32_t brec = (uint32_t)ne_t * RS * sizeof(T), bci = (uint32_t)ne_t * (4 + 2 * (D + 1));
        mbar_arrive_expect_tx(bar + 1, brec + bci);
        const uint64_t pol = l2_evict_first_policy();  // element data is read once per launch
        bulk_g2s_stream(sRec, erec + (int64_t)es * RS, brec, bar + 1, pol);
        bulk_g2s_stream(smem + L.conn, td.ci + (int64_t)es * (4 + 2 * (D + 1)), bci, bar + 1, pol);
    }
    __syncthreads();
    // Everything copied so far is static during a solve; state (u, v) and the
    // CG scalars are read only after the predecessor kernel has completed.
    pdl_wait();
    constexpr int PRE = 4;  // activations a thread holds (tiles of more than PRE x threads elements: the rest later)
    T av[PRE];
    auto activation = [&](int le) {
        if constexpr (MODE == HVP_CALLER) {
            const int32_t pe = td.perm[es + le];
            return pe >= 0 ? T(static_cast<const double *>(act)[pe]) : T(0);
        } else {
            return static_cast<const T *>(act)[es + le];
        }
    };
    if constexpr (!CG) {
#pragma unroll
        for (int j = 0; j < PRE; ++j) {
            const int le = threadIdx.x + j * blockDim.x;
            av[j] = le < ne_t ? activation(le) : T(0);
        }
    }
    // the flag is read before the wait so that its load overlaps the copies
    // in flight; the previous kernel has completed, so every thread reads the
    // same value
    const int cg_done = CG ? sc->done : 0;
    // every thread takes the same decision, so no thread is left at a barrier
    if (__syncthreads_or(!mbar_wait_bounded(bar, 0, td.wait_polls))) {
        if (threadIdx.x == 0) {
            atomicOr(&sc->kerr, 1);
            mbar_wait_bounded(bar, 0);  // give copies in flight a last chance before the CTA exits
            mbar_wait_bounded(bar + 1, 0);
        }
        return;
    }
    if (cg_done) {  // CG already finished: drain the second copy, then leave
        if (threadIdx.x == 0) mbar_wait_bounded(bar + 1, 0);
        return;
    }
    for (int k = threadIdx.x; k < nlv; k += blockDim.x) {
        const int64_t gid = sLv[3 * k];
        const bool fx = ((uint32_t)sLv[3 * k + 2] & kLvPinned) != 0;
        if constexpr (CG && sizeof(T) == 4 && D == 3) {
            // the CG loop's 3D FP32 displacement comes in 16-byte rows
            const float4 u4 = reinterpret_cast<const float4 *>(u)[gid];
            suv[k * 6 + 0] = u4.x;
            suv[k * 6 + 1] = u4.y;
            suv[k * 6 + 2] = u4.z;
        } else if constexpr (MODE == HVP_CALLER) {
#pragma unroll
            for (int c = 0; c < D; ++c) suv[k * 2 * D + c] = T(x[gid * D + c] - vd.X[gid * D + c]);
        } else {
#pragma unroll
            for (int c = 0; c < D; ++c) suv[k * 2 * D + c] = u[gid * D + c];
        }
#pragma unroll
        for (int c = 0; c < D; ++c) suv[k * 2 * D + D + c] = fx ? T(0) : v[gid * D + c];
    }
    if (__syncthreads_or(!mbar_wait_bounded(bar + 1, 0))) {
        if (threadIdx.x == 0) {
            atomicOr(&sc->kerr, 1);
            mbar_wait_bounded(bar + 1, 0);
        }
        return;
    }
    if constexpr (!CG) {  // each thread's own elements: no barrier needed
#pragma unroll
        for (int j = 0; j < PRE; ++j) {
            const int le = threadIdx.x + j * blockDim.x;
            if (le < ne_t) sRec[le * RS + NF] = av[j];
        }
        for (int le = threadIdx.x + PRE * blockDim.x; le < ne_t; le += blockDim.x) sRec[le * RS + NF] = activation(le);
    }
    const T mu = pick<T>(ph.mu, ph.mu_f), lam = pick<T>(ph.lam, ph.lam_f);
    const T sel = pick<T>(ph.s_el, ph.s_el_f), kk = pick<T>(ph.k, ph.k_f);
    // CG: p.Ap of this tile from the element quadratic forms v_e . (H_e v_e)
    // and the owners' vertex terms, in the kernel's precision.  In the mixed
    // kernel the per-thread and block sums stay plain FP32 (GB300's FP64 pipe
    // runs at 1/64 of FP32, and compensating them here cost ~7 % of the
    // kernel's time); k_cg_alpha sums the tiles' partials with compensation.
    T dot = T(0);
    for (int le = threadIdx.x; le < ne_t; le += blockDim.x)
        hvp_element<T, D, CG, SPRING, RS>(sRec + le * RS, le, sConn[le], suv, ph, mu, lam, sel, kk, dot,
                                          sRec + le * RS);
    __syncthreads();
    for (int k = threadIdx.x; k < nlv; k += blockDim.x)
        hvp_vertex<T, D, CG>(sLv[3 * k + 1], (uint32_t)sLv[3 * k + 2], sLv[3 * k], suv + k * 2 * D, sInc, sRec, vd, ph,
                             y, hp, dot);
    pdl_trigger();  // the alpha reduction may be scheduled once every tile is done
    if (CG) {
        const T sum = block_sum(dot);
        if (threadIdx.x == 0) reinterpret_cast<T *>(partials)[t] = sum;  // reduced by k_cg_alpha<T>
    }
}

// Completes y = A v at halo vertices: the tiles' partial sums in tile order
// plus the per-vertex terms.  x: the caller's positions (HVP_CALLER; u unused).
// Latency of a few dependent loads: the table entries come before the wait for
// the tile kernel, and the partial sums four at a time.
template <typename T, int D>
__global__ void __launch_bounds__(256) k_fin_hvp(TileDev td, VertDev vd, Phys ph, const T *__restrict__ u,
                                                 const double *__restrict__ x, const T *__restrict__ v,
                                                 const T *__restrict__ hp, T *__restrict__ y)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = i < td.n_fin;
    const int64_t gid = in ? td.fin_gid[i] : 0;
    const int s0 = in ? td.fin_ptr[i] : 0, s1 = in ? td.fin_ptr[i + 1] : 0;
    const bool fx = in && vd.fixed[gid] != 0;
    pdl_wait();  // everything above is static
    if (!in) return;
    T vv[D];
#pragma unroll
    for (int c = 0; c < D; ++c) vv[c] = fx ? T(0) : v[gid * D + c];
    T acc[D];
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c] = T(0);
    for (int s = s0; s < s1; s += 4) {
        T h[4][D];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < D; ++c) h[q][c] = s + q < s1 ? hp[(int64_t)(s + q) * D + c] : T(0);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < D; ++c) acc[c] += h[q][c];
    }
    if (ph.kc > 0.0) {
        const double ux = x ? (double)T(x[gid * D + 1] - vd.X[gid * D + 1]) : (double)u[gid * D + 1];
        const double yy = vd.X[gid * D + 1] + ux;
        const double pen = yy < 0.0 ? -yy : 0.0;
        const double d2 = pen > 0.0 ? ph.cpow * (ph.cpow - 1) * ph.kc * (ph.cpow == 2 ? 1.0 : pen) : 0.0;
        acc[1] += T(ph.s_el * d2) * vv[1];
    }
    if (ph.dyn) {
        const T m = T(vd.mass[gid]);
        const T mh = ph.fw ? m + T(ph.fw[gid]) : m;
#pragma unroll
        for (int c = 0; c < D; ++c) acc[c] += (c == 1 ? m : mh) * vv[c];
    }
#pragma unroll
    for (int c = 0; c < D; ++c) y[gid * D + c] = fx ? T(0) : acc[c];
}

// ---------------------------------------------------------------- parameter VJP

template <int D>
__global__ void __launch_bounds__(256) k_tile_vjp(TileDev td, ElemDev<double> ed, VertDev vd, Phys ph,
                                                  const double *__restrict__ u, const double *__restrict__ a,
                                                  const double *__restrict__ lam, double *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double *su = reinterpret_cast<double *>(smem);
    double *sl = su + td.max_tv * D;
    const int t = blockIdx.x;
    const int es = td.tile_elem[t], ne_t = td.tile_elem[t + 1] - es;
    const int vs = td.tile_vert[t], nlv = td.tile_vert[t + 1] - vs;
    for (int k = threadIdx.x; k < nlv; k += blockDim.x) {
        const int64_t gid = td.lv_gid[vs + k];
        const bool fx = vd.fixed[gid] != 0;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            su[k * D + c] = u[gid * D + c];
            sl[k * D + c] = fx ? 0.0 : lam[gid * D + c];
        }
    }
    __syncthreads();
    for (int le = threadIdx.x; le < ne_t; le += blockDim.x) {
        const int64_t e = es + le;
        int lid[D + 1];
        unpack<D>(td.conn[e], lid);
        double B[D][D], Du[D][D], Dl[D][D], F[D][D];
        load_B<double, D>(ed, e, B);
        edges<double, D>(su, lid, Du);
        edges<double, D>(sl, lid, Dl);
        mul<double, D>(Du, B, F, true);
        double f[D], gv[D];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            f[i] = __ldg(ed.field(FI<D>::F + i) + e);
            gv[i] = __ldg(ed.field(FI<D>::G + i) + e);
        }
        double dot = 0.0, s2 = 0.0;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            double Ff = 0.0, dFf = 0.0;
#pragma unroll
            for (int q = 0; q < D; ++q) {
                Ff += F[i][q] * f[q];
                dFf += Dl[i][q] * gv[q];  // dF(lam) f = Dlam Dm^-1 f = Dlam g
            }
            dot += Ff * dFf;
            s2 += Ff * Ff;
        }
        const double W = __ldg(ed.field(FI<D>::W) + e);
        const int32_t pe = td.perm[e];
        // d2psi/dq da = k q (contractile) or k (1/a^2 - 2 s/a^3)/s q (spring, s = |q|)
        double kq = ph.k;
        if (ph.muscle && pe >= 0) {
            const double s = sqrt(s2), ia = 1.0 / a[e];
            kq = ph.k * (ia * ia - 2.0 * s * ia * ia * ia) / s;
        }
        if (pe >= 0) out[pe] = -ph.s_el * W * kq * dot;
    }
}

// Material-parameter VJPs per element: -s W (dP/dtheta) : dF(lam) with
// dP/dmu = F - l'(J) cof F, dP/dlambda = l(J) l'(J) cof F, and for the
// muscle stiffness -s W (d2psi_m/dq dk) . dq(lam).  Null outputs are skipped.
template <int D>
__global__ void __launch_bounds__(256) k_tile_mat_vjp(TileDev td, ElemDev<double> ed, VertDev vd, Phys ph,
                                                      const double *__restrict__ u, const double *__restrict__ a,
                                                      const double *__restrict__ lam, double *__restrict__ dmu,
                                                      double *__restrict__ dlam, double *__restrict__ dk)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double *su = reinterpret_cast<double *>(smem);
    double *sl = su + td.max_tv * D;
    const int t = blockIdx.x;
    const int es = td.tile_elem[t], ne_t = td.tile_elem[t + 1] - es;
    const int vs = td.tile_vert[t], nlv = td.tile_vert[t + 1] - vs;
    for (int k = threadIdx.x; k < nlv; k += blockDim.x) {
        const int64_t gid = td.lv_gid[vs + k];
        const bool fx = vd.fixed[gid] != 0;
#pragma unroll
        for (int c = 0; c < D; ++c) {
            su[k * D + c] = u[gid * D + c];
            sl[k * D + c] = fx ? 0.0 : lam[gid * D + c];
        }
    }
    __syncthreads();
    for (int le = threadIdx.x; le < ne_t; le += blockDim.x) {
        const int64_t e = es + le;
        const int32_t pe = td.perm[e];
        if (pe < 0) continue;  // padding
        int lid[D + 1];
        unpack<D>(td.conn[e], lid);
        double B[D][D], Du[D][D], Dl[D][D], F[D][D], dF[D][D], C[D][D];
        load_B<double, D>(ed, e, B);
        edges<double, D>(su, lid, Du);
        edges<double, D>(sl, lid, Dl);
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
        double l, lp;  // l(J) and l'(J)
        if (ph.log_mode == 0) {
            l = log(J);
            lp = 1.0 / J;
        } else {
            l = (J - 1.0) - 0.5 * (J - 1.0) * (J - 1.0);
            lp = 2.0 - J;
        }
        const double sW = -ph.s_el * __ldg(ed.field(FI<D>::W) + e);
        if (dmu) dmu[pe] = sW * (FdF - lp * CdF);
        if (dlam) dlam[pe] = sW * l * lp * CdF;
        if (dk) {
            double qdq = 0.0, s2 = 0.0;
#pragma unroll
            for (int i = 0; i < D; ++i) {
                double q = 0.0, dq = 0.0;
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    q += F[i][k] * __ldg(ed.field(FI<D>::F + k) + e);
                    dq += Dl[i][k] * __ldg(ed.field(FI<D>::G + k) + e);  // dF(lam) f = Dlam g
                }
                qdq += q * dq;
                s2 += q * q;
            }
            double c = a[e];  // d2psi_m/dq dk = c q
            if (ph.muscle) {
                const double sq = sqrt(s2);
                c = (sq / a[e] - 1.0) / (a[e] * sq);
            }
            dk[pe] = sW * c * qdq;
        }
    }
}

// ---------------------------------------------------------------- launchers

static inline size_t smem_verts(const Ctx &c, size_t elt, int nfields)
{
    return (size_t)c.td.max_tv * c.dim * nfields * elt;
}

void launch_energy(const Ctx &c, const Phys &ph, const double *u, const double *dir, const double *uhat,
                   const double *a, const double *t, int n_trials, cudaStream_t s)
{
    c.n_launch += 1;
    TrialT tr;
    tr.n = n_trials;
    for (int j = 0; j < kMaxTrials; ++j) tr.t[j] = j < n_trials ? t[j] : 0.0;
    const size_t sm = smem_verts(c, sizeof(double), 2);
    if (c.dim == 2)
        k_tile_energy<2><<<c.td.n_tiles, c.threads, sm, s>>>(c.td, c.e64, c.vd, ph, u, dir, uhat, a, tr, c.partials, c.sc);
    else
        k_tile_energy<3><<<c.td.n_tiles, c.threads, sm, s>>>(c.td, c.e64, c.vd, ph, u, dir, uhat, a, tr, c.partials, c.sc);
}

// CTAs that share a tile: as many as leave every SM at most one (the FP64 pipe
// is saturated by a tile's four warps, so more than one CTA an SM gains
// nothing).  A backward-Euler step of 5,616 tets, 15 tiles: 3.51 -> 2.80 ms
// together with the fused evaluation; 107 tiles stay whole.
int eval_split(int n_tiles, int sms)
{
    int sp = 8;
    while (sp > 1 && n_tiles * sp > sms) sp /= 2;
    return sp;
}

template <int D, bool EN>
static void grad_k(const Ctx &c, const Phys &ph, const double *u, const double *uhat, const double *a, double *g,
                   double *hp, cudaStream_t s)
{
    c.n_launch += 2;
    const size_t sm = smem_verts(c, sizeof(double), 1) + (size_t)c.td.max_te * c.td.rs * sizeof(double);
    const int n_part = c.td.n_tiles * c.split;
    launch_cluster(c.split, k_tile_grad<D, EN>, dim3(n_part), dim3(c.threads), sm, s, c.td, c.e64, c.vd, ph, u, uhat,
                   a, g, hp, c.partials, c.split);
    launch_k(true, k_fin_grad<D, EN>, dim3(c.n_fin_blocks), dim3(256), 0, s, c.td, c.vd, ph, u, uhat,
             (const double *)hp, g, c.partials, n_part, c.sc);
}

void launch_grad(const Ctx &c, const Phys &ph, const double *u, const double *uhat, const double *a, double *g,
                 double *hp, bool energy, cudaStream_t s)
{
    if (c.dim == 2)
        (energy ? grad_k<2, true> : grad_k<2, false>)(c, ph, u, uhat, a, g, hp, s);
    else
        (energy ? grad_k<3, true> : grad_k<3, false>)(c, ph, u, uhat, a, g, hp, s);
}

template <typename T>
static const T *erec(const Ctx &c);
template <>
const float *erec<float>(const Ctx &c) { return c.rec32; }
template <>
const double *erec<double>(const Ctx &c) { return c.rec64; }

template <typename T>
static const T *eact(const Ctx &c);
template <>
const float *eact<float>(const Ctx &c) { return c.a32; }
template <>
const double *eact<double>(const Ctx &c) { return c.a64; }

template <typename T>
size_t hvp_smem(const Ctx &c)
{
    return c.dim == 2 ? HvpSmem<T, 2>(c.td.max_te, c.td.max_tv, c.td.rs).total
                      : HvpSmem<T, 3>(c.td.max_te, c.td.max_tv, c.td.rs).total;
}

// Resident CTAs per SM that the tile's shared memory allows (at most 4);
// the kernel variant compiled for that count caps registers to match.  (At
// 128 threads and 7 resident tiles, the 64-register FP32 variant measured
// faster in-solve than the 72-register one before the element used paired
// FP32 arithmetic: 66.3 vs 68.4 us on the large body; with it, the CG variant
// spills at 64 and runs at 58.4 us with 72 against 60.7 us.)
template <typename T>
int hvp_blocks_per_sm(const Ctx &c)
{
    const size_t per = hvp_smem<T>(c) + 1024;  // + static shared memory and reserve
    int b = (int)((227 * 1024) / per);
    return b < 1 ? 1 : (b > 4 ? 4 : b);
}

// Tile capacities with a compile-time specialisation (the library defaults).
constexpr int kCap2 = 512, kCap3 = 384;

// What an HVP reads besides v: the handle's displacement and activations, or
// (x set) the caller's positions and activations.
template <typename T>
struct HvpIn {
    const T *u;
    const double *x;
    const void *act;
};

template <typename T, int D, int MODE, int MINB>
static void hvp_tile_v(const Ctx &c, const Phys &ph, const HvpIn<T> &in, const T *v, T *y, T *hp, cudaStream_t s)
{
    constexpr int CAP = D == 2 ? kCap2 : kCap3;
    auto go = [&](auto k) {
        launch_k(c.pdl, k, dim3(c.td.n_tiles), dim3(c.threads), hvp_smem<T>(c), s, c.td, erec<T>(c), c.vd, ph, in.u,
                 in.x, in.act, v, y, hp, c.partials, c.sc);
    };
    if (c.muscle)  // the spring variant exists for the runtime tile capacity only
        go(k_tile_hvp<T, D, MODE, MINB, 0, true>);
    else if (sizeof(T) == 4 && c.td.max_te == CAP)
        go(k_tile_hvp<T, D, MODE, MINB, (sizeof(T) == 4 ? CAP : 0), false>);
    else
        go(k_tile_hvp<T, D, MODE, MINB, 0, false>);
}

template <typename T, int MODE>
static void hvp_tile(const Ctx &c, const Phys &ph, const HvpIn<T> &in, const T *v, T *y, T *hp, cudaStream_t s)
{
    c.n_launch += 1;
    const int b = hvp_blocks_per_sm<T>(c);
    if constexpr (sizeof(T) == 4) {
        if (c.dim == 2)
            (b >= 4 ? hvp_tile_v<T, 2, MODE, 4> : hvp_tile_v<T, 2, MODE, 3>)(c, ph, in, v, y, hp, s);
        else
            // the CG variant also forms p.Ap: at 64 registers it spilled, at
            // the 3-CTA bound it takes 72, which still lets 7 of the
            // 128-thread tiles be resident (shared memory allows 7)
            ((b >= 4 && MODE == HVP_STATE) ? hvp_tile_v<T, 3, MODE, 4> : hvp_tile_v<T, 3, MODE, 3>)(c, ph, in, v, y, hp,
                                                                                                 s);
    } else {
        if (c.dim == 2)
            (b >= 2 ? hvp_tile_v<T, 2, MODE, 2> : hvp_tile_v<T, 2, MODE, 1>)(c, ph, in, v, y, hp, s);
        else
            (b >= 2 ? hvp_tile_v<T, 3, MODE, 2> : hvp_tile_v<T, 3, MODE, 1>)(c, ph, in, v, y, hp, s);
    }
}

template <typename T>
static void hvp_fin(const Ctx &c, const Phys &ph, const HvpIn<T> &in, const T *v, T *y, const T *hp, cudaStream_t s)
{
    c.n_launch += 1;
    if (c.dim == 2)
        launch_k(true, k_fin_hvp<T, 2>, dim3(c.n_fin_blocks), dim3(256), 0, s, c.td, c.vd, ph, in.u, in.x, v, hp, y);
    else
        launch_k(true, k_fin_hvp<T, 3>, dim3(c.n_fin_blocks), dim3(256), 0, s, c.td, c.vd, ph, in.u, in.x, v, hp, y);
}

template <typename T>
void launch_hvp(const Ctx &c, const Phys &ph, const T *u, const T *v, T *y, T *hp, cudaStream_t s)
{
    const HvpIn<T> in{u, nullptr, eact<T>(c)};
    hvp_tile<T, HVP_STATE>(c, ph, in, v, y, hp, s);
    hvp_fin<T>(c, ph, in, v, y, hp, s);
}

template <typename T>
void launch_hvp_at(const Ctx &c, const Phys &ph, const double *x, const double *act, const T *v, T *y, T *hp,
                   cudaStream_t s)
{
    const HvpIn<T> in{nullptr, x, act};
    hvp_tile<T, HVP_CALLER>(c, ph, in, v, y, hp, s);
    hvp_fin<T>(c, ph, in, v, y, hp, s);
}

template <typename T>
void launch_hvp_cg(const Ctx &c, const Phys &ph, const T *u, const T *v, T *y, T *hp, cudaStream_t s)
{
    hvp_tile<T, HVP_CG>(c, ph, HvpIn<T>{u, nullptr, eact<T>(c)}, v, y, hp, s);
}

template <typename T>
void launch_hvp_tile_only(const Ctx &c, const Phys &ph, const T *u, const T *v, T *y, T *hp, cudaStream_t s)
{
    hvp_tile<T, HVP_STATE>(c, ph, HvpIn<T>{u, nullptr, eact<T>(c)}, v, y, hp, s);
}

template <typename T>
void launch_hvp_finalize_only(const Ctx &c, const Phys &ph, const T *u, const T *v, T *y, const T *hp,
                              cudaStream_t s)
{
    hvp_fin<T>(c, ph, HvpIn<T>{u, nullptr, eact<T>(c)}, v, y, hp, s);
}

void launch_param_vjp(const Ctx &c, const Phys &ph, const double *u, const double *a, const double *lam,
                      double *dLda, cudaStream_t s)
{
    c.n_launch += 1;
    const size_t sm = smem_verts(c, sizeof(double), 2);
    if (c.dim == 2)
        k_tile_vjp<2><<<c.td.n_tiles, c.threads, sm, s>>>(c.td, c.e64, c.vd, ph, u, a, lam, dLda);
    else
        k_tile_vjp<3><<<c.td.n_tiles, c.threads, sm, s>>>(c.td, c.e64, c.vd, ph, u, a, lam, dLda);
}

void launch_material_vjp(const Ctx &c, const Phys &ph, const double *u, const double *a, const double *lam,
                         double *dmu, double *dlam, double *dk, cudaStream_t s)
{
    c.n_launch += 1;
    const size_t sm = smem_verts(c, sizeof(double), 2);
    if (c.dim == 2)
        k_tile_mat_vjp<2><<<c.td.n_tiles, c.threads, sm, s>>>(c.td, c.e64, c.vd, ph, u, a, lam, dmu, dlam, dk);
    else
        k_tile_mat_vjp<3><<<c.td.n_tiles, c.threads, sm, s>>>(c.td, c.e64, c.vd, ph, u, a, lam, dmu, dlam, dk);
}

// Opt every kernel that may need more than 48 KB of dynamic shared memory into
// the larger carve-out.
cudaError_t configure_elem_kernels()
{
    const int big = 200 * 1024;
    cudaError_t e = cudaSuccess;
#define SET(k) \
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, big)
    SET((k_tile_energy<2>));
    SET((k_tile_energy<3>));
    SET((k_tile_grad<2, false>));
    SET((k_tile_grad<3, false>));
    SET((k_tile_grad<2, true>));
    SET((k_tile_grad<3, true>));
#define SET_MODE(T, MB, M)                                                \
    SET((k_tile_hvp<T, 2, M, MB, 0, false>));                             \
    SET((k_tile_hvp<T, 3, M, MB, 0, false>));                             \
    SET((k_tile_hvp<T, 2, M, MB, 0, true>));                              \
    SET((k_tile_hvp<T, 3, M, MB, 0, true>));                              \
    SET((k_tile_hvp<T, 2, M, MB, (sizeof(T) == 4 ? kCap2 : 0), false>));  \
    SET((k_tile_hvp<T, 3, M, MB, (sizeof(T) == 4 ? kCap3 : 0), false>));
#define SET_HVP(T, MB)          \
    SET_MODE(T, MB, HVP_STATE)  \
    SET_MODE(T, MB, HVP_CG)     \
    SET_MODE(T, MB, HVP_CALLER)
    SET_HVP(float, 3)
    SET_HVP(float, 4)
    SET_HVP(double, 1)
    SET_HVP(double, 2)
#undef SET_HVP
#undef SET_MODE
    SET((k_tile_vjp<2>));
    SET((k_tile_vjp<3>));
    SET((k_tile_mat_vjp<2>));
    SET((k_tile_mat_vjp<3>));
#undef SET
    return e;
}

template void launch_hvp<float>(const Ctx &, const Phys &, const float *, const float *, float *, float *,
                                cudaStream_t);
template void launch_hvp<double>(const Ctx &, const Phys &, const double *, const double *, double *, double *,
                                 cudaStream_t);
template void launch_hvp_at<float>(const Ctx &, const Phys &, const double *, const double *, const float *, float *,
                                   float *, cudaStream_t);
template void launch_hvp_at<double>(const Ctx &, const Phys &, const double *, const double *, const double *,
                                    double *, double *, cudaStream_t);
template void launch_hvp_cg<float>(const Ctx &, const Phys &, const float *, const float *, float *, float *,
                                   cudaStream_t);
template void launch_hvp_cg<double>(const Ctx &, const Phys &, const double *, const double *, double *, double *,
                                    cudaStream_t);
template void launch_hvp_tile_only<float>(const Ctx &, const Phys &, const float *, const float *, float *, float *,
                                          cudaStream_t);
template void launch_hvp_tile_only<double>(const Ctx &, const Phys &, const double *, const double *, double *,
                                           double *, cudaStream_t);
template void launch_hvp_finalize_only<float>(const Ctx &, const Phys &, const float *, const float *, float *,
                                              const float *, cudaStream_t);
template void launch_hvp_finalize_only<double>(const Ctx &, const Phys &, const double *, const double *,
                                               double *, const double *, cudaStream_t);
template size_t hvp_smem<float>(const Ctx &);
template size_t hvp_smem<double>(const Ctx &);

}  // namespace softsim
