// Batched persistent solver: many independent meshes of uneven size, each
// simulated for n_steps backward-Euler steps (Eq. opt-be) and then
// differentiated by backpropagation through time (Sec. 4: implicit
// differentiation of each step, Eq. dLda-re-ordered, plus plain backprop of
// v1 = (x1 - x0)/h), all inside ONE kernel launch.
//
// Every team -- a thread-block cluster for the largest meshes when meshes are
// few or uneven, then each of its CTAs for itself -- takes the next mesh
// (largest first) from an integer work counter and runs that mesh's whole forward rollout and backward pass: Newton-CG
// with backtracking for every step, then for every step in reverse the
// adjoint CG solve with FP64 refinement and the parameter VJP
// (batched_kernel.cuh).  A mesh is always computed by a team of the same size
// and thread count with fixed-order sums, so results do not depend on which
// team takes it.
//
// Precision follows the single-mesh mixed path: FP32 HVP and CG vectors,
// FP64 state, gradient, energies and adjoint residuals, compensated FP32 dot
// products in CG.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <numeric>
#include <string>
#include <vector>

#include "batched_kernel.cuh"
#include "cg_pcg_host.h"
#include "host_parallel.h"

using namespace softsim;

namespace {

constexpr int kBatchThreads = 256;

thread_local std::string g_batch_error;

}  // namespace

static BatchKernel batch_kernel(int dim, int threads)
{
    return dim == 2 ? batch_kernel_2d(threads) : batch_kernel_3d(threads);
}

struct sim_batch {
    int M = 0, dim = 0;
    int64_t V = 0, E = 0;
    BatchDev dev;
    std::vector<void *> allocs;
    std::vector<int64_t> voff, eoff;
    int threads = kBatchThreads;  // threads per CTA
    size_t smem = 0;              // dynamic shared memory of a CTA
    std::string err;

    cudaLaunchConfig_t config(cudaStream_t s, cudaLaunchAttribute *at) const
    {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(dev.team);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = dev.team;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = dev.team > 1 ? 1 : 0;
        return cfg;
    }
};

static int bfail(sim_batch *b, int code, const std::string &msg)
{
    if (b)
        b->err = msg;
    else
        g_batch_error = msg;
    return code;
}

#define BCK(b, call)                                                                          \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return bfail((b), SIM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

template <typename V>
static V *bupload(sim_batch *b, const std::vector<V> &v)
{
    void *p = nullptr;
    if (cudaMalloc(&p, std::max<size_t>(v.size() * sizeof(V), 16)) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    b->allocs.push_back(p);
    if (!v.empty() && cudaMemcpy(p, v.data(), v.size() * sizeof(V), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return static_cast<V *>(p);
}

template <typename V>
static V *balloc(sim_batch *b, size_t n)
{
    void *p = nullptr;
    if (cudaMalloc(&p, std::max<size_t>(n * sizeof(V), 16)) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    b->allocs.push_back(p);
    return static_cast<V *>(p);
}

extern "C" const char *sim_batch_last_error(const sim_batch *b) { return b ? b->err.c_str() : g_batch_error.c_str(); }

extern "C" int sim_batch_destroy(sim_batch *b)
{
    if (!b) return SIM_EINVAL;
    for (void *p : b->allocs) cudaFree(p);
    delete b;
    return SIM_OK;
}

// How the meshes are shared out: the first n_big of the order (largest first) go
// to teams of `team` CTAs, the others to single CTAs, which the teams' CTAs become
// when the large meshes are done.
struct Share {
    int team = 1, n_big = 0;
};

// A mesh's rollout is one serial chain, so the largest meshes decide when they
// are few or uneven, and small ones waste the CTAs of a team.  The end of the
// launch is modelled from a step's cost, in microseconds (measured at 120 to
// 4,140 vertices on teams of 1, 2 and 4), for every team size and a few sizes of
// n_big.  More than four vertices a thread cost a CG iteration 26 us at 2,070
// vertices a CTA, where four cost 15 at 1,900 (256 bodies of 200 to 8,000
// triangles: 66.7 ms with the iteration taken as linear, 63.5 like this);
// meshes above eight have no assembled CG.
static Share share_out(const std::vector<int64_t> &nv_sorted, const int n_teams[5], int sms, int threads)
{
    const int M = (int)nv_sorted.size();
    auto cost = [&](int64_t nv, int c) {
        const double v = (double)nv / c;
        const double its = 110.0 + (c == 1 ? 0.125 : 0.082) * (double)nv;
        const double it = v > 4.0 * threads - 64.0 ? 21.5 + 2.25e-3 * v : c == 1 ? 4.3 + 6.4e-3 * v : 4.9 + 5.0e-3 * v;
        return (its * it + 270.0 + 1.6 * v) * (v > (double)kBatchVpt * threads - 256.0 ? 10.0 : 1.0);
    };
    Share best;
    double best_t = INFINITY;
    for (int lg = 0; lg < 5; ++lg) {
        const int c = 1 << lg, teams = lg == 0 ? sms : n_teams[lg];
        if (teams < 1) continue;
        for (int q = lg == 0 ? 16 : 0; q <= 16; ++q) {
            // n_big: all (q = 16), or the largest 1, 2, 4, ... meshes
            const int k = lg == 0 ? 0 : q == 16 ? M : std::min<int>(M, 1 << q);
            std::vector<double> end(std::min(teams, std::max(M, 1)), 0.0);  // min-heap of ends
            auto later = [](double a, double b) { return a > b; };
            auto give = [&](double w) {
                std::pop_heap(end.begin(), end.end(), later);
                end.back() += w;
                std::push_heap(end.begin(), end.end(), later);
            };
            for (int m = 0; m < k; ++m) give(cost(nv_sorted[m], c));
            std::vector<double> solo;
            for (double e : end) solo.insert(solo.end(), c, e);
            end.swap(solo);
            std::make_heap(end.begin(), end.end(), later);
            for (int m = k; m < M; ++m) give(cost(nv_sorted[m], 1));
            const double t = *std::max_element(end.begin(), end.end());
            if (t < 0.97 * best_t) {
                best_t = t;
                best.team = c;
                best.n_big = k;
            }
            if (k == M && q < 16) break;
        }
    }
    return best;
}

// Plans of the meshes' CG solves; a mesh that does not fit one is left to the
// matrix-free iteration.
static int build_plans(sim_batch *bt, const sim_mesh *meshes, const std::vector<int32_t> &order)
{
    const int M = bt->M, d = bt->dim, nm = d == 3 ? 6 : 3;
    BatchDev &b = bt->dev;
    const BatchKernel k = batch_kernel(d, bt->threads);
    int dev = 0, sms = 0, n_teams[5] = {0};
    cudaFuncAttributes fa;
    BCK(bt, cudaGetDevice(&dev));
    BCK(bt, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    BCK(bt, cudaFuncGetAttributes(&fa, k));
    bt->smem = kBatchPlanAt + (sizeof(PcgDev) + 15) / 16 * 16;
    if (fa.sharedSizeBytes + bt->smem > kPcgSmem) return bfail(bt, SIM_ECUDA, "shared memory larger than planned");
    BCK(bt, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bt->smem));
    BCK(bt, cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    std::vector<int64_t> nv(M), ne(M);
    for (int m = 0; m < M; ++m) nv[m] = meshes[m].n_vert, ne[m] = meshes[m].n_elem;
    for (int lg = 1; lg < 5; ++lg) {
        cudaLaunchAttribute at[1];
        b.team = 1 << lg;
        const cudaLaunchConfig_t cfg = bt->config(nullptr, at);
        if (cudaOccupancyMaxActiveClusters(&n_teams[lg], k, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n_teams[lg] = 0;
        }
    }
    std::vector<int64_t> nv_sorted(M);
    std::vector<int> place(M);  // of a mesh in the order
    for (int k = 0; k < M; ++k) {
        nv_sorted[k] = nv[order[k]];
        place[order[k]] = k;
    }
    const Share share = share_out(nv_sorted, n_teams, sms, bt->threads);
    b.team = share.team;
    b.n_big = share.n_big;
    std::vector<CgPlan> plans(M);
    std::vector<char> ok(M, 0);
    std::vector<PcgDev> pds(M);
    parallel_for(bt->V, M, 1, [&](int64_t m) {
        std::vector<int32_t> perm(ne[m]);
        std::iota(perm.begin(), perm.end(), 0);
        std::string err;
        const int c = place[m] < b.n_big ? b.team : 1;
        int a = (int)std::max<int64_t>(1, std::min<int64_t>({96 / nm, 16 * c, nv[m] / 18}));
        if (a > c) a = c * aggregates_per_part((nv[m] + c - 1) / c, a / c, bt->threads);
        ok[m] = build_cg_plan(d, nv[m], ne[m], meshes[m].rest_pos, meshes[m].elems, perm.data(), ne[m], c, a, true,
                              sizeof(float), false, plans[m], err) &&
                batch_plan_fits(plans[m], bt->threads);
        if (!ok[m]) return;
        pcg_sizes_of(plans[m], c > 1, true, pds[m]);
        pds[m].threads = bt->threads;
    });
    size_t table_bytes = 0, buffer_bytes = 0;
    for (int m = 0; m < M; ++m)
        if (ok[m]) {
            table_bytes = pcg_place_tables(plans[m], pds[m], nullptr, nullptr, table_bytes);
            buffer_bytes = pcg_place_buffers<float>(plans[m], pds[m], nullptr, buffer_bytes);
        }
    unsigned char *d0 = balloc<unsigned char>(bt, table_bytes), *d1 = d0 ? balloc<unsigned char>(bt, buffer_bytes) : nullptr;
    if (!d1) {  // without the memory for them the matrix-free iteration, which needs none, does the solves
        if (d0) {
            cudaFree(d0);
            bt->allocs.pop_back();
        }
        table_bytes = 0;
        ok.assign(M, 0);
    }
    std::vector<unsigned char> host(table_bytes);
    size_t at = 0, bat = 0;
    for (int m = 0; m < M; ++m) {
        if (!ok[m]) {
            pds[m] = PcgDev();
            continue;
        }
        at = pcg_place_tables(plans[m], pds[m], host.data(), d0, at);
        bat = pcg_place_buffers<float>(plans[m], pds[m], d1, bat);
    }
    if (table_bytes) BCK(bt, cudaMemcpy(d0, host.data(), table_bytes, cudaMemcpyHostToDevice));
    b.pcg = bupload(bt, pds);
    if (!b.pcg) return bfail(bt, SIM_ENOMEM, "device allocation or upload failed");
    // the uploads lie on the default stream, which a rollout on a non-blocking stream does not wait for
    BCK(bt, cudaStreamSynchronize(nullptr));
    return SIM_OK;
}

static int batch_create_impl(sim_batch *bt, int M, const sim_mesh *meshes, const sim_material *mats,
                             const sim_options *opt)
{
    const int d = meshes[0].dim;
    const int nc = d + 1;
    bt->M = M;
    bt->dim = d;
    sim_options o;
    if (opt)
        o = *opt;
    else
        sim_default_options(&o);
    if (o.threads != 0 && o.threads != 128 && o.threads != 256 && o.threads != 512)
        return bfail(bt, SIM_EINVAL, "batched threads per mesh must be 0 (default 256), 128, 256 or 512");
    bt->threads = o.threads ? o.threads : kBatchThreads;
    bt->voff.assign(M + 1, 0);
    bt->eoff.assign(M + 1, 0);
    for (int m = 0; m < M; ++m) {
        if (meshes[m].dim != d) return bfail(bt, SIM_EINVAL, "all meshes of a batch must have the same dim");
        if (meshes[m].n_vert <= 0 || meshes[m].n_elem <= 0 || !meshes[m].rest_pos || !meshes[m].elems)
            return bfail(bt, SIM_EINVAL, "empty mesh in batch");
        if (!(mats[m].dt > 0.0)) return bfail(bt, SIM_EINVAL, "batched rollouts need dt > 0");
        bt->voff[m + 1] = bt->voff[m] + meshes[m].n_vert;
        bt->eoff[m + 1] = bt->eoff[m] + meshes[m].n_elem;
    }
    const sim_material &m0 = mats[0];
    for (int m = 1; m < M; ++m)
        if (mats[m].k_muscle != m0.k_muscle || mats[m].gravity != m0.gravity || mats[m].k_contact != m0.k_contact ||
            mats[m].contact_power != m0.contact_power || mats[m].log_mode != m0.log_mode || mats[m].dt != m0.dt ||
            mats[m].density != m0.density || mats[m].k_friction != m0.k_friction ||
            mats[m].eps_friction != m0.eps_friction || mats[m].muscle_model != m0.muscle_model)
            return bfail(bt, SIM_EINVAL, "batched meshes may differ only in mu and lambda");
    if (!(m0.k_friction >= 0.0) || !std::isfinite(m0.k_friction) || !std::isfinite(m0.eps_friction))
        return bfail(bt, SIM_EINVAL, "k_friction must be finite and >= 0, eps_friction finite");
    if (m0.contact_power != 2 && m0.contact_power != 3) return bfail(bt, SIM_EINVAL, "contact_power must be 2 or 3");
    if (m0.muscle_model != SIM_MUSCLE_CONTRACTILE && m0.muscle_model != SIM_MUSCLE_SPRING)
        return bfail(bt, SIM_EINVAL, "muscle_model must be SIM_MUSCLE_CONTRACTILE or SIM_MUSCLE_SPRING");
    const int64_t V = bt->voff[M], E = bt->eoff[M];
    bt->V = V;
    bt->E = E;
    const int nf = d * d + 2 * d + 1;
    std::vector<double> X(V * d), mass(V, 0.0), e64((size_t)nf * E, 0.0), mu(M), lam(M);
    std::vector<uint8_t> fixed(V, 0);
    std::vector<int32_t> conn(E * nc), vinc(E * nc);
    std::vector<int64_t> vinc_ptr(V + 1, 0);
    for (int m = 0; m < M; ++m) {
        const sim_mesh &mh = meshes[m];
        const int64_t v0 = bt->voff[m], e0 = bt->eoff[m];
        mu[m] = mats[m].mu;
        lam[m] = mats[m].lambda;
        for (int64_t i = 0; i < mh.n_vert * d; ++i) X[v0 * d + i] = mh.rest_pos[i];
        if (mh.fixed)
            for (int64_t i = 0; i < mh.n_vert; ++i) fixed[v0 + i] = mh.fixed[i] ? 1 : 0;
        for (int64_t e = 0; e < mh.n_elem; ++e) {
            const int32_t *t = mh.elems + e * nc;
            for (int k = 0; k < nc; ++k) {
                if (t[k] < 0 || t[k] >= mh.n_vert) return bfail(bt, SIM_EINVAL, "element vertex id out of range");
                conn[(e0 + e) * nc + k] = t[k];
                vinc_ptr[v0 + t[k] + 1] += 1;
            }
            double Dm[3][3] = {{0}}, B[3][3] = {{0}}, det;
            for (int k = 0; k < d; ++k)
                for (int i = 0; i < d; ++i) Dm[i][k] = mh.rest_pos[(int64_t)t[k + 1] * d + i] - mh.rest_pos[(int64_t)t[0] * d + i];
            if (d == 2) {
                det = Dm[0][0] * Dm[1][1] - Dm[0][1] * Dm[1][0];
                B[0][0] = Dm[1][1] / det;
                B[0][1] = -Dm[0][1] / det;
                B[1][0] = -Dm[1][0] / det;
                B[1][1] = Dm[0][0] / det;
            } else {
                double C[3][3];
                for (int j = 0; j < 3; ++j) {
                    const int a = (j + 1) % 3, c = (j + 2) % 3;
                    C[0][j] = Dm[1][a] * Dm[2][c] - Dm[2][a] * Dm[1][c];
                    C[1][j] = Dm[2][a] * Dm[0][c] - Dm[0][a] * Dm[2][c];
                    C[2][j] = Dm[0][a] * Dm[1][c] - Dm[1][a] * Dm[0][c];
                }
                det = Dm[0][0] * C[0][0] + Dm[1][0] * C[1][0] + Dm[2][0] * C[2][0];
                for (int i = 0; i < 3; ++i)
                    for (int j = 0; j < 3; ++j) B[i][j] = C[j][i] / det;
            }
            if (!(det > 0.0)) return bfail(bt, SIM_EINVERTED, "element with non-positive rest volume");
            const double W = det / (d == 2 ? 2.0 : 6.0);
            double f[3] = {0, 0, 0};
            if (mats[m].fiber)
                for (int c = 0; c < d; ++c) f[c] = mats[m].fiber[e * d + c];
            const int64_t ge = e0 + e;
            for (int i = 0; i < d; ++i)
                for (int j = 0; j < d; ++j) e64[(size_t)(i * d + j) * E + ge] = B[i][j];
            for (int i = 0; i < d; ++i) {
                double s = 0.0;
                for (int j = 0; j < d; ++j) s += B[i][j] * f[j];
                e64[(size_t)(d * d + i) * E + ge] = s;
                e64[(size_t)(d * d + d + 1 + i) * E + ge] = f[i];
            }
            e64[(size_t)(d * d + d) * E + ge] = W;
            for (int k = 0; k < nc; ++k) mass[v0 + t[k]] += mats[m].density * W / nc;
        }
    }
    for (int64_t v = 0; v < V; ++v) vinc_ptr[v + 1] += vinc_ptr[v];
    {
        std::vector<int64_t> fill(vinc_ptr.begin(), vinc_ptr.end() - 1);
        for (int m = 0; m < M; ++m) {
            const int64_t v0 = bt->voff[m], e0 = bt->eoff[m], ne = bt->eoff[m + 1] - e0;
            for (int64_t e = 0; e < ne; ++e)
                for (int k = 0; k < nc; ++k) vinc[fill[v0 + conn[(e0 + e) * nc + k]]++] = (int32_t)(e * nc + k);
        }
    }
    std::vector<int32_t> order(M);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
        return bt->eoff[a + 1] - bt->eoff[a] > bt->eoff[c + 1] - bt->eoff[c];
    });
    std::vector<float> e32(e64.begin(), e64.end());
    BatchDev &b = bt->dev;
    b.M = M;
    b.dim = d;
    b.voff = bupload(bt, bt->voff);
    b.eoff = bupload(bt, bt->eoff);
    b.order = bupload(bt, order);
    b.X = bupload(bt, X);
    b.mass = bupload(bt, mass);
    b.fixed = bupload(bt, fixed);
    b.conn = bupload(bt, conn);
    b.vinc_ptr = bupload(bt, vinc_ptr);
    b.vinc = bupload(bt, vinc);
    b.e32 = bupload(bt, e32);
    b.e64 = bupload(bt, e64);
    b.estride = E;
    b.mu = bupload(bt, mu);
    b.lam = bupload(bt, lam);
    b.k = m0.k_muscle;
    b.grav = m0.gravity;
    b.kc = m0.k_contact;
    b.dt = m0.dt;
    b.kf = m0.k_friction;
    b.k_f = (float)m0.k_muscle;
    b.dt2_f = (float)(m0.dt * m0.dt);
    b.feps = m0.eps_friction;
    b.cpow = m0.contact_power;
    b.log_mode = m0.log_mode;
    b.muscle = m0.muscle_model;
    b.newton_rtol = o.newton_rtol;
    b.adj_rtol = o.adjoint_rtol;
    b.max_newton = o.max_newton;
    b.max_cg = o.max_cg;
    b.max_adj_cg = o.max_adjoint_cg > 0 ? o.max_adjoint_cg : 2000;
    b.max_ls = o.max_ls;
    const size_t VD = (size_t)V * d;
    b.u = balloc<double>(bt, VD);
    b.uhat = balloc<double>(bt, VD);
    b.g = balloc<double>(bt, VD);
    b.w64 = balloc<double>(bt, VD);
    b.r64 = balloc<double>(bt, VD);
    b.Hx = balloc<double>(bt, VD);
    b.lacc = balloc<double>(bt, VD);
    b.xbar = balloc<double>(bt, VD);
    b.vbar = balloc<double>(bt, VD);
    if (b.kf > 0.0) {
        b.fw = balloc<double>(bt, V);
        b.u0 = balloc<double>(bt, VD);
    }
    b.u32 = balloc<float>(bt, VD);
    b.a32 = balloc<float>(bt, (size_t)E);
    b.dg32 = balloc<float>(bt, (size_t)2 * V);
    b.d = balloc<float>(bt, VD);
    b.r = balloc<float>(bt, VD);
    b.p = balloc<float>(bt, VD);
    b.Ap = balloc<float>(bt, VD);
    b.c32 = balloc<float>(bt, (size_t)E * nc * d);
    b.c64 = balloc<double>(bt, (size_t)E * nc * d);
    b.counter = balloc<int>(bt, 2);
    b.mstat = balloc<int>(bt, (size_t)4 * M);
    b.mgrad = balloc<double>(bt, (size_t)3 * M);
    const void *ptrs[] = {b.voff, b.eoff, b.order, b.X, b.mass, b.fixed, b.conn, b.vinc_ptr, b.vinc, b.e32, b.e64,
                          b.mu, b.lam, b.u, b.uhat, b.g, b.w64, b.r64, b.Hx, b.lacc, b.xbar, b.vbar, b.u32,
                          b.d, b.r, b.p, b.Ap, b.c32, b.c64, b.counter, b.mstat, b.mgrad, b.a32, b.dg32};
    for (const void *p : ptrs)
        if (!p) return bfail(bt, SIM_ENOMEM, "device allocation or upload failed");
    if (b.kf > 0.0 && (!b.fw || !b.u0)) return bfail(bt, SIM_ENOMEM, "device allocation failed");
    try {
        return build_plans(bt, meshes, order);
    } catch (const std::exception &e) {
        return bfail(bt, SIM_ENOMEM, e.what());
    }
}

extern "C" int sim_batch_create(int n_meshes, const sim_mesh *meshes, const sim_material *mats,
                                const sim_options *opt, sim_batch **out)
{
    if (out) *out = nullptr;
    if (n_meshes <= 0 || !meshes || !mats || !out) return bfail(nullptr, SIM_EINVAL, "bad batch arguments");
    if (meshes[0].dim != 2 && meshes[0].dim != 3) return bfail(nullptr, SIM_EINVAL, "dim must be 2 or 3");
    sim_batch *b = new sim_batch();
    const int rc = batch_create_impl(b, n_meshes, meshes, mats, opt);
    if (rc != SIM_OK) {
        g_batch_error = b->err;
        sim_batch_destroy(b);
        return rc;
    }
    *out = b;
    return SIM_OK;
}

extern "C" int sim_batch_sizes(const sim_batch *b, int *n_meshes, int64_t *total_vert, int64_t *total_elem)
{
    if (!b) return SIM_EINVAL;
    if (n_meshes) *n_meshes = b->M;
    if (total_vert) *total_vert = b->V;
    if (total_elem) *total_elem = b->E;
    return SIM_OK;
}

extern "C" int sim_batch_rollout(sim_batch *bt, int n_steps, double *states_x, double *states_v, const double *a_seq,
                                 const double *xbarT, const double *vbarT, double *abar_seq, double *xbar0,
                                 double *vbar0, int *mesh_stats, double *mat_grad, void *stream)
{
    if (!bt) return SIM_EINVAL;
    if (n_steps <= 0 || !states_x || !states_v || !a_seq || !xbarT || !vbarT || !abar_seq || !xbar0 || !vbar0)
        return bfail(bt, SIM_EINVAL, "null or bad rollout argument");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const BatchDev &b = bt->dev;
    const size_t VD = (size_t)bt->V * bt->dim;
    const BatchKernel kfun = batch_kernel(bt->dim, bt->threads);
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = bt->config(s, at);
    int n_teams = 0;
    if (b.team > 1) {
        BCK(bt, cudaOccupancyMaxActiveClusters(&n_teams, kfun, &cfg));
    } else {
        int dev = 0;
        BCK(bt, cudaGetDevice(&dev));
        BCK(bt, cudaDeviceGetAttribute(&n_teams, cudaDevAttrMultiProcessorCount, dev));
    }
    // no more teams than meshes; a team's CTAs take single meshes after the large ones
    const int want = b.n_big + (bt->M - b.n_big + b.team - 1) / b.team;
    cfg.gridDim = dim3((unsigned)(b.team * std::max(1, std::min(want, n_teams))));
    BCK(bt, cudaMemsetAsync(b.counter, 0, 2 * sizeof(int), s));
    BCK(bt, cudaLaunchKernelEx(&cfg, kfun, b, n_steps, a_seq, states_x, states_v, xbarT, vbarT, abar_seq, bt->V, bt->E));
    BCK(bt, cudaMemcpyAsync(xbar0, b.xbar, VD * sizeof(double), cudaMemcpyDeviceToDevice, s));
    BCK(bt, cudaMemcpyAsync(vbar0, b.vbar, VD * sizeof(double), cudaMemcpyDeviceToDevice, s));
    if (mesh_stats) BCK(bt, cudaMemcpyAsync(mesh_stats, b.mstat, sizeof(int) * 4 * bt->M, cudaMemcpyDeviceToDevice, s));
    if (mat_grad) BCK(bt, cudaMemcpyAsync(mat_grad, b.mgrad, sizeof(double) * 3 * bt->M, cudaMemcpyDeviceToDevice, s));
    return SIM_OK;
}
