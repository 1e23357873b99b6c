// Device side of the preconditioned conjugate gradients on assembled edge
// blocks: the solve of one CTA's part, shared by the persistent solver of one
// mesh (cg_pcg_kernel.cuh) and the batched solver (batched_kernel.cuh).
#pragma once

#include <cstdint>
#include <type_traits>

#include "cg_pcg.h"
#include "grid_sync.cuh"
#include "reduce.cuh"
#include "tma.cuh"

namespace softsim {

namespace {

constexpr int kMaxWarps = 16;

template <typename T, int D>
struct Row;  // published vector row: D values in 8- or 16-byte units
template <>
struct Row<float, 3> {
    static constexpr int N = 4;
};
template <>
struct Row<float, 2> {
    static constexpr int N = 2;
};
template <>
struct Row<double, 3> {
    static constexpr int N = 4;
};
template <>
struct Row<double, 2> {
    static constexpr int N = 2;
};

template <typename T, int D>
__device__ __forceinline__ void put_row(T *z, const T v[D])
{
    if constexpr (sizeof(T) == 4 && D == 3) {
        *reinterpret_cast<float4 *>(z) = make_float4(v[0], v[1], v[2], 0.0f);
    } else if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float2 *>(z) = make_float2(v[0], v[1]);
    } else {
        *reinterpret_cast<double2 *>(z) = make_double2(v[0], v[1]);
        if constexpr (D == 3) z[2] = v[2];
    }
}

template <typename T, int D>
__device__ __forceinline__ void get_row(const T *z, T v[D])
{
    if constexpr (sizeof(T) == 4 && D == 3) {
        const float4 a = __ldcg(reinterpret_cast<const float4 *>(z));
        v[0] = a.x, v[1] = a.y, v[2] = a.z;
    } else if constexpr (sizeof(T) == 4) {
        const float2 a = __ldcg(reinterpret_cast<const float2 *>(z));
        v[0] = a.x, v[1] = a.y;
    } else {
        const double2 a = __ldcg(reinterpret_cast<const double2 *>(z));
        v[0] = a.x, v[1] = a.y;
        if constexpr (D == 3) v[2] = __ldcg(z + 2);
    }
}

// z += Z c at a vertex with arm R (c: the aggregate's coarse values)
template <typename T, int D>
__device__ __forceinline__ void prolong_add(float4 R, const float *c, T z[D])
{
    if constexpr (D == 3) {
        z[0] += T(c[0] + c[4] * R.z - c[5] * R.y);
        z[1] += T(c[1] + c[5] * R.x - c[3] * R.z);
        z[2] += T(c[2] + c[3] * R.y - c[4] * R.x);
    } else {
        z[0] += T(c[0] - c[2] * R.y);
        z[1] += T(c[1] + c[2] * R.x);
    }
}

// acc += Z^T f
template <int D>
__device__ __forceinline__ void restrict_to(float4 R, const float f[D], float *acc)
{
#pragma unroll
    for (int c = 0; c < D; ++c) acc[c] += f[c];
    if constexpr (D == 3) {
        acc[3] += R.y * f[2] - R.z * f[1];
        acc[4] += R.z * f[0] - R.x * f[2];
        acc[5] += R.x * f[1] - R.y * f[0];
    } else {
        acc[2] += R.x * f[1] - R.y * f[0];
    }
}

template <typename V>
__device__ __forceinline__ V warp_all(V v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of eight values over a warp with nine shuffles: each step halves the
// values a lane carries; lane l ends with the total of value (l >> 2) & 7.
__device__ __forceinline__ float warp_sum8(const float v[8])
{
    const int lane = threadIdx.x & 31;
    float a[4], b[2], c;
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        a[i] = (h4 ? v[i + 4] : v[i]) + __shfl_xor_sync(0xffffffffu, h4 ? v[i] : v[i + 4], 16);
#pragma unroll
    for (int i = 0; i < 2; ++i) b[i] = (h3 ? a[i + 2] : a[i]) + __shfl_xor_sync(0xffffffffu, h3 ? a[i] : a[i + 2], 8);
    c = (h2 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h2 ? b[0] : b[1], 4);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    return c + __shfl_xor_sync(0xffffffffu, c, 1);
}

// Inverse of the symmetric block S (xx, xy, yy | xx, xy, xz, yy, yz, zz); a
// block that is not positive definite becomes a multiple of the identity.
template <typename T, int D>
__device__ __forceinline__ void invert_sym(const T *S, T *out)
{
    if constexpr (D == 2) {
        const T det = S[0] * S[2] - S[1] * S[1];
        if (S[0] > T(0) && det > T(1e-6) * S[0] * S[2]) {
            const T i = T(1) / det;
            out[0] = S[2] * i;
            out[1] = -S[1] * i;
            out[2] = S[0] * i;
        } else {
            const T t = fabs(S[0]) + fabs(S[2]), i = t > T(0) ? T(1) / t : T(0);
            out[0] = out[2] = i;
            out[1] = T(0);
        }
    } else {
        const T a = S[3] * S[5] - S[4] * S[4], b = S[2] * S[4] - S[1] * S[5], c = S[1] * S[4] - S[2] * S[3];
        const T det = S[0] * a + S[1] * b + S[2] * c, m = S[0] * S[3] - S[1] * S[1];
        if (S[0] > T(0) && m > T(1e-6) * S[0] * S[3] && det > T(1e-6) * m * S[5]) {
            const T i = T(1) / det;
            out[0] = a * i;
            out[1] = b * i;
            out[2] = c * i;
            out[3] = (S[0] * S[5] - S[2] * S[2]) * i;
            out[4] = (S[1] * S[2] - S[0] * S[4]) * i;
            out[5] = m * i;
        } else {
            const T t = fabs(S[0]) + fabs(S[3]) + fabs(S[5]), i = t > T(0) ? T(1) / t : T(0);
            out[0] = out[3] = out[5] = i;
            out[1] = out[2] = out[4] = T(0);
        }
    }
}

template <typename T, int D>
__device__ __forceinline__ void sym_mul(const T *S, const T r[D], T z[D])
{
    if constexpr (D == 2) {
        z[0] = S[0] * r[0] + S[1] * r[1];
        z[1] = S[1] * r[0] + S[2] * r[1];
    } else {
        z[0] = S[0] * r[0] + S[1] * r[1] + S[2] * r[2];
        z[1] = S[1] * r[0] + S[3] * r[1] + S[4] * r[2];
        z[2] = S[2] * r[0] + S[4] * r[1] + S[5] * r[2];
    }
}

// Inner products of the solver.  FP32: a pair (hi, lo) whose sums are all
// compensated (TwoSum, Knuth), about 48 bits where FP64 would cost 64 times the
// issue slots; FP64: a double.
template <typename T>
struct DotOf {
    using Type = double;
};
template <>
struct DotOf<float> {
    using Type = float2;
};

// s + e == a + b exactly, in intrinsics: contracting a product into the sum would lose its error.
__device__ __forceinline__ void two_sum_rn(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// v += x . y of one vertex.  EXACT: with the rounding errors of the products
// too (dot product of Ogita, Rump and Oishi 2005), else they come from one FMA
// chain.  first: v is zero.
template <int D, bool EXACT>
__device__ __forceinline__ void dot_add(float2 &v, const float *x, const float *y, bool first)
{
    float p = __fmul_rn(x[0], y[0]), e = 0.0f;
    if (EXACT) e = __fmaf_rn(x[0], y[0], -p);
#pragma unroll
    for (int c = 1; c < D; ++c) {
        if (EXACT) {
            const float q = __fmul_rn(x[c], y[c]), eq = __fmaf_rn(x[c], y[c], -q);
            float es;
            two_sum_rn(p, q, p, es);
            e = __fadd_rn(e, __fadd_rn(eq, es));
        } else {
            p = __fmaf_rn(x[c], y[c], p);
        }
    }
    if (first) {
        v = make_float2(p, e);
        return;
    }
    float es;
    two_sum_rn(v.x, p, v.x, es);
    v.y = __fadd_rn(v.y, __fadd_rn(e, es));
}
template <int D, bool EXACT>
__device__ __forceinline__ void dot_add(double &v, const double *x, const double *y, bool)
{
#pragma unroll
    for (int c = 0; c < D; ++c) v += x[c] * y[c];
}

// The sum of two partial dots; the same bits whichever comes first.
__device__ __forceinline__ float2 dot_merge(float2 a, float2 b)
{
    float2 r;
    two_sum(a.x, b.x, r.x, r.y);
    r.y += a.y + b.y;
    return r;
}

__device__ __forceinline__ double dot_merge(double a, double b) { return a + b; }

__device__ __forceinline__ float2 dot_xor(float2 v, int o)
{
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}
__device__ __forceinline__ double dot_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }

// Sums over groups of 2 K lanes, the same in every lane of a group.  (Two digits of
// fixed point added by the integer reduction instructions instead of the shuffles:
// slower, 4.3 to 4.6 us an iteration on the walker.)
template <int K, typename V>
__device__ __forceinline__ V group_dot(V v)
{
#pragma unroll
    for (int o = K; o > 0; o >>= 1) v = dot_merge(v, dot_xor(v, o));
    return v;
}

// The dot rounded to FP32.
__device__ __forceinline__ float dot_value(float2 v) { return v.x + v.y; }
__device__ __forceinline__ double dot_value(double v) { return v; }

// a / b rounded to FP32: a quotient good to a few units and the remainder it leaves.
__device__ __forceinline__ float dot_quot(float2 a, float2 b)
{
    const float bv = dot_value(b), q = __fdividef(dot_value(a), bv);
    const float r = __fadd_rn(__fmaf_rn(-q, b.x, a.x), __fmaf_rn(-q, b.y, a.y));
    return __fadd_rn(q, __fdividef(r, bv));
}

// a - b rounded to FP32 (exact in sign for dots that agree in their leading parts).
__device__ __forceinline__ float dot_minus(float2 a, float2 b) { return (a.x - b.x) + (a.y - b.y); }
__device__ __forceinline__ double dot_minus(double a, double b) { return a - b; }

// What a CTA's threads share in the edge passes.
struct Slice {
    unsigned char *base;             // the slice in shared memory, or the ring
    const unsigned char *rest;       // rows: the steps that stay in global memory
    const uint32_t *meta;            // shared-memory copy of the chunk sizes (colours) or step offsets (rows)
    uint64_t *full, *empty;
    int n_chunks, nthr, stages, ns;
    uint32_t stage_bytes, n_ent, n_rest;
    int tpr, polls0;                 // threads per row; poll limit of the very first wait
    int stage;                       // position in the ring (every thread keeps its own copy)
    uint32_t phase;
    volatile int *bad;
};

__device__ __forceinline__ void csync(int nthr) { asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory"); }

template <typename T, int D>
__device__ __forceinline__ void load_entry(const unsigned char *base, int n, int k, uint32_t &w, T *M)
{
    w = reinterpret_cast<const uint32_t *>(base)[k];
    const T *val = reinterpret_cast<const T *>(base + (size_t)n * 4);
#pragma unroll
    for (int q = 0; q < D * D; ++q) M[q] = val[q * n + k];
}

// One pass over the CTA's edges in colour order: f(target, source, block) for
// every entry, colours separated by barriers.  Two chunks of a colour are
// loaded before either is used.
template <typename T, int D, typename F>
__device__ __forceinline__ void colour_pass(Slice &sl, F f)
{
    constexpr int DD = D * D;
    size_t off = 0;
    for (int c = 0; c < sl.n_chunks;) {
        const int k = threadIdx.x;
        uint32_t w[2] = {kCgPadEntry, kCgPadEntry}, cn = 0;
        T M[2][DD];
        int took = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (u == 1 && ((cn & kCgLastOfColour) || c + 1 >= sl.n_chunks)) break;
            cn = sl.meta[c + u];
            const int n = (int)(cn & ~kCgLastOfColour);
            const unsigned char *base = sl.base + off;
            bool ok = true;
            const int st = sl.stage;
            if (sl.stages) {
                base = sl.base + (size_t)st * sl.stage_bytes;
                ok = mbar_wait_bounded(sl.full + st, sl.phase, sl.polls0);
                if (!ok) *sl.bad = 1;  // nothing of the chunk is touched
                sl.polls0 = kWaitLimit;
                if (++sl.stage == sl.stages) sl.stage = 0, sl.phase ^= 1u;
            } else {
                off += (size_t)n * (4 + DD * sizeof(T));
            }
            if (ok && k < n) load_entry<T, D>(base, n, k, w[u], M[u]);
            if (sl.stages) {
                __syncwarp();
                if ((threadIdx.x & 31) == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(sl.empty + st)) : "memory");
            }
            ++took;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (w[u] != kCgPadEntry) f((int)(w[u] & 0xffff), (int)(w[u] >> 16), M[u]);
        c += took;
        if (cn & kCgLastOfColour) csync(sl.nthr);
    }
}

// One pass over the CTA's rows: tpr threads a row, add(acc, row, source,
// block) for its entries, done(row, acc) once with the row's sum of K values.
// Steps that did not fit in shared memory come from L2, U at a time.
template <typename T, int D, int K, int U, typename A, typename F>
__device__ __forceinline__ void row_pass(const Slice &sl, A add, F done)
{
    constexpr int DD = D * D;
    const int lane = threadIdx.x & 31, nw = sl.nthr >> 5, tpr = sl.tpr, n_vw = sl.ns * tpr >> 5;
    const int sh = 31 - __clz(tpr);
    const uint32_t *rest_at = sl.meta + n_vw + 1;
    for (int vw = threadIdx.x >> 5; vw < n_vw; vw += nw) {
        const int row = (vw * 32 + lane) >> sh;
        T acc[K];
#pragma unroll
        for (int q = 0; q < K; ++q) acc[q] = T(0);
        if (sl.n_rest) {
            const uint32_t e1 = rest_at[vw + 1];
            const uint32_t *idx = reinterpret_cast<const uint32_t *>(sl.rest);
            const T *val = reinterpret_cast<const T *>(sl.rest + (size_t)sl.n_rest * 4);
            for (uint32_t s = rest_at[vw]; s < e1; s += U) {
                uint32_t w[U];
                T M[U][DD];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const size_t e = (size_t)(s + u) * 32 + lane;
                    w[u] = s + u < e1 ? __ldcg(idx + e) : 0u;
#pragma unroll
                    for (int q = 0; q < DD; ++q) M[u][q] = s + u < e1 ? __ldcg(val + (size_t)q * sl.n_rest + e) : T(0);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) add(acc, row, (int)(w[u] >> 16), M[u]);
            }
        }
        const uint32_t s1 = sl.meta[vw + 1];
#pragma unroll 3
        for (uint32_t s = sl.meta[vw]; s < s1; ++s) {
            uint32_t w;
            T M[DD];
            load_entry<T, D>(sl.base, (int)sl.n_ent, (int)(s * 32 + lane), w, M);
            add(acc, row, (int)(w >> 16), M);
        }
        for (int o = 1; o < tpr; o <<= 1)
#pragma unroll
            for (int q = 0; q < K; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
        if ((lane & (tpr - 1)) == 0) done(row, acc);
    }
}

template <typename V>
__device__ __forceinline__ void st_dsmem(void *local, uint32_t rank, V v)
{
    const uint32_t a = dsmem_addr(local, rank);
    if constexpr (std::is_same_v<V, float2>)
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
    else if constexpr (sizeof(V) == 4)
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
    else
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// (value, tag) words of the grid's exchanges: 8-byte scalars, so that a reader
// sees a value with its tag or neither.
__device__ __forceinline__ void put_word(unsigned long long *p, uint32_t v, uint32_t tag)
{
    asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p), "l"((unsigned long long)tag << 32 | v) : "memory");
}
// Two neighbouring words; each carries its own tag.
__device__ __forceinline__ ulonglong2 load_words(const unsigned long long *p)
{
    ulonglong2 w;
    asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
    return w;
}

// Vertex vector in shared memory: 2D FP32 rows in one 8-byte access.
template <typename T, int D>
__device__ __forceinline__ void ld_vec(const T *p, int k, T v[D])
{
    if constexpr (sizeof(T) == 4 && D == 2) {
        const float2 a = reinterpret_cast<const float2 *>(p)[k];
        v[0] = a.x, v[1] = a.y;
    } else {
#pragma unroll
        for (int c = 0; c < D; ++c) v[c] = p[k * D + c];
    }
}
template <typename T, int D>
__device__ __forceinline__ void st_vec(T *p, int k, const T v[D])
{
    if constexpr (sizeof(T) == 4 && D == 2) {
        reinterpret_cast<float2 *>(p)[k] = make_float2(v[0], v[1]);
    } else {
#pragma unroll
        for (int c = 0; c < D; ++c) p[k * D + c] = v[c];
    }
}

// Tables of CTA cta that a solve reads from shared memory (the caller synchronises).
template <int D, typename T, bool ROWS>
__device__ __forceinline__ void pcg_tables(const PcgDev &pd, int cta, bool grid, unsigned char *smem)
{
    const PcgSmem L(D, sizeof(T), pd.ns, pd.max_halo, pd.max_items, pd.n_coarse, pd.n_meta, grid ? pd.n_cta : 0);
    uint32_t *meta = reinterpret_cast<uint32_t *>(smem + L.meta);
    int32_t *shalo = reinterpret_cast<int32_t *>(smem + L.halo);
    const int h0 = pd.halo_ptr[cta], nh = pd.halo_ptr[cta + 1] - h0;
    if constexpr (ROWS) {
        for (int k = threadIdx.x; k < pd.n_meta; k += blockDim.x) meta[k] = pd.row_step[(size_t)cta * pd.n_meta + k];
    } else {
        const int c0 = pd.chunk_ptr[cta], nch = pd.chunk_ptr[cta + 1] - c0;
        for (int k = threadIdx.x; k < nch; k += blockDim.x) meta[k] = pd.chunk_n[c0 + k];
    }
    for (int k = threadIdx.x; k < nh; k += blockDim.x) shalo[k] = pd.halo_slot[h0 + k];
}

// The slice of CTA cta (stored by rows when ROWS) whose shared part or ring starts at smem + L.ring.
template <int D, typename T, bool ROWS>
__device__ __forceinline__ Slice pcg_slice(const PcgDev &pd, int cta, bool grid, unsigned char *smem, int polls,
                                           volatile int *bad)
{
    const PcgSmem L(D, sizeof(T), pd.ns, pd.max_halo, pd.max_items, pd.n_coarse, pd.n_meta, grid ? pd.n_cta : 0);
    const size_t esz = 4 + D * D * sizeof(T);
    const int c0 = pd.chunk_ptr[cta], nch = pd.chunk_ptr[cta + 1] - c0;
    Slice sl;
    sl.n_ent = (uint32_t)(pd.chunk_ent[c0 + (ROWS ? 1 : nch)] - pd.chunk_ent[c0]);
    sl.n_rest = ROWS ? (uint32_t)(pd.chunk_ent[c0 + 2] - pd.chunk_ent[c0 + 1]) : 0u;
    sl.base = smem + L.ring;
    sl.rest = pd.slices + ((size_t)pd.chunk_ent[c0] + sl.n_ent) * esz;
    sl.meta = reinterpret_cast<const uint32_t *>(smem + L.meta);
    sl.full = reinterpret_cast<uint64_t *>(smem);
    sl.empty = sl.full + kPcgMaxStages;
    sl.n_chunks = nch;
    sl.nthr = pd.threads;
    sl.stages = ROWS ? 0 : pd.stages;
    sl.ns = pd.nslot[cta];
    sl.stage_bytes = (uint32_t)(kCgChunk * esz);
    sl.tpr = pd.tpr;
    sl.polls0 = polls;
    sl.stage = 0;
    sl.phase = 0;
    sl.bad = bad;
    return sl;
}

struct PcgResult {
    int iter, neg, fail;
    double rr;
};

// The solve itself, by the consumer threads of one CTA (number cta of pd.n_cta)
// whose slice sl and tables (pcg_tables) are in place: x with A x = sign b to
// |r| <= rtol |b| goes to dout.  ROWS: the slice is stored by rows (see
// cg_plan.h), else by colours.  GRID: the CTAs are a grid, else one cluster or
// one CTA (a variant of its own: the grid's exchange would cost a cluster's
// solver its registers, 4.2 to 4.4 us an iteration on the walker); nb2: |b|^2;
// new_coarse: the coarse inverse is not the one of the CTA's previous solve.
template <typename T, int D, int VPT, bool ROWS, bool GRID>
__device__ __forceinline__ PcgResult pcg_run(const PcgDev &pd, Slice &sl, int cta, unsigned char *smem, const double *b,
                                             double sign, double nb2, T *dout, double rtol, int max_iter,
                                             bool new_coarse)
{
    constexpr bool grid = GRID;
    constexpr int NM = D == 3 ? 6 : 3, ND = D == 3 ? 6 : 3, DD = D * D, RN = Row<T, D>::N;
    constexpr int NI = (NM + 1) / 2;       // pairs of words that hold a CTA's items
    constexpr bool F32 = sizeof(T) == 4;
    using Dot = typename DotOf<T>::Type;
    // A slot's arm, vertex diagonal and inverse block stay in registers where one
    // slot a thread leaves room (walker 4.54 -> 4.09 us an iteration, 70,785
    // vertices 13.0 -> 12.5); with four slots the spills cost more than the loads
    // (2D 20,000 vertices 7.1 -> 7.6 us)
    constexpr bool KEEP_S = F32 && VPT == 1;
    constexpr bool EXACT = VPT <= 2;   // with more slots the products' errors average out (largest body: 61.6 us with, 60.2 without)
    constexpr bool KEEP_Z = VPT <= 2;  // so does z between the phases
    __shared__ float sred[kMaxWarps * VPT][8];  // restriction, per warp or per group of 32 slots
    __shared__ T sbc[3];
    __shared__ Dot sdot[2][kMaxWarps];          // dots of the warps
    __shared__ Dot sdots[3][kMaxWarps];         // dots of the CTAs of a cluster (or of the only CTA), or of 32 CTAs of a grid
    __shared__ float scown[kMaxWarps][8];       // coarse values of this CTA's aggregates
    __shared__ int sgrp[kMaxWarps + 1];         // first group of 32 slots of an item
    __shared__ int sok;
    const int G = pd.n_cta, nthr = sl.nthr, nw = nthr >> 5, tid = threadIdx.x;
    const int lane = tid & 31, wrp = tid >> 5, N = pd.n_coarse;
    const int ns = sl.ns, s0 = cta * pd.ns;
    const int nh = pd.halo_ptr[cta + 1] - pd.halo_ptr[cta];
    const int i0 = pd.item_ptr[cta], ni = pd.item_ptr[cta + 1] - i0, a0 = pd.item_agg[i0];
    const bool one = ni == 1, solo = G == 1;
    // Loads of an exchange in flight per thread: two cover 152 CTAs' words, and with
    // four the registers spill (70,785 vertices: 11.2 against 12.5 us an iteration).
    constexpr int PB = 2;
    const int n_part = grid ? (G + 31) / 32 : 1;  // partial sums of a dot over a grid's CTAs
    const PcgSmem L(D, sizeof(T), pd.ns, pd.max_halo, pd.max_items, N, pd.n_meta, grid ? G : 0);
    T *sp = reinterpret_cast<T *>(smem + L.p), *sy = reinterpret_cast<T *>(smem + L.y);
    float *sE = reinterpret_cast<float *>(smem + L.e);
    // ss: restricted residual, two buffers (a cluster's CTAs write the next one while this one is read)
    float *ss = reinterpret_cast<float *>(smem + L.s), *ss_next = ss + N, *st_ = reinterpret_cast<float *>(smem + L.t);
    const int32_t *shalo = reinterpret_cast<const int32_t *>(smem + L.halo);
    uint32_t *sword = reinterpret_cast<uint32_t *>(smem + L.word);  // [G][kPcgRow] of a grid's exchange
    int fail = 0;
    for (int k = tid; k < kMaxWarps * VPT * 8; k += nthr) (&sred[0][0])[k] = 0.0f;
    for (int k = tid; k < ns / 32; k += nthr) {
        const int it = pd.grp_agg[(s0 >> 5) + k] - a0;
        if (k == 0 || pd.grp_agg[(s0 >> 5) + k - 1] - a0 != it) sgrp[it] = k;
        if (k == ns / 32 - 1) sgrp[ni] = ns / 32;
    }
    if (tid == 0) sok = 1;

    // --- diagonal blocks: minus the sums of the edge blocks, plus the vertex terms
    // per-slot arrays, looked up in the plan where they are used: held in registers
    // their addresses would cost the kernel a dozen
    auto dg = [&](int k) { return static_cast<const T *>(pd.diag2) + 2 * (int64_t)(s0 + k); };
    auto dinv = [&](int q, int k) { return static_cast<T *>(pd.dinv) + (int64_t)q * pd.n_cta * pd.ns + s0 + k; };
    auto zr = [&](int slot) { return static_cast<T *>(pd.zr) + (int64_t)slot * RN; };
    auto pos = [&](int k) { return pd.pos4[s0 + k]; };
    auto gid = [&](int k) { return pd.slot_gid[s0 + k]; };
    {
        T *sd = sp;  // [ND][ns]: fits in p and y
        auto sym = [](const T *M, T *S) {
            if constexpr (D == 3) {
                S[0] = M[0], S[1] = T(0.5) * (M[1] + M[3]), S[2] = T(0.5) * (M[2] + M[6]);
                S[3] = M[4], S[4] = T(0.5) * (M[5] + M[7]), S[5] = M[8];
            } else {
                S[0] = M[0], S[1] = T(0.5) * (M[1] + M[2]), S[2] = M[3];
            }
        };
        if constexpr (ROWS) {
            row_pass<T, D, ND, 2>(
                sl,
                [&](T *acc, int, int, const T *M) {
                    T S[ND];
                    sym(M, S);
#pragma unroll
                    for (int q = 0; q < ND; ++q) acc[q] -= S[q];
                },
                [&](int row, const T *acc) {
#pragma unroll
                    for (int q = 0; q < ND; ++q) sd[q * ns + row] = acc[q];
                });
        } else {
            for (int k = tid; k < ND * ns; k += nthr) sd[k] = T(0);
            csync(nthr);
            colour_pass<T, D>(sl, [&](int i, int j, const T *M) {
                T S[ND];
                sym(M, S);
#pragma unroll
                for (int q = 0; q < ND; ++q) sd[q * ns + i] -= S[q];
                if (j < ns)
#pragma unroll
                    for (int q = 0; q < ND; ++q) sd[q * ns + j] -= S[q];
            });
        }
        csync(nthr);
        for (int k = tid; k < ns; k += nthr) {
            T S[ND], o[ND];
#pragma unroll
            for (int q = 0; q < ND; ++q) S[q] = sd[q * ns + k];
            const T dh = dg(k)[0], dy = dg(k)[1];
            if constexpr (D == 3)
                S[0] += dh, S[3] += dy, S[5] += dh;
            else
                S[0] += dh, S[2] += dy;
            invert_sym<T, D>(S, o);
#pragma unroll
            for (int q = 0; q < ND; ++q) *dinv(q, k) = o[q];
        }
        csync(nthr);
    }
    for (int k = tid; k < (ns + nh) * D; k += nthr) sp[k] = T(0);
    for (int k = tid; new_coarse && k < ni * NM * N; k += nthr) {  // this CTA's rows of E^-1, symmetrised
        const int r = a0 * NM + k / N, n = k % N;
        sE[k] = 0.5f * (pd.Einv[(size_t)r * N + n] + pd.Einv[(size_t)n * N + r]);
    }

    auto rhs = [&](int k, int c) {  // an unused or pinned slot has none
        const int g = k < ns ? gid(k) : -1;
        return g >= 0 && !(__float_as_int(pos(k).w) >> 30) ? sign * b[(int64_t)g * D + c] : 0.0;
    };
    // Per-slot restricted components v (v[6], v[7] are zero).  A CTA of one
    // aggregate sums its slots first.
    auto put_sum = [&](int m, const float v[8]) {
        const float t = warp_sum8(v);
        if ((lane & 3) == 0) sred[one ? wrp : m * nw + wrp][lane >> 2] = t;
    };
    auto put_group = [&](int m, float v[8]) {  // of one group of 32 slots
        put_sum(m, v);
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = 0.0f;
    };
    // Two dots share a warp's sum: the lower half-warp ends with the first, the
    // upper with the second (of one dot, both with it).
    auto half = [&](int nd) { return nd > 1 ? lane >> 4 : 0; };
    auto dot_of = [&](Dot v, int d) -> Dot {
        if constexpr (F32)
            return make_float2(__shfl_sync(0xffffffffu, v.x, 16 * d), __shfl_sync(0xffffffffu, v.y, 16 * d));
        else
            return __shfl_sync(0xffffffffu, v, 16 * d);
    };
    // This warp's nd dots to shared memory; warps without slots have none.
    auto put_dots = [&](int nd, const Dot *dots) {
        Dot v{};
        if (wrp * 32 < ns && nd > 0) {
            const bool up = half(nd) != 0, low = nd > 1 && !up;
            v = dot_merge(up ? dots[1] : dots[0], dot_xor(low ? dots[1] : dots[0], 16));
            v = group_dot<8>(v);
        }
        if ((lane & 15) == 0 && (lane >> 4) < nd) sdot[lane >> 4][wrp] = v;
    };
    // The CTA's nd dots (after put_dots), by one warp.
    auto cta_dot = [&](int nd) -> Dot {
        const int w = lane & 15;
        return group_dot<8>(w < nw ? sdot[half(nd)][w] : Dot{});
    };
    // Exchange of the restricted vector (into dst) and of nd dots (slot base of
    // sdots, or words of the grid).  rows: the CTA has published its rows of z,
    // which others read after it.  buf and tag name the grid's words.
    auto exchange = [&](int nd, const Dot *dots, float *dst, bool rows, int base, int buf, uint32_t tag) -> bool {
        put_dots(nd, dots);
        csync(nthr);
        const int q = lane & 7, h = lane >> 3;
        unsigned long long *mine = pd.words + ((size_t)buf * G + cta) * kPcgWords;
        if (grid && rows && wrp == 0) __threadfence();  // the CTA's rows before its words
        for (int it = wrp; it < ni; it += nw) {
            float v = 0.0f;
            if (one) {
#pragma unroll
                for (int g = 0; g < kMaxWarps; g += 4) v += sred[g + h][q];  // rows of absent warps are zero
            } else {
                for (int g = sgrp[it] + h; g < sgrp[it + 1]; g += 4) v += sred[g][q];
            }
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            if (grid) {  // one aggregate a CTA
                if (h == 0 && q < 2 * NI) put_word(mine + q, __float_as_uint(v), tag);
            } else if (q < NM) {
                const int n = (a0 + it) * NM + q;
                if (solo) {
                    if (h == 0) dst[n] = v;
                } else {
                    for (int k = h; k < G; k += 4) st_dsmem(dst + n, (uint32_t)k, v);
                }
            }
        }
        if (nd > 0 && wrp == nw - 1) {
            const Dot v = cta_dot(nd);
            if (!grid && !solo) {
                for (int k = 0; k < nd; ++k) {
                    const Dot w = dot_of(v, k);
                    if (lane < G) st_dsmem(&sdots[base + k][cta], (uint32_t)lane, w);
                }
            } else {
                const int d = lane >> 4, i = lane & 15;
                if (solo) {
                    if (d < nd && i == 0) sdots[base + d][0] = v;
                } else {  // two words a dot, from neighbouring lanes: the parts of a pair, or the halves of a double
                    uint32_t w;
                    if constexpr (F32)
                        w = __float_as_uint(i ? v.y : v.x);
                    else
                        w = (uint32_t)(i ? __double2hiint(v) : __double2loint(v));
                    if (d < nd && i < 2) put_word(mine + kPcgDots + 2 * d + i, w, tag);
                }
            }
        }
        if (solo) {
            csync(nthr);
            return true;
        }
        if (!grid) {
            cluster_sync();
            return true;
        }
        // the words of every CTA, neighbouring threads on one CTA's line; PB loads in
        // flight before the first is looked at
        const unsigned long long *all = pd.words + (size_t)buf * G * kPcgWords;
        const int nt = NI + nd, n_load = G * nt;
        bool ok = true;
        for (int k0 = tid; k0 < n_load; k0 += PB * nthr) {
            ulonglong2 w[PB];
            int o[PB];  // CTA << 8 | word
#pragma unroll
            for (int u = 0; u < PB; ++u)
                if (k0 + u * nthr < n_load) {
                    const int k = k0 + u * nthr, g = k / nt, j = k - g * nt;
                    o[u] = g << 8 | (j < NI ? 2 * j : kPcgDots + 2 * (j - NI));
                    w[u] = load_words(all + g * kPcgWords + (o[u] & 255));
                }
#pragma unroll
            for (int u = 0; u < PB; ++u) {
                if (k0 + u * nthr >= n_load) break;
                for (int i = 0; ok && ((uint32_t)(w[u].x >> 32) != tag || (uint32_t)(w[u].y >> 32) != tag); ++i) {
                    if (i >= kGridWaitPolls) ok = false;
                    w[u] = load_words(all + (o[u] >> 8) * kPcgWords + (o[u] & 255));
                }
                *reinterpret_cast<uint2 *>(sword + (o[u] >> 8) * kPcgRow + (o[u] & 255)) =
                    make_uint2((uint32_t)w[u].x, (uint32_t)w[u].y);
            }
        }
        if (!ok) sok = 0;
        if (rows) __threadfence();  // the rows read next are those published before the words
        csync(nthr);
        for (int n = tid; n < N; n += nthr) {
            const int a = n / NM, j = n - a * NM, g0 = pd.agg_item[a], g1 = pd.agg_item[a + 1];
            float v = 0.0f;
            for (int g = g0; g < g1; ++g) v += __uint_as_float(sword[g * kPcgRow + j]);
            dst[n] = v;
        }
        for (int u = nw - 1 - wrp; u < nd * n_part; u += nw) {  // meanwhile the last warps: a dot over 32 CTAs each
            const int d = u >= n_part, p = u - d * n_part, g = p * 32 + lane;
            Dot v{};
            if (g < G) {
                const uint2 w = *reinterpret_cast<const uint2 *>(sword + g * kPcgRow + kPcgDots + 2 * d);
                if constexpr (F32)
                    v = make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
                else
                    v = __hiloint2double((int)w.y, (int)w.x);
            }
            v = group_dot<16>(v);
            if (lane == 0) sdots[base + d][p] = v;
        }
        csync(nthr);
        return sok != 0;
    };
    // Sums of the nd dots of the last exchange over the CTAs; every calling warp forms them alike.
    auto dot_sums = [&](int base, int nd, Dot *out) {
        if (grid || solo) {
            for (int d = 0; d < nd; ++d) out[d] = sdots[base + d][0];
            for (int p = 1; p < n_part; ++p)
                for (int d = 0; d < nd; ++d) out[d] = dot_merge(out[d], sdots[base + d][p]);
        } else {
            const int g = lane & 15;
            const Dot v = group_dot<8>(g < G ? sdots[base + half(nd)][g] : Dot{});
            for (int d = 0; d < nd; ++d) out[d] = dot_of(v, d);
        }
    };
    auto swap_s = [&]() {
        float *t = ss;
        ss = ss_next;
        ss_next = t;
    };
    // The coarse values of this CTA's aggregates from the restricted residual ss
    // - alpha st_: a warp per row of E^-1 (the last ones, which often have no
    // slots), or, with more rows than warps, eight lanes per row.
    auto coarse = [&](float alpha, bool with_t) {
        if (ni * NM <= nw) {
            const int row = nw - 1 - wrp;
            if (row < ni * NM) {
                float v = 0.0f;
#pragma unroll
                for (int u = 0; u < kCgMaxCoarse / 32; ++u) {
                    const int n = lane + 32 * u;
                    if (n < N) v = fmaf(sE[row * N + n], with_t ? fmaf(-alpha, st_[n], ss[n]) : ss[n], v);
                }
                v = warp_all(v);
                if (lane == 0) scown[row / NM][row % NM] = v;
            }
        } else {
            const int sub = lane & 7;
            for (int row = wrp * 4 + (lane >> 3); row - (lane >> 3) < ni * NM; row += nw * 4) {
                float v = 0.0f;
                if (row < ni * NM)
#pragma unroll 4
                    for (int n = sub; n < N; n += 8)
                        v = fmaf(sE[row * N + n], with_t ? fmaf(-alpha, st_[n], ss[n]) : ss[n], v);
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                if (sub == 0 && row < ni * NM) scown[row / NM][row % NM] = v;
            }
        }
    };

    T x[VPT][D], r[VPT][D], zk[KEEP_Z ? VPT : 1][D];
    float4 Rk[KEEP_S ? VPT : 1];
    T dk[KEEP_S ? VPT : 1][2], Sk[KEEP_S ? VPT : 1][ND];
    if constexpr (KEEP_S)
#pragma unroll
        for (int m = 0; m < VPT; ++m) {
            const int k = tid + m * nthr;
            Rk[m] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            dk[m][0] = dk[m][1] = T(0);
#pragma unroll
            for (int q = 0; q < ND; ++q) Sk[m][q] = T(0);
            if (k >= ns) continue;
            Rk[m] = pos(k);
            if (pd.has_diag) dk[m][0] = dg(k)[0], dk[m][1] = dg(k)[1];
#pragma unroll
            for (int q = 0; q < ND; ++q) Sk[m][q] = *dinv(q, k);
        }
    auto arm = [&](int m, int k) {
        if constexpr (KEEP_S)
            return Rk[m];
        else
            return pos(k);
    };
    auto inv_block = [&](int m, int k, T *S) {
#pragma unroll
        for (int q = 0; q < ND; ++q) {
            if constexpr (KEEP_S)
                S[q] = Sk[m][q];
            else
                S[q] = *dinv(q, k);
        }
    };
#pragma unroll
    for (int m = 0; m < VPT; ++m)
#pragma unroll
        for (int c = 0; c < D; ++c) x[m][c] = T(0);
    int it = 0, neg = 0;
    Dot rr{}, rz{};
    // rtol^2 |b|^2 with |b| = 1, as a dot
    Dot tol2;
    if constexpr (F32) {
        tol2.x = (float)(rtol * rtol);
        tol2.y = (float)(rtol * rtol - (double)tol2.x);
        rr = make_float2(1.0f, 0.0f);
    } else {
        tol2 = rtol * rtol;
        rr = 1.0;
    }
    bool run = !fail && nb2 > 0.0 && isfinite(nb2) && max_iter > 0 && rtol < 1.0;
    if (*sl.bad) run = false, fail = 1;
    // z = D^-1 r + Z c of slot k with inverse diagonal block S and arm R (zero at an
    // unused or pinned slot): publishes the row, adds r.z to its dot
    auto precondition = [&](int m, int k, const T *S, float4 R, const T *rm, Dot &d_rz) {
        T z[D];
        const int w = __float_as_int(R.w);
        sym_mul<T, D>(S, rm, z);
        prolong_add<T, D>(R, scown[one ? 0 : (w & 0xffff) - a0], z);
#pragma unroll
        for (int c = 0; c < D; ++c) {
            z[c] = (w >> 30) ? T(0) : z[c];
            if constexpr (KEEP_Z) zk[m][c] = z[c];
        }
        put_row<T, D>(zr(s0 + k), z);
        dot_add<D, EXACT>(d_rz, rm, z, m == 0);
    };
    auto restrict_slot = [&](float4 R, const T *rm, float v[8]) {
        float f[D];
#pragma unroll
        for (int c = 0; c < D; ++c) f[c] = (float)rm[c];
        restrict_to<D>(R, f, v);
    };
    uint32_t tag = 1;
    if (run) {
        const double scale = 1.0 / sqrt(nb2);
        float v[8] = {};
        Dot d_rz{};
#pragma unroll
        for (int m = 0; m < VPT; ++m) {
            const int k = tid + m * nthr;
#pragma unroll
            for (int c = 0; c < D; ++c) r[m][c] = T(rhs(k, c) * scale);
            if (k < ns) {
                restrict_slot(arm(m, k), r[m], v);
                if (!one) put_group(m, v);
            }
        }
        if (one) put_sum(0, v);
        if (!exchange(0, nullptr, ss, false, 0, 0, tag)) fail = 1;
        coarse(0.0f, false);
        csync(nthr);
#pragma unroll
        for (int m = 0; m < VPT; ++m) {
            const int k = tid + m * nthr;
            if (k >= ns) continue;
            T S[ND];
            inv_block(m, k, S);
            precondition(m, k, S, arm(m, k), r[m], d_rz);
        }
        // the same restricted vector again, with r.z and the rows of z
        if (!exchange(1, &d_rz, ss_next, true, 1, 1, tag)) fail = 1;
        swap_s();
        dot_sums(1, 1, &rz);
    }
    T beta = T(0);
    while (run && !fail) {
        ++tag;
        // 1. p = z + beta p at own and halo vertices; A p
#pragma unroll 2
        for (int h = tid; h < nh; h += nthr) {
            T z[D], pv[D];
            get_row<T, D>(zr(shalo[h]), z);
            ld_vec<T, D>(sp, ns + h, pv);
#pragma unroll
            for (int c = 0; c < D; ++c) pv[c] = z[c] + beta * pv[c];
            st_vec<T, D>(sp, ns + h, pv);
        }
#pragma unroll
        for (int m = 0; m < VPT; ++m) {
            const int k = tid + m * nthr;
            if (k >= ns) continue;
            T z[D], pv[D];
            if constexpr (KEEP_Z) {
#pragma unroll
                for (int c = 0; c < D; ++c) z[c] = zk[m][c];
            } else {
                get_row<T, D>(zr(s0 + k), z);
            }
            ld_vec<T, D>(sp, k, pv);
#pragma unroll
            for (int c = 0; c < D; ++c) pv[c] = z[c] + beta * pv[c];
            st_vec<T, D>(sp, k, pv);
            if constexpr (!ROWS) {
                const T zero[D] = {};
                st_vec<T, D>(sy, k, zero);
            }
        }
        csync(nthr);
        if constexpr (ROWS) {
            row_pass<T, D, D, (VPT == 1 ? 3 : 2)>(
                sl,
                [&](T *acc, int row, int j, const T *M) {
                    T pi[D], d[D];
                    ld_vec<T, D>(sp, row, pi);
                    ld_vec<T, D>(sp, j, d);
#pragma unroll
                    for (int c = 0; c < D; ++c) d[c] -= pi[c];
#pragma unroll
                    for (int a = 0; a < D; ++a)
#pragma unroll
                        for (int c = 0; c < D; ++c) acc[a] += M[a * D + c] * d[c];
                },
                [&](int row, const T *acc) { st_vec<T, D>(sy, row, acc); });
            csync(nthr);
        } else {
            colour_pass<T, D>(sl, [&](int i, int j, const T *M) {
                T pi[D], d[D], y[D];
                ld_vec<T, D>(sp, i, pi);
                ld_vec<T, D>(sp, j, d);
                ld_vec<T, D>(sy, i, y);
#pragma unroll
                for (int c = 0; c < D; ++c) d[c] -= pi[c];
#pragma unroll
                for (int a = 0; a < D; ++a)
#pragma unroll
                    for (int c = 0; c < D; ++c) y[a] += M[a * D + c] * d[c];
                st_vec<T, D>(sy, i, y);
                if (j < ns) {
                    ld_vec<T, D>(sy, j, y);
#pragma unroll
                    for (int a = 0; a < D; ++a)
#pragma unroll
                        for (int c = 0; c < D; ++c) y[a] -= M[c * D + a] * d[c];
                    st_vec<T, D>(sy, j, y);
                }
            });
        }
        {
            float v[8] = {};
            Dot dot{};
#pragma unroll
            for (int m = 0; m < VPT; ++m) {
                const int k = tid + m * nthr;
                if (k >= ns) continue;
                const float4 R = arm(m, k);
                T dh = T(0), dy = T(0);
                if constexpr (KEEP_S)
                    dh = dk[m][0], dy = dk[m][1];
                else if (pd.has_diag)
                    dh = dg(k)[0], dy = dg(k)[1];
                float f[D];
                T pv[D], y[D];
                const bool fx = (__float_as_int(R.w) >> 30) != 0;
                ld_vec<T, D>(sp, k, pv);
                ld_vec<T, D>(sy, k, y);
#pragma unroll
                for (int c = 0; c < D; ++c) {
                    y[c] = fx ? T(0) : y[c] + (c == 1 ? dy : dh) * pv[c];
                    f[c] = (float)y[c];
                }
                dot_add<D, EXACT>(dot, pv, y, m == 0);
                st_vec<T, D>(sy, k, y);
                restrict_to<D>(R, f, v);
                if (!one) put_group(m, v);
            }
            if (one) put_sum(0, v);
            if (*sl.bad) {  // a chunk never came: the others give up at their next wait
                fail = 1;
                break;
            }
            if (!exchange(1, &dot, st_, false, 0, 0, tag)) {
                fail = 1;
                break;
            }
        }
        // 2. alpha; x, r; the coarse values; z; r.r and r.z
        Dot pAp;
        T alpha;
        if constexpr (F32) {
            dot_sums(0, 1, &pAp);
            alpha = dot_quot(rz, pAp);
        } else {  // one warp forms the FP64 scalars
            if (wrp == 0) {
                dot_sums(0, 1, &pAp);
                if (lane == 0) {
                    sbc[0] = pAp;
                    sbc[1] = rz / pAp;
                }
            }
            csync(nthr);
            pAp = sbc[0];
            alpha = sbc[1];
        }
        if (!(dot_value(pAp) > T(0)) || !isfinite(dot_value(pAp))) {
            neg = 1;
            if (it == 0)  // the preconditioned steepest-descent direction
#pragma unroll
                for (int m = 0; m < VPT; ++m)
#pragma unroll
                    for (int c = 0; c < D; ++c)
                        if (tid + m * nthr < ns) x[m][c] = sp[(tid + m * nthr) * D + c];
            break;
        }
        coarse((float)alpha, true);
        {
            float v[8] = {};
            Dot dots[2] = {};
            // x and r go on while some warps form the coarse values; with one slot a thread
            // (its arm in registers), or two in a CTA of one aggregate, the restriction too
            constexpr bool EARLY = VPT == 1 || (VPT == 2 && !ROWS);
#pragma unroll
            for (int m = 0; m < VPT; ++m) {
                const int k = tid + m * nthr;
                if (k >= ns) continue;
                T pv[D], y[D];
                ld_vec<T, D>(sp, k, pv);
                ld_vec<T, D>(sy, k, y);
#pragma unroll
                for (int c = 0; c < D; ++c) {
                    x[m][c] += alpha * pv[c];
                    r[m][c] -= alpha * y[c];
                }
                dot_add<D, EXACT>(dots[0], r[m], r[m], m == 0);
                if (EARLY) restrict_slot(arm(m, k), r[m], v);
            }
            if (EARLY) put_sum(0, v);
            csync(nthr);
#pragma unroll
            for (int m = 0; m < VPT; ++m) {
                const int k = tid + m * nthr;
                if (k >= ns) continue;
                const float4 R = arm(m, k);
                T S[ND];
                inv_block(m, k, S);
                if (!EARLY) restrict_slot(R, r[m], v);
                precondition(m, k, S, R, r[m], dots[1]);
                if (!EARLY && !one) put_group(m, v);
            }
            if (!EARLY && one) put_sum(0, v);
            if (!exchange(2, dots, ss_next, true, 1, 1, tag)) {
                fail = 1;
                break;
            }
            swap_s();
        }
        ++it;
        Dot rz_new;
        if constexpr (F32) {
            Dot two[2];
            dot_sums(1, 2, two);
            rr = two[0];
            rz_new = two[1];
            beta = dot_quot(rz_new, rz);
        } else {
            if (wrp == 0) {
                Dot two[2];
                dot_sums(1, 2, two);
                if (lane == 0) {
                    sbc[0] = two[0];
                    sbc[1] = two[1];
                    sbc[2] = two[1] / rz;
                }
            }
            csync(nthr);
            rr = sbc[0];
            rz_new = sbc[1];
            beta = sbc[2];
        }
        rz = rz_new;
        if (!(dot_minus(rr, tol2) > T(0)) || it >= max_iter || !isfinite(dot_value(rr)) || !(dot_value(rz) > T(0))) break;
    }
    const double bnorm = nb2 > 0.0 && isfinite(nb2) ? sqrt(nb2) : 0.0;
#pragma unroll
    for (int m = 0; m < VPT; ++m) {
        const int k = tid + m * nthr;
        if (k >= ns || gid(k) < 0) continue;
#pragma unroll
        for (int c = 0; c < D; ++c) dout[(int64_t)gid(k) * D + c] = T((double)x[m][c] * bnorm);
    }
    PcgResult res;
    res.iter = it;
    res.neg = neg;
    res.fail = fail;
    if constexpr (F32)
        res.rr = ((double)rr.x + (double)rr.y) * bnorm * bnorm;
    else
        res.rr = rr * bnorm * bnorm;
    return res;
}

}  // namespace
}  // namespace softsim
