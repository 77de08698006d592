// clustercg.cuh -- what the CG solves that run as one thread-block cluster
// launch share (mass.cu, state.cu): distributed shared memory, the two
// arithmetics (FP64; double-float vectors with an FP32 direction and FP64
// scalars), the sums over the cluster and the scalar step.
#pragma once

#include <cooperative_groups.h>

#include "internal.cuh"
#include "df.cuh"
#include "util.cuh"

namespace cg = cooperative_groups;

#define CLUSTER_MAX 16 // CTAs (above 8: not portable, allowed per kernel)
// a loop that may run longer than this (~0.2 s) is left to the replayed kernels,
// between which the host reads the stop flag
#define CLUSTER_MAX_ITERS 10000

__device__ __forceinline__ uint32_t dsmem_of(const void *p, uint32_t rank)
{
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// address of element p of CTA `owner`; an address of the CTA's own shared
// memory is valid as it stands
__device__ __forceinline__ uint32_t dsmem_at(const void *p, uint32_t owner, uint32_t rank)
{
    return owner == rank ? (uint32_t)__cvta_generic_to_shared(p) : dsmem_of(p, owner);
}
__device__ __forceinline__ float dsmem_ld(uint32_t a, float)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ double dsmem_ld(uint32_t a, double)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void dsmem_st(uint32_t a, float2 v)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void dsmem_st(uint32_t a, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// The two arithmetics: what z and the vectors are, their sums, and a matrix
// entry held in registers.
struct ClusterDf {
    typedef float Z;
    typedef DF V;
    typedef float2 P; // a stored partial sum
    static constexpr bool SCALED = true; // the right side is scaled to norm ~1
    struct Entry {
        float hi, lo;
    };
    __device__ static Entry entry(double v)
    {
        const float h = (float)v;
        return Entry{h, (float)(v - (double)h)};
    }
    __device__ static void term(V &acc, Entry a, Z z) { df_fma(acc, a.hi, a.lo, z); }
    __device__ static V lanes(V v, int o)
    {
        DF w = {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
        df_merge(v, w);
        return v;
    }
    __device__ static V done(V acc)
    {
        V r;
        quick_two_sum(acc.hi, acc.lo, r.hi, r.lo);
        return r;
    }
    __device__ static V zero() { return DF{0.f, 0.f}; }
    __device__ static V add(V a, V b) { return df_add_fast(a, b); }
    __device__ static V shfl_xor(V v, int o)
    {
        return DF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
    }
    __device__ static V shfl(V v, int l)
    {
        return DF{__shfl_sync(0xffffffffu, v.hi, l), __shfl_sync(0xffffffffu, v.lo, l)};
    }
    __device__ static V dot(V a, Z z) { return df_mulf(a, z); }
    __device__ static V sqr(V a) { return df_mul2(a, a); }
    __device__ static P store(V v) { return make_float2(v.hi, v.lo); }
    __device__ static V load(P v) { return DF{v.x, v.y}; }
    __device__ static double value(V v) { return df_to_double(v); }
    __device__ static V scaled(double f, double scale) { return df_from_double(scale * f); }
    __device__ static Z jacobi(Z d, V r) { return r.hi * d; }
    __device__ static double out(V x, double inv) { return df_to_double(x) * inv; }
    // alpha or beta as the updates use it, and v + c w
    typedef DF C;
    __device__ static C coef(double c) { return df_from_double(c); }
    __device__ static C neg(C c) { return DF{-c.hi, -c.lo}; }
    __device__ static V axpy(V v, C c, V w) { return df_add2(v, df_mul2(c, w)); }
    __device__ static V of_z(Z z) { return DF{z, 0.f}; }
};
struct ClusterF64 {
    typedef double Z;
    typedef double V;
    typedef double P;
    static constexpr bool SCALED = false;
    typedef double Entry;
    __device__ static Entry entry(double v) { return v; }
    __device__ static void term(V &acc, Entry a, Z z) { acc += a * z; }
    __device__ static V lanes(V v, int o) { return v + __shfl_xor_sync(0xffffffffu, v, o); }
    __device__ static V done(V acc) { return acc; }
    __device__ static V zero() { return 0.0; }
    __device__ static V add(V a, V b) { return a + b; }
    __device__ static V shfl_xor(V v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
    __device__ static V shfl(V v, int l) { return __shfl_sync(0xffffffffu, v, l); }
    __device__ static V dot(V a, Z z) { return a * z; }
    __device__ static V sqr(V a) { return a * a; }
    __device__ static P store(V v) { return v; }
    __device__ static V load(P v) { return v; }
    __device__ static double value(V v) { return v; }
    __device__ static V scaled(double f, double) { return f; }
    __device__ static Z jacobi(Z d, V r) { return d * r; }
    __device__ static double out(V x, double) { return x; }
    typedef double C;
    __device__ static C coef(double c) { return c; }
    __device__ static C neg(C c) { return -c; }
    __device__ static V axpy(V v, C c, V w) { return v + c * w; }
    __device__ static V of_z(Z z) { return z; }
};

__device__ __forceinline__ bool not_finite(double x) { return !(x == x) || isinf(x); }

// scalars of the CG loop, one copy per CTA, all with the same values
template <typename M>
struct ClusterScal {
    double ff, rr, thr, rz, ra, scale; // ra = rz alpha
    typename M::C al, be;
    int iters, k1, status, done;
};

// warp 0: the stopping test of the iteration before, then alpha and beta of
// the single-reduction CG.  Lane 0 writes alpha's side, lane 1 beta's.
template <typename M>
__device__ __forceinline__ void cluster_step(ClusterScal<M> &s, double g, double d, double rr, double tol2, int maxit,
                                          bool start, double &alpha)
{
    const double thr = start ? tol2 * rr : s.thr;
    const int iters = start ? 0 : s.iters + 1, k1 = s.k1, l = threadIdx.x & 31;
    int status = CG_RUNNING;
    if (!finite64(rr)) status = CG_NUMERIC;
    else if (start ? rr == 0.0 : le64(rr, thr)) status = CG_CONVERGED;
    else if (!start && iters >= maxit) status = CG_MAXIT;
    double beta = 0.0;
    const int step = cg2_scalars(g, d, k1, s.rz, s.ra, alpha, beta);
    if (status == CG_RUNNING) status = step;
    __syncwarp();
    if (l < 2) {
        const typename M::C c = M::coef(l ? beta : alpha);
        if (l) s.be = c;
        else s.al = c;
    }
    if (l == 0) {
        if (start) s.ff = rr;
        s.rr = rr;
        s.thr = thr;
        s.iters = iters;
        s.status = status;
        s.done = status != CG_RUNNING;
    }
}

// warp 0, off the other warps' path: what the next step needs of this one
template <typename M>
__device__ __forceinline__ void cluster_keep(ClusterScal<M> &s, double g, double alpha)
{
    if ((threadIdx.x & 31) == 0) {
        s.rz = g;
        s.ra = g * alpha;
        s.k1 += 1;
    }
}

// Sums over the warp of a, b and c, of which only every STEP-th lane's values
// count: the first two steps hand each half of the lanes one of two values to
// carry on with.  The sums are left in lanes 0 (a), 16 (b) and 8 (c).
template <typename M, int STEP>
__device__ __forceinline__ typename M::V sum3(typename M::V a, typename M::V b, typename M::V c)
{
    const int l = threadIdx.x & 31;
    const bool h16 = l & 16, h8 = l & 8;
    typename M::V v = M::add(h16 ? b : a, M::shfl_xor(h16 ? a : b, 16));
    c = M::add(c, M::shfl_xor(c, 16));
    v = M::add(h8 ? c : v, M::shfl_xor(h8 ? v : c, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
        if (o >= STEP) v = M::add(v, M::shfl_xor(v, o));
    return v;
}

// every CTA's shared memory writes (its own and remote ones) before the
// barrier are visible to all CTAs after it
__device__ __forceinline__ void cluster_barrier(uint32_t ctas)
{
    if (ctas == 1) {
        __syncthreads();
        return;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// shared memory of one CTA for the sums and the scalars
template <typename M>
struct ClusterShared {
    typename M::V shw[3][32];
    typename M::P part[3][CLUSTER_MAX]; // (r, z), (z, A z) and r.r of every CTA
    double part64[CLUSTER_MAX];
    ClusterScal<M> ms;
};

// the power of two nearest 1 / ||f||, an exact scaling; fi is the thread's
// element of f
template <typename M>
__device__ __forceinline__ double cluster_scale(ClusterShared<M> &c, double fi, uint32_t rank, uint32_t ctas)
{
    const int t = threadIdx.x, w = t >> 5, l = t & 31, nw = blockDim.x >> 5;
    double v = warp_sum(fi * fi), *sd = (double *)c.shw[0];
    if (l == 0) sd[w] = v;
    __syncthreads();
    if (w == 0) {
        v = warp_sum(l < nw ? sd[l] : 0.0);
        if (ctas == 1) {
            if (l == 0) c.part64[0] = v;
        } else if (l < (int)ctas) {
            dsmem_st(dsmem_of(&c.part64[rank], (uint32_t)l), v);
        }
    }
    cluster_barrier(ctas);
    if (w == 0) {
        const double nrm = sqrt(warp_sum(l < (int)ctas ? c.part64[l] : 0.0));
        if (l == 0) c.ms.scale = (nrm > 0.0 && !not_finite(nrm)) ? exp2(-rint(log2(nrm))) : 1.0;
    }
    __syncthreads();
    return c.ms.scale;
}

// The sums of a = (r, z), b = (z, A z) and rr = r.r over the cluster (of every
// STEP-th lane's values) and the scalar step on them, taken by every CTA alike.
// Returns whether the loop ends; g and alpha (warp 0) go to cluster_keep.
template <typename M, int STEP>
__device__ __forceinline__ bool cluster_sums(ClusterShared<M> &sh, typename M::V a, typename M::V b,
                                             typename M::V rr, uint32_t rank, uint32_t ctas, double tol2, int maxit,
                                             bool start, double &g, double &alpha)
{
    typedef typename M::V V;
    const int t = threadIdx.x, w = t >> 5, l = t & 31, nw = blockDim.x >> 5;
    V v = sum3<M, STEP>(a, b, rr);
    if ((l & 7) == 0 && l < 24) sh.shw[l >> 3][w] = v; // 0: (r, z), 1: r.r, 2: (z, s)
    __syncthreads();
    if (w == 0) {
        const V none = M::zero();
        v = sum3<M, 1>(l < nw ? sh.shw[0][l] : none, l < nw ? sh.shw[2][l] : none, l < nw ? sh.shw[1][l] : none);
        if (ctas > 1) {
            const V p0 = M::shfl(v, 0), p1 = M::shfl(v, 16), p2 = M::shfl(v, 8);
            if (l < (int)ctas) {
                dsmem_st(dsmem_of(&sh.part[0][rank], (uint32_t)l), M::store(p0));
                dsmem_st(dsmem_of(&sh.part[1][rank], (uint32_t)l), M::store(p1));
                dsmem_st(dsmem_of(&sh.part[2][rank], (uint32_t)l), M::store(p2));
            }
        }
    }
    if (ctas > 1) {
        cluster_barrier(ctas);
        if (w == 0) {
            // the last steps of sum3 on at most 16 partials a value
            const int k = l & 15;
            const bool on = k < (int)ctas, h8 = l & 8;
            V ab = on ? M::load(sh.part[l >> 4][k]) : M::zero(), c = on ? M::load(sh.part[2][k]) : M::zero();
            v = M::add(h8 ? c : ab, M::shfl_xor(h8 ? ab : c, 8));
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) v = M::add(v, M::shfl_xor(v, o));
        }
    }
    g = alpha = 0.0;
    if (w == 0) {
        const double tot = M::value(v), d = __shfl_sync(0xffffffffu, tot, 16), r2 = __shfl_sync(0xffffffffu, tot, 8);
        g = __shfl_sync(0xffffffffu, tot, 0);
        cluster_step(sh.ms, g, d, r2, tol2, maxit, start, alpha);
    }
    __syncthreads();
    return sh.ms.done; // the same values, so the same decision, in every CTA
}

template <typename M>
__device__ __forceinline__ void cluster_init(ClusterScal<M> &ms)
{
    if (threadIdx.x == 0) {
        ms.scale = 1.0;
        ms.iters = ms.k1 = ms.done = 0;
        ms.status = CG_RUNNING;
        ms.rz = ms.ra = 0.0;
    }
}

// the loop's scalars as the host reads them; called by one thread of the cluster
template <typename M>
__device__ __forceinline__ void cluster_report(const ClusterScal<M> &ms, CgScal &sc, int maxit)
{
    sc.rz = ms.rz;
    sc.rr = ms.rr;
    sc.ff = ms.ff;
    sc.thr = ms.thr;
    sc.scale = ms.scale;
    sc.done = 1;
    sc.iters = ms.iters;
    sc.status = ms.status;
    sc.maxit = maxit;
    sc.total_iters += ms.iters;
    sc.k1 = ms.k1;
}
