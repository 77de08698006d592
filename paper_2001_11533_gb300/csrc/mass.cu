// mass.cu -- the Jacobi-preconditioned CG of a mass solve M_{u,l} x = b
// (Sec. 5.2) on a small level as one launch: one thread-block cluster per
// right side keeps the matrix and every vector in registers and shared memory
// for the whole solve.
//
// A mass CG iteration is one product with 7-25 entries a row and a handful of
// vector updates: at most a megabyte on these levels, far below what two
// launches cost (11-20 us an iteration as graph-replayed kernels: launch,
// last-block reductions through global memory, and the host's reads of the
// stop flag).  What is left in one launch is latency: two cluster barriers per
// iteration, one gather, one sum, one scalar step.
//
//   rows     CTA r of the cluster owns rows [r 2^lg, (r+1) 2^lg), so the owner
//            of a column is a shift.  L lanes share a row, at most eight
//            entries each, held in registers for the whole solve with their
//            columns as shared memory addresses; the group's first lane holds
//            the row's x, r, p, q
//   z        in shared memory, gathered across the cluster through distributed
//            shared memory
//   sums     (r, z), (z, A z) and the r.r of the iteration before in one
//            butterfly that halves the values it carries at its first two
//            steps (6 additions instead of 15), then one warp per CTA, whose
//            partial goes to every CTA of the cluster; each CTA adds the
//            partials in the same fixed order and takes the same scalar step,
//            so all of them reach the same stopping decision without a further
//            barrier.  (The stopping test of an iteration so comes beside the
//            scalar step of the next: one product more per solve, one sum and
//            one barrier less per iteration.)
//
// Method, stopping rule and status codes are those of the graph-replayed loop
// in solver.cu (single-reduction CG, blas.cu); so is the precision: FP64, or
// (precision 2) double-float vectors with an FP32 Jacobi direction and FP64
// scalars.  How the sums are grouped depends on the level's size and longest
// row only.
//
// What bounds it: dependent instructions.  At 2,278 rows an iteration is about
// 8,000 cycles: product 1,700, sum 1,900, FP64 scalar step 1,900, update 1,400,
// barriers 1,200.  Measured (one GB300, whole public call of 15-25 iterations,
// graph-replayed kernels -> here): 56 rows 297 -> 73 us, 581 rows 406 -> 110,
// 2,278 rows 421 -> 137, 4,225 rows 384 -> 123 (FP64: 339 -> 86, 459 -> 123,
// 486 -> 198, 439 -> 180).
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "internal.cuh"
#include "df.cuh"
#include "util.cuh"

namespace cg = cooperative_groups;

#define MCG_MAX_CTAS 16
// threads of a CTA whose lanes hold at most E entries of a row
template <typename M, int E>
constexpr int MCG_TPB = M::SCALED && E == 8 ? 1024 : 512;

// right sides: element i of column c at f[i * stride + c], x likewise; the
// final scalars of column c go to sc[c]
struct MassRhs {
    const double *f;
    double *x;
    CgScal *sc;
    int stride;
};

// canonical CSR of the mass matrix
struct MassMat {
    int n;
    const int *rp, *ci;
    const double *v;
};

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
struct MassDf {
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
struct MassF64 {
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
struct MassScal {
    double ff, rr, thr, rz, ra, scale; // ra = rz alpha
    typename M::C al, be;
    int iters, k1, status, done;
};

// warp 0: the stopping test of the iteration before, then alpha and beta of
// the single-reduction CG.  Lane 0 writes alpha's side, lane 1 beta's.
template <typename M>
__device__ __forceinline__ void mass_step(MassScal<M> &s, double g, double d, double rr, double tol2, int maxit,
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
__device__ __forceinline__ void mass_keep(MassScal<M> &s, double g, double alpha)
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
__device__ __forceinline__ void mass_barrier(uint32_t ctas)
{
    if (ctas == 1) {
        __syncthreads();
        return;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename M, int L, int E>
__global__ void __launch_bounds__(MCG_TPB<M, E>)
    k_mass_cg(MassMat A, const typename M::Z *__restrict__ invd, MassRhs rhs, int lg, int ctas_, double tol2, int maxit)
{
    typedef typename M::Z Z;
    typedef typename M::V V;
    typedef typename M::P P;
    __shared__ Z z[MCG_TPB<M, E>];
    __shared__ V shw[3][32];
    __shared__ P part[3][MCG_MAX_CTAS]; // (r, z), (z, A z) and r.r of every CTA
    __shared__ double part64[MCG_MAX_CTAS];
    __shared__ MassScal<M> ms;
    const uint32_t ctas = (uint32_t)ctas_;
    const uint32_t rank = ctas == 1 ? 0u : cg::this_cluster().block_rank();
    const int col = blockIdx.y, n = A.n, t = threadIdx.x, w = t >> 5, l = t & 31, nw = blockDim.x >> 5;
    const int i = t / L, row = ((int)rank << lg) + i; // this lane group's row
    const bool mine = i < (1 << lg) && row < n, lead = mine && t % L == 0;
    // the row: values in registers, columns as shared memory addresses
    typename M::Entry ev[E];
    uint32_t ea[E];
    int ne = 0;
    if (mine) {
        const int k0 = A.rp[row] + t % L, k1 = A.rp[row + 1];
#pragma unroll
        for (int j = 0; j < E; j++)
            if (k0 + j * L < k1) {
                const int c = A.ci[k0 + j * L];
                ev[j] = M::entry(A.v[k0 + j * L]);
                ea[j] = dsmem_at(z + (c & ((1 << lg) - 1)), (uint32_t)(c >> lg), rank);
                ne = j + 1;
            }
    }
    const Z iv = lead ? invd[row] : (Z)0;
    pdl_enter();
    const double fi = lead ? rhs.f[(int64_t)row * rhs.stride + col] : 0.0;
    if (t == 0) {
        ms.scale = 1.0;
        ms.iters = ms.k1 = ms.done = 0;
        ms.status = CG_RUNNING;
        ms.rz = ms.ra = 0.0;
    }
    mass_barrier(ctas); // every CTA runs before any of them is written to
    double scale = 1.0;
    if (M::SCALED) {
        // the power of two nearest 1 / ||f||, an exact scaling
        double v = warp_sum(fi * fi), *sd = (double *)shw[0];
        if (l == 0) sd[w] = v;
        __syncthreads();
        if (w == 0) {
            v = warp_sum(l < nw ? sd[l] : 0.0);
            if (ctas == 1) {
                if (l == 0) part64[0] = v;
            } else if (l < (int)ctas) {
                dsmem_st(dsmem_of(&part64[rank], (uint32_t)l), v);
            }
        }
        mass_barrier(ctas);
        if (w == 0) {
            const double nrm = sqrt(warp_sum(l < (int)ctas ? part64[l] : 0.0));
            if (l == 0) ms.scale = (nrm > 0.0 && !not_finite(nrm)) ? exp2(-rint(log2(nrm))) : 1.0;
        }
        __syncthreads();
        scale = ms.scale;
    }
    V r = lead ? M::scaled(fi, scale) : M::zero(), x = M::zero(), p = M::zero(), q = M::zero(), rr = M::sqr(r);
    Z zi = M::jacobi(iv, r);
    if (lead) z[i] = zi;
    mass_barrier(ctas);
    for (int it = 0;; it++) {
        // ---- s = A z; (r, z), (z, s) and the last r.r over the cluster
        Z zv[E];
#pragma unroll
        for (int j = 0; j < E; j++) zv[j] = j < ne ? dsmem_ld(ea[j], Z()) : (Z)0;
        V s = M::zero();
#pragma unroll
        for (int j = 0; j < E; j++)
            if (j < ne) M::term(s, ev[j], zv[j]);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) s = M::lanes(s, o);
        s = M::done(s);
        V v = sum3<M, L>(lead ? M::dot(r, zi) : M::zero(), lead ? M::dot(s, zi) : M::zero(), rr);
        if ((l & 7) == 0 && l < 24) shw[l >> 3][w] = v; // 0: (r, z), 1: r.r, 2: (z, s)
        __syncthreads();
        if (w == 0) {
            const V none = M::zero();
            v = sum3<M, 1>(l < nw ? shw[0][l] : none, l < nw ? shw[2][l] : none, l < nw ? shw[1][l] : none);
            if (ctas > 1) {
                const V a = M::shfl(v, 0), b = M::shfl(v, 16), c = M::shfl(v, 8);
                if (l < (int)ctas) {
                    dsmem_st(dsmem_of(&part[0][rank], (uint32_t)l), M::store(a));
                    dsmem_st(dsmem_of(&part[1][rank], (uint32_t)l), M::store(b));
                    dsmem_st(dsmem_of(&part[2][rank], (uint32_t)l), M::store(c));
                }
            }
        }
        if (ctas > 1) {
            mass_barrier(ctas);
            if (w == 0) {
                // the last steps of sum3 on at most 16 partials a value
                const int k = l & 15;
                const bool on = k < (int)ctas, h8 = l & 8;
                V ab = on ? M::load(part[l >> 4][k]) : M::zero(), c = on ? M::load(part[2][k]) : M::zero();
                v = M::add(h8 ? c : ab, M::shfl_xor(h8 ? ab : c, 8));
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) v = M::add(v, M::shfl_xor(v, o));
            }
        }
        double g = 0.0, alpha = 0.0;
        if (w == 0) {
            const double tot = M::value(v), d = __shfl_sync(0xffffffffu, tot, 16),
                         r2 = __shfl_sync(0xffffffffu, tot, 8);
            g = __shfl_sync(0xffffffffu, tot, 0);
            mass_step(ms, g, d, r2, tol2, maxit, it == 0, alpha);
        }
        __syncthreads();
        if (ms.done) break; // the same values, so the same decision, in every CTA
        // ---- p = z + beta p, q = s + beta q, x += alpha p, r -= alpha q, z = D^-1 r, r.r
        if (lead) {
            const typename M::C al = ms.al, be = ms.be;
            p = M::axpy(M::of_z(zi), be, p); // beta = 0 and p = q = 0 in the first iteration
            q = M::axpy(s, be, q);
            x = M::axpy(x, al, p);
            r = M::axpy(r, M::neg(al), q);
            rr = M::sqr(r);
            zi = M::jacobi(iv, r);
            z[i] = zi;
        }
        if (w == 0) mass_keep(ms, g, alpha);
        mass_barrier(ctas);
    }
    // every remote access was before the last barrier: CTAs may leave apart
    if (lead) rhs.x[(int64_t)row * rhs.stride + col] = M::out(x, 1.0 / scale);
    if (rank == 0 && t == 0) {
        CgScal &sc = rhs.sc[col];
        sc.rz = ms.rz;
        sc.rr = ms.rr;
        sc.ff = ms.ff;
        sc.thr = ms.thr;
        sc.scale = scale;
        sc.done = 1;
        sc.iters = ms.iters;
        sc.status = ms.status;
        sc.maxit = maxit;
        sc.total_iters += ms.iters;
        sc.k1 = ms.k1;
    }
}

// ------------------------------------------------------------------ host side
struct MassShape {
    int entries, lanes, lg, ctas, threads;
};

// Lanes per row so that none has more than `entries`, and rows per CTA so that
// its lanes cover them at once: one CTA where `one` lanes suffice, else up to
// 16 with at least `least` lanes each and at most `most`.
static bool mass_shape_for(const DevCsr &a, int entries, int one, int least, int most, MassShape *out)
{
    const int n = a.rows;
    if (n < 1 || a.longest < 1 || a.longest > 32 * entries) return false;
    int L = 1, lg = 0;
    while (L * entries < a.longest) L *= 2;
    if ((int64_t)n * L <= one) {
        while ((1 << lg) < n) lg++;
    } else {
        while ((L << lg) < least || (int64_t)MCG_MAX_CTAS << lg < n) lg++;
    }
    if ((int64_t)L << lg > most) return false;
    out->entries = entries;
    out->lanes = L;
    out->lg = lg;
    out->ctas = ceil_div(n, 1 << lg);
    out->threads = std::max(64, L << lg);
    return true;
}

// Which form: eight entries a lane while the lanes are few (the sum over a
// lane's entries is a dependent chain), then sixteen (half the lanes to sum and
// update over), then eight again in CTAs of 1024 threads, which reach furthest.
// Measured, us a mass solve of ~20 iterations to 1e-10 through the public call,
// 8 / 16 entries: 478 rows 99 / 113, 2278 rows 148 / 139, graph-replayed
// kernels 335 and 421.  FP64 spreads wider (its units, at 1/64 of the FP32
// rate, are what it waits for: 198 rows on 4 CTAs 106, on one 147) and ends
// where a 512-thread CTA does.
static bool mass_shape(const DevCsr &a, bool df, MassShape *out)
{
    if (df)
        return mass_shape_for(a, 8, 256, 256, 256, out) ||
               mass_shape_for(a, 16, 512, 256, MCG_TPB<MassDf, 16>, out) ||
               mass_shape_for(a, 8, 512, 256, MCG_TPB<MassDf, 8>, out);
    return mass_shape_for(a, 8, 128, 64, 256, out) || mass_shape_for(a, 16, 128, 64, MCG_TPB<MassF64, 16>, out);
}

template <typename M, int L, int E>
static int mass_launch_as(amgh_problem *p, const MassShape &sh, const DevCsr &a, const void *invd,
                          const MassRhs &rhs, double tol, int maxit)
{
    auto kern = k_mass_cg<M, L, E>;
    // clusters above 8 CTAs: allowed once per instantiation and device
    static std::atomic<uint64_t> allowed{0};
    int dev = 0;
    CU(cudaGetDevice(&dev));
    const uint64_t bit = 1ull << (dev & 63);
    if (!(allowed.load() & bit)) {
        CU(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        allowed.fetch_or(bit);
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = sh.ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(sh.ctas, rhs.stride, 1);
    cfg.blockDim = dim3(sh.threads, 1, 1);
    cfg.stream = p->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const MassMat A = {a.rows, a.rp, a.ci, a.v};
    CU(cudaLaunchKernelEx(&cfg, kern, A, (const typename M::Z *)invd, rhs, sh.lg, sh.ctas, tol * tol, maxit));
    LAUNCH_CHECK();
    return AMGH_OK;
}

template <typename M, int L>
static int mass_launch(amgh_problem *p, const MassShape &sh, const DevCsr &a, const void *invd, const MassRhs &rhs,
                       double tol, int maxit)
{
    if (sh.entries == 8) return mass_launch_as<M, L, 8>(p, sh, a, invd, rhs, tol, maxit);
    return mass_launch_as<M, L, 16>(p, sh, a, invd, rhs, tol, maxit);
}

template <typename M>
static int mass_dispatch(amgh_problem *p, const MassShape &sh, const DevCsr &a, const void *invd, const MassRhs &rhs,
                         double tol, int maxit)
{
    switch (sh.lanes) {
    case 2: return mass_launch<M, 2>(p, sh, a, invd, rhs, tol, maxit);
    case 4: return mass_launch<M, 4>(p, sh, a, invd, rhs, tol, maxit);
    case 8: return mass_launch<M, 8>(p, sh, a, invd, rhs, tol, maxit);
    case 16: return mass_launch<M, 16>(p, sh, a, invd, rhs, tol, maxit);
    case 32: return mass_launch<M, 32>(p, sh, a, invd, rhs, tol, maxit);
    default: return mass_launch<M, 1>(p, sh, a, invd, rhs, tol, maxit);
    }
}

bool mass_cluster_fits(const DevCsr &a, bool df)
{
    MassShape sh;
    return mass_shape(a, df, &sh);
}

int mass_cluster(amgh_problem *p, const CtrlLevel &C, bool df, const double *b, double *x, CgScal *sc, int cols,
                 double tol, int maxit)
{
    MassShape sh;
    if (!mass_shape(C.Mu, df, &sh)) return AMGH_ERR_INVALID_ARG;
    const MassRhs rhs = {b, x, sc, cols};
    return df ? mass_dispatch<MassDf>(p, sh, C.Mu, C.mu_invdiag32, rhs, tol, maxit)
              : mass_dispatch<MassF64>(p, sh, C.Mu, C.mu_invdiag, rhs, tol, maxit);
}
