// state.cu -- the AMG-preconditioned CG of a state solve A_l y = f on a small
// level as one launch: one thread-block cluster runs every iteration with its
// whole V-cycle, the hierarchy from level l down and all vectors in shared
// memory, vectors gathered across the cluster through distributed shared memory.
//
// Graph-replayed, an iteration of such a level is 7-15 launches (1.3 us each, of
// which the work is a fraction), and a solve also pays its start graph and the
// host's reads of the stop flag.  Here a phase (one sweep over the rows of one
// level) is a cluster barrier, a gather and a short sum.
//
//   rows      level k's rows are dealt in runs of 2^lg_k to the CTAs, so the owner
//             of a column is a shift; as many lanes share a row as the CTA has
//             threads for, so a lane has one or two to a few entries
//   matrices  of every level in the owner's shared memory, copied once per solve,
//             columns as the addresses of their vector elements.  (Read from L2
//             in each phase, rows loaded ahead of the barrier, the solves were
//             slower than graph-replayed: 33^2 FP64 cost and gradient 2.38 ms
//             against 1.71.)
//   vectors   of level k: two iterates, b, d, the residual and D^-1; the CG's x, r,
//             p and q in registers of the thread that owns the row
//   coarsest  the dense inverse's rows in shared memory; a phase copies b to every
//             CTA and takes a warp per row
//
// Method, stopping rule and precision are those of the loop in solver.cu
// (single-reduction CG; FP64, or double-float vectors with an FP32 V-cycle), the
// V-cycle's point-wise arithmetic that of spmv.cuh; row sums are grouped by the
// lanes of a row, which depend on the hierarchy only.  The stopping test comes
// beside the next scalar step, as in mass.cu.
//
// What bounds it: dependent latency and issue.  A phase is about 1,400 cycles (a
// cluster barrier 600, the gather 300, the sum over a row's lanes, the point-wise
// step), the sums and the scalar step of an iteration 5,000.  Measured (one GB300,
// whole public call to 1e-10, 16-19 iterations, us, graph-replayed -> here): FP32
// V-cycles 49 rows 339 -> 182, 441 rows 468 -> 319, 961 rows 379 -> 240, 2,025 rows
// 541 -> 356; FP64 461 -> 243, 709 -> 390, 524 -> 307, 771 -> 452.  Rows per CTA
// from 32 to 128 make no difference beyond 5 %.
#include <algorithm>

#include "clustercg.cuh"
#include "spmv.cuh"

// Threads of a CTA.  FP64: with 512 and a lane per entry the FP64 units are held
// by butterflies over nearly empty lanes, one addition of a whole warp a step;
// with 256, at least two entries a lane and idle warps skipping the phase 2,025
// rows take 452 us instead of 665 (33^2 cost and gradient 1.40 -> 1.12 ms).  FP32
// additions are cheap, so its lanes pay: 512 threads -> 256 and two entries a lane
// are 243 -> 230 us on short rows (33^2) but 84 -> 94 on a level of 115 rows of up
// to 24 entries, and a lane's 16 entries then end at rows half as long, so that
// hierarchies fall back to the replayed kernels: 47^2 over four levels 444 -> 683
// us, a cube's level of 449 rows of up to 78 entries 318 -> 428.  Whole calls on
// short rows cannot tell them apart (65^2 solve 13.59 and 13.64 ms, 201^2
// preconditioner 4.48 and 4.49).
template <typename T>
constexpr int SCG_TPB = sizeof(T) == 8 ? 256 : 512;
#define SCG_ROWS 128 // rows of the solved level per CTA
#define SCG_LEVELS 6
#define SCG_SMEM (200 << 10)
#define SCG_CHUNK 4 // entries of a lane read together
#define SCG_MAX_ENTRIES 16
#define SCG_NONE 0xffffffffu

// A matrix's rows of one CTA in shared memory: 2^lgl lanes share a row, lane
// entry e of thread t at [e * width + t], its value (and, for the solved level
// in double-float, the low part) and the address of its column's element in
// the first vector of level x
struct ScgMat {
    const int *rp, *ci;
    const double *v;
    int rows, lg; // rows dealt in runs of 2^lg
    int lgl, entries, width;
    int val, lo, addr; // byte offsets
};
struct ScgLevel {
    ScgMat A, St, S; // St: rows of the next level
    const void *invd;
    int n, lg, off; // off: first byte of the level's vectors
};
template <typename T>
struct ScgArgs {
    ScgLevel lv[SCG_LEVELS];
    const T *inv; // dense inverse of the last level
    int ld, inv_off, b_off;
    int levels, steps, ctas;
    T cd[16], cr[16];
};

enum { SV_XA, SV_XB, SV_B, SV_D, SV_R, SV_IV, SV_COUNT };

template <typename T>
struct ScgCta {
    unsigned char *sm;
    uint32_t rank, ctas;
    __device__ __forceinline__ T *vec(const ScgLevel &L, int which) const
    {
        return (T *)(sm + L.off) + (which << L.lg);
    }
};

// cluster_barrier in two halves: what needs nothing of the other CTAs goes between.
// Warps without entries wait at a place of their own (scg_row).  PTX barriers count
// the warps that arrive wherever they do; __syncthreads() is defined for one place
// only, so a single CTA waits by barrier.cta.sync (all warps at one place instead:
// 31^2 FP64 Hessian apply 727 us against 718).
__device__ __forceinline__ void scg_arrive(uint32_t ctas)
{
    if (ctas > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void scg_wait(uint32_t ctas)
{
    if (ctas > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    else asm volatile("barrier.cta.sync.aligned 0;" ::: "memory");
}

// the CTA's rows of m to shared memory
template <typename T>
__device__ __noinline__ void scg_load(const ScgCta<T> c, const ScgMat &m, const ScgLevel &X)
{
    const int t = threadIdx.x, L = 1 << m.lgl, i = t >> m.lgl, row = ((int)c.rank << m.lg) + i;
    if (t >= m.width) return;
    const bool mine = i < (1 << m.lg) && row < m.rows;
    const int k0 = mine ? m.rp[row] + (t & (L - 1)) : 0, k1 = mine ? m.rp[row + 1] : 0;
    T *val = (T *)(c.sm + m.val) + t, *lo = (T *)(c.sm + m.lo) + t;
    uint32_t *addr = (uint32_t *)(c.sm + m.addr) + t;
#pragma unroll 4
    for (int e = 0; e < m.entries; e++) {
        const int k = k0 + (e << m.lgl);
        const bool ok = k < k1;
        const double v = ok ? m.v[k] : 0.0;
        const int j = ok ? m.ci[k] : 0;
        val[e * m.width] = (T)v;
        if (m.lo >= 0) lo[e * m.width] = (T)(v - (double)(T)v);
        addr[e * m.width] = ok ? dsmem_of((T *)(c.sm + X.off) + (j & ((1 << X.lg) - 1)), (uint32_t)(j >> X.lg)) : SCG_NONE;
    }
}

// Row sums of m times vector `which` of its columns' level, after the cluster
// barrier; the row's first lane has the sum.  PROD: in the accuracy of the CG
// vectors (double-float from value pairs), else plain.
template <typename M, bool PROD>
struct ScgSum {
    typedef typename M::Z V;
    __device__ static V zero() { return (V)0; }
    __device__ static void term(V &s, V v, V, V x) { s = rfma(v, x, s); }
    __device__ static V lanes(V s, int o) { return s + __shfl_xor_sync(0xffffffffu, s, o); }
    __device__ static V done(V s) { return s; }
};
template <>
struct ScgSum<ClusterDf, true> {
    typedef DF V;
    __device__ static V zero() { return DF{0.f, 0.f}; }
    __device__ static void term(V &s, float hi, float lo, float x) { df_fma(s, hi, lo, x); }
    __device__ static V lanes(V s, int o) { return ClusterDf::lanes(s, o); }
    __device__ static V done(V s) { return ClusterDf::done(s); }
};

template <typename M, bool PROD>
__device__ __forceinline__ typename ScgSum<M, PROD>::V scg_row(const ScgCta<typename M::Z> &c, const ScgMat &m,
                                                               uint32_t which_off)
{
    typedef typename M::Z T;
    typedef ScgSum<M, PROD> Sum;
    constexpr bool PAIR = PROD && M::SCALED;
    const int t = threadIdx.x, ne = t < m.width ? m.entries : 0;
    const T *val = (const T *)(c.sm + m.val) + t, *lo = (const T *)(c.sm + m.lo) + t;
    const uint32_t *addr = (const uint32_t *)(c.sm + m.addr) + t;
    T v[SCG_CHUNK], w[SCG_CHUNK], x[SCG_CHUNK];
    uint32_t a[SCG_CHUNK];
    auto load = [&](int e0) {
#pragma unroll
        for (int j = 0; j < SCG_CHUNK; j++) {
            const bool ok = e0 + j < ne;
            a[j] = ok ? addr[(e0 + j) * m.width] : SCG_NONE;
            v[j] = ok ? val[(e0 + j) * m.width] : (T)0;
            w[j] = PAIR && ok ? lo[(e0 + j) * m.width] : (T)0;
        }
    };
    scg_arrive(c.ctas);
    if (sizeof(T) == 8 && t >= m.width) { // a warp without entries (the width is a multiple of 32)
        scg_wait(c.ctas);
        return Sum::zero();
    }
    load(0);
    scg_wait(c.ctas);
    typename Sum::V s = Sum::zero();
    for (int e = 0;;) {
#pragma unroll
        for (int j = 0; j < SCG_CHUNK; j++) x[j] = a[j] != SCG_NONE ? dsmem_ld(a[j] + which_off, T()) : (T)0;
#pragma unroll
        for (int j = 0; j < SCG_CHUNK; j++)
            if (a[j] != SCG_NONE) Sum::term(s, v[j], w[j], x[j]);
        e += SCG_CHUNK;
        if (e >= m.entries) break;
        load(e);
    }
    for (int o = 1 << m.lgl >> 1; o > 0; o >>= 1) s = Sum::lanes(s, o);
    return Sum::done(s);
}

// whether this thread is the first lane of one of the CTA's rows of m
__device__ __forceinline__ bool scg_lead(const ScgMat &m, uint32_t rank)
{
    const int t = threadIdx.x, i = t >> m.lgl;
    return t < m.width && (t & ((1 << m.lgl) - 1)) == 0 && i < (1 << m.lg) && ((int)rank << m.lg) + i < m.rows;
}

// the dense coarsest solve: b to every CTA, then a warp per row
template <typename T>
__device__ __forceinline__ void scg_dense(const ScgCta<T> &c, const ScgArgs<T> &a)
{
    const ScgLevel &L = a.lv[a.levels - 1];
    const int t = threadIdx.x, n = L.n, first = (int)c.rank << L.lg, mine = min(1 << L.lg, n - first);
    const T *b = c.vec(L, SV_B), *inv = (const T *)(c.sm + a.inv_off);
    T *all = (T *)(c.sm + a.b_off), *x = c.vec(L, SV_XB);
    cluster_barrier(c.ctas);
    for (int j = t; j < n; j += SCG_TPB<T>)
        all[j] = dsmem_ld(dsmem_of(b + (j & ((1 << L.lg) - 1)), (uint32_t)(j >> L.lg)), T());
    __syncthreads();
    for (int i = t >> 5; i < mine; i += SCG_TPB<T> / 32) {
        T s0 = 0, s1 = 0;
        int j = t & 31;
        for (; j + 32 < n; j += 64) {
            s0 = rfma(inv[i * n + j], all[j], s0);
            s1 = rfma(inv[i * n + j + 32], all[j + 32], s1);
        }
        if (j < n) s0 = rfma(inv[i * n + j], all[j], s0);
        s0 += s1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        if ((t & 31) == 0) x[i] = s0;
    }
}

// V-cycle on the level's b; its first step (d and the iterate SV_XA) is taken
// already, the result is left in SV_XB (2 ns - 1 alternations of the iterates).
// Every phase starts with a barrier and gathers only what the phase before
// wrote, and writes nothing that it gathers.
template <typename M>
__device__ __forceinline__ void scg_vcycle(const ScgCta<typename M::Z> &c, const ScgArgs<typename M::Z> &a)
{
    typedef typename M::Z T;
    const int last = a.levels - 1, ns = a.steps;
    // a level's phases going down: ns - 1 steps, residual, restriction; going
    // up: prolongation, ns steps
    int k = 0, j = 0;
    bool up = false;
    for (;;) {
        if (k == last) {
            scg_dense<T>(c, a);
            up = true;
            k--;
            j = 0;
        }
        if (k < 0) break;
        const ScgLevel &L = a.lv[k], &C = a.lv[k + 1];
        const bool smooth = up ? j > 0 : j < ns - 1, restr = !up && j == ns, prolong = up && j == 0;
        const int step = up ? j - 1 : j + 1, odd = up ? (ns - 1 + max(step, 0)) & 1 : min(j, ns - 1) & 1;
        const int cur = odd ? SV_XB : SV_XA, nxt = odd ? SV_XA : SV_XB;
        const ScgMat &m = restr ? L.St : prolong ? L.S : L.A;
        const int which = restr ? SV_R : prolong ? SV_XB : cur, xlg = prolong ? C.lg : L.lg;
        const T v = scg_row<M, false>(c, m, (uint32_t)(which << xlg) * (uint32_t)sizeof(T));
        if (scg_lead(m, c.rank)) {
            const int i = threadIdx.x >> m.lgl;
            if (smooth) {
                T dn, xn, *d = c.vec(L, SV_D);
                cheb_point(c.vec(L, SV_B)[i], v, c.vec(L, SV_IV)[i], d[i], c.vec(L, cur)[i],
                           up && step == 0 ? (T)0 : a.cd[step], a.cr[step], dn, xn);
                d[i] = dn;
                c.vec(L, nxt)[i] = xn;
            } else if (prolong) {
                T *x = c.vec(L, cur);
                x[i] = radd(x[i], v);
            } else if (restr) { // with the coarse level's first step
                c.vec(C, SV_B)[i] = v;
                if (k + 1 < last)
                    c.vec(C, SV_D)[i] = c.vec(C, SV_XA)[i] = cheb_first_point(v, c.vec(C, SV_IV)[i], a.cr[0]);
            } else {
                c.vec(L, SV_R)[i] = rsub(c.vec(L, SV_B)[i], v);
            }
        }
        if (j++ == ns) {
            j = 0;
            k += up ? -1 : 1;
        }
    }
}

__device__ __forceinline__ float scg_head(DF r) { return r.hi; }
__device__ __forceinline__ double scg_head(double r) { return r; }

template <typename M>
__global__ void __launch_bounds__(SCG_TPB<typename M::Z>, 1)
    k_state_cg(const __grid_constant__ ScgArgs<typename M::Z> a, const double *f, double *__restrict__ y,
               CgScal *scal, double tol2, int maxit)
{
    typedef typename M::Z T;
    typedef typename M::V V;
    extern __shared__ __align__(16) unsigned char scg_sm[];
    __shared__ V sv[SCG_ROWS];
    __shared__ ClusterShared<M> sh;
    const int t = threadIdx.x;
    ScgCta<T> c;
    c.sm = scg_sm;
    c.ctas = (uint32_t)a.ctas;
    c.rank = a.ctas == 1 ? 0u : cg::this_cluster().block_rank();
    // what only the setup writes: matrices, D^-1, the dense rows
    for (int k = 0; k < a.levels; k++) {
        const ScgLevel &L = a.lv[k];
        if (k < a.levels - 1 || k == 0) scg_load<T>(c, L.A, L);
        if (k == a.levels - 1) break;
        scg_load<T>(c, L.St, L);
        scg_load<T>(c, L.S, a.lv[k + 1]);
        const int row = ((int)c.rank << L.lg) + t;
        if (t < (1 << L.lg) && row < L.n) c.vec(L, SV_IV)[t] = ((const T *)L.invd)[row];
    }
    {
        const ScgLevel &L = a.lv[a.levels - 1];
        const int first = (int)c.rank << L.lg, mine = min(1 << L.lg, L.n - first);
        T *inv = (T *)(c.sm + a.inv_off);
        for (int i = t >> 5; i < mine; i += SCG_TPB<T> / 32)
            for (int j = t & 31; j < L.n; j += 32) inv[i * L.n + j] = a.inv[(int64_t)(first + i) * a.ld + j];
    }
    const ScgLevel &L = a.lv[0];
    const int row = ((int)c.rank << L.lg) + t;
    const bool own = t < (1 << L.lg) && row < L.n, smooths = a.levels > 1;
    pdl_enter();
    const double fi = own ? f[row] : 0.0;
    cluster_init(sh.ms);
    cluster_barrier(c.ctas); // every CTA runs before any of them is written to
    const double scale = M::SCALED ? cluster_scale(sh, fi, c.rank, c.ctas) : 1.0;
    V r = own ? M::scaled(fi, scale) : M::zero(), x = M::zero(), p = M::zero(), q = M::zero(), rr = M::sqr(r);
    T *z = c.vec(L, SV_XB);
    for (int it = 0;; it++) {
        if (own) {
            const T rh = scg_head(r);
            c.vec(L, SV_B)[t] = rh;
            if (smooths) c.vec(L, SV_D)[t] = c.vec(L, SV_XA)[t] = cheb_first_point(rh, c.vec(L, SV_IV)[t], a.cr[0]);
        }
        scg_vcycle<M>(c, a);
        const V row_s = scg_row<M, true>(c, L.A, (uint32_t)(SV_XB << L.lg) * (uint32_t)sizeof(T));
        if (scg_lead(L.A, c.rank)) sv[t >> L.A.lgl] = row_s;
        __syncthreads();
        const V s = own ? sv[t] : M::zero();
        const T zi = own ? z[t] : (T)0;
        double g, alpha;
        if (cluster_sums<M, 1>(sh, own ? M::dot(r, zi) : M::zero(), own ? M::dot(s, zi) : M::zero(), rr, c.rank,
                               c.ctas, tol2, maxit, it == 0, g, alpha))
            break;
        if (own) {
            const typename M::C al = sh.ms.al, be = sh.ms.be;
            p = M::axpy(M::of_z(zi), be, p);
            q = M::axpy(s, be, q);
            x = M::axpy(x, al, p);
            r = M::axpy(r, M::neg(al), q);
            rr = M::sqr(r);
        }
        if (t < 32) cluster_keep(sh.ms, g, alpha);
    }
    // every remote access was before the last barrier: CTAs may leave apart
    if (own) y[row] = M::out(x, 1.0 / scale);
    if (c.rank == 0 && t == 0) cluster_report(sh.ms, *scal, maxit);
}

// ------------------------------------------------------------------ host side
// Place m's rows (dealt in runs of 2^lg) in shared memory: as many lanes a row
// as the threads allow and its longest row fills (FP64: with two entries each).
static bool scg_place(const DevCsr &a, int lg, size_t vb, bool pair, ScgMat *m, int64_t *off)
{
    if (a.rows < 1 || a.longest < 1) return false;
    const int tpb = vb == 8 ? SCG_TPB<double> : SCG_TPB<float>, least = vb == 8 ? 2 : 1; // entries a lane
    int lgl = 0;
    while (lgl < 5 && (2 << lgl << lg) <= tpb && (least << lgl) < a.longest) lgl++;
    const int width = std::max(32, 1 << lg << lgl), entries = ceil_div(a.longest, 1 << lgl);
    if (width > tpb || entries > SCG_MAX_ENTRIES) return false;
    const int64_t each = (int64_t)entries * width;
    *m = ScgMat{a.rp, a.ci, a.v, a.rows, lg, lgl, entries, width, (int)*off, -1, 0};
    *off += each * vb;
    if (pair) {
        m->lo = (int)*off;
        *off += each * vb;
    }
    m->addr = (int)*off;
    *off += each * 4;
    return *off <= SCG_SMEM;
}

// Levels of at most 2,048 rows (16 CTAs of 128) whose hierarchy fits in shared
// memory.  Larger ones stay with the replayed kernels, which spread a phase's
// rows over the whole GPU and are what the fuse_coarse option chooses among.
// The rows placed are the canonical ones: exact zeros, which the replayed kernels
// leave out (a quarter of a regular 2D grid's entries, half of a Kuhn cube's),
// take a lane's slot here.  Graph-replayed -> here all the same (us to 1e-10, FP32
// / FP64): regular 33^2 square 411 -> 241 / 523 -> 307; 13^3 cube, 2,028 rows, 429
// -> 269 / 562 -> 379, its coarse level of 206 rows of up to 72 entries above a
// level of 14 400 -> 291 / 614 -> 364.
template <typename T>
static bool scg_shape(const amgh_problem *p, int l, ScgArgs<T> *a, size_t *smem)
{
    const int n = p->sl[l].A.rows, levels = p->Ls - l;
    if (n < 1 || n > CLUSTER_MAX * SCG_ROWS || levels > SCG_LEVELS) return false;
    if (l == 0 && p->aopts.matrix_free) return false;
    int lg = sizeof(T) == 4 ? 6 : 5;
    while ((int64_t)CLUSTER_MAX << lg < n) lg++;
    const int ctas = ceil_div(n, 1 << lg);
    int64_t off = 0; // multiples of 8: every size is a multiple of 32 elements or rounded
    for (int k = 0; k < levels; k++) {
        ScgLevel &L = a->lv[k];
        L.n = p->sl[l + k].A.rows;
        L.lg = 0;
        while ((int64_t)ctas << L.lg < L.n) L.lg++;
        if (k == 0) L.lg = lg;
        L.off = (int)off;
        off += ((int64_t)SV_COUNT * sizeof(T) << L.lg) + 15 & ~15ll;
        if (off > SCG_SMEM) return false;
    }
    for (int k = 0; k < levels; k++) {
        const StateLevel &S = p->sl[l + k];
        ScgLevel &L = a->lv[k];
        const bool last = k == levels - 1;
        if ((!last || k == 0) && !scg_place(S.A, L.lg, sizeof(T), k == 0 && sizeof(T) == 4, &L.A, &off)) return false;
        if (last) break;
        if (!scg_place(S.St, a->lv[k + 1].lg, sizeof(T), false, &L.St, &off)) return false;
        if (!scg_place(S.S, L.lg, sizeof(T), false, &L.S, &off)) return false;
    }
    const ScgLevel &E = a->lv[levels - 1];
    a->inv_off = (int)off;
    off += (int64_t)E.n * sizeof(T) << E.lg;
    a->b_off = (int)off;
    off += (int64_t)E.n * sizeof(T);
    if (off > SCG_SMEM) return false;
    a->levels = levels;
    a->ctas = ctas;
    a->steps = p->nsteps;
    for (int s = 0; s < p->nsteps; s++) {
        a->cd[s] = (T)p->cd[s];
        a->cr[s] = (T)p->cr[s];
    }
    *smem = (size_t)off;
    return true;
}

template <typename M>
static int scg_launch(amgh_problem *p, int l, ScgArgs<typename M::Z> &a, size_t smem, const double *f, double *y,
                      double tol, int maxit, bool *done)
{
    auto kern = k_state_cg<M>;
    *done = cluster_fits((const void *)kern, a.ctas, SCG_TPB<typename M::Z>, smem, SCG_SMEM);
    if (!*done) return AMGH_OK;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = a.ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(a.ctas, 1, 1);
    cfg.blockDim = dim3(SCG_TPB<typename M::Z>, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = p->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    CU(cudaLaunchKernelEx(&cfg, kern, a, f, y, p->sl[l].scal, tol * tol, maxit));
    LAUNCH_CHECK();
    return AMGH_OK;
}

// The state CG of level l as one cluster launch, its scalars left in the
// level's scal; *done = false (and nothing launched) where the level does not fit
// or the device cannot place the cluster
int state_cluster(amgh_problem *p, int l, const double *f, double *y, double tol, int maxit, bool *done)
{
    *done = false;
    size_t smem = 0;
    if (p->aopts.precision == 2 && maxit <= CLUSTER_MAX_ITERS) {
        ScgArgs<float> a = {};
        if (scg_shape<float>(p, l, &a, &smem)) {
            for (int k = 0; k < a.levels; k++) a.lv[k].invd = p->sl[l + k].invd32;
            a.inv = p->Acoarse.inv32;
            a.ld = p->Acoarse.ld32;
            return scg_launch<ClusterDf>(p, l, a, smem, f, y, tol, maxit, done);
        }
    } else if (p->aopts.precision == 0 && maxit <= CLUSTER_MAX_ITERS) {
        ScgArgs<double> a = {};
        if (scg_shape<double>(p, l, &a, &smem)) {
            for (int k = 0; k < a.levels; k++) a.lv[k].invd = p->sl[l + k].invd;
            a.inv = p->Acoarse.inv;
            a.ld = p->Acoarse.n;
            return scg_launch<ClusterF64>(p, l, a, smem, f, y, tol, maxit, done);
        }
    }
    return AMGH_OK;
}
