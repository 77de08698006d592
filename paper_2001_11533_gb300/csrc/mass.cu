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
#include <algorithm>

#include "internal.cuh"
#include "clustercg.cuh"

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

template <typename M, int L, int E>
__global__ void __launch_bounds__(MCG_TPB<M, E>)
    k_mass_cg(MassMat A, const typename M::Z *__restrict__ invd, MassRhs rhs, int lg, int ctas_, double tol2, int maxit)
{
    typedef typename M::Z Z;
    typedef typename M::V V;
    __shared__ Z z[MCG_TPB<M, E>];
    __shared__ ClusterShared<M> sh;
    const uint32_t ctas = (uint32_t)ctas_;
    const uint32_t rank = ctas == 1 ? 0u : cg::this_cluster().block_rank();
    const int col = blockIdx.y, n = A.n, t = threadIdx.x;
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
    cluster_init(sh.ms);
    cluster_barrier(ctas); // every CTA runs before any of them is written to
    const double scale = M::SCALED ? cluster_scale(sh, fi, rank, ctas) : 1.0;
    V r = lead ? M::scaled(fi, scale) : M::zero(), x = M::zero(), p = M::zero(), q = M::zero(), rr = M::sqr(r);
    Z zi = M::jacobi(iv, r);
    if (lead) z[i] = zi;
    cluster_barrier(ctas);
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
        double g, alpha;
        if (cluster_sums<M, L>(sh, lead ? M::dot(r, zi) : M::zero(), lead ? M::dot(s, zi) : M::zero(), rr, rank,
                               ctas, tol2, maxit, it == 0, g, alpha))
            break;
        // ---- p = z + beta p, q = s + beta q, x += alpha p, r -= alpha q, z = D^-1 r, r.r
        if (lead) {
            const typename M::C al = sh.ms.al, be = sh.ms.be;
            p = M::axpy(M::of_z(zi), be, p); // beta = 0 and p = q = 0 in the first iteration
            q = M::axpy(s, be, q);
            x = M::axpy(x, al, p);
            r = M::axpy(r, M::neg(al), q);
            rr = M::sqr(r);
            zi = M::jacobi(iv, r);
            z[i] = zi;
        }
        if (t < 32) cluster_keep(sh.ms, g, alpha);
        cluster_barrier(ctas);
    }
    // every remote access was before the last barrier: CTAs may leave apart
    if (lead) rhs.x[(int64_t)row * rhs.stride + col] = M::out(x, 1.0 / scale);
    if (rank == 0 && t == 0) cluster_report(sh.ms, rhs.sc[col], maxit);
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
        while ((L << lg) < least || (int64_t)CLUSTER_MAX << lg < n) lg++;
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
               mass_shape_for(a, 16, 512, 256, MCG_TPB<ClusterDf, 16>, out) ||
               mass_shape_for(a, 8, 512, 256, MCG_TPB<ClusterDf, 8>, out);
    return mass_shape_for(a, 8, 128, 64, 256, out) || mass_shape_for(a, 16, 128, 64, MCG_TPB<ClusterF64, 16>, out);
}

template <typename M, int L, int E>
static int mass_launch_as(amgh_problem *p, const MassShape &sh, const DevCsr &a, const void *invd,
                          const MassRhs &rhs, double tol, int maxit, bool *done)
{
    auto kern = k_mass_cg<M, L, E>;
    *done = cluster_fits((const void *)kern, sh.ctas, sh.threads, 0, 0);
    if (!*done) return AMGH_OK;
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
                       double tol, int maxit, bool *done)
{
    if (sh.entries == 8) return mass_launch_as<M, L, 8>(p, sh, a, invd, rhs, tol, maxit, done);
    return mass_launch_as<M, L, 16>(p, sh, a, invd, rhs, tol, maxit, done);
}

template <typename M>
static int mass_dispatch(amgh_problem *p, const MassShape &sh, const DevCsr &a, const void *invd, const MassRhs &rhs,
                         double tol, int maxit, bool *done)
{
    switch (sh.lanes) {
    case 2: return mass_launch<M, 2>(p, sh, a, invd, rhs, tol, maxit, done);
    case 4: return mass_launch<M, 4>(p, sh, a, invd, rhs, tol, maxit, done);
    case 8: return mass_launch<M, 8>(p, sh, a, invd, rhs, tol, maxit, done);
    case 16: return mass_launch<M, 16>(p, sh, a, invd, rhs, tol, maxit, done);
    case 32: return mass_launch<M, 32>(p, sh, a, invd, rhs, tol, maxit, done);
    default: return mass_launch<M, 1>(p, sh, a, invd, rhs, tol, maxit, done);
    }
}

int mass_cluster(amgh_problem *p, const CtrlLevel &C, bool df, const double *b, double *x, CgScal *sc, int cols,
                 double tol, int maxit, bool *done)
{
    MassShape sh;
    *done = false;
    if (maxit > CLUSTER_MAX_ITERS || !mass_shape(C.Mu, df, &sh)) return AMGH_OK;
    const MassRhs rhs = {b, x, sc, cols};
    return df ? mass_dispatch<ClusterDf>(p, sh, C.Mu, C.mu_invdiag32, rhs, tol, maxit, done)
              : mass_dispatch<ClusterF64>(p, sh, C.Mu, C.mu_invdiag, rhs, tol, maxit, done);
}
