// transfer.cu -- the V-cycle's transfers fused with the products beside them.
//
// With the Galerkin setup's own product A S at hand, neither the residual nor
// the prolonged iterate has to exist as a vector:
//   restriction   b_c = S^T (b - A x) = S^T b - (A S)^T x,
//   prolongation  with e the coarse correction, x' = x + S e and the first
//                 post-smoothing step on it,
//                 d = c D^-1 (b - A x - (A S) e),  x'' = x + S e + d.
// A level so takes one launch to its coarse level and one back instead of two
// each (residual, restriction; prolongation, first step), the residual product
// with A (the longest rows of the level) is replaced by the shorter (A S)^T,
// and A and e are gathered once.  S has entries only where A S has (A_ii S_ik
// is a term of (A S)_ik), so both coefficients of a pair (i, k) are stored side
// by side in A S's layout: `m` holds A S and `s` the matching entries of S
// (zero where S has none); pairs that are zero in both are left out.
//
// Only FP32 cycles do this: in FP64 the pair rows cost as many FP64 instructions
// (1/64 of the FP32 rate) as the launches they save (129^2 step 35.7 -> 35.6 ms,
// 257^2 Hessian apply 4.41 -> 4.38 ms).
#include "internal.cuh"
#include "spmv.cuh"
#include "util.cuh"

// ------------------------------------------------------------------ setup
// entries of row i of A S that are kept, and S's entry for each
template <bool FILL>
__global__ void k_pair_rows(int rows, const int *__restrict__ rp, const int *__restrict__ ci,
                            const double *__restrict__ v, const int *__restrict__ srp, const int *__restrict__ sci,
                            const double *__restrict__ sv, int *__restrict__ cnt, const int *__restrict__ orp,
                            int *__restrict__ oci, double *__restrict__ ov, double *__restrict__ os)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows) return;
    int q = FILL ? orp[i] : 0, j = srp[i];
    const int je = srp[i + 1];
    for (int k = rp[i]; k < rp[i + 1]; k++) {
        const int c = ci[k];
        while (j < je && sci[j] < c) j++;
        const bool in = j < je && sci[j] == c;
        if (!in && v[k] == 0.0) continue;
        if (FILL) {
            oci[q] = c;
            ov[q] = v[k];
            os[q] = in ? sv[j] : 0.0;
        }
        q++;
    }
    if (!FILL) cnt[i] = q;
}

// S^T's entry for every entry of (A S)^T, one warp per row (both rows sorted)
__global__ void k_pair_lookup(int rows, const int *__restrict__ rp, const int *__restrict__ ci,
                              const int *__restrict__ srp, const int *__restrict__ sci,
                              const double *__restrict__ sv, double *__restrict__ os)
{
    const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (i >= rows) return;
    for (int k = rp[i] + lane; k < rp[i + 1]; k += 32) {
        const int c = ci[k];
        int lo = srp[i], hi = srp[i + 1];
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (sci[mid] < c) lo = mid + 1;
            else hi = mid;
        }
        os[k] = lo < srp[i + 1] && sci[lo] == c ? sv[lo] : 0.0;
    }
}

// second values of a SELL-32 layout (padding zero, as k_sell_fill)
__global__ void k_pair_sell(int rows, const int *__restrict__ rp, const double *__restrict__ s,
                            const int *__restrict__ slp, float *__restrict__ out, int nslices)
{
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nslices * 32) return;
    const int base = slp[r >> 5], w = (slp[(r >> 5) + 1] - base) >> 5, lane = r & 31;
    const int beg = r < rows ? rp[r] : 0, len = r < rows ? rp[r + 1] - beg : 0;
    for (int k = 0; k < w; k++) out[base + 32 * k + lane] = k < len ? (float)s[beg + k] : 0.f;
}

static int pair_layout(amgh_problem *p, Arena &ar, PairMat &w, const double *s, int force_tpr)
{
    cudaStream_t st = p->stream;
    TRY(prepare_layout(ar, w.m, st, force_tpr));
    const int64_t n = w.m.tpr <= 1 ? w.m.sell_nnz : w.m.nnz;
    TRY(ar.alloc(&w.s, n));
    if (n == 0) return AMGH_OK;
    if (w.m.tpr > 1) return to_f32(p, s, n, w.s);
    k_pair_sell<<<ceil_div(w.m.nslices * 32, 256), 256, 0, st>>>(w.m.rows, w.m.rp, s, w.m.sl_ptr, w.s, w.m.nslices);
    LAUNCH_CHECK();
    return AMGH_OK;
}

// Levels whose V-cycle is bound by launches (1.3 us each, two of six a level
// saved) rather than by bytes, of which the pair rows have more than the rows
// they replace; and A S rows short enough that the transposed ones stay short:
// 5-11 entries in 2D, 8 on the finest level and 20-35 below it in 3D.
// Measured, without pairs -> up to 65,536 rows -> up to 262,144: 65^2 solve 16.4
// -> 14.7 -> 14.7 ms, refinement form on 513^2 6.27 -> 5.83 -> 5.70, 1025^2 step
// 149.0 -> 145.8 -> 146.7 (their setup); with 3D coarse levels too, 65^3 cost
// and gradient 4.54 -> 4.62 -> 5.20.
#define PAIR_MAX_ROWS 65536
#define PAIR_MAX_AVG 12
bool transfer_fits(const amgh_problem *p, int l)
{
    return p->aopts.precision != 0 && p->sl[l].A.rows <= PAIR_MAX_ROWS;
}

// Both pair matrices of a level from as = A S (canonical CSR, not kept), or
// neither where its rows are long.  The prolongation's rows are read by the lane
// groups that read A's.
int transfer_setup(amgh_problem *p, Arena &ar, StateLevel &S, const DevCsr &as)
{
    cudaStream_t st = p->stream;
    const int n = as.rows;
    Scratch sc;
    int *cnt = nullptr, *rp = nullptr;
    double *s = nullptr, *t = nullptr;
    DevCsr m;
    m.rows = n;
    m.cols = as.cols;
    TRY(sc.alloc(&cnt, n + 1));
    TRY(sc.alloc(&rp, n + 1));
    k_pair_rows<false><<<ceil_div(n, 256), 256, 0, st>>>(n, as.rp, as.ci, as.v, S.S.rp, S.S.ci, S.S.v, cnt, nullptr,
                                                         nullptr, nullptr, nullptr);
    LAUNCH_CHECK();
    TRY(exclusive_scan<int>(cnt, rp, n, st, &m.nnz));
    if (m.nnz > (int64_t)PAIR_MAX_AVG * n) return AMGH_OK;
    TRY(ar.alloc(&m.rp, n + 1));
    CU(cudaMemcpyAsync(m.rp, rp, sizeof(int) * (n + 1), cudaMemcpyDeviceToDevice, st));
    TRY(ar.alloc(&m.ci, m.nnz));
    TRY(ar.alloc(&m.v, m.nnz));
    TRY(sc.alloc(&s, m.nnz));
    k_pair_rows<true><<<ceil_div(n, 256), 256, 0, st>>>(n, as.rp, as.ci, as.v, S.S.rp, S.S.ci, S.S.v, nullptr, m.rp,
                                                        m.ci, m.v, s);
    LAUNCH_CHECK();
    S.up.m = m;
    TRY(csr_transpose(ar, m, S.down.m, st));
    TRY(sc.alloc(&t, m.nnz));
    k_pair_lookup<<<ceil_div((int64_t)S.down.m.rows * 32, 256), 256, 0, st>>>(S.down.m.rows, S.down.m.rp,
                                                                              S.down.m.ci, S.St.rp, S.St.ci, S.St.v, t);
    LAUNCH_CHECK();
    TRY(pair_layout(p, ar, S.up, s, S.A.tpr < 1 ? 1 : S.A.tpr));
    TRY(pair_layout(p, ar, S.down, t, 0));
    S.paired = true;
    return AMGH_OK;
}

// ------------------------------------------------------------------ kernels
// b_c = S^T b - (A S)^T x, with the coarse level's first smoother step from
// zero d_c = x_c = c0 D_c^-1 b_c where that level smooths (d not null)
template <typename T, int TPR>
__global__ void k_restrict_pair(MatView<T> W, const T *__restrict__ sv, const T *b, const T *x,
                                T *__restrict__ bc, const T *__restrict__ invd, T *__restrict__ d,
                                T *__restrict__ xc, T c0, const int *skip)
{
    int i = my_row<TPR>();
    bool lead = i < W.rows && row_leader<TPR>();
    RowPrePair<T> pre;
    T ir = 0;
    PDL_ENTER_LOADING(skip, (row_prefetch_pair<T, TPR>(W, sv, i, pre)); if (lead && d) ir = invd[i])
    T v = row_restrict_pair<T, TPR>(
        W, sv, i, pre, [&](int c) { return b[c]; }, [&](int c) { return x[c]; });
    if (lead) {
        bc[i] = v;
        if (d) {
            T z = cheb_first_point(v, ir, c0);
            d[i] = z;
            xc[i] = z;
        }
    }
}

// x_n = x + S e + d, d = c D^-1 (b - A x - (A S) e)
template <typename T, int TPR>
__global__ void k_prolong_pair(MatView<T> A, MatView<T> W, const T *__restrict__ sv, const T *__restrict__ invd,
                               const T *b, const T *x, const T *e, T *__restrict__ d, T *__restrict__ xn, T c,
                               const int *skip)
{
    int r = my_row<TPR>();
    bool lead = r < A.rows && row_leader<TPR>();
    RowPre<T> pa;
    RowPrePair<T> pw;
    T ir = 0;
    PDL_ENTER_LOADING(skip, (row_prefetch<T, TPR>(A, r, pa)); (row_prefetch_pair<T, TPR>(W, sv, r, pw));
                      if (lead) ir = invd[r])
    T br = 0, xr = 0;
    if (lead) {
        br = b[r];
        xr = x[r];
    }
    T ax = row_sum_pre<T, TPR>(A, r, pa, [&](int j) { return x[j]; });
    T ase, se;
    row_prolong_pair<T, TPR>(W, sv, r, pw, [&](int j) { return e[j]; }, ase, se);
    if (lead) {
        T dn, xv;
        prolong_point(br, ax, ase, se, ir, xr, c, dn, xv);
        d[r] = dn;
        xn[r] = xv;
    }
}

int restrict_pair(amgh_problem *p, const StateLevel &S, const float *b, const float *x, float *bc,
                  const float *invd_c, float *d_c, float *x_c, double c0, const int *skip)
{
    const DevCsr &m = S.down.m;
    if (m.rows == 0) return AMGH_OK;
    MatView<float> W = view<float>(m);
    const int cls = m.cols == p->m ? KC_RESTRICT0 : KC_RESTRICT;
    timer_begin(p, cls);
    LAUNCH_TPR(k_restrict_pair, float, W.tpr, W.rows, p->stream, W, (const float *)S.down.s, b, x, bc, invd_c, d_c,
               x_c, (float)c0, skip);
    LAUNCH_CHECK();
    // both coefficients of a pair, b and x gathered; the coarse level's D^-1, d and x
    timer_end(p, cls, spmv_bytes(m, 4) + 4.0 * ((double)m.nnz + m.cols + (d_c ? 3.0 * m.rows : 0.0)));
    return AMGH_OK;
}

int prolong_pair(amgh_problem *p, const StateLevel &S, const float *b, const float *x, const float *e, float *d,
                 float *xn, double c, const int *skip)
{
    const DevCsr &m = S.up.m;
    if (m.rows == 0) return AMGH_OK;
    MatView<float> A = view<float>(S.A), W = view<float>(m);
    const int cls = m.rows == p->m ? KC_PROLONG0 : KC_PROLONG;
    timer_begin(p, cls);
    LAUNCH_TPR(k_prolong_pair, float, A.tpr, A.rows, p->stream, A, W, (const float *)S.up.s,
               (const float *)S.invd32, b, x, e, d, xn, (float)c, skip);
    LAUNCH_CHECK();
    // A x, both coefficients of a pair with e gathered, b and D^-1 read, d and x_n written
    timer_end(p, cls, spmv_bytes(S.A, 4) + spmv_bytes(m, 4) + 4.0 * ((double)m.nnz + 2.0 * m.rows));
    return AMGH_OK;
}
