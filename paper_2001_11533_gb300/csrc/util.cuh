// util.cuh -- device helpers: fixed-order warp/block reductions, scans.
#pragma once

#include "internal.cuh"

template <typename T>
int exclusive_scan(const T *in, T *out, int64_t n, cudaStream_t s, T *total_host);

// Butterfly sum inside a warp: the same lanes combine in the same order on
// every run, so the result is deterministic.
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ int warp_max_int(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Sum over a block of blockDim.x (multiple of 32, <= 1024) threads; result
// valid in thread 0.  Fixed order: warp butterflies, then warp 0 sums the
// per-warp values.
__device__ __forceinline__ double block_sum(double v, double *sh32)
{
    v = warp_sum(v);
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh32[w] = v;
    __syncthreads();
    int nw = blockDim.x >> 5;
    double t = 0.0;
    if (w == 0) {
        t = l < nw ? sh32[l] : 0.0;
        t = warp_sum(t);
    }
    __syncthreads();
    return t;
}

// Last-block finalisation of a two-stage reduction with NV values per block.
// Returns true in the first warp of the block that finished last; `tot` then
// holds the fixed-order sums of all partials.  partials layout: [NV][gridDim.x].
template <int NV>
__device__ bool reduce_last_block(const double (&val)[NV], double *partials, unsigned *ticket,
                                  double (&tot)[NV])
{
    __shared__ double sh32[NV][32];
    __shared__ bool is_last;
    int nb = gridDim.x;
#pragma unroll
    for (int q = 0; q < NV; q++) {
        double v = warp_sum(val[q]);
        int w = threadIdx.x >> 5, l = threadIdx.x & 31;
        if (l == 0) sh32[q][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int nw = blockDim.x >> 5;
#pragma unroll
        for (int q = 0; q < NV; q++) {
            double t = (int)threadIdx.x < nw ? sh32[q][threadIdx.x] : 0.0;
            t = warp_sum(t);
            if (threadIdx.x == 0) partials[q * nb + blockIdx.x] = t;
        }
    }
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned t = atomicAdd(ticket, 1u);
        is_last = (t == (unsigned)nb - 1);
    }
    __syncthreads();
    if (!is_last) return false;
    __threadfence();
    // fixed-order sum of the nb partials: thread t sums t, t+B, ...; then tree
#pragma unroll
    for (int q = 0; q < NV; q++) {
        double s = 0.0;
        for (int b = threadIdx.x; b < nb; b += blockDim.x) s += ((volatile double *)partials)[q * nb + b];
        s = warp_sum(s);
        int w = threadIdx.x >> 5, l = threadIdx.x & 31;
        if (l == 0) sh32[q][w] = s;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int nw = blockDim.x >> 5;
#pragma unroll
        for (int q = 0; q < NV; q++) {
            double t = (int)threadIdx.x < nw ? sh32[q][threadIdx.x] : 0.0;
            tot[q] = warp_sum(t);
        }
    }
    if (threadIdx.x == 0) *ticket = 0u;
    return threadIdx.x < 32;
}

// Order of non-negative FP64 numbers by their bits: an FP64 comparison, like
// every FP64 instruction, holds its unit for ~65 cycles here.
__device__ __forceinline__ bool pos64(double x) // 0 < x <= infinity
{
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool finite64(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool le64(double x, double y) // x <= y, both >= 0
{
    return __double_as_longlong(x) <= __double_as_longlong(y);
}

// alpha and beta of the single-reduction CG (Chronopoulos & Gear) from
// g = (r, z), d = (z, A z) and, from the step before (k1 > 0), rz = g' and
// ra = g' alpha':
//   beta = g / g',  alpha = g / (d - beta g / alpha') = g ra / (d ra - g^2).
// Called by all lanes of a warp, lanes 2c and 2c + 1 with the scalars of loop c
// (the same for all lanes where there is one loop); both get the result.  An
// FP64 division takes ten dependent FP64 instructions, so the two divisions
// are made by two lanes of one instruction sequence (in the textbook order
// three divisions follow each other).  The products are formed on g and ra
// scaled by the power of two of g, so that no square over- or underflows where
// g itself does not.  Returns CG_RUNNING, or the status that ends the loop.
__device__ __forceinline__ int cg2_scalars(double g, double d, int k1, double rz, double ra, double &alpha,
                                           double &beta)
{
    double num = g, den = d;
    if (k1) {
        const int e = (__double2hiint(g) >> 20) & 0x7ff; // biased exponent
        const double s = __hiloint2double(min(max(2046 - e, 1), 2046) << 20, 0);
        const double gs = g * s, rs = ra * s;
        num = gs * rs;
        den = fma(d * s, rs, -(gs * gs));
    }
    const bool second = threadIdx.x & 1;
    const double quo = (second ? g : num) / (second ? rz : den);
    const double other = __shfl_xor_sync(0xffffffffu, quo, 1);
    alpha = second ? other : quo;
    beta = second ? quo : other;
    if (!k1) beta = 0.0;
    if (pos64(g) && pos64(d) && pos64(den)) return CG_RUNNING;
    return finite64(g) && finite64(d) && finite64(den) ? CG_INDEFINITE : CG_NUMERIC;
}
