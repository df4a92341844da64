// common.cuh -- shared device types, copies and reductions of the propagator,
// EPD and force passes of the hybrid LB/EPD step (arXiv:1804.02883).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

namespace epdlb {

// ---------------------------------------------------------------------------
// complex pairs
// ---------------------------------------------------------------------------
template <typename T> struct V2Of;
template <> struct V2Of<float> { using type = float2; };
template <> struct V2Of<double> { using type = double2; };
template <typename T> using V2 = typename V2Of<T>::type;

template <typename T> __host__ __device__ __forceinline__ V2<T> mk(T x, T y) { V2<T> r; r.x = x; r.y = y; return r; }
template <typename V> __device__ __forceinline__ V cadd(V a, V b) { a.x += b.x; a.y += b.y; return a; }
template <typename V> __device__ __forceinline__ V csub(V a, V b) { a.x -= b.x; a.y -= b.y; return a; }
template <typename V> __device__ __forceinline__ V cmul(V a, V b)
{
    V r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}
template <typename V, typename S> __device__ __forceinline__ V cscale(V a, S s) { a.x *= s; a.y *= s; return a; }

// Quotient of 0 <= n < 2^24 by a positive d through the float reciprocal,
// corrected to the exact integer quotient (a runtime integer division costs
// tens of instructions; this one a handful).
struct FastDiv {
    int d;
    float inv;
    __device__ __forceinline__ explicit FastDiv(int d_) : d(d_), inv(1.0f / (float)d_) {}
    __device__ __forceinline__ int div(int n) const
    {
        int q = __float2int_rz((float)n * inv);
        if ((q + 1) * d <= n) ++q;
        if (q * d > n) --q;
        return q;
    }
};

// 8-byte asynchronous copy global -> shared (the thread's own staging
// slot), and the commit / wait of the thread's copy groups
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
// 16-byte asynchronous copy global -> shared, not cached in L1
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Block-wide sum of one double per thread (blockDim.x a multiple of 32, at
// most 1024).  Fixed order: deterministic.  Result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double *scratch32)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) scratch32[warp] = v;
    __syncthreads();
    double r = 0.0;
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        r = lane < nw ? scratch32[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    }
    return r;
}

// Sum of cnt partial sums, identical in every block that calls it (the
// warp-0 lanes take fixed strided slices).  Result valid in thread 0 of warp 0
// and broadcast through the returned value of every thread after the call.
__device__ __forceinline__ double sum_partials(const double *part, int cnt, int stride_el, double *bcast)
{
    if (threadIdx.x < 32) {
        double v = 0.0;
        for (int i = threadIdx.x; i < cnt; i += 32) v += part[(size_t)i * stride_el];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (threadIdx.x == 0) *bcast = v;
    }
    __syncthreads();
    double r = *bcast;
    __syncthreads();
    return r;
}

__host__ __device__ __forceinline__ int ilog2(int v)
{
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

// Signed index of FFT bin m on an axis of n points.
__device__ __forceinline__ int signed_bin(int m, int n) { return m <= (n >> 1) ? m : m - n; }

constexpr int kThreads = 256;

} // namespace epdlb
