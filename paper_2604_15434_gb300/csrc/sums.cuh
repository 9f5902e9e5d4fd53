// sums.cuh -- sums over a whole field (included by mg.cu).
#pragma once

#include "internal.cuh"

namespace pmeft {

// The sum of four values, or of the one FP64 value that is loaded at a time.
__device__ __forceinline__ float vec_sum(const float (&e)[4]) { return (e[0] + e[1]) + (e[2] + e[3]); }
__device__ __forceinline__ double vec_sum(const double (&e)[1]) { return e[0]; }

// Sum of x, four loads in flight per thread: FP32 data (the library's own buffers) by 16-byte loads, FP64
// data (the caller's density among it) by aligned 8-byte loads.  The sixteen FP32 values of a step are
// added pairwise, four additions deep, and everything beyond that is FP64, so that the sum's error does
// not grow with the field (an FP32 accumulator per thread took 221 additions one after the other at 512^3,
// 1800 at 1024^3): one conversion and one FP64 addition per sixteen values, which HBM hides.
template <typename T>
__global__ void __launch_bounds__(256) k_sum(const T* __restrict__ x, size_t total, double* __restrict__ partials,
                                             double* __restrict__ fin_out)
{
    constexpr int W = sizeof(T) == 4 ? 4 : 1;
    struct alignas(W * sizeof(T)) Vec {
        T e[W];
    };
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    const size_t nv = total / W;  // total is a multiple of 512
    const Vec* xv = reinterpret_cast<const Vec*>(x);
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    size_t c = tid;
    for (; c + 3 * stride < nv; c += 4 * stride) {
        Vec q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k] = xv[c + k * stride];
        if constexpr (W == 4) {
            a[0] += (double)((vec_sum(q[0].e) + vec_sum(q[1].e)) + (vec_sum(q[2].e) + vec_sum(q[3].e)));
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) a[k] += vec_sum(q[k].e);
        }
    }
    for (; c < nv; c += stride) a[0] += (double)vec_sum(xv[c].e);
    const double v[1] = {(a[0] + a[1]) + (a[2] + a[3])};
    block_sums<1>(v, partials, fin_out, (double)total);
}

// sum of (x - mean)^2 with the mean read from the device (sums[1], as k_sum leaves it)
__global__ void __launch_bounds__(256) k_sum_centred(const double* __restrict__ x, size_t total,
                                                     const double* __restrict__ sums, double* __restrict__ partials,
                                                     double* __restrict__ fin_out)
{
    const double mean = sums[1];
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; c + 3 * stride < total; c += 4 * stride) {
        double q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k] = x[c + k * stride];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double d = q[k] - mean;
            a[k] += d * d;
        }
    }
    for (; c < total; c += stride) {
        const double d = x[c] - mean;
        a[0] += d * d;
    }
    const double v[1] = {(a[0] + a[1]) + (a[2] + a[3])};
    block_sums<1>(v, partials, fin_out, 1.0);
}

}  // namespace pmeft
