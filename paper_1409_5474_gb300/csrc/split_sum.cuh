// K3, the sums of j-split partials, shared by the 4th- and 6th-order force paths.
#pragma once

#include <cuda_runtime.h>

#include "ds.cuh"

namespace nb {

// A partial is a double-single float2, or a double.
__device__ __forceinline__ dsf split_value(float2 x) { return dsf{x.x, x.y}; }
__device__ __forceinline__ double split_value(double x) { return x; }
__device__ __forceinline__ double split_total(dsf x) { return ds_to_double(x); }
__device__ __forceinline__ double split_total(double x) { return x; }

// Outputs up to which a split reduction takes eight threads per output: above, one
// thread per output gives every SM more than two CTAs.
constexpr long long SPLIT_WIDE_OUTS = 1 << 17;

// The sum of the nsplit partials p[0], p[stride], ... of a thread's output in a fixed order.
// A CTA of 256 threads is 256 / G consecutive outputs (their partials are adjacent, so the
// loads of a warp are coalesced) times G groups of splits: group g adds the splits g, g + G,
// ..., eight at a time, all eight loads in flight and added in pairs (FP64: 114 splits one
// after the other doubled the rounding error of small i-sets), and the groups are added in
// order through shared memory. G = 1 where the outputs alone fill the GPU; with G = 8 a small
// due set's many splits cost one or two round trips to L2 and not nsplit / 8 of them (64
// slots, 152 splits at N = 65536: force and reduction 27.0 -> 18.8 us, 14.3 as a dependent
// launch). Every thread of the CTA calls this; the total is in group 0's threads (true).
template <class T, int G>
__device__ __forceinline__ bool split_sum(const T *p, size_t stride, int nsplit, bool valid,
                                          double &total)
{
    using V = decltype(split_value(T{}));
    constexpr int NQ = 256 / G;
    __shared__ V s_sum[G > 1 ? G - 1 : 1][NQ];
    const int o = threadIdx.x % NQ, g = threadIdx.x / NQ;
    V sum{};
    if (valid)
        for (int sp = g; sp < nsplit; sp += 8 * G) {
            V x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                x[u] = split_value(sp + u * G < nsplit ? __ldcg(p + (size_t)(sp + u * G) * stride)
                                                       : T{});
#pragma unroll
            for (int h = 1; h < 8; h <<= 1)
#pragma unroll
                for (int u = 0; u < 8; u += 2 * h) sum_into(x[u], x[u + h]);
            sum_into(sum, x[0]);
        }
    if (G > 1) {
        if (g > 0) s_sum[g - 1][o] = sum;
        __syncthreads();
        if (g > 0) return false;
#pragma unroll
        for (int u = 1; u < G; ++u) sum_into(sum, s_sum[u - 1][o]);
    }
    total = split_total(sum);
    return valid;
}

}  // namespace nb
