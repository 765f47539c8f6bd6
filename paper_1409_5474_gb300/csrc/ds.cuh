// Double-single arithmetic of the pair kernels (force.cu) and the fused
// block-step kernel (persist.cu).
#pragma once

#include <cuda_runtime.h>

namespace nb {

// ---------------------------------------------------------------------------
// Double-single accumulation (Knuth/Moller TwoSum + fast renormalisation).
// ---------------------------------------------------------------------------

__device__ __forceinline__ void ds_add(float &hi, float &lo, float x)
{
    const float s = hi + x;
    const float bb = s - hi;
    const float e = (hi - (s - bb)) + (x - bb);
    const float t = lo + e;
    hi = s + t;
    lo = t - (hi - s);
}

// A double-single value hi + lo (two FP32 numbers). On GB300 a warp-wide FP64
// instruction holds an SMSP's FP64 pipe for ~64 cycles, so partial sums are
// combined in double-single FP32 arithmetic and only final results are FP64.
struct dsf {
    float hi, lo;
};

// a += b for double-single values (TwoSum of the high parts, low parts added,
// renormalised).
__device__ __forceinline__ void ds_acc(dsf &a, dsf b)
{
    const float s = a.hi + b.hi;
    const float bb = s - a.hi;
    float e = (a.hi - (s - bb)) + (b.hi - bb);
    e += a.lo + b.lo;
    a.hi = s + e;
    a.lo = e - (a.hi - s);
}

__device__ __forceinline__ dsf ds_shfl_xor(dsf a, int o)
{
    return dsf{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

__device__ __forceinline__ void sum_into(dsf &a, dsf b) { ds_acc(a, b); }
__device__ __forceinline__ void sum_into(float &a, float b) { a += b; }
__device__ __forceinline__ void sum_into(double &a, double b) { a += b; }
__device__ __forceinline__ dsf lane_xor(dsf a, int o) { return ds_shfl_xor(a, o); }
__device__ __forceinline__ double lane_xor(double a, int o)
{
    return __shfl_xor_sync(0xffffffffu, a, o);
}
__device__ __forceinline__ float lane_xor(float a, int o)
{
    return __shfl_xor_sync(0xffffffffu, a, o);
}

// The sums of P (a power of two, at most 32) values over the warp's lanes: lane l returns the
// sum of value l % P. A butterfly over every value costs 5 P exchanges and sums; here
// the lanes halve the values they hold with every exchange (P / 2 + P / 4 + ... + 1, then
// one each up to 32 lanes), and the exchange distances 16, 8, ... of P = 32 add in the
// butterfly's order, to the same bits. 28 double-single values: 31 sums for 140.
template <int P, class T>
__device__ __forceinline__ T warp_scatter_sum(T (&v)[P])
{
    static_assert(P >= 1 && P <= 32 && (P & (P - 1)) == 0, "a power of two");
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = P / 2; h >= 1; h >>= 1) {
        const bool up = (lane & h) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            T keep = up ? v[i + h] : v[i];
            const T send = up ? v[i] : v[i + h];
            sum_into(keep, lane_xor(send, h));
            v[i] = keep;
        }
    }
#pragma unroll
    for (int o = P; o < 32; o <<= 1) sum_into(v[0], lane_xor(v[0], o));
    return v[0];
}

__device__ __forceinline__ double ds_to_double(dsf a) { return (double)a.hi + (double)a.lo; }

}  // namespace nb
