// The FP32 pair term of two j-particles at a time, shared by the kernels that
// read their j-records as j-pairs (force.cu, persist.cu).
//
// Blackwell's packed FP32x2 instructions do two IEEE operations per lane at the
// scalar rate per operation in half the issue slots. A j-pair holds the values of
// records 2q and 2q + 1 side by side in six float4; every lane keeps its
// i-particle, negated, in both halves, so each instruction computes the same
// term for two j.
#pragma once

#include <cuda_runtime.h>

#include "ds.cuh"
#include "nb_internal.cuh"

namespace nb {

// 1 / sqrt(x) on the SFU. SOFT promises x >= FLT_MIN, a normal number: then the instruction
// rsqrt.approx.ftz.f32 gives rsqrtf's bits (tests/test_gpu_soft_pairs.py) in fewer
// instructions (N = 262144, with the totals in shared memory: 76.3 -> 67.8 ms).
template <bool SOFT>
__device__ __forceinline__ float rsqrt_pair(float x)
{
    if (!SOFT) return rsqrtf(x);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Whether every |r|^2 + eps^2 is a normal FP32 number whatever r is (rounding is
// monotone, so the sum is at least eps2f).
__host__ __device__ __forceinline__ bool soft_pairs(float eps2f)
{
    return eps2f >= 1.17549435e-38f;
}

// An i-particle, negated, in both halves.
struct IPair {
    float2 xh, yh, zh, xl, yl, zl, vx, vy, vz;
};

__device__ __forceinline__ IPair ipair_of(const float4 &a, const float4 &b, const float4 &c)
{
    IPair r;
    r.xh = make_float2(-a.x, -a.x);
    r.yh = make_float2(-a.y, -a.y);
    r.zh = make_float2(-a.z, -a.z);
    r.xl = make_float2(-b.x, -b.x);
    r.yl = make_float2(-b.y, -b.y);
    r.zl = make_float2(-b.z, -b.z);
    r.vx = make_float2(-c.x, -c.x);
    r.vy = make_float2(-c.y, -c.y);
    r.vz = make_float2(-c.z, -c.z);
    return r;
}

// FP32 sums of an i-particle, one per half: acc, the jerk's m v / s^3 and
// m (r.v) r / s^5 parts, and the positive potential.
struct PairSum {
    float2 a[3], ja[3], jb[3], p;
};

__device__ __forceinline__ void pair_zero(PairSum &t)
{
#pragma unroll
    for (int c = 0; c < 3; ++c) t.a[c] = t.ja[c] = t.jb[c] = make_float2(0.f, 0.f);
    t.p = make_float2(0.f, 0.f);
}

// One j-pair: {x_hi y_hi} {z_hi m} {x_lo y_lo} {z_lo -} {vx vy} {vz -}, each value
// twice (records 2q, 2q + 1).
struct JPair {
    float4 q0, q1, q2, q3, q4, q5;
};

template <bool DS>
__device__ __forceinline__ JPair jpair_load(const float4 *P)
{
    JPair j;
    j.q0 = P[0];
    j.q1 = P[1];
    if (DS) {
        j.q2 = P[2];
        j.q3 = P[3];
    }
    j.q4 = P[4];
    j.q5 = P[5];
    return j;
}

__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }

// Add the pair terms of j on i to t. mask(rinv) may zero halves (self pair, ragged end).
template <bool DS, bool SOFT, class Mask>
__device__ __forceinline__ void pair_add(const JPair &j, const IPair &i, float2 e2, PairSum &t,
                                         Mask mask)
{
    float2 dx, dy, dz;
    if (DS) {
        dx = __fadd2_rn(__fadd2_rn(lo2(j.q0), i.xh), __fadd2_rn(lo2(j.q2), i.xl));
        dy = __fadd2_rn(__fadd2_rn(hi2(j.q0), i.yh), __fadd2_rn(hi2(j.q2), i.yl));
        dz = __fadd2_rn(__fadd2_rn(lo2(j.q1), i.zh), __fadd2_rn(lo2(j.q3), i.zl));
    } else {
        dx = __fadd2_rn(lo2(j.q0), i.xh);
        dy = __fadd2_rn(hi2(j.q0), i.yh);
        dz = __fadd2_rn(lo2(j.q1), i.zh);
    }
    const float2 dvx = __fadd2_rn(lo2(j.q4), i.vx);
    const float2 dvy = __fadd2_rn(hi2(j.q4), i.vy);
    const float2 dvz = __fadd2_rn(lo2(j.q5), i.vz);
    float2 r2 = __ffma2_rn(dx, dx, e2);
    r2 = __ffma2_rn(dy, dy, r2);
    r2 = __ffma2_rn(dz, dz, r2);
    float2 rv = __fmul2_rn(dx, dvx);
    rv = __ffma2_rn(dy, dvy, rv);
    rv = __ffma2_rn(dz, dvz, rv);
    float2 rinv = make_float2(rsqrt_pair<SOFT>(r2.x), rsqrt_pair<SOFT>(r2.y));
    mask(rinv);
    const float2 rinv2 = __fmul2_rn(rinv, rinv);
    const float2 mrinv = __fmul2_rn(hi2(j.q1), rinv);
    const float2 mr3 = __fmul2_rn(mrinv, rinv2);
    const float2 beta = __fmul2_rn(__fmul2_rn(mr3, rinv2), rv);
    t.p = __fadd2_rn(t.p, mrinv);
    t.a[0] = __ffma2_rn(mr3, dx, t.a[0]);
    t.a[1] = __ffma2_rn(mr3, dy, t.a[1]);
    t.a[2] = __ffma2_rn(mr3, dz, t.a[2]);
    t.ja[0] = __ffma2_rn(mr3, dvx, t.ja[0]);
    t.ja[1] = __ffma2_rn(mr3, dvy, t.ja[1]);
    t.ja[2] = __ffma2_rn(mr3, dvz, t.ja[2]);
    t.jb[0] = __ffma2_rn(beta, dx, t.jb[0]);
    t.jb[1] = __ffma2_rn(beta, dy, t.jb[1]);
    t.jb[2] = __ffma2_rn(beta, dz, t.jb[2]);
}

struct NoMask {
    __device__ __forceinline__ void operator()(float2 &) const {}
};

// The self pair and records past the end of a ragged tile contribute nothing: records
// ja and ja + 1 of the j-set, the i-particle's own index, the end of the tile.
struct PairMask {
    int ja, own, end;
    __device__ __forceinline__ void operator()(float2 &rinv) const
    {
        rinv.x = (ja == own || ja >= end) ? 0.f : rinv.x;
        rinv.y = (ja + 1 == own || ja + 1 >= end) ? 0.f : rinv.y;
    }
};

// The self pair alone (a pair with both records).
struct OwnMask {
    int ja, own;
    __device__ __forceinline__ void operator()(float2 &rinv) const
    {
        rinv.x = ja == own ? 0.f : rinv.x;
        rinv.y = ja + 1 == own ? 0.f : rinv.y;
    }
};

// Rewrite cnt records (of a tile of JT) at T as j-pairs at s_pair, by NT threads;
// records past the end become zeros (their pairs are masked).
template <int JT, int NT>
__device__ __forceinline__ void tile_to_pairs(const float4 *T, int cnt, float4 *s_pair, int tid)
{
    constexpr int NPAIR = JT / 2;
    auto put = [&](int x, bool full) {
        const int q = x % NPAIR, part = x / NPAIR;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 u = full || 2 * q < cnt ? T[DS_REC * (2 * q) + part] : zero;
        const float4 v = full || 2 * q + 1 < cnt ? T[DS_REC * (2 * q + 1) + part] : zero;
        float4 *P = s_pair + 6 * q + 2 * part;
        P[0] = make_float4(u.x, v.x, u.y, v.y);
        P[1] = make_float4(u.z, v.z, u.w, v.w);
    };
    if (cnt == JT) {
        for (int x = tid; x < DS_REC * NPAIR; x += NT) put(x, true);
    } else {
        for (int x = tid; x < DS_REC * NPAIR; x += NT) put(x, false);
    }
}

// The pair terms of the j-pairs q0, q0 + step, ... of a tile (first record jbase, cnt
// records) on IPT i-particles; own: their indices. masked: the tile is ragged or
// holds one of the warp's own particles.
template <bool DS, int IPT, int JT, bool SOFT>
__device__ __forceinline__ void tile_pairs(const float4 *s_pair, int q0, int step, int jbase,
                                           int cnt, bool masked, const IPair (&ip)[IPT],
                                           const int (&own)[IPT], float2 e2, PairSum (&ts)[IPT])
{
    if (masked) {
        const int npair = (cnt + 1) / 2;
#pragma unroll 2
        for (int q = q0; q < npair; q += step) {
            const JPair j = jpair_load<DS>(s_pair + 6 * q);
#pragma unroll
            for (int p = 0; p < IPT; ++p)
                pair_add<DS, SOFT>(j, ip[p], e2, ts[p],
                                   PairMask{jbase + 2 * q, own[p], jbase + cnt});
        }
    } else {
#pragma unroll 4
        for (int q = q0; q < JT / 2; q += step) {
            const JPair j = jpair_load<DS>(s_pair + 6 * q);
#pragma unroll
            for (int p = 0; p < IPT; ++p) pair_add<DS, SOFT>(j, ip[p], e2, ts[p], NoMask{});
        }
    }
}

// The sums of component c (0-2 acc, 3-5 jerk, 6 the positive potential) over both halves.
__device__ __forceinline__ float pair_total(const PairSum &t, int c)
{
    if (c < 3) return t.a[c].x + t.a[c].y;
    if (c < 6)
        return fmaf(-3.f, t.jb[c - 3].x + t.jb[c - 3].y, t.ja[c - 3].x + t.ja[c - 3].y);
    return t.p.x + t.p.y;
}

}  // namespace nb
