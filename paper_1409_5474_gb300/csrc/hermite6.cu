// The 6th-order Hermite scheme on the GPU (Sect. II: direct-summation codes
// pair with integrators of 4th or higher order and individual time steps; the
// scheme is the two-point Hermite one of Nitadori & Makino's 6th-order paper,
// which the same passage cites).
//
// What differs from the 4th-order path: every pair also yields the snap, the
// second time derivative of its acceleration,
//   alpha = (r.v) / r2,   beta = (|v|^2 + r.a) / r2 + alpha^2,
//   A = m r / r2^(3/2),   J = m v / r2^(3/2) - 3 alpha A,
//   S = m a / r2^(3/2) - 6 alpha J - 3 beta A,
// with r, v, a the j-minus-i position, velocity and predicted acceleration and
// r2 = |r|^2 + eps^2. The FP32 kernels evaluate it expanded in r, v and a, so
// that every term is one FMA into its running sum: with q = m / r2^(3/2),
// a3 = -3 alpha and u3 = -3 (|v|^2 + r.a) / r2,
//   J = q v + (a3 q) r,   S = q a + (2 a3 q) v + ((5/3) a3^2 + u3) q r
// (57 FP32 operations per pair against 64 for the nested form). So the j-records carry the predicted acceleration (64
// bytes instead of 48), the prediction runs through the crackle term, and the
// corrector is the order-6 two-point quadrature with the crackle, pop and 5th
// derivative of the acceleration taken from the quintic through (a, jerk,
// snap) at both ends of the step; the step criterion uses the crackle only (see
// k_correct6).
//
// Kernels:
//   k_predict6           K1 for all particles (the block scheduler has its own
//                        order-6 instantiation in step.cu)
//   k_force6_tile32<DS, NWJ>
//                        K2, FP32 / double-single pairs: a CTA of 8 warps holds
//                        one i-particle per thread in 8/NWJ warp columns, NWJ
//                        warp rows share each j-tile; j-tiles of 128 records
//                        stream through a 3-stage ring of bulk copies (TMA
//                        engine, mbarrier completion, bounded waits); a
//                        tile is transposed into j-pairs and its pair terms run
//                        on packed FP32x2 arithmetic, two j per instruction;
//                        FP32 sums per tile are folded into double-single
//                        totals; grid.y splits the j-range
//   k_force6_tile64      K2, FP64 pairs (the correctness variant)
//   k_force6_sums        K3: the splits of each output added in fixed order
//   k_correct6           K4: corrector, end-of-step crackle, step criterion,
//                        block quantization
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "ds.cuh"
#include "nb_internal.cuh"
#include "pair.cuh"
#include "split_sum.cuh"
#include "step_body.cuh"
#include "tma.cuh"

namespace nb {

namespace {

constexpr int H6_VALS = 10;     // acc 3, jerk 3, snap 3, pot 1 per i-particle
constexpr int H6_JT = 128;      // j-records per FP32 fold, and per tile unless split coarsely
constexpr int H6_JT_BIG = 256;  // j-records per tile of long splits (plan6_jt)
constexpr int H6_NS = 3;        // ring stages
constexpr int H6_NWARP = 8;     // warps per FP32 CTA
constexpr int H6_T64 = 128;     // threads per FP64 CTA
constexpr int H6_JT64 = 128;    // j per FP64 shared tile
constexpr int CORRECT6_THREADS = 128;  // 4 warps x 10 slots (3 lanes per slot)
constexpr float F53 = 5.f / 3.f;        // S's r coefficient: (15 alpha^2 - 3 u) = 5/3 a3^2 + u3

// ---- K1 ----------------------------------------------------------------------

template <bool REC>
__global__ void k_predict6(StateDev s, double t, unsigned *err)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    cudaGridDependencySynchronize();
    if (t < s.t[i]) atomicOr(err, DERR_BACKWARD);
    predict6_one<REC>(s, i, t);
}

// Member index of slot k; an index outside [0, n) is flagged and replaced by 0.
__device__ __forceinline__ int member6(const int *idx, int k, int n, unsigned *err)
{
    const int r = idx ? idx[k] : k;
    if ((unsigned)r >= (unsigned)n) {
        atomicOr(err, DERR_BADINDEX);
        return 0;
    }
    return r;
}

// Store the 10 totals of slot k (v[9] is the positive potential sum P; pot = -P).
__device__ __forceinline__ void store6(const Out6 &out, int k, double v[H6_VALS], unsigned *err)
{
    v[9] = -v[9];
    bool ok = true;
#pragma unroll
    for (int c = 0; c < H6_VALS; ++c) ok = ok && isfinite(v[c]);
    if (!ok) atomicOr(err, DERR_NONFINITE);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (out.acc) out.acc[c * out.ld + k] = v[c];
        if (out.jerk) out.jerk[c * out.ld + k] = v[3 + c];
        if (out.snap) out.snap[c * out.ld + k] = v[6 + c];
    }
    if (out.pot) out.pot[k] = v[9];
}

// ---- K2, FP32 / double-single ---------------------------------------------------

// An i-particle, negated, in both halves; the FP32 sums of its ten outputs, one per half;
// a j-pair {x_hi y_hi} {z_hi m} {x_lo y_lo} {z_lo -} {vx vy} {vz -} {ax ay} {az -}.
struct IPair6 {
    IPair p;
    float2 ax, ay, az;
};

template <bool DS, bool SOFT, class Mask>
__device__ __forceinline__ void pair6_add(const float4 *Pp, const IPair6 &i, float2 e2,
                                          float2 (&t)[H6_VALS], Mask mask)
{
    const float4 q0 = Pp[0], q1 = Pp[1], q4 = Pp[4], q5 = Pp[5], q6 = Pp[6], q7 = Pp[7];
    float2 dx, dy, dz;
    if (DS) {
        const float4 q2 = Pp[2], q3 = Pp[3];
        dx = __fadd2_rn(__fadd2_rn(lo2(q0), i.p.xh), __fadd2_rn(lo2(q2), i.p.xl));
        dy = __fadd2_rn(__fadd2_rn(hi2(q0), i.p.yh), __fadd2_rn(hi2(q2), i.p.yl));
        dz = __fadd2_rn(__fadd2_rn(lo2(q1), i.p.zh), __fadd2_rn(lo2(q3), i.p.zl));
    } else {
        dx = __fadd2_rn(lo2(q0), i.p.xh);
        dy = __fadd2_rn(hi2(q0), i.p.yh);
        dz = __fadd2_rn(lo2(q1), i.p.zh);
    }
    const float2 dvx = __fadd2_rn(lo2(q4), i.p.vx);
    const float2 dvy = __fadd2_rn(hi2(q4), i.p.vy);
    const float2 dvz = __fadd2_rn(lo2(q5), i.p.vz);
    const float2 dax = __fadd2_rn(lo2(q6), i.ax);
    const float2 day = __fadd2_rn(hi2(q6), i.ay);
    const float2 daz = __fadd2_rn(lo2(q7), i.az);
    float2 r2 = __ffma2_rn(dx, dx, e2);
    r2 = __ffma2_rn(dy, dy, r2);
    r2 = __ffma2_rn(dz, dz, r2);
    float2 rv = __fmul2_rn(dx, dvx);
    rv = __ffma2_rn(dy, dvy, rv);
    rv = __ffma2_rn(dz, dvz, rv);
    float2 w2 = __fmul2_rn(dvx, dvx);  // |v|^2 + r.a
    w2 = __ffma2_rn(dvy, dvy, w2);
    w2 = __ffma2_rn(dvz, dvz, w2);
    w2 = __ffma2_rn(dx, dax, w2);
    w2 = __ffma2_rn(dy, day, w2);
    w2 = __ffma2_rn(dz, daz, w2);
    float2 rinv = make_float2(rsqrt_pair<SOFT>(r2.x), rsqrt_pair<SOFT>(r2.y));
    mask(rinv);
    const float2 rinv2 = __fmul2_rn(rinv, rinv);
    const float2 mrinv = __fmul2_rn(hi2(q1), rinv);
    const float2 mr3 = __fmul2_rn(mrinv, rinv2);
    const float2 r3 = __fmul2_rn(rinv2, make_float2(-3.f, -3.f));
    const float2 m3a = __fmul2_rn(rv, r3);  // -3 alpha
    const float2 m3u = __fmul2_rn(w2, r3);  // -3 (|v|^2 + r.a) / r^2
    const float2 k1 = __fmul2_rn(m3a, mr3);
    const float2 c1 = __fadd2_rn(k1, k1);
    const float2 c2 =
        __fmul2_rn(__ffma2_rn(m3a, __fmul2_rn(m3a, make_float2(F53, F53)), m3u), mr3);
    t[0] = __ffma2_rn(mr3, dx, t[0]);
    t[1] = __ffma2_rn(mr3, dy, t[1]);
    t[2] = __ffma2_rn(mr3, dz, t[2]);
    t[3] = __ffma2_rn(k1, dx, __ffma2_rn(mr3, dvx, t[3]));
    t[4] = __ffma2_rn(k1, dy, __ffma2_rn(mr3, dvy, t[4]));
    t[5] = __ffma2_rn(k1, dz, __ffma2_rn(mr3, dvz, t[5]));
    t[6] = __ffma2_rn(c2, dx, __ffma2_rn(c1, dvx, __ffma2_rn(mr3, dax, t[6])));
    t[7] = __ffma2_rn(c2, dy, __ffma2_rn(c1, dvy, __ffma2_rn(mr3, day, t[7])));
    t[8] = __ffma2_rn(c2, dz, __ffma2_rn(c1, dvz, __ffma2_rn(mr3, daz, t[8])));
    t[9] = __fadd2_rn(t[9], mrinv);
}

// The pair terms of the j-pairs q0, q0 + step, ... of H6_JT records (the first of them
// jbase, cnt in all) on one i-particle (index own).
template <bool DS, bool SOFT>
__device__ __forceinline__ void tile6_pairs(const float4 *pairs, int q0, int step, int jbase,
                                            int cnt, bool masked, const IPair6 &ip, int own,
                                            float2 e2, float2 (&t)[H6_VALS])
{
    if (masked) {
        const int npair = (cnt + 1) / 2;
#pragma unroll 2
        for (int q = q0; q < npair; q += step)
            pair6_add<DS, SOFT>(pairs + 2 * DS6_REC * q, ip, e2, t,
                                PairMask{jbase + 2 * q, own, jbase + cnt});
    } else {
#pragma unroll 4
        for (int q = q0; q < H6_JT / 2; q += step)
            pair6_add<DS, SOFT>(pairs + 2 * DS6_REC * q, ip, e2, t, NoMask{});
    }
}

// One i-particle per thread shares each j-record loaded from shared memory (a second one
// spills). The CTA's 8 warps are NWI warp columns (different i-particles) x NWJ warp rows
// (the same i-particles, sharing out each j-tile: row g takes pairs g, g + NWJ,
// ...), so that a small due set still spreads over the SM; rows are added in
// shared memory at the end, in fixed order. Two CTAs per SM (16 warps) hide the
// pair arithmetic's latencies better than one. A j-tile is rewritten once in
// shared memory as j-pairs (each float4 part of records 2q and 2q + 1 interleaved
// component by component), so that the pair terms of two j run on the packed
// FP32x2 instructions (half the issue slots of scalar FP32 at the same lane rate),
// with the i-particle's values duplicated in both lanes; tiles that are ragged or
// hold one of a warp's own particles mask halves. As in the 4th-order tile kernel the
// totals live in shared memory and softened pairs take the bare reciprocal square root:
// bound by the FP32 pipe (57 operations per interaction, 706 G/s). N = 20011, all i: 881 ->
// 789 us with the splits' sums, N = 65536: 8.68 -> 7.76 ms.
template <bool DS, int NWJ, int JT>
__global__ void __launch_bounds__(32 * H6_NWARP, 2)
    k_force6_tile32(const float4 *jrec, int nj, const int *idx, int n_i, float eps2f, int ntiles,
                    float2 *part, long long pld,
                    Out6 out, unsigned *err)
{
    // H6_NS ring stages of JT records, the current tile as j-pairs, the running totals
    extern __shared__ __align__(128) float4 s_tile6[];
    __shared__ __align__(8) uint64_t s_full[H6_NS];
    __shared__ int s_abort;

    constexpr int NT = 32 * H6_NWARP;
    constexpr int NWI = H6_NWARP / NWJ;
    constexpr int IB = 32 * NWI;
    constexpr int NPAIR = JT / 2;
    static_assert(NWI * NWJ == H6_NWARP, "warp grid");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wi = warp % NWI, wj = warp / NWI;
    const int nsplit = gridDim.y, split = blockIdx.y;
    const int tile0 = (int)((long long)ntiles * split / nsplit);
    const int tile1 = (int)((long long)ntiles * (split + 1) / nsplit);
    const int my_tiles = tile1 - tile0;
    float4 *s_pair = s_tile6 + (size_t)H6_NS * JT * DS6_REC;
    // running totals (double-single, or plain FP32 in .x), this thread's own column
    float2 *s_tot = reinterpret_cast<float2 *>(s_pair + (size_t)JT * DS6_REC) + tid;
#pragma unroll
    for (int c = 0; c < H6_VALS; ++c) s_tot[c * NT] = make_float2(0.f, 0.f);
    if (tid == 0) {
        s_abort = 0;
#pragma unroll
        for (int q = 0; q < H6_NS; ++q) mbar_init(&s_full[q], 1);
        fence_mbar_init();
    }
    cudaGridDependencySynchronize();  // nothing above reads what another launch wrote

    // this thread's i-particle (idle slots past n_i compute a copy of the last one)
    const int kk = blockIdx.x * IB + wi * 32 + lane;
    const bool idle = blockIdx.x * IB + wi * 32 >= n_i;  // no slot of this warp is written
    const int ii = member6(idx, min(kk, n_i - 1), nj, err);
    IPair6 ip;
    {
        const float4 *r = jrec + (size_t)DS6_REC * ii;
        const float4 d = r[3];
        ip.p = ipair_of(r[0], r[1], r[2]);
        ip.ax = make_float2(-d.x, -d.x);
        ip.ay = make_float2(-d.y, -d.y);
        ip.az = make_float2(-d.z, -d.z);
    }
    const float2 e2 = make_float2(eps2f, eps2f);
    const bool soft = soft_pairs(eps2f);
    __syncthreads();

    auto issue = [&](int kt) {
        const int stage = kt % H6_NS;
        const int tt = tile0 + kt;
        const int cnt = min(JT, nj - tt * JT);
        const uint32_t bytes = (uint32_t)cnt * DS6_REC * 16u;
        mbar_expect_tx(&s_full[stage], bytes);
        bulk_g2s(s_tile6 + (size_t)stage * JT * DS6_REC, jrec + (size_t)tt * JT * DS6_REC,
                 bytes, &s_full[stage]);
    };
    if (tid == 0)
        for (int kt = 0; kt < H6_NS && kt < my_tiles; ++kt) issue(kt);

    for (int kt = 0; kt < my_tiles; ++kt) {
        const int stage = kt % H6_NS;
        if (!mbar_wait(&s_full[stage], (uint32_t)((kt / H6_NS) & 1))) s_abort = 1;
        const float4 *T = s_tile6 + (size_t)stage * JT * DS6_REC;
        const int jbase = (tile0 + kt) * JT;
        const int cnt = min(JT, nj - jbase);
        const bool masked =
            __any_sync(0xffffffffu, ii >= jbase && ii < jbase + cnt) || cnt < JT;
        // the tile as j-pairs; records past the end become zeros (their pairs are masked)
        for (int x = tid; x < DS6_REC * NPAIR; x += NT) {
            const int q = x % NPAIR, part6 = x / NPAIR;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 u = 2 * q < cnt ? T[DS6_REC * (2 * q) + part6] : zero;
            const float4 v = 2 * q + 1 < cnt ? T[DS6_REC * (2 * q + 1) + part6] : zero;
            float4 *Pp = s_pair + 2 * DS6_REC * q + 2 * part6;
            Pp[0] = make_float4(u.x, v.x, u.y, v.y);
            Pp[1] = make_float4(u.z, v.z, u.w, v.w);
        }
        __syncthreads();
        // FP32 sums of every H6_JT records (at most 64 terms per half), folded into the totals
#pragma unroll 1
        for (int f = 0; f < cnt && !idle; f += H6_JT) {
            const float4 *pairs = s_pair + (size_t)DS6_REC * f;
            const int fcnt = min(H6_JT, cnt - f);
            float2 t[H6_VALS];
#pragma unroll
            for (int c = 0; c < H6_VALS; ++c) t[c] = make_float2(0.f, 0.f);
            if (soft)
                tile6_pairs<DS, true>(pairs, wj, NWJ, jbase + f, fcnt, masked, ip, ii, e2, t);
            else
                tile6_pairs<DS, false>(pairs, wj, NWJ, jbase + f, fcnt, masked, ip, ii, e2, t);
#pragma unroll
            for (int c = 0; c < H6_VALS; ++c) {
                float2 &h = s_tot[c * NT];
                float2 v = h;
                if (DS)
                    ds_add(v.x, v.y, t[c].x + t[c].y);
                else
                    v.x += t[c].x + t[c].y;
                h = v;
            }
        }

        __syncthreads();  // every warp is done with this stage and the pairs
        if (s_abort) {
            if (tid == 0) {
                drain_ring<H6_NS>(s_full, 0u, kt, my_tiles);
                atomicOr(err, DERR_TIMEOUT);
            }
            return;
        }
        if (tid == 0 && kt + H6_NS < my_tiles) issue(kt + H6_NS);
    }
    if (wj != 0 || kk >= n_i) return;
    // the warp rows' totals in order 0..NWJ-1 (columns 32 NWI threads apart)
    dsf v[H6_VALS];
#pragma unroll
    for (int c = 0; c < H6_VALS; ++c) {
        const float2 *h = s_tot + c * NT;
        v[c] = dsf{h[0].x, h[0].y};
#pragma unroll
        for (int g = 1; g < NWJ; ++g) ds_acc(v[c], dsf{h[32 * NWI * g].x, h[32 * NWI * g].y});
    }
    if (nsplit == 1) {
        double d[H6_VALS];
#pragma unroll
        for (int c = 0; c < H6_VALS; ++c) d[c] = ds_to_double(v[c]);
        store6(out, kk, d, err);
    } else {
#pragma unroll
        for (int c = 0; c < H6_VALS; ++c)
            part[((size_t)split * H6_VALS + c) * pld + kk] = make_float2(v[c].hi, v[c].lo);
    }
}

// ---- K2, FP64 ---------------------------------------------------------------

// One i-particle per thread; the j-set (predicted FP64 position, velocity,
// acceleration and mass: 80 bytes per particle) goes through shared memory in
// tiles of H6_JT64. grid.y splits the j-range.
__global__ void __launch_bounds__(H6_T64)
    k_force6_tile64(StateDev s, const int *__restrict__ idx, int n_i, double eps2,
                    double *__restrict__ part, long long pld, Out6 out, unsigned *err)
{
    __shared__ double sj[10][H6_JT64];
    const int nj = s.n;
    const int nsplit = gridDim.y, split = blockIdx.y;
    const int ntiles = (nj + H6_JT64 - 1) / H6_JT64;
    const int tile0 = (int)((long long)ntiles * split / nsplit);
    const int tile1 = (int)((long long)ntiles * (split + 1) / nsplit);
    const int k = min(blockIdx.x * H6_T64 + (int)threadIdx.x, n_i - 1);
    const int ii = member6(idx, k, nj, err);
    double xi[3], vi[3], ai[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        xi[c] = s.pos_p[c * s.ld + ii];
        vi[c] = s.vel_p[c * s.ld + ii];
        ai[c] = s.acc_p[c * s.ld + ii];
    }
    double acc[H6_VALS];
#pragma unroll
    for (int c = 0; c < H6_VALS; ++c) acc[c] = 0.0;
    for (int tt = tile0; tt < tile1; ++tt) {
        const int jbase = tt * H6_JT64;
        const int cnt = min(H6_JT64, nj - jbase);
        __syncthreads();
        for (int q = threadIdx.x; q < cnt; q += H6_T64) {
            const int j = jbase + q;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                sj[c][q] = s.pos_p[c * s.ld + j];
                sj[3 + c][q] = s.vel_p[c * s.ld + j];
                sj[6 + c][q] = s.acc_p[c * s.ld + j];
            }
            sj[9][q] = s.m[j];
        }
        __syncthreads();
        for (int q = 0; q < cnt; ++q) {
            if (jbase + q == ii) continue;
            const double dx = sj[0][q] - xi[0], dy = sj[1][q] - xi[1], dz = sj[2][q] - xi[2];
            const double dvx = sj[3][q] - vi[0], dvy = sj[4][q] - vi[1], dvz = sj[5][q] - vi[2];
            const double dax = sj[6][q] - ai[0], day = sj[7][q] - ai[1], daz = sj[8][q] - ai[2];
            const double r2 = eps2 + dx * dx + dy * dy + dz * dz;
            const double rinv = rsqrt(r2);
            const double rinv2 = rinv * rinv;
            const double mrinv = sj[9][q] * rinv;
            const double mr3 = mrinv * rinv2;
            const double alpha = (dx * dvx + dy * dvy + dz * dvz) * rinv2;
            const double beta =
                (dvx * dvx + dvy * dvy + dvz * dvz + dx * dax + dy * day + dz * daz) * rinv2 +
                alpha * alpha;
            const double A[3] = {mr3 * dx, mr3 * dy, mr3 * dz};
            const double dv[3] = {dvx, dvy, dvz}, da[3] = {dax, day, daz};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double J = mr3 * dv[c] - 3.0 * alpha * A[c];
                acc[c] += A[c];
                acc[3 + c] += J;
                acc[6 + c] += mr3 * da[c] - 6.0 * alpha * J - 3.0 * beta * A[c];
            }
            acc[9] += mrinv;
        }
    }
    const int kk = blockIdx.x * H6_T64 + threadIdx.x;
    if (kk >= n_i) return;
    if (nsplit == 1) {
        store6(out, kk, acc, err);
    } else {
#pragma unroll
        for (int c = 0; c < H6_VALS; ++c) part[((size_t)split * H6_VALS + c) * pld + kk] = acc[c];
    }
}

// ---- K3 --------------------------------------------------------------------------

// Output q = component c of slot k (split_sum).
template <class T, int G>
__global__ void __launch_bounds__(256)
    k_force6_sums(const T *part, long long pld, int nsplit, int n_i, Out6 out, unsigned *err)
{
    const long long q = (long long)blockIdx.x * (256 / G) + threadIdx.x % (256 / G);
    const int c = (int)(q / n_i), k = (int)(q % n_i);
    double v;
    cudaGridDependencySynchronize();
    if (!split_sum<T, G>(part + (size_t)c * pld + k, (size_t)H6_VALS * pld, nsplit,
                         q < (long long)H6_VALS * n_i, v))
        return;
    if (c == 9) {
        v = -v;
        if (out.pot) out.pot[k] = v;
    } else {
        double *dst = c < 3 ? out.acc : (c < 6 ? out.jerk : out.snap);
        if (dst) dst[(c % 3) * out.ld + k] = v;
    }
    if (!isfinite(v)) atomicOr(err, DERR_NONFINITE);
}

template <class T>
cudaError_t go_force6_sums(const double *part, int n_i, int nsplit, const Out6 &out, unsigned *err,
                           cudaStream_t st)
{
    const long long outs = (long long)H6_VALS * n_i;
    const T *p = reinterpret_cast<const T *>(part);
    if (nsplit > 8 && outs <= SPLIT_WIDE_OUTS)
        return launch_dependent(k_force6_sums<T, 8>, dim3((unsigned)((outs + 31) / 32)), 256, 0, st,
                                p, (long long)n_i, nsplit, n_i, out, err);
    return launch_dependent(k_force6_sums<T, 1>, dim3((unsigned)((outs + 255) / 256)), 256, 0, st, p,
                            (long long)n_i, nsplit, n_i, out, err);
}

// ---- K4 --------------------------------------------------------------------------

// Slot k: the order-6 corrector (correct6_lanes_pre) from the start-of-step state
// and the new a1, j1, s1 (f, slot-indexed).
__global__ void __launch_bounds__(CORRECT6_THREADS)
    k_correct6(StateDev s, const int *act, int na, double t_new, Out6 f,
               StepParams prm, SchedDev *sd, unsigned *err, unsigned long long *dtmin_hits)
{
    cudaGridDependencySynchronize();
    // three lanes per slot (component c = lane % 3 of slot lane / 3; lanes 30, 31
    // idle), so that the FP64 dependency chains of the three components run side by side
    const int lane = threadIdx.x & 31;
    const int warp_g = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int k = warp_g * 10 + lane / 3;
    const int c = lane % 3;
    const bool mine = lane < 30 && k < na;
    C6State q{};
    double a1 = 0.0, j1 = 0.0, s1 = 0.0;
    int i = 0;
    if (mine) {
        i = act ? act[k] : k;
        c6state_load(s, i, c, q);
        a1 = f.acc[c * f.ld + k];
        j1 = f.jerk[c * f.ld + k];
        s1 = f.snap[c * f.ld + k];
    }
    correct6_lanes_pre(s, i, k, c, lane - c, mine, t_new, q, a1, j1, s1, prm, sd, err,
                       dtmin_hits);
}

// Shared memory of the tile kernel: the ring, the transposed tile and the running totals
// (52 or 84 KB).
template <int JT>
constexpr size_t h6_smem()
{
    return (size_t)(H6_NS + 1) * JT * DS6_REC * sizeof(float4) +
           (size_t)32 * H6_NWARP * H6_VALS * sizeof(float2);
}

// Resident CTAs per SM of a FP32 / double-single variant (occupancy API, cached).
template <bool DS, int NWJ>
int occ6()
{
    static int v = -1;
    if (v < 0) {
        int b = 0;
        constexpr auto kern = k_force6_tile32<DS, NWJ, H6_JT>;
        constexpr size_t smem = h6_smem<H6_JT>();
        if (allow_smem<kern>(smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, 32 * H6_NWARP, smem) !=
                cudaSuccess) {
            cudaGetLastError();
            b = 1;
        }
        v = std::max(b, 1);
    }
    return v;
}

template <bool DS, int NWJ, int JT = H6_JT>
cudaError_t go_tile6(const StateDev &s, const int *idx, int n_i, float e2, int nsplit, float2 *part,
                     const Out6 &out, unsigned *err, cudaStream_t st)
{
    constexpr auto kern = k_force6_tile32<DS, NWJ, JT>;
    constexpr int ib = 32 * (H6_NWARP / NWJ);
    const cudaError_t e = allow_smem<kern>(h6_smem<JT>());
    if (e != cudaSuccess) return e;
    return launch_dependent(kern, dim3((n_i + ib - 1) / ib, nsplit), 32 * H6_NWARP, h6_smem<JT>(),
                            st, s.rec6, s.n, idx, n_i, e2, (s.n + JT - 1) / JT, part,
                            (long long)n_i, out, err);
}

// Tile depth: 256 records where one warp row takes splits of eight 128-record tiles or more
// (half the barriers: N = 65536, all i, 8.12 -> 7.69 ms), else 128 (finer splits: 520 of
// 2500 14.5 us against 23).
int plan6_jt(int nwj, int nsplit, int n_j)
{
    const long long ntiles = (n_j + H6_JT - 1) / H6_JT;
    return nwj == 1 && ntiles >= 8LL * nsplit ? H6_JT_BIG : H6_JT;
}

int occ6_of(bool ds, int nwj)
{
    switch (nwj) {
    case 8: return ds ? occ6<true, 8>() : occ6<false, 8>();
    case 4: return ds ? occ6<true, 4>() : occ6<false, 4>();
    case 2: return ds ? occ6<true, 2>() : occ6<false, 2>();
    default: return ds ? occ6<true, 1>() : occ6<false, 1>();
    }
}

}  // namespace

// ---- host side ---------------------------------------------------------------------

cudaError_t launch_predict6(const StateDev &s, double t, bool want_rec, unsigned *err,
                            cudaStream_t st)
{
    if (s.n <= 0) return cudaSuccess;
    const int bs = 256, g = (s.n + bs - 1) / bs;
    return launch_dependent(want_rec ? k_predict6<true> : k_predict6<false>, dim3(g), bs, 0, st, s, t,
                            err);
}


// The warp rows of sets of 257 to 511 i-particles: of the shapes (and split counts just within
// one to eight waves of two CTAs an SM, four j-tiles a split at least) the one of least waves x
// (pairs of a CTA + 16384). A row of eight sums 8 FP32 terms a half between folds, one of four
// 16, a single one 64, so the rows carry accuracy: this rule laid these sets out before the
// cost model did, and with the model's rows the median jerk error for 498 of 65536 was 2.08e-7
// and not 1.74e-7 (64 bits; Plummer sphere with a mass spectrum). The smaller and larger sets' rows
// are as many as before, or more. 498 of 65536 74.8 -> 107 us (before the model 112), 300 of
// 2500 7.6 -> 9.2 (18.8).
int few_waves_rows(int n_i, int n_j, long long sms)
{
    const long long ntiles = (n_j + H6_JT - 1) / H6_JT;
    const long long cap = std::max(1LL, std::min(ntiles / 4, 1024LL)), slots = 2 * sms;
    int rows = 1;
    long long best = -1;
    for (int nwj = 1; nwj <= 8; nwj *= 2) {
        const long long ib = 32LL * (H6_NWARP / nwj), nblk = (n_i + ib - 1) / ib;
        for (int k = 0; k <= 9; ++k) {
            const long long ns =
                k == 0 ? 1 : (k == 9 ? cap : std::max(1LL, std::min(cap, k * slots / nblk)));
            const long long jpc = (ntiles + ns - 1) / ns * H6_JT;
            const long long t = (nblk * ns + slots - 1) / slots * (ib * jpc + 16384);
            if (best < 0 || t < best) {
                best = t;
                rows = nwj;
            }
        }
    }
    return rows;
}

// FP32 kinds: the warp rows (8, 4, 2 or 1: 32, 64, 128 or 256 i-particles per CTA) and
// j-splits of least estimated time, as the 4th-order plan: an SM's count of CTAs (at most
// ceil(CTAs / SMs)) times the tiles of a split times the SM's time for a tile of that shape,
// a little more where a CTA is left alone at the end; the splits' partials cost their traffic.
// Only split counts that fill a whole number of CTAs per SM are tried. Within 5% of the best
// of a sweep at N = 2500 to 65536, mostly. Against the rule before it (shape by size, two
// waves) and with the kernel as it was: 130 of 65536 51.5 -> 40 us, 520 127 -> 101, 1531 242
// -> 207; 300 of 2500 18.8 -> 8.1.
// Sets of 257 to 511 keep the rows of few_waves_rows.
// FP64: at least two waves of resident CTAs, then the fewest splits, up to eight times that
// many, whose last wave is at least 97% full, else the fullest.
ForcePlan plan_force6(int variant, int n_i, int n_j, int num_sms, size_t max_part)
{
    ForcePlan p{};
    // the most splits whose partials (H6_VALS doubles an i-particle each) fit
    const long long fit = std::max<long long>(
        1, (long long)std::min<size_t>(max_part / (H6_VALS * (size_t)n_i), 1 << 20));
    p.kind = 0;
    p.nwj = 1;
    p.ipt = 1;  // the packed pair terms already give each thread two j per step
    const long long sms = std::max(num_sms, 1);
    if (variant != NB_F64) {
        const long long ntiles = (n_j + H6_JT - 1) / H6_JT;
        double best = 1e300;
        const int few = n_i > 256 && n_i < 512 ? few_waves_rows(n_i, n_j, sms) : 0;
        for (int nwj = few ? few : 8; nwj >= (few ? few : 1); nwj /= 2) {
            const long long ib = 32LL * (H6_NWARP / nwj);
            const long long nblk = (n_i + ib - 1) / ib;
            // microseconds of an SM per 128-record tile
            const double t_tile = nwj == 8 ? 1.55 : (nwj == 4 ? 2.6 : (nwj == 2 ? 4.7 : 8.7));
            long long last = 0;
            for (const int per_sm : {1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 14, 16, 20, 24, 32, 40, 48}) {
                long long ns = std::max(1LL, std::min({per_sm * sms / nblk, ntiles, 512LL}));
                if (!splits_fit(fit, last, ns)) continue;
                const long long on_sm = (nblk * ns + sms - 1) / sms;
                const bool big = plan6_jt(nwj, (int)ns, n_j) == H6_JT_BIG;
                const long long tiles =
                    big ? 2 * (((ntiles + 1) / 2 + ns - 1) / ns) : (ntiles + ns - 1) / ns;
                const double alone = on_sm % 2 ? 0.10 : 0.04;
                const double t =
                    ((double)on_sm + alone) * (double)tiles * t_tile * (big ? 0.95 : 1.0) +
                    0.5 * (double)on_sm +
                    (ns > 1 ? 2.0 + 0.01 * (double)ns + 3e-5 * (double)(ns * n_i) : 0.0);
                if (t < best) {
                    best = t;
                    p.nwj = nwj;
                    p.nsplit = (int)ns;
                }
            }
        }
        p.threads = 32 * (H6_NWARP / p.nwj);  // i-particles per CTA
        p.jt = plan6_jt(p.nwj, p.nsplit, n_j);
        return p;
    }
    p.threads = H6_T64;
    p.jt = H6_JT64;
    const long long nblk = (n_i + p.threads - 1) / p.threads;
    const long long ntiles = (n_j + p.jt - 1) / p.jt;
    const long long cap = std::min(fit, std::max(1LL, ntiles / 4));
    const long long slots = 4 * sms;
    const long long ns0 = std::min(cap, std::max(1LL, (2 * slots + nblk - 1) / nblk));
    long long best = ns0;
    double best_eff = 0.0;
    for (long long ns = ns0; ns <= std::min(cap, 8 * ns0); ++ns) {
        const double waves = (double)(nblk * ns) / (double)slots;
        const double eff = waves / std::ceil(waves);
        if (eff > best_eff + 1e-9) {
            best_eff = eff;
            best = ns;
        }
        if (eff >= 0.97) break;  // the fewest splits whose last wave is nearly full
    }
    p.nsplit = (int)std::min(best, 1024LL);
    return p;
}

// The plan of a table entry (F32 / double-single kinds: warp rows nwj in {1, 2, 4,
// 8}, nsplit j-splits clamped to the j-tiles and to 1024; FP64: one warp row).
ForcePlan plan6_from_entry(int variant, int nwj, int nsplit, int n_i, int n_j)
{
    ForcePlan p{};
    p.kind = 0;
    p.ipt = 1;
    if (variant == NB_F64) {
        p.nwj = 1;
        p.threads = H6_T64;
        p.jt = H6_JT64;
    } else {
        p.nwj = (nwj == 2 || nwj == 4 || nwj == 8) ? nwj : 1;
        p.threads = 32 * (H6_NWARP / p.nwj);
        p.jt = H6_JT;
    }
    const long long ntiles = std::max(1LL, ((long long)n_j + p.jt - 1) / p.jt);
    p.nsplit = (int)std::max(1LL, std::min<long long>({(long long)nsplit, ntiles, 1024LL}));
    if (variant != NB_F64) p.jt = plan6_jt(p.nwj, p.nsplit, n_j);
    (void)n_i;
    return p;
}

int occ6_blocks(int variant, int nwj)
{
    return occ6_of(variant == NB_F32DS, nwj);
}

size_t plan6_partial_doubles(const ForcePlan &p, int n_i)
{
    if (p.nsplit <= 1) return 0;
    return (size_t)p.nsplit * H6_VALS * (size_t)n_i;  // float2 (DS) or double: 8 bytes each
}

cudaError_t launch_force6(int variant, const ForcePlan &p, const StateDev &s, const int *idx,
                          int n_i, double eps2, double *part, const Out6 &out, unsigned *err,
                          cudaStream_t st, cudaEvent_t *ev)
{
    if (n_i <= 0) return cudaSuccess;
    const long long pld = n_i;
    if (ev) cudaEventRecord(ev[0], st);
    cudaError_t e;
    if (variant == NB_F64) {
        dim3 grid((n_i + H6_T64 - 1) / H6_T64, p.nsplit);
        k_force6_tile64<<<grid, H6_T64, 0, st>>>(s, idx, n_i, eps2, part, pld, out, err);
        e = cudaGetLastError();
    } else {
        float2 *pp = reinterpret_cast<float2 *>(part);
        const float e2 = (float)eps2;
        const bool ds = (variant == NB_F32DS);
        const auto go = p.nwj == 8   ? (ds ? go_tile6<true, 8> : go_tile6<false, 8>)
                        : p.nwj == 4 ? (ds ? go_tile6<true, 4> : go_tile6<false, 4>)
                        : p.nwj == 2 ? (ds ? go_tile6<true, 2> : go_tile6<false, 2>)
                        : p.jt == H6_JT_BIG
                            ? (ds ? go_tile6<true, 1, H6_JT_BIG> : go_tile6<false, 1, H6_JT_BIG>)
                            : (ds ? go_tile6<true, 1> : go_tile6<false, 1>);
        e = go(s, idx, n_i, e2, p.nsplit, pp, out, err, st);
    }
    if (e != cudaSuccess) return e;
    if (ev) {
        cudaEventRecord(ev[1], st);
        cudaEventRecord(ev[2], st);
    }
    if (p.nsplit > 1)
        e = variant == NB_F64 ? go_force6_sums<double>(part, n_i, p.nsplit, out, err, st)
                              : go_force6_sums<float2>(part, n_i, p.nsplit, out, err, st);
    if (ev) cudaEventRecord(ev[3], st);
    return e;
}

cudaError_t launch_correct6(const StateDev &s, const int *act, int n_a, double t_new,
                            const Out6 &f, const StepParams &p, SchedDev *sd, unsigned *err,
                            unsigned long long *dtmin_hits, cudaStream_t st)
{
    const int slots = 10 * (CORRECT6_THREADS / 32);
    const int g = std::max(1, (n_a + slots - 1) / slots);
    return launch_dependent(k_correct6, dim3(g), CORRECT6_THREADS, 0, st, s, act, n_a, t_new, f, p, sd,
                            err, dtmin_hits);
}

}  // namespace nb
