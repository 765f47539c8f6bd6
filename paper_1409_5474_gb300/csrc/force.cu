// Pair-force kernels (K2) and the partial-sum reduction (K3).
//
// Direct summation of softened gravity from a j-set onto an i-set (paper
// Sect. III.A): for every i and every j != i,
//   r = x_j - x_i, v = v_j - v_i, s2 = |r|^2 + eps^2, rinv = s2^(-1/2),
//   acc += m_j rinv^3 r,  jerk += m_j rinv^3 (v - 3 (r.v) rinv^2 r),  pot -= m_j rinv.
//
// Two mappings of the (i, j) work onto the GPU, as the paper discusses:
//  - tile kernels ("i-parallel", Sect. III.A): each thread owns IPT
//    i-particles in registers; the CTA streams its j-range through shared
//    memory in tiles of JT records, staged by 1-D bulk copies (the TMA engine,
//    cp.async.bulk) into an NS-deep ring of mbarrier-guarded buffers. The
//    j-range is split across grid.y (the paper's j-parallel split for small
//    N_i, after Makino's scheme), and the partial sums are reduced by K3.
//  - j-parallel warp kernels for tiny i-sets (FP32: N_i <= 4, or 8 above 65536 j; FP64:
//    N_i <= 32 where that is faster; block-step tails): every thread holds the same few
//    i-particles and a different j; partial sums are combined by warp shuffles, then
//    across warps (double-single, FP64), then across CTAs by K3.
//
// Precision variants (Sect. III.A: emulated double precision for the
// inter-particle distance, native FP64 for extreme mass ratios):
//  - NB_F32DS: positions as double-single (hi + lo FP32) records; the relative
//    coordinate is (x_j.hi - x_i.hi) + (x_j.lo - x_i.lo), which keeps close
//    pairs far from the origin accurate; pair math in FP32 with rsqrtf on the
//    SFU; per-tile FP32 sums folded into double-single accumulators (TwoSum).
//  - NB_F32: the same kernel with FP32 positions (hi only) and FP32 sums.
//  - NB_F64: IEEE binary64 throughout.
//
// Self pair: for i-particles that are members of the j-set the i == j pair is
// masked by index (its potential term m_i/eps would otherwise swamp the FP32
// sums, and with eps = 0 it is 0/0). The mask is applied only in the j-tiles
// that contain one of the warp's own i-particles or are ragged (a warp-uniform
// branch), so the inner loop of every other tile carries no compare. A warp holds
// consecutive slots, so a sorted due set meets its own particles in few tiles.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "nb_internal.cuh"
#include "ds.cuh"
#include "pair.cuh"
#include "split_sum.cuh"
#include "tma.cuh"

namespace nb {

__device__ __forceinline__ bool finite7(const double *v)
{
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 7; ++c) ok = ok && isfinite(v[c]);
    return ok;
}

// Write the 7 totals of slot k: acc (3), jerk (3) and the positive potential
// sum P (pot = -P).
__device__ __forceinline__ void write_final(const Out3 &out, int k, double v[7], unsigned *err)
{
    v[6] = -v[6];
    if (!finite7(v)) atomicOr(err, DERR_NONFINITE);
    if (out.acc) {
        out.acc[k] = v[0];
        out.acc[out.ld + k] = v[1];
        out.acc[2 * out.ld + k] = v[2];
    }
    if (out.jerk) {
        out.jerk[k] = v[3];
        out.jerk[out.ld + k] = v[4];
        out.jerk[2 * out.ld + k] = v[5];
    }
    if (out.pot) out.pot[k] = v[6];
}

// Store the reduced value s of component c of slot k (c == 6: the positive
// potential sum, stored negated).
__device__ __forceinline__ void store_component(const Out3 &out, int c, int k, double s,
                                                unsigned *err)
{
    if (c == 6) {
        s = -s;
        if (out.pot) out.pot[k] = s;
    } else if (c < 3) {
        if (out.acc) out.acc[c * out.ld + k] = s;
    } else {
        if (out.jerk) out.jerk[(c - 3) * out.ld + k] = s;
    }
    if (!isfinite(s)) atomicOr(err, DERR_NONFINITE);
}

// K3, folded into the warp-group and the allocation-free FP64 kernels: after a CTA has
// written its partial sums for slots [slot0, slot0 + nslots), the last of the nsplit CTAs that share
// these slots (counted in *counter) reduces them and re-arms the counter. One
// warp per (slot, component): lane l adds splits l, l + 32, ... in order, then a
// fixed xor tree, so the result does not depend on which CTA finished last.
// The same with double-single partials (float2 {hi, lo} in the part buffer)
// combined in FP32 arithmetic; the final value is converted once.
template <int NT, int U = 8>
__device__ __forceinline__ void finish_split_ds(int nsplit, int slot0, int nslots, int n_i,
                                                const float2 *part, long long pld,
                                                unsigned *counter, const Out3 &out,
                                                unsigned *err)
{
    __shared__ int s_last_ds;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last_ds = (atomicAdd(counter, 1u) == (unsigned)nsplit - 1u);
    __syncthreads();
    if (!s_last_ds) return;
    __threadfence();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int valid = min(nslots, n_i - slot0);
    const int total = valid * 7;
    for (int q0 = warp * U; q0 < total; q0 += (NT / 32) * U) {
        dsf acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u] = dsf{0.f, 0.f};
        for (int sp = lane; sp < nsplit; sp += 32) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int q = q0 + u;
                if (q < total) {
                    const int c = q / valid, k = slot0 + q % valid;
                    const float2 v = __ldcg(part + ((size_t)sp * 7 + c) * pld + k);
                    ds_acc(acc[u], dsf{v.x, v.y});
                }
            }
        }
        const dsf v = warp_scatter_sum<U>(acc);
        const int q = q0 + lane;
        if (lane < U && q < total)
            store_component(out, q / valid, slot0 + q % valid, ds_to_double(v), err);
    }
    if (threadIdx.x == 0) *counter = 0u;
}

template <int NT>
__device__ __forceinline__ void finish_split(int nsplit, int slot0, int nslots, int n_i,
                                             const double *part, long long pld,
                                             unsigned *counter, const Out3 &out, unsigned *err)
{
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(counter, 1u) == (unsigned)nsplit - 1u);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int valid = min(nslots, n_i - slot0);
    const int total = valid * 7;
    constexpr int U = 8;  // outputs per warp pass: 8 independent loads in flight per lane
    for (int q0 = warp * U; q0 < total; q0 += (NT / 32) * U) {
        double acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u] = 0.0;
        for (int sp = lane; sp < nsplit; sp += 32) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int q = q0 + u;
                if (q < total) {
                    const int c = q / valid, k = slot0 + q % valid;
                    acc[u] += __ldcg(part + ((size_t)sp * 7 + c) * pld + k);
                }
            }
        }
        const double v = warp_scatter_sum<U>(acc);
        const int q = q0 + lane;
        if (lane < U && q < total) store_component(out, q / valid, slot0 + q % valid, v, err);
    }
    if (threadIdx.x == 0) *counter = 0u;
}

// Record row of i-slot k: the slot itself for a gathered or external i-set,
// else the member's particle index.
__device__ __forceinline__ int member_index(const ISet &is, int k, unsigned *err);
__device__ __forceinline__ int i_row(const ISet &is, int k, unsigned *err)
{
    if (is.gathered || !is.member) return k;
    return member_index(is, k, err);
}

// Particle index of an i-record (self-pair mask): from the record for a
// gathered set, the row for members, none (-1) for an external set.
__device__ __forceinline__ int i_id(const ISet &is, int row, float id_bits)
{
    if (is.gathered) return __float_as_int(id_bits);
    return is.member ? row : -1;
}

// Member index of slot k; an index outside the j-set is flagged and replaced by 0.
__device__ __forceinline__ int member_index(const ISet &is, int k, unsigned *err)
{
    const int r = is.idx ? is.idx[k] : k;
    if ((unsigned)r >= (unsigned)is.nj) {
        atomicOr(err, DERR_BADINDEX);
        return 0;
    }
    return r;
}

// ---------------------------------------------------------------------------
// FP32 / double-single tile kernel.
//
// A CTA is NWI x NWJ warps. The NWI warp columns own different i-particles
// (IPT per lane, an i-block of IB = 32 NWI IPT); the NWJ warp rows hold the
// same i-particles and share out every j-tile (row g takes j = g, g + NWJ,
// ...), so that a few hundred i-particles still fill an SM without cutting
// the j-range into many grid-level pieces. Rows are added in shared memory at
// the end, in fixed order.
//
// Bound by the FP32 pipe: 33 operations per interaction (27 for plain FP32), 1220 G/s at
// 2070 MHz. The running totals live in shared memory (touched once per fold) and
// not in 28 registers, so the packed loop, unrolled four pairs deep, runs without
// spills at two CTAs per SM; with eps^2 >= FLT_MIN the reciprocal square root is the one
// instruction rsqrt.approx.ftz.f32 (pair.cuh).
// N = 262144, F32-DS: 76.3 -> 67.8 ms, FMA pipe 84% of cycles (unroll 2: 68.7 ms, 1:
// 68.5 ms). Tiles that are ragged or hold a warp's own particle stay on the packed path
// with their halves masked, and warps without slots skip the arithmetic: 67.8 ->
// 66.0 ms at N = 262144, 47.4 -> 43.3 us for N_i = 300 at N = 65536.
// ---------------------------------------------------------------------------

__host__ __device__ constexpr bool tile_ahead(int nwj) { return nwj == 8; }

template <int VAR, int IPT, int NWI, int NWJ, int JT, int NS, int RUN>
__global__ void __launch_bounds__(32 * NWI * NWJ, 2)
    k_force_tile32(const float4 *jrec, int nj, ISet is, float eps2f, int ntiles, double *part,
                   long long pld, Out3 out, unsigned *err)
{
    // NS ring stages of JT records (bulk-copy destinations), one or (AHEAD) two tiles as
    // j-pairs (JT / 2 pairs x 6 float4 each), the running totals
    extern __shared__ __align__(128) float4 s_tile[];
    __shared__ __align__(8) uint64_t s_full[NS];
    __shared__ int s_abort;

    constexpr bool DS = (VAR == NB_F32DS);
    constexpr int NT = 32 * NWI * NWJ;
    constexpr int IB = 32 * NWI * IPT;
    // pairs that a warp row takes of a tile; a run ends with a tile, or several of them
    // make up a tile (of RUNS each)
    constexpr int ROW = JT / 2 / NWJ;
    constexpr int FOLD = RUN > ROW ? RUN / ROW : 1;
    constexpr int RUNS = RUN < ROW ? ROW / RUN : 1;
    constexpr int JR = JT / RUNS;  // records of a run, of all warp rows
    constexpr int PAIRS = JT * DS_REC;  // float4 of a pair buffer
    constexpr bool AHEAD = tile_ahead(NWJ);
    float4 *s_pair = s_tile + (size_t)NS * PAIRS;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wi = warp % NWI, wj = warp / NWI;
    const int nsplit = gridDim.y;
    const int split = blockIdx.y;
    const int tile0 = (int)((long long)ntiles * split / nsplit);
    const int tile1 = (int)((long long)ntiles * (split + 1) / nsplit);
    const int my_tiles = tile1 - tile0;

    // running totals (double-single, or plain FP32 in .x), this thread's own column
    float2 *s_tot = reinterpret_cast<float2 *>(s_pair + (AHEAD ? 2 : 1) * PAIRS) + tid;
#pragma unroll
    for (int q = 0; q < 7 * IPT; ++q) s_tot[q * NT] = make_float2(0.f, 0.f);
    if (tid == 0) {
        s_abort = 0;
#pragma unroll
        for (int s = 0; s < NS; ++s) mbar_init(&s_full[s], 1);
        fence_mbar_init();
    }
    cudaGridDependencySynchronize();  // nothing above reads what another launch wrote

    // i-particles of this thread
    IPair ip[IPT];
    int iid[IPT];
#pragma unroll
    for (int p = 0; p < IPT; ++p) {
        int k = blockIdx.x * IB + (wi * IPT + p) * 32 + lane;
        if (k >= is.n) k = is.n - 1;  // idle slots compute a copy, never written
        const int r = i_row(is, k, err);
        const float4 a = is.rec32[(size_t)DS_REC * r];
        const float4 b = is.rec32[(size_t)DS_REC * r + 1];
        const float4 c = is.rec32[(size_t)DS_REC * r + 2];
        ip[p] = ipair_of(a, b, c);
        iid[p] = i_id(is, r, b.w);
    }
    const float2 e2 = make_float2(eps2f, eps2f);
    const bool soft = soft_pairs(eps2f);
    const bool idle = blockIdx.x * IB + wi * IPT * 32 >= is.n;

    // FP32 partial sums between folds, two lanes each (even and odd j of a pair)
    PairSum ts[IPT];
#pragma unroll
    for (int p = 0; p < IPT; ++p) pair_zero(ts[p]);

    __syncthreads();

    auto issue = [&](int kt) {
        const int stage = kt % NS;
        const int t = tile0 + kt;
        const int cnt = min(JT, nj - t * JT);
        const uint32_t bytes = (uint32_t)cnt * DS_REC * 16u;
        mbar_expect_tx(&s_full[stage], bytes);
        bulk_g2s(s_tile + (size_t)stage * JT * DS_REC, jrec + (size_t)t * JT * DS_REC, bytes,
                 &s_full[stage]);
    };
    if (tid == 0) {
        for (int kt = 0; kt < NS && kt < my_tiles; ++kt) issue(kt);
    }

    // AHEAD (eight warp rows): tile kt + 1 is rewritten as j-pairs into one buffer before
    // the pair terms of tile kt are taken from the other, so there is one barrier per tile
    // and the rewriting of some warps overlaps the arithmetic of others. A warp then has
    // only 16 pairs of a tile: N_i = 300 and 1531 at N = 65536 take 41.3 and 133 us
    // against 43.3 and 135.5 with one buffer and two barriers. With 128 or 32 pairs per
    // warp and tile the second buffer's traffic costs more than the barrier (4.24 against
    // 4.13 ms at N_i = 65536, 582 against 574 us at N_i = 8200).
    auto fetch = [&](int kt) {
        const int stage = kt % NS;
        if (!mbar_wait(&s_full[stage], (uint32_t)((kt / NS) & 1))) s_abort = 1;
        tile_to_pairs<JT, NT>(s_tile + (size_t)stage * JT * DS_REC,
                              min(JT, nj - (tile0 + kt) * JT),
                              s_pair + (AHEAD ? (kt & 1) * PAIRS : 0), tid);
    };
    if (AHEAD) {
        if (my_tiles > 0) fetch(0);
        __syncthreads();
        if (s_abort) {
            if (tid == 0) {
                drain_ring<NS>(s_full, 0u, 0, my_tiles);
                atomicOr(err, DERR_TIMEOUT);
            }
            return;
        }
        if (tid == 0 && NS < my_tiles) issue(NS);
    }

    for (int kt = 0; kt < my_tiles; ++kt) {
        const int got = AHEAD ? kt + 1 : kt;  // the tile this iteration fetches
        if (got < my_tiles) fetch(got);
        if (!AHEAD) __syncthreads();
        const float4 *pairs = s_pair + (AHEAD ? (kt & 1) * PAIRS : 0);
        const int jbase = (tile0 + kt) * JT;
        const int cnt = min(JT, nj - jbase);

        // self pair in this tile for any lane of the warp? (warp-uniform)
        bool own = false;
#pragma unroll
        for (int p = 0; p < IPT; ++p) own = own || (iid[p] >= jbase && iid[p] < jbase + cnt);
        own = __any_sync(0xffffffffu, own);

        const bool masked = own || cnt < JT;
#pragma unroll 1
        for (int r = 0; r < (idle ? 0 : RUNS); ++r) {  // idle: no slot of this warp is written
            const int f = r * JR;
            if (RUNS > 1 && f >= cnt) break;
            const float4 *P = pairs + DS_REC * f;
            const int fcnt = min(JR, cnt - f);
            if (soft)
                tile_pairs<DS, IPT, JR, true>(P, wj, NWJ, jbase + f, fcnt, masked, ip, iid, e2, ts);
            else
                tile_pairs<DS, IPT, JR, false>(P, wj, NWJ, jbase + f, fcnt, masked, ip, iid, e2, ts);

            // fold the FP32 partial sums (both lanes) into the running totals
            if (FOLD > 1 && (kt + 1) % FOLD != 0 && kt + 1 != my_tiles) continue;
#pragma unroll
            for (int p = 0; p < IPT; ++p) {
#pragma unroll
                for (int c = 0; c < 7; ++c) {
                    float2 &h = s_tot[(p * 7 + c) * NT];
                    float2 v = h;
                    if (DS)
                        ds_add(v.x, v.y, pair_total(ts[p], c));
                    else
                        v.x += pair_total(ts[p], c);
                    h = v;
                }
                pair_zero(ts[p]);
            }
        }

        // every warp is done with the pairs of tile kt and the stage of tile got
        __syncthreads();
        if (s_abort) {
            if (tid == 0) {
                drain_ring<NS>(s_full, 0u, got, my_tiles);
                atomicOr(err, DERR_TIMEOUT);
            }
            return;
        }
        if (tid == 0 && got + NS < my_tiles) issue(got + NS);
    }

    if (wj == 0) {
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
            const int k = blockIdx.x * IB + (wi * IPT + p) * 32 + lane;
            if (k >= is.n) continue;
            // the warp rows' totals in order 0..NWJ-1 (columns 32 NWI threads apart)
            dsf v[7];
#pragma unroll
            for (int c = 0; c < 7; ++c) {
                const float2 *h = s_tot + (p * 7 + c) * NT;
                v[c] = dsf{h[0].x, h[0].y};
#pragma unroll
                for (int g = 1; g < NWJ; ++g)
                    ds_acc(v[c], dsf{h[32 * NWI * g].x, h[32 * NWI * g].y});
            }
            if (nsplit == 1) {
                double d[7];
#pragma unroll
                for (int c = 0; c < 7; ++c) d[c] = ds_to_double(v[c]);
                write_final(out, k, d, err);
            } else {
                float2 *pp = reinterpret_cast<float2 *>(part);
#pragma unroll
                for (int c = 0; c < 7; ++c)
                    pp[((size_t)split * 7 + c) * pld + k] = make_float2(v[c].hi, v[c].lo);
            }
        }
    }
    // with nsplit > 1 the partials are summed by k_split_sums, launched next
}

// K3 of the tile and FP64 kernels (split_sum): output q = component c of slot k.
template <class T, int G>
__global__ void __launch_bounds__(256)
    k_split_sums(const T *part, long long pld, int nsplit, int n_i, Out3 out, unsigned *err)
{
    const long long q = (long long)blockIdx.x * (256 / G) + threadIdx.x % (256 / G);
    const int c = (int)(q / n_i), k = (int)(q % n_i);
    double v;
    cudaGridDependencySynchronize();
    if (split_sum<T, G>(part + (size_t)c * pld + k, (size_t)7 * pld, nsplit, q < 7LL * n_i, v))
        store_component(out, c, k, v, err);
}

// ---------------------------------------------------------------------------
// FP64 tile kernel.
//
// Bound by the FP64 pipe: a warp-wide FP64 instruction holds an SMSP's pipe for 64
// cycles, and a pair takes about 32 of them, so one j costs a warp of 32 i-particles 1 us
// and a GB300 does 19.7 G/s at most (17.3 measured at N = 20011). What is
// left is to keep all 608 pipes busy to the end: a CTA is 32 i-particles times four warp rows (one warp per
// SMSP; row g takes j = g, g + 4, ... of every tile, the rows are added in order through
// shared memory), so an SM's four pipes always carry the same load and the plan divides
// the j-range in units of 16. The splits are summed by k_split_sums. N = 1024, all
// i: 316 -> 75.7 us; 100 of 20011 688 -> 158 us; N = 6007, all i: 2380 -> 2123 us.
// ---------------------------------------------------------------------------

constexpr int T64_ROWS = 4;   // warp rows of a CTA
constexpr int T64_UNIT = 16;  // j-ranges are whole units (16-byte aligned rows)

template <int JT, int NS>
__global__ void __launch_bounds__(32 * T64_ROWS)
    k_force_tile64(JSet js, ISet is, double eps2, int nunits, double *part, long long pld,
                   Out3 out, unsigned *err)
{
    extern __shared__ __align__(128) double s_t64[];  // NS * 7 * JT
    __shared__ __align__(8) uint64_t s_full[NS];
    __shared__ int s_abort;
    __shared__ double s_row[T64_ROWS - 1][7][32];

    const int tid = threadIdx.x, lane = tid & 31, row = tid >> 5;
    const int nsplit = gridDim.y;
    const int split = blockIdx.y;
    const int j0 = (int)((long long)nunits * split / nsplit) * T64_UNIT;
    const int j1 = min(js.n, (int)((long long)nunits * (split + 1) / nsplit) * T64_UNIT);
    const int my_tiles = (j1 - j0 + JT - 1) / JT;

    if (tid == 0) {
        s_abort = 0;
#pragma unroll
        for (int s = 0; s < NS; ++s) mbar_init(&s_full[s], 1);
        fence_mbar_init();
    }
    cudaGridDependencySynchronize();  // nothing above reads what another launch wrote

    const int k = blockIdx.x * 32 + lane;
    const int kc = min(k, is.n - 1);  // idle lanes compute a copy, never written
    const int r = is.member ? member_index(is, kc, err) : kc;
    const int iid = is.member ? r : -1;
    double xi[3], vi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        xi[c] = is.pos64[c * is.ld64 + r];
        vi[c] = is.vel64[c * is.ld64 + r];
    }
    double v[7];  // acc, jerk, positive potential
#pragma unroll
    for (int c = 0; c < 7; ++c) v[c] = 0.0;
    __syncthreads();

    // 7 rows per stage: x, y, z, vx, vy, vz, m
    auto issue = [&](int kt) {
        const int stage = kt % NS;
        const int cnt = min(JT, j1 - j0 - kt * JT);
        const uint32_t bytes = (uint32_t)(((cnt * 8) + 15) & ~15);  // rows are padded
        mbar_expect_tx(&s_full[stage], 7u * bytes);
        double *dst = s_t64 + (size_t)stage * 7 * JT;
        const size_t off = (size_t)j0 + (size_t)kt * JT;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            bulk_g2s(dst + c * JT, js.pos64 + c * js.ld + off, bytes, &s_full[stage]);
            bulk_g2s(dst + (3 + c) * JT, js.vel64 + c * js.ld + off, bytes, &s_full[stage]);
        }
        bulk_g2s(dst + 6 * JT, js.m64 + off, bytes, &s_full[stage]);
    };
    if (tid == 0) {
        for (int kt = 0; kt < NS && kt < my_tiles; ++kt) issue(kt);
    }

    for (int kt = 0; kt < my_tiles; ++kt) {
        const int stage = kt % NS;
        const uint32_t parity = (uint32_t)((kt / NS) & 1);
        if (!mbar_wait(&s_full[stage], parity)) s_abort = 1;
        const double *T = s_t64 + (size_t)stage * 7 * JT;
        const int jbase = j0 + kt * JT;
        const int cnt = min(JT, j1 - jbase);
        double ta[3], tja[3], tjb[3], tp = 0.0;
#pragma unroll
        for (int c = 0; c < 3; ++c) ta[c] = tja[c] = tjb[c] = 0.0;
#pragma unroll 2
        for (int jj = row; jj < cnt; jj += T64_ROWS) {
            const double dx = T[jj] - xi[0], dy = T[JT + jj] - xi[1], dz = T[2 * JT + jj] - xi[2];
            const double dvx = T[3 * JT + jj] - vi[0], dvy = T[4 * JT + jj] - vi[1],
                         dvz = T[5 * JT + jj] - vi[2];
            double r2 = fma(dx, dx, eps2);
            r2 = fma(dy, dy, r2);
            r2 = fma(dz, dz, r2);
            double rv = dx * dvx;
            rv = fma(dy, dvy, rv);
            rv = fma(dz, dvz, rv);
            const double rinv = jbase + jj == iid ? 0.0 : rsqrt(r2);
            const double rinv2 = rinv * rinv;
            const double mrinv = T[6 * JT + jj] * rinv;
            const double mr3 = mrinv * rinv2;
            const double beta = (mr3 * rinv2) * rv;
            tp += mrinv;
            ta[0] = fma(mr3, dx, ta[0]);
            ta[1] = fma(mr3, dy, ta[1]);
            ta[2] = fma(mr3, dz, ta[2]);
            tja[0] = fma(mr3, dvx, tja[0]);
            tja[1] = fma(mr3, dvy, tja[1]);
            tja[2] = fma(mr3, dvz, tja[2]);
            tjb[0] = fma(beta, dx, tjb[0]);
            tjb[1] = fma(beta, dy, tjb[1]);
            tjb[2] = fma(beta, dz, tjb[2]);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] += ta[c];
            v[3 + c] += fma(-3.0, tjb[c], tja[c]);
        }
        v[6] += tp;
        __syncthreads();
        if (s_abort) {
            if (tid == 0) {
                drain_ring<NS>(s_full, 0u, kt, my_tiles);
                atomicOr(err, DERR_TIMEOUT);
            }
            return;
        }
        if (tid == 0 && kt + NS < my_tiles) issue(kt + NS);
    }

    if (row > 0) {
#pragma unroll
        for (int c = 0; c < 7; ++c) s_row[row - 1][c][lane] = v[c];
    }
    __syncthreads();
    if (row > 0 || k >= is.n) return;
#pragma unroll
    for (int c = 0; c < 7; ++c)
        v[c] = (v[c] + s_row[0][c][lane]) + (s_row[1][c][lane] + s_row[2][c][lane]);
    if (nsplit == 1) {
        write_final(out, k, v, err);
    } else {
#pragma unroll
        for (int c = 0; c < 7; ++c) part[((size_t)split * 7 + c) * pld + k] = v[c];
    }
}

// ---------------------------------------------------------------------------
// j-parallel kernels for small i-sets (lanes over j).
// ---------------------------------------------------------------------------

// FP32 / double-single warp-group kernel for small and mid-size i-sets: each
// warp owns its own IPT i-particles (every lane holds the same ones) and its
// lanes stride over the CTA's j-range, reading the j-records straight from
// L1/L2 (the warps of a CTA share one j-range, so it is read from L2 once per
// CTA). A warp needs no block barrier: its lanes' sums meet in one xor tree.
// Grid: i-groups of NWARP warps (x) times j-splits (y); the splits are reduced
// by the last CTA of each group (finish_split).
template <int VAR, int IPT, int NWARP>
__global__ void __launch_bounds__(32 * NWARP)
    k_force_wgrp32(const float4 *__restrict__ jrec, int nj, ISet is, float eps2f,
                   double *__restrict__ part, long long pld, unsigned *counters, Out3 out,
                   unsigned *err)
{
    constexpr bool DS = (VAR == NB_F32DS);
    constexpr int NT = 32 * NWARP;
    constexpr int CHUNK = 32 * 32;  // j per FP32 partial sum (32 per lane)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nsplit = gridDim.y, split = blockIdx.y;
    const int j0 = (int)((long long)nj * split / nsplit);
    const int j1 = (int)((long long)nj * (split + 1) / nsplit);
    const int slot0 = (blockIdx.x * NWARP + warp) * IPT;

    float xh[IPT], yh[IPT], zh[IPT], xl[IPT], yl[IPT], zl[IPT], vx[IPT], vy[IPT], vz[IPT];
    int iid[IPT];
#pragma unroll
    for (int p = 0; p < IPT; ++p) {
        const int k = min(slot0 + p, is.n - 1);
        const int r = i_row(is, k, err);
        const float4 a = __ldg(is.rec32 + (size_t)DS_REC * r);
        const float4 b = __ldg(is.rec32 + (size_t)DS_REC * r + 1);
        const float4 c = __ldg(is.rec32 + (size_t)DS_REC * r + 2);
        xh[p] = a.x; yh[p] = a.y; zh[p] = a.z;
        xl[p] = b.x; yl[p] = b.y; zl[p] = b.z;
        vx[p] = c.x; vy[p] = c.y; vz[p] = c.z;
        iid[p] = i_id(is, r, b.w);
    }
    float A_h[IPT][3], A_l[IPT][3], J_h[IPT][3], J_l[IPT][3], P_h[IPT], P_l[IPT];
#pragma unroll
    for (int p = 0; p < IPT; ++p) {
#pragma unroll
        for (int c = 0; c < 3; ++c) A_h[p][c] = A_l[p][c] = J_h[p][c] = J_l[p][c] = 0.f;
        P_h[p] = P_l[p] = 0.f;
    }

    for (int c0 = j0; c0 < j1; c0 += CHUNK) {
        const int c1 = min(c0 + CHUNK, j1);
        float ta[IPT][3], tja[IPT][3], tjb[IPT][3], tp[IPT];
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
#pragma unroll
            for (int c = 0; c < 3; ++c) ta[p][c] = tja[p][c] = tjb[p][c] = 0.f;
            tp[p] = 0.f;
        }
#pragma unroll 4
        for (int j = c0 + lane; j < c1; j += 32) {
            const float4 a = __ldg(jrec + (size_t)DS_REC * j);
            const float4 c = __ldg(jrec + (size_t)DS_REC * j + 2);
            float4 b;
            if (DS) b = __ldg(jrec + (size_t)DS_REC * j + 1);
#pragma unroll
            for (int p = 0; p < IPT; ++p) {
                float dx, dy, dz;
                if (DS) {
                    dx = (a.x - xh[p]) + (b.x - xl[p]);
                    dy = (a.y - yh[p]) + (b.y - yl[p]);
                    dz = (a.z - zh[p]) + (b.z - zl[p]);
                } else {
                    dx = a.x - xh[p];
                    dy = a.y - yh[p];
                    dz = a.z - zh[p];
                }
                const float dvx = c.x - vx[p], dvy = c.y - vy[p], dvz = c.z - vz[p];
                float r2 = fmaf(dx, dx, eps2f);
                r2 = fmaf(dy, dy, r2);
                r2 = fmaf(dz, dz, r2);
                float rv = dx * dvx;
                rv = fmaf(dy, dvy, rv);
                rv = fmaf(dz, dvz, rv);
                float rinv = rsqrtf(r2);
                rinv = (j == iid[p]) ? 0.f : rinv;
                const float rinv2 = rinv * rinv;
                const float mrinv = a.w * rinv;
                const float mr3 = mrinv * rinv2;
                const float beta = (mr3 * rinv2) * rv;
                tp[p] += mrinv;
                ta[p][0] = fmaf(mr3, dx, ta[p][0]);
                ta[p][1] = fmaf(mr3, dy, ta[p][1]);
                ta[p][2] = fmaf(mr3, dz, ta[p][2]);
                tja[p][0] = fmaf(mr3, dvx, tja[p][0]);
                tja[p][1] = fmaf(mr3, dvy, tja[p][1]);
                tja[p][2] = fmaf(mr3, dvz, tja[p][2]);
                tjb[p][0] = fmaf(beta, dx, tjb[p][0]);
                tjb[p][1] = fmaf(beta, dy, tjb[p][1]);
                tjb[p][2] = fmaf(beta, dz, tjb[p][2]);
            }
        }
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float jt = fmaf(-3.f, tjb[p][c], tja[p][c]);
                if (DS) {
                    ds_add(A_h[p][c], A_l[p][c], ta[p][c]);
                    ds_add(J_h[p][c], J_l[p][c], jt);
                } else {
                    A_h[p][c] += ta[p][c];
                    J_h[p][c] += jt;
                }
            }
            if (DS)
                ds_add(P_h[p], P_l[p], tp[p]);
            else
                P_h[p] += tp[p];
        }
    }

    // lanes -> warp total (double-single xor tree); lane 0 stores
#pragma unroll
    for (int p = 0; p < IPT; ++p) {
        dsf v[7];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] = dsf{A_h[p][c], A_l[p][c]};
            v[3 + c] = dsf{J_h[p][c], J_l[p][c]};
        }
        v[6] = dsf{P_h[p], P_l[p]};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < 7; ++c) ds_acc(v[c], ds_shfl_xor(v[c], o));
        const int k = slot0 + p;
        if (lane == 0 && k < is.n) {
            if (nsplit == 1) {
                double d[7];
#pragma unroll
                for (int c = 0; c < 7; ++c) d[c] = ds_to_double(v[c]);
                write_final(out, k, d, err);
            } else {
                float2 *pp = reinterpret_cast<float2 *>(part);
#pragma unroll
                for (int c = 0; c < 7; ++c)
                    pp[((size_t)split * 7 + c) * pld + k] = make_float2(v[c].hi, v[c].lo);
            }
        }
    }
    if (nsplit > 1)
        finish_split_ds<NT>(nsplit, blockIdx.x * NWARP * IPT, NWARP * IPT, is.n,
                            reinterpret_cast<float2 *>(part), pld, counters + blockIdx.x, out,
                            err);
}


// FP32 / double-single kernel for tiny i-sets (block-step tails): every thread
// holds the same IPT i-particles and JPT j-records of its own, all loaded
// before any arithmetic so the whole j-set costs one L2 round trip; sums go
// through a double-single warp tree, then across the CTA's warps, one
// partial per CTA.
// Groups of IPT (<= 4) i-particles are processed in turn (the j-records stay
// in registers).
template <int VAR, int IPT, int JPT>
__global__ void __launch_bounds__(256)
    k_force_tiny32(const float4 *jrec, int nj, ISet is, float eps2f, double *part, long long pld,
                   unsigned *counters, Out3 out, unsigned *err)
{
    constexpr bool DS = (VAR == NB_F32DS);
    constexpr int NT = 256, NW = NT / 32;
    __shared__ float2 s_red[NW][IPT * 7];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nsplit = gridDim.x, split = blockIdx.x;
    cudaGridDependencySynchronize();

    // this thread's j-records: j = split * NT * JPT + r * NT + tid
    float4 ja[JPT], jb[JPT], jc[JPT];
    int jidx[JPT];
#pragma unroll
    for (int r = 0; r < JPT; ++r) {
        const int j = split * NT * JPT + r * NT + tid;
        jidx[r] = j;
        if (j < nj) {
            ja[r] = jrec[(size_t)DS_REC * j];
            jc[r] = jrec[(size_t)DS_REC * j + 2];
            if (DS) jb[r] = jrec[(size_t)DS_REC * j + 1];
        } else {
            ja[r] = make_float4(0.f, 0.f, 0.f, 0.f);  // massless: contributes nothing
            jc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
            jb[r] = make_float4(0.f, 0.f, 0.f, 0.f);
            jidx[r] = -2;
        }
    }

    for (int g0 = 0; g0 < is.n; g0 += IPT) {
        float xh[IPT], yh[IPT], zh[IPT], xl[IPT], yl[IPT], zl[IPT], vx[IPT], vy[IPT], vz[IPT];
        int iid[IPT];
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
            const int k = min(g0 + p, is.n - 1);
            const int r = i_row(is, k, err);
            const float4 a = is.rec32[(size_t)DS_REC * r];
            const float4 b = is.rec32[(size_t)DS_REC * r + 1];
            const float4 c = is.rec32[(size_t)DS_REC * r + 2];
            xh[p] = a.x; yh[p] = a.y; zh[p] = a.z;
            xl[p] = b.x; yl[p] = b.y; zl[p] = b.z;
            vx[p] = c.x; vy[p] = c.y; vz[p] = c.z;
            iid[p] = i_id(is, r, b.w);
        }
        constexpr int P = IPT == 1 ? 8 : (IPT == 2 ? 16 : 32);
        dsf v[P];
#pragma unroll
        for (int q = 0; q < P; ++q) v[q] = dsf{0.f, 0.f};
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
            float ta0 = 0.f, ta1 = 0.f, ta2 = 0.f, tj0 = 0.f, tj1 = 0.f, tj2 = 0.f;
            float tb0 = 0.f, tb1 = 0.f, tb2 = 0.f, tp = 0.f;
#pragma unroll
            for (int r = 0; r < JPT; ++r) {
                float dx, dy, dz;
                if (DS) {
                    dx = (ja[r].x - xh[p]) + (jb[r].x - xl[p]);
                    dy = (ja[r].y - yh[p]) + (jb[r].y - yl[p]);
                    dz = (ja[r].z - zh[p]) + (jb[r].z - zl[p]);
                } else {
                    dx = ja[r].x - xh[p];
                    dy = ja[r].y - yh[p];
                    dz = ja[r].z - zh[p];
                }
                const float dvx = jc[r].x - vx[p], dvy = jc[r].y - vy[p], dvz = jc[r].z - vz[p];
                float r2 = fmaf(dx, dx, eps2f);
                r2 = fmaf(dy, dy, r2);
                r2 = fmaf(dz, dz, r2);
                float rv = dx * dvx;
                rv = fmaf(dy, dvy, rv);
                rv = fmaf(dz, dvz, rv);
                float rinv = rsqrtf(r2);
                // self pair and padding records (jidx -2) contribute nothing
                rinv = (jidx[r] == iid[p] || jidx[r] < 0) ? 0.f : rinv;
                const float rinv2 = rinv * rinv;
                const float mrinv = ja[r].w * rinv;
                const float mr3 = mrinv * rinv2;
                const float beta = (mr3 * rinv2) * rv;
                tp += mrinv;
                ta0 = fmaf(mr3, dx, ta0);
                ta1 = fmaf(mr3, dy, ta1);
                ta2 = fmaf(mr3, dz, ta2);
                tj0 = fmaf(mr3, dvx, tj0);
                tj1 = fmaf(mr3, dvy, tj1);
                tj2 = fmaf(mr3, dvz, tj2);
                tb0 = fmaf(beta, dx, tb0);
                tb1 = fmaf(beta, dy, tb1);
                tb2 = fmaf(beta, dz, tb2);
            }
            v[7 * p + 0] = dsf{ta0, 0.f};
            v[7 * p + 1] = dsf{ta1, 0.f};
            v[7 * p + 2] = dsf{ta2, 0.f};
            v[7 * p + 3] = dsf{fmaf(-3.f, tb0, tj0), 0.f};
            v[7 * p + 4] = dsf{fmaf(-3.f, tb1, tj1), 0.f};
            v[7 * p + 5] = dsf{fmaf(-3.f, tb2, tj2), 0.f};
            v[7 * p + 6] = dsf{tp, 0.f};
        }
        // double-single sums over the lanes: lane 7 p + c holds component c of slot p
        const dsf wsum = warp_scatter_sum<P>(v);
        if (lane < IPT * 7) s_red[warp][lane] = make_float2(wsum.hi, wsum.lo);
        __syncthreads();
        if (tid < IPT * 7) {
            const int p = tid / 7, c = tid % 7;
            const int k = g0 + p;
            dsf sum{0.f, 0.f};
#pragma unroll
            for (int w = 0; w < NW; ++w) ds_acc(sum, dsf{s_red[w][tid].x, s_red[w][tid].y});
            if (k < is.n) {
                if (nsplit == 1)
                    store_component(out, c, k, ds_to_double(sum), err);
                else
                    reinterpret_cast<float2 *>(part)[((size_t)split * 7 + c) * pld + k] =
                        make_float2(sum.hi, sum.lo);
            }
        }
        __syncthreads();
    }
    if (nsplit <= 1) return;
    // the last CTA sums the partials, as k_split_sums does (32 outputs a pass, eight threads
    // each: one or two round trips to L2). A launch of its own for 7 to 56 outputs takes no
    // less time on the GPU and 1.5 us more of the host's (3 of 65536, a call and its copy: 25.3 -> 24.1 us).
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(counters, 1u) == (unsigned)nsplit - 1u);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int q0 = 0; q0 < 7 * is.n; q0 += NT / 8) {
        const int q = q0 + tid % (NT / 8);
        const bool valid = q < 7 * is.n;
        const int c = valid ? q / is.n : 0, k = valid ? q - c * is.n : 0;
        double sum;
        if (split_sum<float2, 8>(reinterpret_cast<const float2 *>(part) + (size_t)c * pld + k,
                                 (size_t)7 * pld, nsplit, valid, sum))
            store_component(out, c, k, sum, err);
        __syncthreads();  // the groups' sums are read before the next pass writes its own
    }
    if (tid == 0) *counters = 0u;
}

// FP64 j-parallel kernel: thread = j, all threads share IPT i's.
template <int IPT, int NT>
__global__ void __launch_bounds__(NT)
    k_force_jmode64(JSet js, ISet is, double eps2, double *part, long long pld,
                    unsigned *counters, Out3 out, unsigned *err)
{
    constexpr int NW = NT / 32;
    __shared__ double s_red[NW][IPT * 7];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nsplit = gridDim.x, split = blockIdx.x;
    const int nj = js.n;
    const int j0 = (int)((long long)nj * split / nsplit);
    const int j1 = (int)((long long)nj * (split + 1) / nsplit);
    cudaGridDependencySynchronize();

    for (int g0 = 0; g0 < is.n; g0 += IPT) {
        double xi[IPT][3], vi[IPT][3], mi[IPT];
        int iid[IPT];
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
            const int k = min(g0 + p, is.n - 1);
            const int r = is.member ? member_index(is, k, err) : k;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                xi[p][c] = is.pos64[c * is.ld64 + r];
                vi[p][c] = is.vel64[c * is.ld64 + r];
            }
            mi[p] = is.member ? is.m64[r] : 0.0;
            iid[p] = is.member ? r : -1;
        }
        double ta[IPT][3], tja[IPT][3], tjb[IPT][3], tp[IPT];
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
#pragma unroll
            for (int c = 0; c < 3; ++c) ta[p][c] = tja[p][c] = tjb[p][c] = 0.0;
            tp[p] = 0.0;
        }
        for (int j = j0 + tid; j < j1; j += NT) {
            const double xj = js.pos64[j], yj = js.pos64[js.ld + j], zj = js.pos64[2 * js.ld + j];
            const double uj = js.vel64[j], wj = js.vel64[js.ld + j], qj = js.vel64[2 * js.ld + j];
            const double mj = js.m64[j];
#pragma unroll
            for (int p = 0; p < IPT; ++p) {
                const double dx = xj - xi[p][0], dy = yj - xi[p][1], dz = zj - xi[p][2];
                const double dvx = uj - vi[p][0], dvy = wj - vi[p][1], dvz = qj - vi[p][2];
                double r2 = fma(dx, dx, eps2);
                r2 = fma(dy, dy, r2);
                r2 = fma(dz, dz, r2);
                double rv = dx * dvx;
                rv = fma(dy, dvy, rv);
                rv = fma(dz, dvz, rv);
                const double rinv = j == iid[p] ? 0.0 : rsqrt(r2);
                const double rinv2 = rinv * rinv;
                const double mrinv = mj * rinv;
                const double mr3 = mrinv * rinv2;
                const double beta = (mr3 * rinv2) * rv;
                tp[p] += mrinv;
                ta[p][0] = fma(mr3, dx, ta[p][0]);
                ta[p][1] = fma(mr3, dy, ta[p][1]);
                ta[p][2] = fma(mr3, dz, ta[p][2]);
                tja[p][0] = fma(mr3, dvx, tja[p][0]);
                tja[p][1] = fma(mr3, dvy, tja[p][1]);
                tja[p][2] = fma(mr3, dvz, tja[p][2]);
                tjb[p][0] = fma(beta, dx, tjb[p][0]);
                tjb[p][1] = fma(beta, dy, tjb[p][1]);
                tjb[p][2] = fma(beta, dz, tjb[p][2]);
            }
        }
        // lane 7 p + c of a warp holds its sum of component c of slot p
        constexpr int P = IPT == 1 ? 8 : (IPT == 2 ? 16 : 32);
        double v[P];
#pragma unroll
        for (int q = 0; q < P; ++q) v[q] = 0.0;
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[7 * p + c] = ta[p][c];
                v[7 * p + 3 + c] = fma(-3.0, tjb[p][c], tja[p][c]);
            }
            v[7 * p + 6] = tp[p];
        }
        const double wsum = warp_scatter_sum<P>(v);
        if (lane < IPT * 7) s_red[warp][lane] = wsum;
        __syncthreads();
        if (tid < IPT * 7) {
            const int p = tid / 7, c = tid % 7;
            const int k = g0 + p;
            if (k < is.n) {
                double s = 0.0;
#pragma unroll
                for (int w = 0; w < NW; ++w) s += s_red[w][tid];
                if (nsplit == 1) {
                    if (c == 6) {
                        s = -s;
                        if (out.pot) out.pot[k] = s;
                    } else if (c < 3) {
                        if (out.acc) out.acc[c * out.ld + k] = s;
                    } else {
                        if (out.jerk) out.jerk[(c - 3) * out.ld + k] = s;
                    }
                    if (!isfinite(s)) atomicOr(err, DERR_NONFINITE);
                } else {
                    part[((size_t)split * 7 + c) * pld + k] = s;
                }
            }
        }
        __syncthreads();
    }
    // counters == null: the partials are summed by k_split_sums, launched next
    if (nsplit > 1 && counters)
        finish_split<NT>(nsplit, 0, is.n, is.n, part, pld, counters, out, err);
}

// ---------------------------------------------------------------------------
// Batched force kernel: many independent systems in one launch (the batched
// clusters, and the requests of the serving loop). A work item is a block of
// i-rows of one system against a range of the same system's j-records, with
// its own pointers (WorkItem). The persistent CTAs take the items of the list (sorted
// by decreasing work on the host) by tickets, so that they finish together.
// i-parallel items stage the j-tiles through the same bulk-copy ring as the
// tile kernel (the mbarrier phases run on across items); j-parallel items read
// the j-records straight from L1/L2. Items of a j-split group leave
// double-single partials that the group's last item sums in split order.
// ---------------------------------------------------------------------------

// One j-parallel item (kind 1): every thread takes j = j0 + tid, j0 + tid + NT,
// ... against the same four i-rows at a time. FP32 sums over at most JPAR_RUN
// j per thread meet in a fixed xor tree per warp (double-single) and a
// fixed-order sum over the warps, added to double-single totals in shared
// memory; the totals are the item's outputs, or its partials when its j-range
// is one split of a group.
constexpr int JPAR_RUN = 32;

template <bool DS, int NT>
__device__ __forceinline__ void item_jpar(const WorkItem &w, float2 (*s_red)[28], float2 *s_tot)
{
    constexpr int G = 4;
    constexpr int NW = NT / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float eps2f = w.eps2;
    const int jend = w.j0 + w.nj;
    for (int g0 = 0; g0 < w.ni; g0 += G) {
        float xh[G], yh[G], zh[G], xl[G], yl[G], zl[G], vx[G], vy[G], vz[G];
        int iid[G];
#pragma unroll
        for (int p = 0; p < G; ++p) {
            const int r = w.i0 + min(g0 + p, w.ni - 1);  // idle slots copy the last i
            const float4 a = __ldg(w.irec + (size_t)DS_REC * r);
            const float4 b = __ldg(w.irec + (size_t)DS_REC * r + 1);
            const float4 c = __ldg(w.irec + (size_t)DS_REC * r + 2);
            xh[p] = a.x; yh[p] = a.y; zh[p] = a.z;
            xl[p] = b.x; yl[p] = b.y; zl[p] = b.z;
            vx[p] = c.x; vy[p] = c.y; vz[p] = c.z;
            iid[p] = w.gathered ? __float_as_int(b.w) : r;
        }
        if (tid < G * 7) s_tot[tid] = make_float2(0.f, 0.f);
        for (int jb = w.j0; jb < jend; jb += NT * JPAR_RUN) {
            float ta[G][3], tjv[G][3], tp[G];
#pragma unroll
            for (int p = 0; p < G; ++p) {
#pragma unroll
                for (int c = 0; c < 3; ++c) ta[p][c] = tjv[p][c] = 0.f;
                tp[p] = 0.f;
            }
            const int jstop = min(jend, jb + NT * JPAR_RUN);
#pragma unroll 2
            for (int j = jb + tid; j < jstop; j += NT) {
                const float4 a = __ldg(w.jrec + (size_t)DS_REC * j);
                const float4 c = __ldg(w.jrec + (size_t)DS_REC * j + 2);
                float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
                if (DS) b = __ldg(w.jrec + (size_t)DS_REC * j + 1);
#pragma unroll
                for (int p = 0; p < G; ++p) {
                    float dx, dy, dz;
                    if (DS) {
                        dx = (a.x - xh[p]) + (b.x - xl[p]);
                        dy = (a.y - yh[p]) + (b.y - yl[p]);
                        dz = (a.z - zh[p]) + (b.z - zl[p]);
                    } else {
                        dx = a.x - xh[p];
                        dy = a.y - yh[p];
                        dz = a.z - zh[p];
                    }
                    const float dvx = c.x - vx[p], dvy = c.y - vy[p], dvz = c.z - vz[p];
                    float r2 = fmaf(dx, dx, eps2f);
                    r2 = fmaf(dy, dy, r2);
                    r2 = fmaf(dz, dz, r2);
                    float rv = dx * dvx;
                    rv = fmaf(dy, dvy, rv);
                    rv = fmaf(dz, dvz, rv);
                    float rinv = rsqrtf(r2);
                    rinv = (j == iid[p]) ? 0.f : rinv;
                    const float rinv2 = rinv * rinv;
                    const float mrinv = a.w * rinv;
                    const float mr3 = mrinv * rinv2;
                    const float beta = -3.f * ((mr3 * rinv2) * rv);
                    tp[p] += mrinv;
                    ta[p][0] = fmaf(mr3, dx, ta[p][0]);
                    ta[p][1] = fmaf(mr3, dy, ta[p][1]);
                    ta[p][2] = fmaf(mr3, dz, ta[p][2]);
                    // per pair: m v / s^3 - 3 m (r.v) r / s^5
                    tjv[p][0] = fmaf(beta, dx, fmaf(mr3, dvx, tjv[p][0]));
                    tjv[p][1] = fmaf(beta, dy, fmaf(mr3, dvy, tjv[p][1]));
                    tjv[p][2] = fmaf(beta, dz, fmaf(mr3, dvz, tjv[p][2]));
                }
            }
            // lanes -> warp (fixed tree), warps -> CTA (fixed order) -> totals
            dsf v[32];
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = dsf{0.f, 0.f};
#pragma unroll
            for (int p = 0; p < G; ++p)
#pragma unroll
                for (int c = 0; c < 7; ++c)
                    v[7 * p + c].hi = c < 3 ? ta[p][c] : (c < 6 ? tjv[p][c - 3] : tp[p]);
            const dsf wsum = warp_scatter_sum<32>(v);
            if (lane < G * 7) s_red[warp][lane] = make_float2(wsum.hi, wsum.lo);
            __syncthreads();
            if (tid < G * 7) {
                dsf sum{s_tot[tid].x, s_tot[tid].y};
#pragma unroll
                for (int q = 0; q < NW; ++q) ds_acc(sum, dsf{s_red[q][tid].x, s_red[q][tid].y});
                s_tot[tid] = make_float2(sum.hi, sum.lo);
            }
            __syncthreads();
        }
        if (tid < G * 7) {
            const int p = tid / 7, c = tid % 7, k = g0 + p;
            if (k < w.ni) {
                const float2 t = s_tot[tid];
                if (w.nsplit <= 1) {
                    const Out3 out{w.acc, w.jerk, w.pot, w.ld};
                    store_component(out, c, w.i0 + k, ds_to_double(dsf{t.x, t.y}), w.err);
                } else {
                    w.part[((size_t)w.split * 7 + c) * w.ni + k] = t;
                }
            }
        }
        __syncthreads();
    }
}

// The j-parallel items of a batched evaluation (kind 1), in a kernel of their
// own so that their register needs do not lower the occupancy of the
// i-parallel kernel; the two run concurrently on two streams.
template <int VAR, int NT>
__global__ void __launch_bounds__(NT)
    k_force_items_jpar32(const WorkItem *__restrict__ items, int nitems)
{
    __shared__ float2 s_red[NT / 32][28];
    __shared__ float2 s_tot[28];
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const WorkItem w = items[it];
        item_jpar<VAR == NB_F32DS, NT>(w, s_red, s_tot);
    }
}

// The j-split groups of a batched evaluation, after the items: each group's
// outputs are the sums of its nsplit double-single partials in the order
// split = 0..nsplit-1 (one thread per output, consecutive outputs coalesced).
__global__ void __launch_bounds__(256)
    k_split_reduce(const SplitGroup *__restrict__ groups, int ngroups)
{
    for (int gi = blockIdx.x; gi < ngroups; gi += gridDim.x) {
        const SplitGroup g = groups[gi];
        const int total = 7 * g.ni;
        const Out3 out{g.acc, g.jerk, g.pot, g.ld};
        for (int q = threadIdx.x; q < total; q += blockDim.x) {
            const int c = q / g.ni, k = q % g.ni;
            dsf sum{0.f, 0.f};
            for (int sp = 0; sp < g.nsplit; ++sp) {
                const float2 v = __ldcg(g.part + ((size_t)sp * 7 + c) * g.ni + k);
                ds_acc(sum, dsf{v.x, v.y});
            }
            store_component(out, c, g.i0 + k, ds_to_double(sum), g.err);
        }
    }
}


// The last CTA of a batched launch to finish (or to give up) puts the ticket back to zero for
// the next launch on the stream. ticket: {items handed out, CTAs finished}.
__device__ __forceinline__ void items_done(unsigned *ticket)
{
    if (atomicAdd(ticket + 1, 1u) == gridDim.x - 1u) {
        ticket[0] = 0u;
        ticket[1] = 0u;
    }
}

// As the tile kernel: bound by the FP32 pipe, totals in shared memory, ragged tiles and
// tiles with a warp's own particles on the packed path (a 1000-particle system has a
// quarter of its tiles of either kind), warps without rows skip the arithmetic. 512
// clusters of 16-4096: a pass of eight steps 11.2 -> 10.3 ms.
// CHUNKS: items may take several j-ranges one after the other (WorkItem::chunk); the sums
// between ranges wait as double-single pairs in the item's own output elements, which are as
// wide, so that no other memory is needed.
template <int VAR, int IPT, int NT, int JT, int NS, bool CHUNKS>
__global__ void __launch_bounds__(NT, 512 / NT)
    k_force_items32(const WorkItem *__restrict__ items, int nitems, unsigned *ticket)
{
    // NS ring stages of JT records, then the current full tile as j-pairs
    extern __shared__ __align__(128) float4 s_tile[];
    __shared__ __align__(8) uint64_t s_full[NS];
    __shared__ int s_abort, s_next;
    constexpr bool DS = (VAR == NB_F32DS);
    float4 *s_pair = s_tile + (size_t)NS * JT * DS_REC;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the running totals (double-single, or plain FP32 in .x), this thread's own column
    float2 *s_tot = reinterpret_cast<float2 *>(s_pair + (size_t)JT * DS_REC) + tid;

    if (tid == 0) {
        s_abort = 0;
#pragma unroll
        for (int s = 0; s < NS; ++s) mbar_init(&s_full[s], 1);
        fence_mbar_init();
    }
    __syncthreads();

    unsigned seq = 0;  // tiles consumed so far by this CTA (ring position and phase)
    for (int it = blockIdx.x, next = 0; it < nitems; it = next) {
        // the item after this one, taken now so that its number is there in time
        if (tid == 0) s_next = (int)(gridDim.x + atomicAdd(ticket, 1u));
        const WorkItem w = items[it];
        unsigned *err = w.err;
        const float eps2f = w.eps2;
        const float2 e2 = make_float2(eps2f, eps2f);
        const bool soft = soft_pairs(eps2f);
        const float4 *__restrict__ jrec = w.jrec;
        const int ntiles = (w.nj + JT - 1) / JT;

        // the i-particles
        IPair ip[IPT];
        int iid[IPT];
#pragma unroll
        for (int p = 0; p < IPT; ++p) {
            const int k = min((warp * IPT + p) * 32 + lane, w.ni - 1);  // idle slots copy the last i
            const int r = w.i0 + k;
            const float4 a = __ldg(w.irec + (size_t)DS_REC * r);
            const float4 b = __ldg(w.irec + (size_t)DS_REC * r + 1);
            const float4 c = __ldg(w.irec + (size_t)DS_REC * r + 2);
            ip[p] = ipair_of(a, b, c);
            iid[p] = w.gathered ? __float_as_int(b.w) : r;
        }
#pragma unroll
        for (int q = 0; q < 7 * IPT; ++q) s_tot[q * NT] = make_float2(0.f, 0.f);

        auto issue = [&](int kt) {
            const unsigned sq = seq + (unsigned)kt;
            const int stage = (int)(sq % NS);
            const int cnt = min(JT, w.nj - kt * JT);
            const uint32_t bytes = (uint32_t)cnt * DS_REC * 16u;
            mbar_expect_tx(&s_full[stage], bytes);
            bulk_g2s(s_tile + (size_t)stage * JT * DS_REC,
                     jrec + ((size_t)w.j0 + (size_t)kt * JT) * DS_REC, bytes, &s_full[stage]);
        };
        if (tid == 0) {
            for (int kt = 0; kt < NS && kt < ntiles; ++kt) issue(kt);
        }
        for (int kt = 0; kt < ntiles; ++kt) {
            const unsigned sq = seq + (unsigned)kt;
            const int stage = (int)(sq % NS);
            if (!mbar_wait(&s_full[stage], (sq / NS) & 1u)) s_abort = 1;
            const float4 *T = s_tile + (size_t)stage * JT * DS_REC;
            const int jbase = w.j0 + kt * JT;
            const int cnt = min(JT, w.nj - kt * JT);
            bool own = false;
#pragma unroll
            for (int p = 0; p < IPT; ++p) own = own || (iid[p] >= jbase && iid[p] < jbase + cnt);
            own = __any_sync(0xffffffffu, own);
            // FP32 sums of this tile, two lanes each (even and odd j of a pair)
            PairSum ts[IPT];
#pragma unroll
            for (int p = 0; p < IPT; ++p) pair_zero(ts[p]);
            const bool masked = own || cnt < JT;
            tile_to_pairs<JT, NT>(T, cnt, s_pair, tid);
            __syncthreads();
            next = s_next;  // thread 0 writes it again after the barrier below at the earliest
            if (warp * IPT * 32 >= w.ni)
                ;  // no row of this warp is written
            else if (soft)
                tile_pairs<DS, IPT, JT, true>(s_pair, 0, 1, jbase, cnt, masked, ip, iid, e2, ts);
            else
                tile_pairs<DS, IPT, JT, false>(s_pair, 0, 1, jbase, cnt, masked, ip, iid, e2, ts);
#pragma unroll
            for (int p = 0; p < IPT; ++p)
#pragma unroll
                for (int c = 0; c < 7; ++c) {
                    float2 &h = s_tot[(p * 7 + c) * NT];
                    float2 v = h;
                    if (DS)
                        ds_add(v.x, v.y, pair_total(ts[p], c));
                    else
                        v.x += pair_total(ts[p], c);
                    h = v;
                }
            if (CHUNKS && w.chunk > 0 && (kt + 1 == ntiles || (kt + 1) * JT % w.chunk == 0)) {
                // the end of a j-range: its sums join those of the ranges before it, as
                // k_split_reduce adds them
#pragma unroll 1
                for (int p = 0; p < IPT; ++p) {
                    const int k = (warp * IPT + p) * 32 + lane;
                    if (k >= w.ni) continue;
#pragma unroll 1
                    for (int c = 0; c < 7; ++c) {
                        double *slot = c < 3 ? w.acc + c * w.ld : c < 6 ? w.jerk + (c - 3) * w.ld : w.pot;
                        float2 *kept = reinterpret_cast<float2 *>(slot + w.i0 + k);
                        float2 &h = s_tot[(p * 7 + c) * NT];
                        const float2 was = kt * JT < w.chunk ? make_float2(0.f, 0.f) : *kept;
                        dsf sum{was.x, was.y};
                        ds_acc(sum, dsf{h.x, h.y});
                        if (kt + 1 == ntiles) {
                            h = make_float2(sum.hi, sum.lo);
                        } else {
                            *kept = make_float2(sum.hi, sum.lo);
                            h = make_float2(0.f, 0.f);
                        }
                    }
                }
            }
            __syncthreads();  // the stage and the pair buffer are free
            if (s_abort) {
                if (tid == 0) {
                    drain_ring<NS>(s_full, seq, kt, ntiles);
                    atomicOr(err, DERR_TIMEOUT);
                    items_done(ticket);
                }
                return;
            }
            if (tid == 0 && kt + NS < ntiles) issue(kt + NS);
        }
        seq += (unsigned)ntiles;
        if (w.nsplit <= 1) {
#pragma unroll
            for (int p = 0; p < IPT; ++p) {
                const int k = (warp * IPT + p) * 32 + lane;
                if (k >= w.ni) continue;
                double d[7];
#pragma unroll
                for (int c = 0; c < 7; ++c) {
                    const float2 h = s_tot[(p * 7 + c) * NT];
                    d[c] = ds_to_double(dsf{h.x, h.y});
                }
                write_final(Out3{w.acc, w.jerk, w.pot, w.ld}, w.i0 + k, d, err);
            }
        } else {
            float2 *pp = w.part + (size_t)w.split * 7 * w.ni;
#pragma unroll
            for (int p = 0; p < IPT; ++p) {
                const int k = (warp * IPT + p) * 32 + lane;
                if (k >= w.ni) continue;
#pragma unroll
                for (int c = 0; c < 7; ++c) pp[(size_t)c * w.ni + k] = s_tot[(p * 7 + c) * NT];
            }
        }
    }
    if (tid == 0) items_done(ticket);
}

// ---------------------------------------------------------------------------
// Plans and launchers.
// ---------------------------------------------------------------------------

constexpr int JT32 = 128;    // j-tile of the batched items
constexpr int JT_TILE = 256;  // j-tile of the tile kernel
constexpr int NS32 = 3;

// Runs of the tile kernel: the terms of each half of a packed FP32 sum before the two halves
// are folded into the running totals. Sets of fewer than 4096 i-particles (every due set but the
// largest) took the scalar warp groups once, whose lanes fold after 32 terms, and are to be as
// accurate: the median jerk error for 2516 of 65536 is 1.79e-7 with runs of 16 (64 bits; Plummer
// sphere with a mass spectrum), 1.89e-7 with 32, 2.4e-7 with 128, and 1.89e-7 by the warp
// groups; for 1531 1.80e-7, 1.89e-7, 2.04e-7 (64) and 1.88e-7. The folds cost 132.6 us for 1531
// (32: 125.8, 64: 123.4; the warp groups 184), 203 for 2516 (32: 195, 128: 189; 411). Larger sets
// were taken by this kernel with runs of 128 (one warp row) and are not less accurate.
constexpr int TILE_FINE_NI = 4096;
constexpr int RUN_FINE = 16;
constexpr int RUN_ROWS = 64;   // larger sets, several warp rows
constexpr int RUN_WHOLE = 128;  // larger sets, one warp row: a tile
constexpr int WGRP_NJ = 576;  // most j-particles of the warp groups' sets
constexpr int JT64 = 64;
constexpr int NS64 = 3;

// Warp-group layout (FP32 kind 1): ipt i-particles per warp, nwarp warps per CTA.
static void wgrp_shape(int n_i, ForcePlan &p)
{
    p.ipt = n_i <= 1 ? 1 : 2;
    const int groups = (n_i + p.ipt - 1) / p.ipt;
    const int nwarp = groups <= 1 ? 1 : groups <= 2 ? 2 : groups <= 4 ? 4 : 8;
    p.threads = 32 * nwarp;
}

static long long clampll(long long v, long long lo, long long hi)
{
    return v < lo ? lo : (v > hi ? hi : v);
}

// Whether the split count ns of a plan search is to be tried: not the one before it (last)
// again, and none whose partials do not fit; where the first does not, the most that fit.
bool splits_fit(long long fit, long long &last, long long &ns)
{
    if (ns > fit && last == 0) ns = fit > 1 ? fit : 1;
    if (ns == last || (ns > fit && ns > 1)) return false;
    last = ns;
    return true;
}

// Tiny-set layout (FP32 kind 2): ipt i-particles per pass, jt = j per thread;
// one j-split per CTA of 256 threads.
static void tiny_shape(int n_i, int n_j, ForcePlan &p)
{
    p.kind = 2;
    p.ipt = n_i <= 1 ? 1 : (n_i <= 2 ? 2 : 4);
    p.threads = 256;
    p.jt = n_j >= 256 * 4 * 32 ? 4 : (n_j >= 256 * 2 * 32 ? 2 : 1);
    p.nsplit = (n_j + 256 * p.jt - 1) / (256 * p.jt);
}

// i-particles per thread of the tile kernel: two, but one for the sets that then fill one
// warp column of eight warp rows (16 of 262144: 24.2 against 32.8 us).
static int tile_ipt(int n_i, int nwj) { return nwj == 8 && n_i <= 32 ? 1 : 2; }

ForcePlan plan_force(int variant, int n_i, int n_j, int num_sms, size_t max_part)
{
    ForcePlan p{};
    p.nwj = 1;
    // the most splits whose partials (7 doubles an i-particle each) fit
    const long long fit = (long long)std::min<size_t>(max_part / (7 * (size_t)n_i), 1 << 20);
    if (variant == NB_F64) {
        // j-parallel below 32 i-particles where it is faster: a pass over the j-set for
        // every four (1 us for each pair of a lane, and the lanes' sums), one j per lane while
        // that takes two CTAs per SM at most; the tile kernel takes as long for one
        // i-particle as for 32 (a j on every SM's four warps is 1 us):
        // 4 of 20011 39.5 -> 21.0 us, 32 of 20011 265 -> 52 us (tiles).
        if (n_i <= 32) {
            const long long ns = clampll((n_j + 127LL) / 128, 1, 2LL * num_sms);
            const bool room = ns == 1 || ns <= fit;
            const double passes = (double)((n_i + 3) / 4);
            const double per_sm = (double)((n_j + 128LL * num_sms - 1) / (128LL * num_sms));
            const double pass = per_sm * (double)(n_i < 4 ? n_i : 4) + 3.0;
            if (room && passes * pass <= (double)n_j / (4.0 * num_sms) + 5.0) {
                p.kind = 1;
                p.ipt = n_i <= 1 ? 1 : n_i <= 2 ? 2 : 4;
                p.threads = 128;
                p.nsplit = (int)ns;
                return p;
            }
        }
        // CTAs of 32 i-particles: the split count of least time, an SM's CTAs (at most
        // ceil(CTAs / SMs)) times the units of a split (4 us each: four warps, four j each),
        // with two CTAs per SM or more to cover the FP64 latencies where the j-range allows
        p.kind = 0;
        p.ipt = 1;
        p.threads = 32;
        p.jt = T64_UNIT;
        const long long nblk = (n_i + 31) / 32;
        const long long nunits = (n_j + T64_UNIT - 1) / T64_UNIT;
        double best = 1e300;
        long long last = 0;
        for (const int per_sm : {1, 2, 3, 4, 5, 6, 8, 10, 12, 16, 24, 32, 48}) {
            long long ns = clampll((long long)per_sm * num_sms / nblk, 1,
                                   nunits < 512 ? nunits : 512);
            if (!splits_fit(fit, last, ns)) continue;
            const long long on_sm = (nblk * ns + num_sms - 1) / num_sms;
            const long long units = (nunits + ns - 1) / ns;
            const double t = ((double)on_sm + (on_sm == 1 ? 0.15 : 0.0)) * (double)units * 4.0 +
                             (double)on_sm +
                             (ns > 1 ? 4.0 + 0.02 * (double)ns + 3e-5 * (double)(ns * n_i) : 0.0);
            if (t < best) {
                best = t;
                p.nsplit = (int)ns;
            }
        }
        return p;
    }
    // Tiny sets: the j-set in registers, a pass over them for every four i-particles. The
    // tile kernel costs the same from one i-particle to 32: 4 of 65536 7.1 us against 9.4, 4 of
    // 262144 11.0 against 18.9; a second pass pays on a large j-set only: 8 of 32768 9.4
    // against 7.6, 8 of 65536 9.9 against 9.7, 8 of 262144 14.8 against 18.6.
    if (n_i <= (n_j > 65536 ? 8 : 4)) {
        tiny_shape(n_i, n_j, p);
        if (p.nsplit == 1 || p.nsplit <= fit) return p;
    }
    // A small j-set: the warp groups, whose lanes then add 18 terms at most. The tile kernel's runs, 32
    // with both halves, are longer: its median jerk error for whole systems (60 Plummer spheres each) is 4%
    // larger at 128, 5% at 200 and 256, 4% at 300, 1% at 500, 1% smaller at 600 and 3% at 800; and one
    // launch without partials is as fast (a call for a whole system of 300 51.5 -> 49.9 us, of 512 52.6
    // -> 51.2; for 2000 outside positions on 512 81 -> 86).
    if (n_j <= WGRP_NJ && n_i < TILE_FINE_NI) {
        p.kind = 1;
        wgrp_shape(n_i, p);
        p.nsplit = 1;
        return p;
    }
    // Tiles: the warp rows (8, 4 or 1: 64, 128 or 512 i-particles per CTA) and j-splits of
    // least estimated time. An SM's CTAs share its pipes, so its time is its count of CTAs
    // (at most ceil(CTAs / SMs)) times the tiles of a split times the SM's time for one
    // tile of that shape, a little more where a CTA is left alone at the end (its eight
    // warps do not fill the pipe); the splits' partials cost their traffic. Only split
    // counts that fill a whole number of CTAs per SM are tried. Within 3% of the best of a
    // sweep over shapes and splits at N = 2500 to 262144, almost everywhere. Against the rule
    // before it (warp groups below 4096 i-particles, 16 tiles or more per split above),
    // at N = 65536: N_i = 260 49.8 -> 39.4 us, 1531 184 -> 127 us, 3000 415 -> 234 us.
    p.kind = 0;
    p.threads = 256;
    p.jt = JT_TILE;
    const long long ntiles = (n_j + p.jt - 1) / p.jt;
    double best = 1e300;
    for (const int nwj : {8, 4, 1}) {
        const long long ib = 512 / nwj;
        const long long nblk = (n_i + ib - 1) / ib;
        // microseconds of an SM per 256-record tile (measured with whole waves at N = 65536)
        const double t_tile = nwj == 8 ? 2.57 : (nwj == 4 ? 4.97 : 18.8);
        long long last = 0;
        for (const int per_sm : {1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 14, 16, 20, 24, 32, 40, 48}) {
            long long ns =
                clampll((long long)per_sm * num_sms / nblk, 1, ntiles < 512 ? ntiles : 512);
            if (!splits_fit(fit, last, ns)) continue;
            const long long on_sm = (nblk * ns + num_sms - 1) / num_sms;
            const long long tiles = (ntiles + ns - 1) / ns;
            const double alone = on_sm % 2 ? 0.10 : 0.04;
            const double t = ((double)on_sm + alone) * (double)tiles * t_tile + 0.5 * (double)on_sm +
                             (ns > 1 ? 2.0 + 0.01 * (double)ns + 2e-5 * (double)(ns * n_i) : 0.0);
            if (t < best) {
                best = t;
                p.nwj = nwj;
                p.nsplit = (int)ns;
            }
        }
    }
    p.ipt = tile_ipt(n_i, p.nwj);
    return p;
}

ForcePlan plan_from_entry(const nb_plan &e, int variant, int n_i, int n_j)
{
    ForcePlan p{};
    p.nwj = 1;
    if (e.kind == 2 && variant != NB_F64) {
        tiny_shape(n_i, n_j, p);  // its split count follows from the j per thread
        return p;
    }
    if (e.kind == 1 || e.kind == 2) {
        p.kind = 1;
        if (variant == NB_F64) {
            p.ipt = n_i <= 1 ? 1 : n_i <= 2 ? 2 : 4;
            p.threads = 128;
        } else {
            wgrp_shape(n_i, p);
        }
        p.nsplit = (int)clampll(e.nsplit, 1, n_j);
        return p;
    }
    p.kind = 0;
    if (variant == NB_F64) {
        p.ipt = 1;
        p.threads = 32;  // i-particles of a CTA
        p.jt = T64_UNIT;
    } else {
        p.threads = 256;
        p.jt = JT_TILE;
        p.nwj = (e.nwj == 4 || e.nwj == 8) ? e.nwj : 1;
        p.ipt = tile_ipt(n_i, p.nwj);
    }
    // FP64 units are 16 records: above 2^20 of them there are more than a grid has rows (65535)
    const int ntiles = (n_j + p.jt - 1) / p.jt;
    p.nsplit = (int)clampll(e.nsplit, 1, variant == NB_F64 && ntiles > 65535 ? 65535 : ntiles);
    return p;
}

size_t plan_partial_doubles(const ForcePlan &p, int n_i)
{
    if (p.nsplit <= 1) return 0;
    return (size_t)p.nsplit * 7 * (size_t)n_i;
}

template <class T>
static cudaError_t go_split_sums(const double *part, int n_i, int nsplit, const Out3 &out,
                                 unsigned *err, cudaStream_t st)
{
    const long long outs = 7LL * n_i;
    const T *p = reinterpret_cast<const T *>(part);
    if (nsplit > 8 && outs <= SPLIT_WIDE_OUTS)
        return launch_dependent(k_split_sums<T, 8>, dim3((unsigned)((outs + 31) / 32)), 256, 0, st, p,
                                (long long)n_i, nsplit, n_i, out, err);
    return launch_dependent(k_split_sums<T, 1>, dim3((unsigned)((outs + 255) / 256)), 256, 0, st, p,
                            (long long)n_i, nsplit, n_i, out, err);
}

// Shared memory of the tile kernel: the ring (36 KB), one or two transposed tiles
// (12 KB each) and the running totals of two i-particles per thread (28 KB).
template <int NT, int NWJ>
static constexpr size_t tile_smem()
{
    return (size_t)(NS32 + (tile_ahead(NWJ) ? 2 : 1)) * JT_TILE * DS_REC * sizeof(float4) +
           (size_t)NT * 14 * sizeof(float2);
}

template <int VAR, int IPT, int NWI, int NWJ, int RUN>
static cudaError_t go_tile32(const JSet &js, const ISet &is, float eps2f, int nsplit,
                             double *part, Out3 out, unsigned *err,
                             cudaStream_t st)
{
    constexpr auto kern = k_force_tile32<VAR, IPT, NWI, NWJ, JT_TILE, NS32, RUN>;
    constexpr int NT = 32 * NWI * NWJ;
    constexpr int IB = 32 * NWI * IPT;
    const size_t smem = tile_smem<NT, NWJ>();
    const cudaError_t attr = allow_smem<kern>(smem);
    if (attr != cudaSuccess) return attr;
    const int ntiles = (js.n + JT_TILE - 1) / JT_TILE;
    dim3 grid((is.n + IB - 1) / IB, nsplit);
    const cudaError_t e = launch_dependent(kern, grid, NT, smem, st, js.rec32, js.n, is, eps2f,
                                           ntiles, part, (long long)is.n, out, err);
    if (e != cudaSuccess || nsplit <= 1) return e;
    return go_split_sums<float2>(part, is.n, nsplit, out, err, st);
}

template <int VAR, int IPT, int NWARP>
static cudaError_t go_wgrp32(const JSet &js, const ISet &is, float eps2f, int nsplit,
                             double *part, unsigned *cnt, Out3 out, unsigned *err,
                             cudaStream_t st)
{
    const int groups = (is.n + IPT - 1) / IPT;
    dim3 grid((groups + NWARP - 1) / NWARP, nsplit);
    k_force_wgrp32<VAR, IPT, NWARP><<<grid, 32 * NWARP, 0, st>>>(js.rec32, js.n, is, eps2f, part,
                                                                  is.n, cnt, out, err);
    return cudaGetLastError();
}

template <int VAR, int IPT, int JPT>
static cudaError_t go_tiny32(const JSet &js, const ISet &is, float eps2f, double *part,
                             unsigned *cnt, Out3 out, unsigned *err, cudaStream_t st)
{
    const int g = (js.n + 256 * JPT - 1) / (256 * JPT);
    return launch_dependent(k_force_tiny32<VAR, IPT, JPT>, dim3(g), 256, 0, st, js.rec32, js.n, is,
                            eps2f, part, (long long)is.n, cnt, out, err);
}

template <int VAR, int IPT>
static cudaError_t go_tiny32_j(int jpt, const JSet &js, const ISet &is, float eps2f,
                               double *part, unsigned *cnt, Out3 out, unsigned *err,
                               cudaStream_t st)
{
    switch (jpt) {
    case 1: return go_tiny32<VAR, IPT, 1>(js, is, eps2f, part, cnt, out, err, st);
    case 2: return go_tiny32<VAR, IPT, 2>(js, is, eps2f, part, cnt, out, err, st);
    default: return go_tiny32<VAR, IPT, 4>(js, is, eps2f, part, cnt, out, err, st);
    }
}

static cudaError_t go_tile64(const JSet &js, const ISet &is, double eps2, int nsplit, double *part,
                             Out3 out, unsigned *err, cudaStream_t st)
{
    const size_t smem = (size_t)NS64 * 7 * JT64 * sizeof(double);  // 10.5 KB
    const int nunits = (js.n + T64_UNIT - 1) / T64_UNIT;
    const cudaError_t e =
        launch_dependent(k_force_tile64<JT64, NS64>, dim3((is.n + 31) / 32, nsplit), 32 * T64_ROWS,
                         smem, st, js, is, eps2, nunits, part, (long long)is.n, out, err);
    if (e != cudaSuccess || nsplit <= 1) return e;
    return go_split_sums<double>(part, is.n, nsplit, out, err, st);
}

template <int VAR>
static cudaError_t dispatch32(const ForcePlan &p, const JSet &js, const ISet &is, float eps2f,
                              double *part, unsigned *cnt, Out3 out, unsigned *err,
                              cudaStream_t st)
{
    if (p.kind == 2) {
        switch (p.ipt) {
        case 1: return go_tiny32_j<VAR, 1>(p.jt, js, is, eps2f, part, cnt, out, err, st);
        case 2: return go_tiny32_j<VAR, 2>(p.jt, js, is, eps2f, part, cnt, out, err, st);
        default: return go_tiny32_j<VAR, 4>(p.jt, js, is, eps2f, part, cnt, out, err, st);
        }
    }
    if (p.kind == 1) {
        const int nw = p.threads / 32;
        if (p.ipt == 1) return go_wgrp32<VAR, 1, 1>(js, is, eps2f, p.nsplit, part, cnt, out, err, st);
        switch (nw) {
        case 1: return go_wgrp32<VAR, 2, 1>(js, is, eps2f, p.nsplit, part, cnt, out, err, st);
        case 2: return go_wgrp32<VAR, 2, 2>(js, is, eps2f, p.nsplit, part, cnt, out, err, st);
        case 4: return go_wgrp32<VAR, 2, 4>(js, is, eps2f, p.nsplit, part, cnt, out, err, st);
        default: return go_wgrp32<VAR, 2, 8>(js, is, eps2f, p.nsplit, part, cnt, out, err, st);
        }
    }
    const bool fine = is.n < TILE_FINE_NI;
    const auto go = p.nwj == 1   ? (fine ? go_tile32<VAR, 2, 8, 1, RUN_FINE> : go_tile32<VAR, 2, 8, 1, RUN_WHOLE>)
                    : p.nwj == 4 ? (fine ? go_tile32<VAR, 2, 2, 4, RUN_FINE> : go_tile32<VAR, 2, 2, 4, RUN_ROWS>)
                    : p.ipt == 1 ? go_tile32<VAR, 1, 1, 8, RUN_FINE>
                                 : (fine ? go_tile32<VAR, 2, 1, 8, RUN_FINE> : go_tile32<VAR, 2, 1, 8, RUN_ROWS>);
    return go(js, is, eps2f, p.nsplit, part, out, err, st);
}

cudaError_t warm_force_jmode64(cudaStream_t st)
{
    cudaFuncAttributes fa;
    cudaError_t e;
    if ((e = cudaFuncGetAttributes(&fa, k_force_jmode64<1, 128>)) != cudaSuccess ||
        (e = cudaFuncGetAttributes(&fa, k_force_jmode64<2, 128>)) != cudaSuccess ||
        (e = cudaFuncGetAttributes(&fa, k_force_jmode64<4, 128>)) != cudaSuccess)
        return e;
    // an empty i-set: the i-loop does not run and one CTA writes nothing
    const JSet js{};
    ISet is{};
    is.member = true;
    k_force_jmode64<1, 128><<<1, 128, 0, st>>>(js, is, 0.0, nullptr, 0, nullptr, Out3{}, nullptr);
    k_force_jmode64<2, 128><<<1, 128, 0, st>>>(js, is, 0.0, nullptr, 0, nullptr, Out3{}, nullptr);
    k_force_jmode64<4, 128><<<1, 128, 0, st>>>(js, is, 0.0, nullptr, 0, nullptr, Out3{}, nullptr);
    return cudaGetLastError();
}

static cudaError_t dispatch64(const ForcePlan &p, const JSet &js, const ISet &is, double eps2,
                              double *part, unsigned *cnt, Out3 out, unsigned *err,
                              cudaStream_t st)
{
    if (p.kind != 1) return go_tile64(js, is, eps2, p.nsplit, part, out, err, st);
    const auto kern = p.ipt == 1   ? k_force_jmode64<1, 128>
                      : p.ipt == 2 ? k_force_jmode64<2, 128>
                                   : k_force_jmode64<4, 128>;
    const cudaError_t e = launch_dependent(kern, dim3(p.nsplit), 128, 0, st, js, is, eps2, part,
                                           (long long)is.n, cnt, out, err);
    if (e != cudaSuccess || p.nsplit <= 1 || cnt) return e;
    return go_split_sums<double>(part, is.n, p.nsplit, out, err, st);
}

// Shared memory of the batched kernel: the ring (18 KB), the transposed tile (6 KB)
// and the running totals of two i-particles per thread.
static size_t items_smem(int threads)
{
    return (size_t)(NS32 + 1) * JT32 * DS_REC * sizeof(float4) +
           (size_t)threads * 14 * sizeof(float2);
}

template <int VAR, int NT, bool CHUNKS>
static cudaError_t go_items(const WorkItem *items, int nitems, int grid, unsigned *ticket,
                            cudaStream_t st)
{
    constexpr auto kern = k_force_items32<VAR, 2, NT, JT32, NS32, CHUNKS>;
    const size_t smem = items_smem(NT);
    const cudaError_t attr = allow_smem<kern>(smem);
    if (attr != cudaSuccess) return attr;
    kern<<<grid, NT, smem, st>>>(items, nitems, ticket);
    return cudaGetLastError();
}

template <int VAR, bool CHUNKS>
static cudaError_t go_items_of(int threads, const WorkItem *items, int nitems, int grid,
                               unsigned *ticket, cudaStream_t st)
{
    switch (threads) {
    case 64: return go_items<VAR, 64, CHUNKS>(items, nitems, grid, ticket, st);
    case 128: return go_items<VAR, 128, CHUNKS>(items, nitems, grid, ticket, st);
    default: return go_items<VAR, 256, CHUNKS>(items, nitems, grid, ticket, st);
    }
}

cudaError_t launch_force_items(int variant, int threads, const WorkItem *items, int nitems,
                               int grid, unsigned *ticket, cudaStream_t st, bool chunks)
{
    if (nitems <= 0) return cudaSuccess;
    const auto go = variant == NB_F32DS
                        ? (chunks ? go_items_of<NB_F32DS, true> : go_items_of<NB_F32DS, false>)
                        : (chunks ? go_items_of<NB_F32, true> : go_items_of<NB_F32, false>);
    return go(threads, items, nitems, grid, ticket, st);
}

cudaError_t launch_force_items_jpar(int variant, const WorkItem *items, int nitems, int grid,
                                    cudaStream_t st)
{
    if (nitems <= 0) return cudaSuccess;
    if (variant == NB_F32DS)
        k_force_items_jpar32<NB_F32DS, JPAR_THREADS><<<grid, JPAR_THREADS, 0, st>>>(items, nitems);
    else
        k_force_items_jpar32<NB_F32, JPAR_THREADS><<<grid, JPAR_THREADS, 0, st>>>(items, nitems);
    return cudaGetLastError();
}

cudaError_t launch_split_reduce(const SplitGroup *groups, int ngroups, int grid,
                                cudaStream_t st)
{
    if (ngroups <= 0) return cudaSuccess;
    k_split_reduce<<<grid, 256, 0, st>>>(groups, ngroups);
    return cudaGetLastError();
}

int jpar_blocks_per_sm(int variant)
{
    int nb = 0;
    const cudaError_t e =
        variant == NB_F32DS
            ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                  &nb, k_force_items_jpar32<NB_F32DS, JPAR_THREADS>, JPAR_THREADS, 0)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                  &nb, k_force_items_jpar32<NB_F32, JPAR_THREADS>, JPAR_THREADS, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return nb > 0 ? nb : 1;
}

// Self-check of the bounded copy wait: an mbarrier that no copy or arrival
// completes; the wait gives up after limit_ns and reports DERR_TIMEOUT.
__global__ void k_selftest_mbar(unsigned *err, unsigned long long limit_ns)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait(&bar, 0u, limit_ns)) atomicOr(err, DERR_TIMEOUT);
}

cudaError_t launch_selftest_mbar(unsigned *err, unsigned long long limit_ns, cudaStream_t st)
{
    k_selftest_mbar<<<1, 32, 0, st>>>(err, limit_ns);
    return cudaGetLastError();
}

template <int VAR, int NWI, int NWJ>
static int tile_occ()
{
    constexpr int NT = 32 * NWI * NWJ;
    const size_t smem = tile_smem<NT, NWJ>();
    constexpr auto kern = k_force_tile32<VAR, 2, NWI, NWJ, JT_TILE, NS32, NWJ == 1 ? RUN_WHOLE : RUN_ROWS>;
    int nb = 0;
    if (allow_smem<kern>(smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, NT, smem) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return nb > 0 ? nb : 1;
}

int tile_blocks_per_sm(int variant, int nwj)
{
    if (variant == NB_F32DS)
        return nwj == 1 ? tile_occ<NB_F32DS, 8, 1>()
                        : (nwj == 4 ? tile_occ<NB_F32DS, 2, 4>() : tile_occ<NB_F32DS, 1, 8>());
    return nwj == 1 ? tile_occ<NB_F32, 8, 1>()
                    : (nwj == 4 ? tile_occ<NB_F32, 2, 4>() : tile_occ<NB_F32, 1, 8>());
}

template <int VAR, int NT>
static int items_occ()
{
    constexpr auto kern = k_force_items32<VAR, 2, NT, JT32, NS32, false>;
    const size_t smem = items_smem(NT);
    int nb = 0;
    if (allow_smem<kern>(smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, NT, smem) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return nb > 0 ? nb : 1;
}

int batch_blocks_per_sm(int variant, int threads)
{
    if (variant == NB_F32DS)
        return threads == 64    ? items_occ<NB_F32DS, 64>()
               : threads == 128 ? items_occ<NB_F32DS, 128>()
                                : items_occ<NB_F32DS, 256>();
    return threads == 64    ? items_occ<NB_F32, 64>()
           : threads == 128 ? items_occ<NB_F32, 128>()
                            : items_occ<NB_F32, 256>();
}

size_t plan_counters(const ForcePlan &p, int n_i)
{
    if (p.nsplit <= 1 || p.kind != 1) return 1;
    const long long ib = (long long)(p.threads / 32) * p.ipt;  // FP32 warp groups (FP64: one)
    return (size_t)((n_i + ib - 1) / ib);
}

cudaError_t launch_force(int variant, const ForcePlan &plan, const JSet &js, const ISet &is,
                         double eps2, double *part, unsigned *counters, Out3 out, unsigned *err,
                         cudaStream_t st, cudaEvent_t *ev)
{
    if (is.n <= 0) return cudaSuccess;
    const float eps2f = (float)eps2;
    cudaError_t e;
    if (ev) cudaEventRecord(ev[0], st);
    if (variant == NB_F64)
        e = dispatch64(plan, js, is, eps2, part, counters, out, err, st);
    else if (variant == NB_F32DS)
        e = dispatch32<NB_F32DS>(plan, js, is, eps2f, part, counters, out, err, st);
    else
        e = dispatch32<NB_F32>(plan, js, is, eps2f, part, counters, out, err, st);
    if (ev) cudaEventRecord(ev[1], st);
    return e;
}

}  // namespace nb
