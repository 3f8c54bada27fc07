// reduce.cuh -- reductions over the aggregates of each pile.
//
// Opening (after the drift): mass, COM and mean velocity, which become the
// next step's frame, and the planet's drift.  Nothing before the closing pass
// reads them, so they ride along: blocks of k_lists sum the chunks of
// kAggChunk aggregates beside the gather, blocks of the contact pass add each
// pile's chunk sums.  Closing: the planet's reaction, the next frame, counters
// and flags, done by the last of the pile's blocks of k_agg_end (counted in
// pile_arrive, which goes back to zero).  Every sum has a fixed
// order -- virtual thread t of 128 adds t, t + 128, ... in order, then each
// virtual warp's lanes by a fixed tree, then the warps -- so no result depends
// on which block came last or on how many threads a block has.
//
// As kernels of their own the two reductions were 20 us of a 384 us step on
// the 1M lattice and 13 and 6 us (ncu) of a 1,000-sphere step.  Finishing the
// opening sums at the end of k_agg_begin instead, by its last blocks, put
// their chain of fences, atomics and FP64 divisions on the step's: 96 us per
// step of 7,466 spheres with a planet, at the end of k_lists 83, as it is 73 (60
// with the other kernels as they are now).
#pragma once

#include "dem_internal.h"
#include "devmath.cuh"

namespace dem {

__device__ __forceinline__ bool pile_active(const Arrays &a, int p)
{
    return a.enabled[p] != 0 && a.pd[p].failed == 0;
}

// Pile of sphere or aggregate i: in a world of one pile no load that all
// others wait for (1,048,576 spheres: k_lists 51.1 -> 47.1 us, contact pass
// 200.7 -> 196.6 us, step 334 -> 327.6 us).
__device__ __forceinline__ int sphere_pile(const Arrays &a, const Sizes &z, int64_t i)
{
    return z.P == 1 ? 0 : a.sph_pile[i];
}
__device__ __forceinline__ int aggregate_pile(const Arrays &a, const Sizes &z, int64_t g)
{
    return z.P == 1 ? 0 : a.agg_pile[g];
}

constexpr int kSumThreads = 128;   // virtual threads of a sum
static_assert(kAggChunk % kSumThreads == 0, "whole rounds per chunk");

__device__ __forceinline__ double add2(double x, double y) { return x + y; }
__device__ __forceinline__ ff add2(ff x, ff y) { return ff_add(x, y); }
__device__ __forceinline__ double to_double(double x) { return x; }
__device__ __forceinline__ double to_double(ff x) { return ff_value(x); }
__device__ __forceinline__ double shfl_down(double x, int o) { return __shfl_down_sync(0xffffffffu, x, o); }
__device__ __forceinline__ ff shfl_down(ff x, int o)
{
    return ff{__shfl_down_sync(0xffffffffu, x.hi, o), __shfl_down_sync(0xffffffffu, x.lo, o)};
}

// Sum of NC values over kSumThreads virtual threads, NT real ones (a multiple
// of 32, at most kSumThreads): term(t, v) adds virtual thread t's values to v
// (zeros).  The sum is thread 0's; ws: shared scratch, 4 NC values.
template <int NC, int NT, typename T, typename Fn>
__device__ __forceinline__ void block_sum(T (&out)[NC], T *ws, Fn term)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int w = threadIdx.x >> 5; w < kSumThreads / 32; w += NT / 32) {
        T v[NC] = {};
        term(32 * w + lane, v);
        for (int o = 16; o > 0; o >>= 1)
            for (int k = 0; k < NC; ++k) v[k] = add2(v[k], shfl_down(v[k], o));
        if (lane == 0)
            for (int k = 0; k < NC; ++k) ws[NC * w + k] = v[k];
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int k = 0; k < NC; ++k)
            out[k] = add2(add2(ws[k], ws[NC + k]), add2(ws[2 * NC + k], ws[3 * NC + k]));
}

// Aggregates [beg, end) of chunk ch.
__device__ __forceinline__ void chunk_range(const Arrays &a, int64_t ch, int p, int64_t &beg, int64_t &end)
{
    const PileStatic &S = a.ps[p];
    beg = S.a0 + (ch - S.ch0) * kAggChunk;
    end = min(beg + kAggChunk, S.a0 + S.na);
}

// Opening: sums of M, M r, M v of chunk ch, from the drifted state.
// (Mixed path: float-float on the FP32 units, M as FP32: the sums fix the
// frame origin and velocity, whose exact values enter no result, since
// positions and velocities are taken relative to them exactly.)
template <bool FP64, int NT>
__device__ __forceinline__ void open_chunk(const Arrays &a, int64_t ch)
{
    const int p = a.chunk_pile[ch];
    if (!pile_active(a, p)) return;
    int64_t beg, end;
    chunk_range(a, ch, p, beg, end);
    double *out = a.chunk_part + ch * kPartialDoubles;
    __shared__ double ws[28];
    __syncthreads();   // ws of the block's previous chunk
    if constexpr (FP64) {
        double s[7];
        block_sum<7, NT>(s, ws, [&](int t, double (&v)[7]) {
            for (int64_t g = beg + t; g < end; g += kSumThreads) {
                const double M = a.M[g];
                v[0] += M;
                for (int c = 0; c < 3; ++c) {
                    v[1 + c] += M * a.r[3 * g + c];
                    v[4 + c] += M * a.v[3 * g + c];
                }
            }
        });
        if (threadIdx.x == 0)
            for (int k = 0; k < 7; ++k) out[k] = s[k];
    } else {
        ff s[7];
        block_sum<7, NT>(s, (ff *)ws, [&](int t, ff (&v)[7]) {
            constexpr int kPer = kAggChunk / kSumThreads;
            float M[kPer];
            ff rv[kPer][6];
#pragma unroll
            for (int q = 0; q < kPer; ++q) {   // loaded together, added in order
                const int64_t g = min(beg + t + kSumThreads * q, end - 1);
                M[q] = (float)a.M[g];
                for (int c = 0; c < 3; ++c) {
                    rv[q][c] = ldff(a.r + 3 * g + c);
                    rv[q][3 + c] = ldff(a.v + 3 * g + c);
                }
            }
#pragma unroll
            for (int q = 0; q < kPer; ++q) {
                if (beg + t + kSumThreads * q >= end) break;
                v[0] = ff_addf(v[0], M[q]);
                for (int c = 0; c < 6; ++c) v[1 + c] = ff_add(v[1 + c], ff_mul(ff{M[q], 0.f}, rv[q][c]));
            }
        });
        if (threadIdx.x == 0)
            for (int k = 0; k < 7; ++k) out[k] = ff_value(s[k]);
    }
}

// Sums of the pile's chunk records (the first NC values), in thread 0.
template <int NC, int NT>
__device__ __forceinline__ void pile_sum(const Arrays &a, const PileStatic &S, double (&s)[NC], double *ws)
{
    block_sum<NC, NT>(s, ws, [&](int t, double (&v)[NC]) {
        for (int64_t c = S.ch0 + t; c < S.ch0 + S.nch; c += kSumThreads)
            for (int k = 0; k < NC; ++k) v[k] += __ldcg(a.chunk_part + c * kPartialDoubles + k);
    });
}

// Opening: COM and mean velocity of pile p from its chunk sums, and the
// planet's kick (with the stored acceleration) and drift; three threads take
// a component each.
template <int NT>
__device__ __forceinline__ void open_pile(const Arrays &a, int p)
{
    if (!pile_active(a, p)) return;
    const PileStatic &S = a.ps[p];
    PileDyn &D = a.pd[p];
    __shared__ double ws[28], tot[7];
    double s[7];
    pile_sum<7, NT>(a, S, s, ws);
    if (threadIdx.x == 0)
        for (int k = 0; k < 7; ++k) tot[k] = s[k];
    __syncthreads();
    const int c = threadIdx.x;
    if (c >= 3) return;
    const double rc = tot[1 + c] / tot[0], vc = tot[4 + c] / tot[0];
    D.Rc[c] = rc;
    D.Vc[c] = vc;
    const ff rf = ff_of(rc);
    D.Rcf[c] = make_float2(rf.hi, rf.lo);
    if (S.ext_mass > 0) {
        const double h = S.h;
        D.P_vel[c] += 0.5 * h * D.P_acc[c];
        D.P_pos[c] += h * D.P_vel[c];
    }
}

// Count one of `n` arrivals at `counter`; true in every thread of the last
// one's block (with the others' writes visible, in L2).
__device__ __forceinline__ bool last_to_arrive(int32_t *counter, int n)
{
    __shared__ int last;
    __syncthreads();   // the block's writes and flags
    if (n == 1) return true;
    if (threadIdx.x == 0) {
        __threadfence();   // they are visible before this block is counted
        last = atomicAdd(counter, 1) == n - 1;
        if (last) *counter = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last != 0;
}

// Closing reduction, called by every block (NT threads, NT consecutive
// aggregates of chunk ch of pile p each) after its stores; Fe: the planet's
// force on the thread's aggregate (zeros where there is none).  Each warp's 32
// aggregates are summed by a fixed tree, and the pile's last block adds the
// warps' sums.
template <int NT, typename T>
__device__ __forceinline__ void close_pile(const Arrays &a, int64_t ch, int p, T (&Fe)[3])
{
    const PileStatic &S = a.ps[p];
    PileDyn &D = a.pd[p];
    const bool planet = S.ext_mass > 0;
    __shared__ double ws[12], tot[3];
    if (planet) {
        for (int o = 16; o > 0; o >>= 1)
            for (int k = 0; k < 3; ++k) Fe[k] = add2(Fe[k], shfl_down(Fe[k], o));
        if ((threadIdx.x & 31) == 0) {
            const int w = (int)(blockIdx.x % (kAggChunk / NT)) * (NT / 32) + (threadIdx.x >> 5);
            for (int k = 0; k < 3; ++k) a.warp_part[(ch * kChunkWarps + w) * 3 + k] = to_double(Fe[k]);
        }
    }
    if (!last_to_arrive(a.pile_arrive + p, (int)((S.na + NT - 1) / NT))) return;
    if (planet) {
        double s[3];
        const int64_t w0 = S.ch0 * kChunkWarps, nw = (S.na + 31) / 32;
        block_sum<3, NT>(s, ws, [&](int t, double (&v)[3]) {
            for (int64_t w = t; w < nw; w += kSumThreads)
                for (int k = 0; k < 3; ++k) v[k] += __ldcg(a.warp_part + (w0 + w) * 3 + k);
        });
        if (threadIdx.x == 0)
            for (int k = 0; k < 3; ++k) tot[k] = s[k];
        __syncthreads();
    }
    const int c = threadIdx.x;
    const double h = S.h;
    if (c < 3) {
        if (planet) {   // reaction of the pile, closing kick
            D.P_acc[c] = -tot[c] / S.ext_mass;
            D.P_vel[c] += 0.5 * h * D.P_acc[c];
        }
        D.O[c] = D.Rc[c];
        D.V[c] = D.Vc[c];
        D.hVf[c] = (float)(h * D.Vc[c]);
        D.Of[c] = D.Rcf[c];
        const ff vc = ff_of(D.Vc[c]);
        D.Vf[c] = make_float2(vc.hi, vc.lo);
    } else if (c == NT - 1) {
        D.steps += 1;
        D.parity ^= 1;
        if (__ldcg(&D.flags) & (DEM_FLAG_SLOTS | DEM_FLAG_NONFINITE | DEM_FLAG_GRAV_RANGE)) D.failed = 1;
        if (D.rebuild) {
            D.rebuilds += 1;
            D.cpar ^= 1;   // the lists built this step become the current ones
        }
        D.rebuilt_prev = D.rebuild;
        D.rebuild = S.skin <= 0.0 ? 1 : 0;
    }
}

}  // namespace dem
