// kernels_lists.cu -- from the aggregates' records to what the contact pass
// and gravity read: sphere centres, predicted velocities and spins in sorted
// order and, in the steps that rebuild them, the cell sort and the candidate
// lists.
//
// One kernel, k_lists.  In most steps no pile rebuilds and it only expands
// and gathers the spheres (HBM-bound: about 250 B per sphere).  In a step in
// which some pile does (its aggregates may have moved half the skin, or the
// host wrote its state), the same launch also sorts that pile's spheres into
// cells and builds its lists, in phases, each of which starts when all of the
// one before is done.  As eleven kernels of their own -- clear, keys, three
// scans, scatter, order, count, scan, fill, link -- the rebuild phases cost a
// launch each in every step, although they returned at once in all but one of
// several hundred.  A step of 1,000 spheres went from 50.8 to 33.3 us with this
// launch and the reductions folded into it and its neighbours (19 kernels ->
// 5; 31.2 with its programmatic launch), of 7,466 spheres with a planet from
// 98.7 to 61 us.
//
// The phases' order (run_phase).  A phase is cut into items, which the blocks
// draw from a counter; a block that finds none left waits until all drawn ones
// are done.  A block never waits while it holds an item, so every item that was
// drawn gets done, and the block that does a phase's last one goes on to the
// next whatever the others do.  Nothing therefore depends on how many blocks
// run at the same time (an ordinary launch: the grid need not be resident, and
// kernels of other streams take their share of the chip), nor on how long a
// wait lasts: it is bounded, and a block that gives up leaves the rest of the
// rebuild to those still working.
//
// Cells: a wrapped uniform grid numbered brick by brick (cell_id); a counting
// sort, each cell ordered by home index, so the order of neighbours is
// deterministic.
//
// Candidate lists: every sphere lists the spheres of other aggregates whose
// centres are closer than the radii sum plus the skin, in the order of their
// home indices; every entry then gets the position of the same pair in the
// partner's list, the entries whose sphere owns the pair (the lower home
// index) are marked, and the contact history is carried over by partner.  The
// candidate test is exact and symmetric, so both spheres of a pair always
// list each other.
#include "dem_internal.h"
#include "devmath.cuh"
#include "expand.cuh"
#include "launch.cuh"
#include "reduce.cuh"

namespace dem {

constexpr int kLB = kCTile;   // threads per block

template <bool FP64> struct HistT;
template <> struct HistT<false> { typedef float4 H; };
template <> struct HistT<true> { typedef dbl4 H; };

__device__ __forceinline__ bool pile_rebuilds(const Arrays &a, int p)
{
    return pile_active(a, p) && a.pd[p].rebuild;
}

// Whether any pile rebuilds this step (the block's threads read the piles'
// flags together; the same answer in every block).
__device__ __forceinline__ bool any_rebuild(const Arrays &a, const Sizes &z)
{
    int mine = 0;
    for (int p = threadIdx.x; p < z.P; p += blockDim.x) mine |= pile_rebuilds(a, p) ? 1 : 0;
    return __syncthreads_or(mine) != 0;
}

// Phases of a rebuild, in order, and the words of Arrays::lbar: per phase the
// next item and the items done, then the blocks that are done with the launch.
enum { kKeys, kScanTiles, kScanPiles, kScanCells, kScatter, kPlace, kCount, kListScan, kFill, kLink, kPhases };
static_assert(2 * kPhases < kListWords, "the words of all phases and the last one");

// Count n items at `done`, with the block's writes before it (those of the
// threads it has synchronised with) visible to whoever sees the count.
__device__ __forceinline__ void count_done(unsigned *done, unsigned n)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(done), "r"(n) : "memory");
}

// Phase ph (see the file comment): f(item), by the whole block, for the items
// of [0, items) that this block draws, then the wait for those of the others.
// False if the wait ran out.  sh: a shared word.  Where there are several items
// for every block, a draw takes some together in the phases whose items are
// alike and short; a tile's candidates take long and unlike times and are drawn
// one by one.  Measured, us of a step that rebuilds, with twelve phases, a fixed
// share of the items for every block, barriers over a resident grid and cells
// sorted by a thread each -> this, ten phases: 1,000 spheres 105 -> 103, 100,000
// 268 -> 247, 1,048,576 1,710 -> 1,726 (always one a draw 1,747, several in every
// phase 1,911), 256 piles of 1.1 million a few of which rebuild 3,250 -> 3,265.
// The next item drawn while one is worked on: 163 at 1,000.
template <typename Fn>
__device__ __forceinline__ bool run_phase(const Arrays &a, const Sizes &z, int ph, int64_t items, unsigned *sh, Fn f)
{
    unsigned *next = a.lbar + 2 * ph, *done = next + 1;
    const unsigned n = (unsigned)items, per = ph <= kPlace ? max(1u, n / (2 * gridDim.x)) : 1u;
    for (unsigned held = 0;;) {
        __syncthreads();   // the block has done what it held (and read *sh)
        if (threadIdx.x == 0) {
            if (held) count_done(done, held);
            *sh = atomicAdd(next, per);
        }
        __syncthreads();
        const unsigned beg = *sh;
        if (beg >= n) break;
        const unsigned end = min(beg + per, n);
        for (unsigned i = beg; i < end; ++i) f((int64_t)i);
        held = end - beg;
    }
    int ok = 1;
    if (threadIdx.x == 0) {
        const volatile unsigned *w = done;
        for (int it = 0; *w < n; ++it) {
            if (it >= z.lwait) {
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

// The last block of a launch that rebuilds puts the words back to zero.
__device__ __forceinline__ void phases_done(const Arrays &a)
{
    __syncthreads();
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicAdd(a.lbar + kListWords - 1, 1u) == gridDim.x - 1)
        for (int k = 0; k < kListWords; ++k) a.lbar[k] = 0;
}

// Exclusive prefix sum over the block's kLB threads; *total gets the sum.
template <typename T>
__device__ __forceinline__ T block_scan(T v, T *ws, T *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();   // ws is free
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    T before = 0, all = 0;
    for (int k = 0; k < kLB / 32; ++k) {
        if (k < wid) before += ws[k];
        all += ws[k];
    }
    *total = all;
    return before + x - v;
}

// ---------------------------------------------------------------- cells
__device__ __forceinline__ int wrapc(int c, int n) { return c < 0 ? c + n : (c >= n ? c - n : c); }

__device__ __forceinline__ int cellc_f(float x, float inv_cell, int n)
{
    float f = floorf(__fmul_rn(x, inv_cell));
    f = fminf(fmaxf(f, -1.0e9f), 1.0e9f);
    int m = ((int)f) % n;
    return m < 0 ? m + n : m;
}

__device__ __forceinline__ int cellc_d(double x, double inv_cell, int n)
{
    double f = floor(__dmul_rn(x, inv_cell));
    f = fmin(fmax(f, -1.0e9), 1.0e9);
    int m = ((int)f) % n;
    return m < 0 ? m + n : m;
}


// Pile of scan tile t (tiles of kScanTile cells never straddle piles).
__device__ __forceinline__ int tile_pile(const Arrays &a, const Sizes &z, int64_t t)
{
    int lo = 0, hi = (int)z.P - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (a.ps[mid].t0 <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// f(i, p) for the spheres of rebuilding piles among the kLB of an item (index
// i in all piles)
template <typename Fn>
__device__ __forceinline__ void rebuilding_spheres(const Arrays &a, const Sizes &z, int64_t item, Fn f)
{
    const int64_t i = item * kLB + threadIdx.x;
    if (i >= z.N) return;
    const int p = sphere_pile(a, z, i);
    if (pile_rebuilds(a, p)) f(i, p);
}

// New neighbour-list reference of a chunk's aggregates (as the test in the
// drift forms it).
template <bool FP64>
__device__ __forceinline__ void reference_chunk(const Arrays &a, int64_t ch)
{
    const int p = a.chunk_pile[ch];
    if (!pile_rebuilds(a, p)) return;
    const PileStatic &S = a.ps[p];
    const PileDyn &D = a.pd[p];
    const int64_t beg = S.a0 + (ch - S.ch0) * kAggChunk, end = min(beg + kAggChunk, S.a0 + S.na);
    for (int64_t g = beg + threadIdx.x; g < end; g += kLB) {
        float *ar = a.aref + 8 * g;
        if constexpr (FP64) {
            for (int c = 0; c < 3; ++c) ar[c] = (float)(a.r[3 * g + c] - D.O[c] - S.h * D.V[c]);
            for (int c = 0; c < 4; ++c) ar[3 + c] = (float)a.q[4 * g + c];
        } else {
            for (int c = 0; c < 3; ++c) ar[c] = ff_sub(ldff(a.r + 3 * g + c), ff_of2(D.Of[c])).hi - D.hVf[c];
            for (int c = 0; c < 4; ++c) ar[3 + c] = ldff(a.q + 4 * g + c).hi;
        }
    }
}

// Zero cell counts of scan tile t, for the next rebuild.
__device__ __forceinline__ void clear_tile(const Arrays &a, const Sizes &z, int64_t t)
{
    if (!pile_rebuilds(a, tile_pile(a, z, t))) return;
    int4 *c = (int4 *)(a.ccount + t * kScanTile);
    for (int k = threadIdx.x; k < kScanTile / 4; k += kLB) c[k] = make_int4(0, 0, 0, 0);
}

// Cell key and rank among the spheres counted into the cell (the rank waits
// in sagg, which the gather writes anew).
template <bool FP64>
__device__ __forceinline__ void key_sphere(const Arrays &a, int64_t i, int p)
{
    const PileStatic &S = a.ps[p];
    const int64_t g = S.a0 + a.sph_agg[i];
    int cx, cy, cz;
    if constexpr (FP64) {
        const double3 pos = expand_64(a.rec64[g], a.b64 + 3 * i);
        cx = cellc_d(pos.x, S.inv_cell, S.nx);
        cy = cellc_d(pos.y, S.inv_cell, S.ny);
        cz = cellc_d(pos.z, S.inv_cell, S.nz);
    } else {
        ff px, py, pz;
        expand_mixed(a.rec32[g], a.bh[i], a.bl[i], px, py, pz);
        const float ic = (float)S.inv_cell;
        cx = cellc_f(px.hi, ic, S.nx);
        cy = cellc_f(py.hi, ic, S.ny);
        cz = cellc_f(pz.hi, ic, S.nz);
    }
    const int key = (int)cell_id(cx, cy, cz, S.nx, S.ny);
    a.key[i] = key;
    a.sagg[i] = atomicAdd(a.ccount + S.c0 + key, 1);
}

// Sum of scan tile t's cell counts.
__device__ __forceinline__ void sum_tile(const Arrays &a, const Sizes &z, int64_t t, int *ws)
{
    if (!pile_rebuilds(a, tile_pile(a, z, t))) return;
    const int4 *c = (const int4 *)(a.ccount + t * kScanTile);
    int s = 0, tot;
    for (int k = threadIdx.x; k < kScanTile / 4; k += kLB) {
        const int4 v = c[k];
        s += (v.x + v.y) + (v.z + v.w);
    }
    block_scan(s, ws, &tot);
    if (threadIdx.x == 0) a.tile_sum[t] = tot;
}

// Exclusive scan of pile p's tile sums, in place.
__device__ __forceinline__ void scan_pile(const Arrays &a, int p, int *ws)
{
    if (!pile_rebuilds(a, p)) return;
    const PileStatic &S = a.ps[p];
    int carry = 0;
    for (int64_t base = 0; base < S.nt; base += kLB) {
        const int64_t t = base + threadIdx.x;
        int tot;
        const int at = block_scan(t < S.nt ? a.tile_sum[S.t0 + t] : 0, ws, &tot);
        if (t < S.nt) a.tile_sum[S.t0 + t] = carry + at;
        carry += tot;
    }
}

// Start of every cell of scan tile t: exclusive scan inside the tile plus the
// tile's offset.
__device__ __forceinline__ void scan_cells(const Arrays &a, const Sizes &z, int64_t t, int *ws)
{
    constexpr int kPer = kScanTile / kLB;
    if (!pile_rebuilds(a, tile_pile(a, z, t))) return;
    const int4 *c = (const int4 *)(a.ccount + t * kScanTile) + threadIdx.x * (kPer / 4);
    int4 *o = (int4 *)(a.cstart + t * kScanTile) + threadIdx.x * (kPer / 4);
    int loc = 0, tot;
    for (int k = 0; k < kPer / 4; ++k) {
        const int4 v = c[k];
        loc += (v.x + v.y) + (v.z + v.w);
    }
    int run = a.tile_sum[t] + block_scan(loc, ws, &tot);
    for (int k = 0; k < kPer / 4; ++k) {
        const int4 v = c[k];
        o[k] = make_int4(run, run + v.x, run + v.x + v.y, run + v.x + v.y + v.z);
        run += (v.x + v.y) + (v.z + v.w);
    }
}

// The pile's spheres (home indices) by cell, not yet ordered inside the cells:
// in the buffer for the carried-over history, which the last phase writes.
template <bool FP64>
__device__ __forceinline__ int32_t *unordered(const Arrays &a, const PileStatic &S)
{
    if constexpr (FP64) return (int32_t *)(a.hist64_rm + S.e0);
    else return (int32_t *)(a.hist32_rm + S.e0);
}

template <bool FP64>
__device__ __forceinline__ void scatter_sphere(const Arrays &a, int64_t i, int p)
{
    const PileStatic &S = a.ps[p];
    const int slot = a.cstart[S.c0 + a.key[i]] + a.sagg[i];
    unordered<FP64>(a, S)[slot] = (int32_t)(i - S.s0);
}

// The sphere in place k of the cells, and its place by home index: the number of
// its cell's spheres with a smaller one (returned with the sphere in hl).  Cells
// hold a handful of spheres,
// but a wide range of radii, a large cell_size or a fragment far away can put
// a whole pile into a few, and sorting such a cell in one thread takes seconds
// (40,000 spheres beside one of 60 times their radius: 13 s for the step that
// rebuilds, 0.03 s so).
template <bool FP64>
__device__ __forceinline__ int64_t order_sphere(const Arrays &a, int64_t k, int p, int &hl)
{
    const PileStatic &S = a.ps[p];
    const int32_t *un = unordered<FP64>(a, S);
    const int me = un[k - S.s0];
    const int key = a.key[S.s0 + me];
    const int start = a.cstart[S.c0 + key], n = a.ccount[S.c0 + key];
    int r = 0;
#pragma unroll 4
    for (int x = 0; x < n; ++x) r += un[start + x] < me ? 1 : 0;
    hl = me;
    a.sorted[S.s0 + start + r] = me;
    return S.s0 + start + r;
}

// ---------------------------------------------------------------- gather
// Sorted copies for the contact pass: position (fixed point in the mixed
// path), predicted velocity v_i = [v_A + h/2 a_A] + w_A x (r_i - r_A) (Eq.
// pred-vel), spin, ids; and the gravity input (position relative to the pile
// frame, mass) at the sphere's home index.  k: sorted position of home sphere hl
// of an active pile.
template <bool FP64>
__device__ __forceinline__ void gather_sphere(const Arrays &a, int64_t k, int p, int hl)
{
    const PileStatic &S = a.ps[p];
    const int64_t i = S.s0 + hl;
    // the sorted order changes only at rebuilds: the sorted aggregate ids are
    // written in a rebuild step (and read here otherwise); the home -> sorted
    // map, which the linking reads at the next rebuild to find each sphere's
    // previous list, is double-buffered by parity and written in a rebuild
    // step and the step after it
    const PileDyn &D = a.pd[p];
    const bool grav = S.G != 0.0;
    const bool fresh = D.rebuild != 0, refresh = fresh || D.rebuilt_prev != 0;
    const int al = fresh ? a.sph_agg[i] : a.sagg[k];
    const int64_t g = S.a0 + al;
    if (refresh) a.pos_of_home[D.parity ^ 1][i] = (int32_t)(k - S.s0);
    if (fresh) a.sagg[k] = al;
    if constexpr (FP64) {
        const AggRec64 &rec = a.rec64[g];
        const double *b = a.b64 + 3 * i;
        double3 pos = expand_64(rec, b);
        double3 rb = mat_mul(rec.R, d3(b[0], b[1], b[2]));
        double3 w = ld3(rec.w);
        double3 v = ld3(rec.vb) + cross(w, rb);
        a.dp_[k] = make_dbl4(pos.x, pos.y, pos.z, a.s64[i]);
        a.dv_[k] = make_dbl4(v.x, v.y, v.z, (double)al);
        a.dw_[k] = make_dbl4(w.x, w.y, w.z, (double)hl);
        if (grav) a.gpos64[i] = make_dbl4(pos.x, pos.y, pos.z, a.m64[i]);
    } else {
        float4 bh = a.bh[i], bl = a.bl[i];
        const AggRecMixed rec = load_rec(a.rec32, g);
        ff px, py, pz;
        expand_mixed(rec, bh, bl, px, py, pz);
        float3 rb = f3(rec.Rh[0] * bh.x + rec.Rh[1] * bh.y + rec.Rh[2] * bh.z,
                       rec.Rh[3] * bh.x + rec.Rh[4] * bh.y + rec.Rh[5] * bh.z,
                       rec.Rh[6] * bh.x + rec.Rh[7] * bh.y + rec.Rh[8] * bh.z);
        float3 w = f3(rec.w[0], rec.w[1], rec.w[2]);
        float3 v = f3(rec.vb[0], rec.vb[1], rec.vb[2]) + cross(w, rb);
        // fixed point in quanta q = 2^qexp: low 32 bits of round((r_i - O) / q)
        // per axis (differences of nearby spheres are exact int32) and
        // round(radius / q), with what the rounding left in FP32
        const int e = -S.qexp;
        float4 rm;
        const int X = ff_to_fixed(px, e, rm.x), Y = ff_to_fixed(py, e, rm.y), Z = ff_to_fixed(pz, e, rm.z);
        const int Sr = ff_to_fixed(ff{bh.w, bl.w}, e, rm.w);
        a.xqr[2 * k] = make_int4(X, Y, Z, Sr);
        a.xqr[2 * k + 1] = make_int4(__float_as_int(rm.x), __float_as_int(rm.y), __float_as_int(rm.z),
                                     __float_as_int(rm.w));
        if (fresh) a.sph_[k] = make_float4(px.hi, py.hi, pz.hi, bh.w);
        a.svw[2 * k] = make_float4(v.x, v.y, v.z, __int_as_float(al));
        a.svw[2 * k + 1] = make_float4(w.x, w.y, w.z, __int_as_float(hl));
        if (grav) a.gpos32[i] = make_float4(px.hi, py.hi, pz.hi, (float)a.m64[i]);
        if (S.ext_mass > 0) {
            // the planet's force, in FP64: a thread per sphere (in k_agg_end, a
            // thread per aggregate, that pass took 34 us at 7,466 spheres, 28
            // so; ncu); the planet as open_pile drifts it later in the step
            const double h = S.h;
            double P[3];
            for (int c = 0; c < 3; ++c) P[c] = D.P_pos[c] + h * (D.P_vel[c] + 0.5 * h * D.P_acc[c]);
            const double3 r = ld3(D.O) + d3((double)px.hi + (double)px.lo, (double)py.hi + (double)py.lo,
                                            (double)pz.hi + (double)pz.lo);
            const double3 f = planet_force(S.G * S.ext_mass, a.m64[i], d3(P[0], P[1], P[2]), r);
            a.fe[i] = make_dbl4(f.x, f.y, f.z, 0.0);
        }
    }
}

// ---------------------------------------------------------------- candidate lists
// Candidate test of sphere k (own data) against sorted position kk.  Exact and
// symmetric: swapping the spheres gives the same answer.
struct CandMe {
    int4 xq;        // mixed
    float4 ph;      // mixed: position hi, radius hi
    dbl4 p;         // fp64
    int agg;
};

template <bool FP64>
__device__ __forceinline__ bool cand_test(const Arrays &a, const PileStatic &S, const CandMe &m, int64_t kk)
{
    if constexpr (FP64) {
        const dbl4 q = a.dp_[kk];
        const double dx = q.x - m.p.x, dy = q.y - m.p.y, dz = q.z - m.p.z;
        const double t = m.p.w + q.w + S.skin;
        return __fma_rn(dz, dz, __fma_rn(dy, dy, __dmul_rn(dx, dx))) < __dmul_rn(t, t);
    } else {
        // FP32 test first (it rejects the spheres of other wraps of the grid,
        // whose 32-bit fixed-point difference would alias): the FP32 centres
        // are the rounded float-float positions, so a margin of a few units in
        // the last place of both keeps every candidate; the margin depends on
        // both spheres alike, so the test stays symmetric
        const float4 q = a.sph_[kk];
        const float dx = __fsub_rn(q.x, m.ph.x), dy = __fsub_rn(q.y, m.ph.y), dz = __fsub_rn(q.z, m.ph.z);
        const float big = __fadd_rn(fmaxf(fabsf(q.x), fmaxf(fabsf(q.y), fabsf(q.z))),
                                    fmaxf(fabsf(m.ph.x), fmaxf(fabsf(m.ph.y), fabsf(m.ph.z))));
        const float sr = __fadd_rn(q.w, m.ph.w);
        const float tc = __fadd_rn(__fadd_rn(sr, (float)S.skin), __fmaf_rn(1e-6f, big, __fmul_rn(1e-5f, sr)));
        if (!(__fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx))) < __fmul_rn(tc, tc))) return false;
        const int4 B = a.xqr[2 * kk];
        const int ex = (int)((unsigned)B.x - (unsigned)m.xq.x);
        const int ey = (int)((unsigned)B.y - (unsigned)m.xq.y);
        const int ez = (int)((unsigned)B.z - (unsigned)m.xq.z);
        const long long D = (long long)ex * ex + (long long)ey * ey + (long long)ez * ez;
        // two quanta more than the skin: the rounding remainders cannot hide a contact
        const long long t = (long long)m.xq.w + B.w + S.skin_q + 2;
        return D < t * t;
    }
}

// Visit every sphere of the 27 neighbour cells of sorted position k (the
// three x-neighbours of a (y, z) row as one index range when they are
// consecutive), calling f(kk) for the candidates.
template <bool FP64, typename Fn>
__device__ __forceinline__ void for_candidates(const Arrays &a, const PileStatic &S, int64_t k,
                                               const CandMe &m, Fn f)
{
    int cx, cy, cz;
    if constexpr (FP64) {
        cx = cellc_d(m.p.x, S.inv_cell, S.nx);
        cy = cellc_d(m.p.y, S.inv_cell, S.ny);
        cz = cellc_d(m.p.z, S.inv_cell, S.nz);
    } else {
        const float ic = (float)S.inv_cell;
        cx = cellc_f(m.ph.x, ic, S.nx);
        cy = cellc_f(m.ph.y, ic, S.ny);
        cz = cellc_f(m.ph.z, ic, S.nz);
    }
    const int32_t *cstart = a.cstart + S.c0, *ccount = a.ccount + S.c0;
    const int64_t s0 = S.s0;
    // without wrap-around the three x-neighbours are consecutive cell ids
    // except across a brick boundary: one or two index ranges
    const bool nowrap = cx >= 1 && cx + 1 < S.nx;
    const int split = (cx & 3) == 0 ? 1 : (cx & 3) == 3 ? 2 : 3;   // first cell of the second range
    for (int dz = -1; dz <= 1; ++dz)
        for (int dy = -1; dy <= 1; ++dy) {
            const int yy = wrapc(cy + dy, S.ny), zz = wrapc(cz + dz, S.nz);
            int beg[3], end[3], nr;
            if (nowrap) {
                const int64_t cl = cell_id(cx - 1, yy, zz, S.nx, S.ny);
                const int64_t cs = cell_id(cx - 1 + split, yy, zz, S.nx, S.ny);
                const int64_t ce = cell_id(cx + 1, yy, zz, S.nx, S.ny);
                if (split == 3) {
                    beg[0] = cstart[cl];
                    end[0] = cstart[ce] + ccount[ce];
                    nr = 1;
                } else {
                    const int64_t cm = split == 1 ? cl : cell_id(cx, yy, zz, S.nx, S.ny);
                    beg[0] = cstart[cl];
                    end[0] = cstart[cm] + ccount[cm];
                    beg[1] = cstart[cs];
                    end[1] = cstart[ce] + ccount[ce];
                    nr = 2;
                }
            } else {
                nr = 0;
                for (int ddx = -1; ddx <= 1; ++ddx) {
                    const int64_t c = cell_id(wrapc(cx + ddx, S.nx), yy, zz, S.nx, S.ny);
                    beg[nr] = cstart[c];
                    end[nr] = cstart[c] + ccount[c];
                    ++nr;
                }
            }
            for (int r = 0; r < nr; ++r)
                for (int t = beg[r]; t < end[r]; ++t) {
                    const int64_t kk = s0 + t;
                    if (kk == k || a.sagg[kk] == m.agg) continue;
                    if (cand_test<FP64>(a, S, m, kk)) f(t);
                }
        }
}

template <bool FP64>
__device__ __forceinline__ void load_me(const Arrays &a, int64_t k, CandMe &m)
{
    if constexpr (FP64) m.p = a.dp_[k];
    else {
        m.xq = a.xqr[2 * k];
        m.ph = a.sph_[k];
    }
    m.agg = a.sagg[k];
}

// Slices: the 32 consecutive sorted spheres a warp takes; slice s of tile t
// (four to a tile) has entry 4 t + s of ctile_cnt and ctile_base.
// f(p, first sorted position, spheres, slice) for the slices of tile t, one
// warp each, if its pile rebuilds; whole warps call it.
template <typename Fn>
__device__ __forceinline__ void rebuilding_slices(const Arrays &a, int64_t t, Fn f)
{
    const int wid = threadIdx.x >> 5;
    const int4 tl = a.ctile[t];
    if (pile_rebuilds(a, tl.x)) f(tl.x, tl.y + 32 * wid, min(32, tl.z - 32 * wid), 4 * t + wid);
}

// Candidates per sphere (new list buffer) and entries per slice: a slice is
// as wide as its longest list.
template <bool FP64>
__device__ __forceinline__ void count_tile(const Arrays &a, int64_t t)
{
    rebuilding_slices(a, t, [&](int p, int first, int ns, int64_t slice) {
        const PileStatic &S = a.ps[p];
        const int lp = a.pd[p].cpar ^ 1, lane = threadIdx.x & 31;
        int n = 0;
        if (lane < ns) {
            const int64_t k = S.s0 + first + lane;
            CandMe m;
            load_me<FP64>(a, k, m);
            for_candidates<FP64>(a, S, k, m, [&](int) { ++n; });
            a.ccnt[lp][k] = n;
        }
        const int wmax = __reduce_max_sync(0xffffffffu, n);
        if (lane == 0) a.ctile_cnt[slice] = 32 * wmax;
    });
}

// Exclusive scan of pile p's slices.  Lists that do not fit the pile's
// entries flag the pile (frozen at the end of the step).
__device__ __forceinline__ void scan_lists(const Arrays &a, int p, long long *ws)
{
    constexpr int kPer = 8;
    if (!pile_rebuilds(a, p)) return;
    const PileStatic &S = a.ps[p];
    const int64_t n = 4 * S.nct, o = 4 * S.ct0;
    long long carry = 0;
    for (int64_t base = 0; base < n; base += kPer * kLB) {
        const int64_t t = base + (int64_t)kPer * threadIdx.x;
        long long v[kPer], loc = 0, tot;
        for (int k = 0; k < kPer; ++k) {
            v[k] = t + k < n ? a.ctile_cnt[o + t + k] : 0;
            loc += v[k];
        }
        long long run = carry + block_scan(loc, ws, &tot);
        for (int k = 0; k < kPer; ++k) {
            if (t + k < n) a.ctile_base[o + t + k] = (int32_t)run;
            run += v[k];
        }
        carry += tot;
    }
    if (carry > S.ne) {
        if (threadIdx.x == 0) atomicOr(&a.pd[p].flags, DEM_FLAG_SLOTS);
        __syncthreads();
        for (int64_t t = threadIdx.x; t < n; t += kLB) a.ctile_base[o + t] = -1;
    }
}

// Offsets, then the candidates themselves, sorted by partner home index.
// Sliced layout: the 32 spheres of a slice store entry e of their lists side
// by side, so sphere k's entry e is at coff[k] + 32 e (coalesced when a warp
// walks its lists together).
constexpr int kFillCap = 20;   // candidates sorted in shared memory per sphere (more: in place)

template <bool FP64>
__device__ __forceinline__ void fill_sphere(const Arrays &a, const PileStatic &S, int lp, int64_t k, int off, int2 *l)
{
    const int n = a.ccnt[lp][k];
    a.coff[lp][k] = off;
    int32_t *ids = a.cand_id[lp] + S.e0 + off;
    int2 *cd = a.cand[lp] + S.e0 + off;
    const int32_t *srt = a.sorted + S.s0;
    CandMe m;
    load_me<FP64>(a, k, m);
    int j = 0;
    if (n <= kFillCap) {
        // insertion by partner home index in shared memory, then one write
        for_candidates<FP64>(a, S, k, m, [&](int t) {
            if (j >= n) return;   // (the count pass visited the same candidates)
            const int id = srt[t];
            int y = j++;
            while (y > 0 && l[(y - 1) * kLB].x > id) {
                l[y * kLB] = l[(y - 1) * kLB];
                --y;
            }
            l[y * kLB] = make_int2(id, t);
        });
        for (int y = 0; y < j; ++y) {
            const int2 v = l[y * kLB];
            ids[32 * y] = v.x;
            cd[32 * y] = make_int2(v.y, 0);
        }
        return;
    }
    for_candidates<FP64>(a, S, k, m, [&](int t) {
        if (j >= n) return;
        // long list: insertion by partner home index in place
        const int id = srt[t];
        int y = j++;
        while (y > 0 && ids[32 * (y - 1)] > id) {
            ids[32 * y] = ids[32 * (y - 1)];
            cd[32 * y] = cd[32 * (y - 1)];
            --y;
        }
        ids[32 * y] = id;
        cd[32 * y] = make_int2(t, 0);
    });
}

template <bool FP64>
__device__ __forceinline__ void fill_tile(const Arrays &a, int64_t t, int2 (*s_list)[kLB])
{
    rebuilding_slices(a, t, [&](int p, int first, int ns, int64_t slice) {
        const PileStatic &S = a.ps[p];
        const int lane = threadIdx.x & 31, base = a.ctile_base[slice];
        if (base < 0 || lane >= ns) return;
        fill_sphere<FP64>(a, S, a.pd[p].cpar ^ 1, S.s0 + first + lane, base + lane, &s_list[0][threadIdx.x]);
    });
}

// Owner bit and mirror entry of every list entry; history carried from the
// previous lists (by the home indices of both spheres) into hist_rm.
template <bool FP64>
__device__ __forceinline__ void cand_link_sphere(const Arrays &a, int p, int kl)
{
    typedef typename HistT<FP64>::H H;
    const PileStatic &S = a.ps[p];
    const PileDyn &D = a.pd[p];
    const int lp = D.cpar ^ 1, op = D.cpar, par = D.parity;
    const int64_t s0 = S.s0, e0 = S.e0;
    const int me = a.sorted[s0 + kl];
    const int n = a.ccnt[lp][s0 + kl], off = a.coff[lp][s0 + kl];
    // the previous list of this home sphere
    const int kprev = a.pos_of_home[par][s0 + me];
    const int pn = a.ccnt[op][s0 + kprev], poff = a.coff[op][s0 + kprev];
    const int32_t *pids = a.cand_id[op] + e0 + poff;
    const H *hprev;
    H *hrm;
    if constexpr (FP64) { hprev = a.hist64[par] + e0; hrm = a.hist64_rm + e0; }
    else { hprev = a.hist32[par] + e0; hrm = a.hist32_rm + e0; }
    int cursor = 0;
    for (int e = 0; e < n; ++e) {
        const int f = off + 32 * e;
        const int2 c = a.cand[lp][e0 + f];
        const int kk = c.x;
        const int id = a.cand_id[lp][e0 + f];
        // my entry in the partner's list: binary search by home index
        const int pn2 = a.ccnt[lp][s0 + kk], po2 = a.coff[lp][s0 + kk];
        const int32_t *ids2 = a.cand_id[lp] + e0 + po2;
        int lo = 0, hi = pn2 - 1, mir = -1;
        while (lo <= hi) {
            const int mid = (lo + hi) >> 1;
            const int v = ids2[32 * mid];
            if (v == me) { mir = po2 + 32 * mid; break; }
            if (v < me) lo = mid + 1; else hi = mid - 1;
        }
        if (mir < 0) atomicOr(&a.pd[p].flags, DEM_FLAG_SLOTS);   // lists not symmetric: cannot happen
        const bool owned = me < id;
        a.cand[lp][e0 + f] = make_int2(kk | (owned ? (int)0x80000000u : 0), mir < 0 ? 0 : mir);
        // carried history: the same partner in the previous list (both lists
        // are in partner order, so one forward cursor finds it)
        H h;
        if constexpr (FP64) h = make_dbl4(0.0, 0.0, 0.0, 0.0);
        else h = make_float4(0.f, 0.f, 0.f, 0.f);
        while (cursor < pn && pids[32 * cursor] < id) ++cursor;
        if (cursor < pn && pids[32 * cursor] == id) {
            const H g = hprev[poff + 32 * cursor];
            if (g.w != 0) h = g;
        }
        hrm[f] = h;
    }
}

template <bool FP64>
__device__ __forceinline__ void link_tile(const Arrays &a, int64_t t)
{
    rebuilding_slices(a, t, [&](int p, int first, int ns, int64_t slice) {
        const int lane = threadIdx.x & 31;
        if (a.ctile_base[slice] >= 0 && lane < ns) cand_link_sphere<FP64>(a, p, first + lane);
    });
}

// ---------------------------------------------------------------- the kernel
// Blocks that run the opening reductions: one per chunk, at most an eighth of
// the resident blocks.
__host__ __device__ __forceinline__ int64_t lists_reducers(const Sizes &z)
{
    const int64_t most = z.LB / 8 > 1 ? z.LB / 8 : 1;
    return z.CH < most ? z.CH : most;
}

// (7 blocks an SM: 72 registers; left alone the compiler takes 64 and spills,
// 59 us for the gather of the 1M lattice, 51 so)
template <bool FP64>
__global__ void __launch_bounds__(kLB, 7) k_lists(Arrays a, Sizes z)
{
    pdl_enter();
    __shared__ int2 s_list[kFillCap][kLB];   // (partner home index, sorted position)
    __shared__ long long ws[kLB / 32];
    int *wsi = (int *)ws;
    const int64_t nsb = (z.N + kLB - 1) / kLB;   // blocks' worth of spheres
    if (!any_rebuild(a, z)) {
        // the first blocks sum the piles' chunks (a long chain of loads and
        // shuffles beside the others' gather), the rest gather
        const int64_t nred = lists_reducers(z), b = (int64_t)blockIdx.x - nred;
        if (b < 0)
            for (int64_t ch = blockIdx.x; ch < z.CH; ch += nred) open_chunk<FP64, kLB>(a, ch);
        else
            for (int64_t k = b * kLB + threadIdx.x; k < z.N; k += (gridDim.x - nred) * kLB) {
                const int p = sphere_pile(a, z, k);
                if (pile_active(a, p)) gather_sphere<FP64>(a, k, p, a.sorted[k]);
            }
        return;
    }
    __shared__ unsigned drawn;
    auto phase = [&](int ph, int64_t items, auto f) { return run_phase(a, z, ph, items, &drawn, f); };
    if (phase(kKeys, z.CH + nsb, [&](int64_t t) {
            if (t < z.CH) reference_chunk<FP64>(a, t);
            else rebuilding_spheres(a, z, t - z.CH, [&](int64_t i, int p) { key_sphere<FP64>(a, i, p); });
        }) &&
        phase(kScanTiles, z.T, [&](int64_t t) { sum_tile(a, z, t, wsi); }) &&
        phase(kScanPiles, z.P, [&](int64_t p) { scan_pile(a, (int)p, wsi); }) &&
        phase(kScanCells, z.T, [&](int64_t t) { scan_cells(a, z, t, wsi); }) &&
        phase(kScatter, nsb, [&](int64_t t) {
            rebuilding_spheres(a, z, t, [&](int64_t i, int p) { scatter_sphere<FP64>(a, i, p); });
        }) &&
        // the gather of every pile and, in the same pass, the order inside the
        // cells of those that rebuild
        phase(kPlace, z.CH + nsb, [&](int64_t t) {
            if (t < z.CH) {
                open_chunk<FP64, kLB>(a, t);
                return;
            }
            int64_t k = (t - z.CH) * kLB + threadIdx.x;
            if (k >= z.N) return;
            const int p = sphere_pile(a, z, k);
            if (!pile_active(a, p)) return;
            int hl;
            if (a.pd[p].rebuild) k = order_sphere<FP64>(a, k, p, hl);
            else hl = a.sorted[k];
            gather_sphere<FP64>(a, k, p, hl);
        }) &&
        phase(kCount, z.CT, [&](int64_t t) { count_tile<FP64>(a, t); }) &&
        phase(kListScan, z.P, [&](int64_t p) { scan_lists(a, (int)p, ws); }) &&
        phase(kFill, z.CT, [&](int64_t t) { fill_tile<FP64>(a, t, s_list); }))
        phase(kLink, z.CT + z.T, [&](int64_t t) {
            if (t < z.CT) link_tile<FP64>(a, t);
            else clear_tile(a, z, t - z.CT);
        });
    phases_done(a);
}

int lists_blocks_per_sm(bool fp64)
{
    int n = 0;
    if (fp64) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_lists<true>, kLB, 0);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_lists<false>, kLB, 0);
    return n;
}

void launch_lists(const Arrays &a, const Sizes &z, bool fp64, cudaStream_t st)
{
    if (z.N == 0) return;
    const int64_t want = (z.N + kLB - 1) / kLB + lists_reducers(z);
    const unsigned nb = (unsigned)(want < z.LB ? want : z.LB);
    if (fp64) launch_pdl(k_lists<true>, nb, kLB, 0, st, a, z);
    else launch_pdl(k_lists<false>, nb, kLB, 0, st, a, z);
}

}  // namespace dem
