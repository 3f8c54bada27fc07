// kernels_tree.cu -- tree gravity (the paper's gravity method, Sec. 2.1: a
// tree code with multipole expansions), as an option beside the direct sum.
//
// Per pile and step: a cubic box around the pile (min/max of the sphere
// centres), an implicit octree of depth D over it (level L has 8^L cells in
// Morton order, so the parent of cell m is m >> 3), spheres counted into the
// leaf cells and ordered by leaf (counting sort, each leaf ordered by home
// index, deterministic), leaf moments from their spheres and upper moments
// from 8 children: mass, centre of mass and the raw moments of ranks 2-4
// about the COM (shifted exactly from child to parent), kept for evaluation
// as their traceless parts -- quadrupole, octupole and hexadecapole, the
// expansion order of the paper's tree code (Sec. 2.1) -- then each warp
// walks the tree for 32 spheres at once.  A cell is accepted when
// the group of spheres is farther from its COM than size/theta +
// |COM - centre| (so no sphere is inside an accepted cell) and contributes
// the gradient of its multipole potential up to rank 4 (or rank 2, the
// cheaper option); an opened leaf is summed directly
// with Plummer softening, skipping the sphere itself and its aggregate mates
// (pairs inside one aggregate cancel in its totals, Sec. 2.2.3).  Mates that
// fall in an accepted distant cell are not removed: their share cancels in
// the aggregate totals to the accuracy of the expansion.  FP32 throughout
// (positions relative to the pile frame); the result is written to the same
// per-sphere gravity array as the direct sum.
#include "dem_internal.h"
#include "devmath.cuh"
#include "f32x2.cuh"
#include "launch.cuh"

namespace dem {

// order-preserving map of floats to ints (min/max by integer atomics)
__device__ __forceinline__ int f2o(float f)
{
    int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float o2f(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

__device__ __forceinline__ bool tree_pile(const Arrays &a, int p)
{
    return a.enabled[p] != 0 && a.pd[p].failed == 0 && a.ps[p].tD > 0;
}

// level offset inside a pile's node block: sum_{k<L} 8^k
__host__ __device__ __forceinline__ int64_t lvl_off(int L) { return ((int64_t)1 << (3 * L)) / 7; }

__device__ __forceinline__ uint32_t spread3(uint32_t v)
{
    v &= 0x3ff;
    v = (v | (v << 16)) & 0x030000ff;
    v = (v | (v << 8)) & 0x0300f00f;
    v = (v | (v << 4)) & 0x030c30c3;
    v = (v | (v << 2)) & 0x09249249;
    return v;
}

// Reset the boxes and the leaf counts.
__global__ void k_tree_init(Arrays a, Sizes z)
{
    pdl_enter();
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < 6 * z.P) {
        const int p = (int)(g / 6), c = (int)(g % 6);
        a.tbox[8 * p + c] = f2o(c < 3 ? 3.0e38f : -3.0e38f);
    }
    if (g >= z.TL) return;
    const int p = a.tleaf_pile[g];
    if (p >= 0 && tree_pile(a, p)) a.tleaf[g] = make_int2(0, 0);
}

// Box of each pile: every warp reduces its spheres' min/max (piles are
// contiguous, so a warp holds one or two), a block that lies in one pile its
// warps', then one atomic per component (min/max do not depend on the order).
// An atomic per warp and component was 16 us at 100,000 spheres (ncu).
constexpr int kBoxThreads = 256;
__global__ void __launch_bounds__(kBoxThreads) k_tree_box(Arrays a, Sizes z)
{
    pdl_enter();
    const unsigned FULL = 0xffffffffu;
    const int64_t b0 = (int64_t)blockIdx.x * kBoxThreads, i = b0 + threadIdx.x;
    const int p = i < z.N ? a.sph_pile[i] : -1;
    const bool act = p >= 0 && tree_pile(a, p);
    const float4 x = act ? a.gpos32[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int o[3] = {f2o(x.x), f2o(x.y), f2o(x.z)};
    __shared__ int sh[kBoxThreads / 32][6];
    const int p0 = a.sph_pile[b0], lane = threadIdx.x & 31;
    const int64_t e = b0 + kBoxThreads < z.N ? b0 + kBoxThreads : z.N;
    const bool one = a.sph_pile[e - 1] == p0;   // uniform over the block
    unsigned todo = __ballot_sync(FULL, act);
    if (one && !tree_pile(a, p0)) return;
    int v[6];
    if (one) {
        for (int c = 0; c < 3; ++c) {
            v[c] = __reduce_min_sync(FULL, act ? o[c] : 0x7fffffff);
            v[3 + c] = __reduce_max_sync(FULL, act ? o[c] : (int)0x80000000);
        }
        if (lane == 0)
            for (int c = 0; c < 6; ++c) sh[threadIdx.x >> 5][c] = v[c];
        __syncthreads();
        if (threadIdx.x < 6) {
            const int c = threadIdx.x;
            int m = sh[0][c];
            for (int w = 1; w < kBoxThreads / 32; ++w) m = c < 3 ? min(m, sh[w][c]) : max(m, sh[w][c]);
            if (c < 3) atomicMin(&a.tbox[8 * p0 + c], m);
            else atomicMax(&a.tbox[8 * p0 + c], m);
        }
        return;
    }
    while (todo) {
        const int leader = __ffs(todo) - 1;
        const int pp = __shfl_sync(FULL, p, leader);
        const bool mine = act && p == pp;
        todo &= ~__ballot_sync(FULL, mine);
        for (int c = 0; c < 3; ++c) {
            v[c] = __reduce_min_sync(FULL, mine ? o[c] : 0x7fffffff);
            v[3 + c] = __reduce_max_sync(FULL, mine ? o[c] : (int)0x80000000);
        }
        if (lane == leader)
            for (int c = 0; c < 6; ++c) {
                if (c < 3) atomicMin(&a.tbox[8 * pp + c], v[c]);
                else atomicMax(&a.tbox[8 * pp + c], v[c]);
            }
    }
}

// cube of the pile: lower corner and edge
__device__ __forceinline__ void tree_cube(const Arrays &a, int p, float3 &lo, float &edge)
{
    const int *b = a.tbox + 8 * p;
    lo = f3(o2f(b[0]), o2f(b[1]), o2f(b[2]));
    const float ex = o2f(b[3]) - lo.x, ey = o2f(b[4]) - lo.y, ez = o2f(b[5]) - lo.z;
    edge = fmaxf(fmaxf(ex, ey), fmaxf(ez, 1e-6f)) * 1.0001f;
}

__global__ void k_tree_keys(Arrays a, Sizes z)
{
    pdl_enter();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= z.N) return;
    const int p = a.sph_pile[i];
    if (!tree_pile(a, p)) return;
    const PileStatic &S = a.ps[p];
    float3 lo;
    float edge;
    tree_cube(a, p, lo, edge);
    const int n1 = 1 << S.tD;
    const float sc = (float)n1 / edge;
    const float4 x = a.gpos32[i];
    const int cx = min(max((int)((x.x - lo.x) * sc), 0), n1 - 1);
    const int cy = min(max((int)((x.y - lo.y) * sc), 0), n1 - 1);
    const int cz = min(max((int)((x.z - lo.z) * sc), 0), n1 - 1);
    const int key = (int)(spread3(cx) | (spread3(cy) << 1) | (spread3(cz) << 2));
    a.tkey[i] = key;
    a.trank[i] = atomicAdd(&a.tleaf[S.tleaf0 + key].y, 1);
}

// Exclusive scan of each pile's leaf counts by blocks of kLeafTile leaves
// (blockIdx.x: pile): first the tiles' sums, then every block adds the sums
// before its own (at most 128) and scans its leaves.  One block per pile, each
// thread walking its own range of leaves, was 60 us at 32,768 leaves (ncu).
constexpr int kLeafTile = 2048, kScanThreads = 256;
// scratch before the walk writes its partial sums: the leaf-sorted but not yet
// ordered spheres, then the leaf tiles' sums (fewer than the pile's spheres)
__device__ __forceinline__ int *tree_unordered(const Arrays &a) { return (int *)a.tpart; }
__device__ __forceinline__ int *tree_tile_sums(const Arrays &a, const Sizes &z, const PileStatic &S)
{
    return (int *)a.tpart + z.N + S.s0;
}

// Inclusive prefix sum over the block's kScanThreads threads.
__device__ __forceinline__ int scan256(int v, int *ws)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) ws[wid] = v;
    __syncthreads();
    for (int k = 0; k < kScanThreads / 32; ++k)
        if (k < wid) v += ws[k];
    return v;
}

__global__ void __launch_bounds__(kScanThreads) k_tree_sums(Arrays a, Sizes z)
{
    pdl_enter();
    const int p = blockIdx.x;
    if (!tree_pile(a, p)) return;
    const PileStatic &S = a.ps[p];
    const int nl = 1 << (3 * S.tD), l0 = blockIdx.y * kLeafTile;
    if (l0 >= nl || nl <= kLeafTile) return;
    __shared__ int ws[kScanThreads / 32];
    int s = 0;
    for (int k = threadIdx.x; k < kLeafTile; k += kScanThreads) s += a.tleaf[S.tleaf0 + l0 + k].y;
    s = scan256(s, ws);
    if (threadIdx.x == kScanThreads - 1) tree_tile_sums(a, z, S)[blockIdx.y] = s;
}

__global__ void __launch_bounds__(kScanThreads) k_tree_scan(Arrays a, Sizes z)
{
    pdl_enter();
    const int p = blockIdx.x;
    if (!tree_pile(a, p)) return;
    const PileStatic &S = a.ps[p];
    const int nl = 1 << (3 * S.tD), l0 = blockIdx.y * kLeafTile;
    if (l0 >= nl) return;
    constexpr int kPer = kLeafTile / kScanThreads;
    __shared__ int ws[kScanThreads / 32], before;
    int2 *leaf = a.tleaf + S.tleaf0 + l0;
    // tiles before this one (at most 127)
    int s = threadIdx.x < blockIdx.y ? tree_tile_sums(a, z, S)[threadIdx.x] : 0;
    s = scan256(s, ws);
    if (threadIdx.x == kScanThreads - 1) before = s;
    __syncthreads();
    int c[kPer], loc = 0;
    for (int k = 0; k < kPer; ++k) {
        const int l = threadIdx.x * kPer + k;
        c[k] = l0 + l < nl ? leaf[l].y : 0;
        loc += c[k];
    }
    int run = before + scan256(loc, ws) - loc;
    for (int k = 0; k < kPer; ++k) {
        const int l = threadIdx.x * kPer + k;
        if (l0 + l < nl) leaf[l].x = run;
        run += c[k];
    }
}

__global__ void k_tree_scatter(Arrays a, Sizes z)
{
    pdl_enter();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= z.N) return;
    const int p = a.sph_pile[i];
    if (!tree_pile(a, p)) return;
    const PileStatic &S = a.ps[p];
    tree_unordered(a)[S.s0 + a.tleaf[S.tleaf0 + a.tkey[i]].x + a.trank[i]] = (int32_t)(i - S.s0);
}

// Every sphere finds its place in its leaf, ordered by home index (the number
// of the leaf's spheres with a smaller one: leaves hold a handful), which makes
// the sums deterministic, and puts its position (+mass) and aggregate there,
// so that a leaf's spheres are contiguous for the moments and the walk.
// (An insertion sort by each leaf's first thread and a gather after it were 20
// and 6 us at 100,000 spheres.)
__global__ void k_tree_gather(Arrays a, Sizes z)
{
    pdl_enter();
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= z.N) return;
    const int p = a.sph_pile[k];
    if (!tree_pile(a, p)) return;
    const PileStatic &S = a.ps[p];
    const int64_t s0 = S.s0;
    const int *un = tree_unordered(a) + s0;
    const int i = un[k - s0];
    const int2 L = a.tleaf[S.tleaf0 + a.tkey[s0 + i]];
    const float4 x = a.gpos32[s0 + i];
    const int ag = a.sph_agg[s0 + i];
    int r = 0;
    for (int m = 0; m < L.y; ++m) r += un[L.x + m] < i ? 1 : 0;
    const int64_t o = s0 + L.x + r;
    a.tsorted[o] = i;
    a.tpos[o] = x;
    a.tagg[o] = ag;
}

// ---- multipole moments up to the hexadecapole
// A symmetric tensor of rank n is kept as its (n+1)(n+2)/2 distinct
// components, component (a, b, c) having a x-, b y- and c z-indices, in the
// order of mono_idx.  Raw moments of a node about its COM, R_abc = sum m x^a
// y^b z^c (rank 1 vanishes), ranks 2..4 at offsets 0, 6, 16 (31 floats,
// traw: 8 float4 per node).  Node record (tnode: 9 float4 = 36 floats): COM
// 0..2, M 3, opening radius^2 4, then the evaluation tensors T_n = c_n
// detrace(R_n) of ranks 2, 3, 4 at 5, 11, 21 with c_n = (2n-1)!!/n!
// (3/2, 5/2, 35/8), so that the potential of the node at offset x from its
// COM is -G (M / r + sum_n T_n . x^n / r^(2n+1)).
constexpr int kNodeF4 = 9, kRawF4 = 8;
__host__ __device__ constexpr int mono_idx(int a, int b, int c)
{
    int n = a + b + c, i = 0;
    for (int aa = n; aa > a; --aa) i += n - aa + 1;
    return i + (n - a) - b;
}
__host__ __device__ constexpr int raw_off(int n) { return n == 2 ? 0 : n == 3 ? 6 : 16; }
__host__ __device__ constexpr int node_off(int n) { return n == 2 ? 5 : n == 3 ? 11 : 21; }
__host__ __device__ constexpr float binomf(int n, int k)
{
    return (k < 0 || k > n) ? 0.f : (k == 0 || k == n) ? 1.f : (n == 2 ? 2.f : n == 3 ? 3.f : (k == 2 ? 6.f : 4.f));
}
__host__ __device__ constexpr float factf(int n) { return n <= 1 ? 1.f : n == 2 ? 2.f : n == 3 ? 6.f : 24.f; }
// number of ways to pair up 4 indices so that both pairs have equal axes
__host__ __device__ constexpr float pairings4(int a, int b, int c)
{
    return ((a & 1) || (b & 1) || (c & 1)) ? 0.f : (a == 4 || b == 4 || c == 4) ? 3.f : 1.f;
}

__device__ __forceinline__ void powers4(float x, float *p)
{
    p[0] = 1.f;
    p[1] = x;
    p[2] = x * x;
    p[3] = p[2] * x;
    p[4] = p[2] * p[2];
}

// trace over one index pair of the rank-n raw moment, component f (rank n - 2)
template <int N>
__device__ __forceinline__ float trace1(const float *R, int fa, int fb, int fc)
{
    return R[raw_off(N) + mono_idx(fa + 2, fb, fc)] + R[raw_off(N) + mono_idx(fa, fb + 2, fc)] +
           R[raw_off(N) + mono_idx(fa, fb, fc + 2)];
}

// Evaluation tensors from raw moments: the traceless part of each rank
// (subtract the symmetrised traces: 1/(2n-1) of single traces, plus 1/35 of
// the double trace at rank 4), scaled by (2n-1)!!/n!.
template <int N>
__device__ __forceinline__ void detrace_scaled(const float *R, float *T)
{
    constexpr float cn = N == 2 ? 1.5f : N == 3 ? 2.5f : 4.375f;
    float W = 0.f;
    if (N == 4) W = trace1<4>(R, 2, 0, 0) + trace1<4>(R, 0, 2, 0) + trace1<4>(R, 0, 0, 2);
#pragma unroll
    for (int a = N; a >= 0; --a)
#pragma unroll
        for (int b = N - a; b >= 0; --b) {
            const int c = N - a - b;
            float tr = 0.f;
            if (a >= 2) tr += binomf(a, 2) * trace1<N>(R, a - 2, b, c);
            if (b >= 2) tr += binomf(b, 2) * trace1<N>(R, a, b - 2, c);
            if (c >= 2) tr += binomf(c, 2) * trace1<N>(R, a, b, c - 2);
            float v = R[raw_off(N) + mono_idx(a, b, c)] - tr * (1.f / (2 * N - 1));
            if (N == 4) v += pairings4(a, b, c) * W * (1.f / 35.f);
            T[node_off(N) - 5 + mono_idx(a, b, c)] = cn * v;
        }
}

__device__ __forceinline__ void put_node(const Arrays &a, int64_t n, float3 c, float M, const float *R,
                                         float ropen2)
{
    float nd[4 * kNodeF4];
    nd[0] = c.x; nd[1] = c.y; nd[2] = c.z; nd[3] = M; nd[4] = ropen2;
    detrace_scaled<2>(R, nd + 5);
    detrace_scaled<3>(R, nd + 5);
    detrace_scaled<4>(R, nd + 5);
    float4 *o = a.tnode + kNodeF4 * n;
#pragma unroll
    for (int k = 0; k < kNodeF4; ++k) o[k] = make_float4(nd[4 * k], nd[4 * k + 1], nd[4 * k + 2], nd[4 * k + 3]);
    float4 *r = a.traw + kRawF4 * n;
#pragma unroll
    for (int k = 0; k < kRawF4; ++k)
        r[k] = make_float4(R[4 * k], R[4 * k + 1], R[4 * k + 2], k == kRawF4 - 1 ? 0.f : R[4 * k + 3]);
}

// centre of cell m (Morton) at level L of pile p's cube
__device__ __forceinline__ float3 cell_centre(float3 lo, float edge, int L, uint32_t m)
{
    uint32_t x = 0, y = 0, zz = 0;
    for (int b = 0; b < L; ++b) {
        x |= ((m >> (3 * b)) & 1u) << b;
        y |= ((m >> (3 * b + 1)) & 1u) << b;
        zz |= ((m >> (3 * b + 2)) & 1u) << b;
    }
    const float s = edge / (float)(1 << L);
    return f3(lo.x + (x + 0.5f) * s, lo.y + (y + 0.5f) * s, lo.z + (zz + 0.5f) * s);
}

__device__ __forceinline__ float opening2(float3 com, float3 ctr, float size, float theta)
{
    const float dx = com.x - ctr.x, dy = com.y - ctr.y, dz = com.z - ctr.z;
    const float r = size / theta + sqrtf(dx * dx + dy * dy + dz * dz);
    return r * r;
}

// Leaf moments: one thread per leaf of every tree pile.
__global__ void k_tree_leaves(Arrays a, Sizes z)
{
    pdl_enter();
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= z.TL) return;
    const int p = a.tleaf_pile[g];
    if (p < 0 || !tree_pile(a, p)) return;
    const PileStatic &S = a.ps[p];
    const uint32_t m = (uint32_t)(g - S.tleaf0);
    const int2 L = a.tleaf[g];
    const int64_t n = S.tnode0 + lvl_off(S.tD) + m;
    float R[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) R[k] = 0.f;
    if (L.y == 0) {
        put_node(a, n, f3(0, 0, 0), 0.f, R, 0.f);
        return;
    }
    const float4 *tp = a.tpos + S.s0;
    float M = 0.f;
    float3 c = f3(0, 0, 0);
    const float4 x0 = tp[L.x];
    for (int k = 0; k < L.y; ++k) {   // COM about the first sphere
        const float4 x = tp[L.x + k];
        M += x.w;
        c = c + x.w * f3(x.x - x0.x, x.y - x0.y, x.z - x0.z);
    }
    c = f3(x0.x, x0.y, x0.z) + (1.0f / M) * c;
    for (int k = 0; k < L.y; ++k) {
        const float4 x = tp[L.x + k];
        float px[5], py[5], pz[5];
        powers4(x.x - c.x, px);
        powers4(x.y - c.y, py);
        powers4(x.z - c.z, pz);
#pragma unroll
        for (int r = 2; r <= 4; ++r)
#pragma unroll
            for (int ea = r; ea >= 0; --ea)
#pragma unroll
                for (int eb = r - ea; eb >= 0; --eb) {
                    const int ec = r - ea - eb;
                    R[raw_off(r) + mono_idx(ea, eb, ec)] += x.w * (px[ea] * py[eb] * pz[ec]);
                }
    }
    float3 lo;
    float edge;
    tree_cube(a, p, lo, edge);
    const float size = edge / (float)(1 << S.tD);
    put_node(a, n, c, M, R, opening2(c, cell_centre(lo, edge, S.tD, m), size, S.theta));
}

// Moments of level L from the 8 children: raw moments shifted from each
// child's COM to the parent's, R_e += sum_{f <= e} C(e, f) R_child,f s^(e-f)
// with s = child COM - parent COM (rank-1 terms vanish about a COM).  Eight
// lanes per node, one per child, summed by a fixed tree; blockIdx.x:
// pile.  With a thread per node a level of 4,096 nodes was 16
// blocks, each thread shifting its 8 children in turn: 22 us a level (ncu).
// Levels below the walk's start (kSplitL) are not needed.
__global__ void __launch_bounds__(128) k_tree_up(Arrays a, Sizes z, int L)
{
    pdl_enter();
    const int p = blockIdx.x;
    if (!tree_pile(a, p)) return;
    const PileStatic &S = a.ps[p];
    const uint32_t t = blockIdx.y * 128 + threadIdx.x, m = t >> 3;
    if (L >= S.tD || (blockIdx.y * 128 >> 3) >= (1u << (3 * L))) return;   // 16 nodes a block: whole blocks
    const int64_t g = S.tnode0 + lvl_off(L) + m;
    const int64_t cn = S.tnode0 + lvl_off(L + 1) + t;   // this lane's child
    auto sum8 = [](float v) {
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        return v + __shfl_xor_sync(0xffffffffu, v, 4);
    };
    const float4 A = a.tnode[kNodeF4 * cn];
    float R[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) R[k] = 0.f;
    const float M = sum8(A.w);
    float3 c = f3(sum8(A.w * A.x), sum8(A.w * A.y), sum8(A.w * A.z));
    if (M > 0.f) c = (1.0f / M) * c;
    if (A.w != 0.f) {
        float Rc[32];
        const float4 *r = a.traw + kRawF4 * cn;
#pragma unroll
        for (int q = 0; q < kRawF4; ++q) {
            const float4 v = r[q];
            Rc[4 * q] = v.x; Rc[4 * q + 1] = v.y; Rc[4 * q + 2] = v.z; Rc[4 * q + 3] = v.w;
        }
        float sx[5], sy[5], sz[5];
        powers4(A.x - c.x, sx);
        powers4(A.y - c.y, sy);
        powers4(A.z - c.z, sz);
#pragma unroll
        for (int n = 2; n <= 4; ++n)
#pragma unroll
            for (int ea = n; ea >= 0; --ea)
#pragma unroll
                for (int eb = n - ea; eb >= 0; --eb) {
                    const int ec = n - ea - eb;
                    float v = 0.f;
#pragma unroll
                    for (int fa = 0; fa <= ea; ++fa)
#pragma unroll
                        for (int fb = 0; fb <= eb; ++fb)
#pragma unroll
                            for (int fc = 0; fc <= ec; ++fc) {
                                const int deg = fa + fb + fc;
                                if (deg == 1) continue;
                                const float Rf = deg == 0 ? A.w : Rc[raw_off(deg) + mono_idx(fa, fb, fc)];
                                v += (binomf(ea, fa) * binomf(eb, fb) * binomf(ec, fc)) * Rf *
                                     (sx[ea - fa] * sy[eb - fb] * sz[ec - fc]);
                            }
                    R[raw_off(n) + mono_idx(ea, eb, ec)] = v;
                }
    }
#pragma unroll
    for (int k = 0; k < 31; ++k) R[k] = sum8(R[k]);
    if ((t & 7) != 0) return;
    if (M == 0.f) {
        put_node(a, g, f3(0, 0, 0), 0.f, R, 0.f);
        return;
    }
    float3 lo;
    float edge;
    tree_cube(a, p, lo, edge);
    put_node(a, g, c, M, R, opening2(c, cell_centre(lo, edge, L, m), edge / (float)(1 << L), S.theta));
}

// The walk of each group of spheres starts from the 64 cells of level kSplitL,
// dealt round robin to kTreeParts warps (so that the cells around the group,
// the long walks, go to different warps).  Measured, us per step with 8 / 16 /
// 32 / 64 warps: 100,000-sphere cloud (theta 0.7) 530 / 508 / 545 / 632, dense
// 50,000-sphere pile (0.5) 495 / 436 / 422 / 437, 10,000-sphere cloud 132 /
// 116 / 118 / 122, dense 200,000-sphere pile (0.5) 1,766 / 1,814 / 1,840 /
// 1,881; with four neighbouring cells each instead of every 16th, the first
// two were 621 and 529.
constexpr int kSplitL = 2;

// Traversal stack per warp: opened cells whose children are still to be
// tested.  A round takes the 4 top entries (or what is left) and puts at most
// 32 children in their place, so a child lies at most 31 places above its
// parent.  The walk's first cells fill at most 64 / kTreeParts places, and
// the cells on the stack are of the levels kSplitL .. kTreeMaxDepth - 1 (the
// deepest level's are leaves): no place above the last is ever used.
constexpr int kTreeStack = 64 / kTreeParts + 31 * (kTreeMaxDepth - 1 - kSplitL);

// The multipoles up to rank ORDER of two cells on the sphere at x: a / G, one
// cell in each half of the packed operands.  With u the unit vector from the
// cell's COM to x and r the distance,
//   a / G = -M u / r^2 + sum_n (n T_n . u^(n-1) - (2n+1) (T_n . u^n) u) / r^(n+2),
// the gradient of the potential -G (M / r + sum_n T_n . x^n / r^(2n+1))
// (unit-vector form: no power of r above the sixth is formed).
template <int ORDER>
__device__ __forceinline__ void node_force2(const f2_t *nd, f2_t x, f2_t y, f2_t z, f2_t &ax, f2_t &ay, f2_t &az)
{
    const f2_t dx = f2_sub(x, nd[0]), dy = f2_sub(y, nd[1]), dz = f2_sub(z, nd[2]);
    float ra, rb;
    f2_unpack(f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx))), ra, rb);
    const f2_t inv = f2_pack(rsqrtf(ra), rsqrtf(rb));
    f2_t px[4], py[4], pz[4];
    const f2_t one = f2_dup(1.f), zero = f2_dup(0.f);
    auto powers = [&](f2_t d, f2_t *p) {
        p[0] = one;
        p[1] = f2_mul(d, inv);
        p[2] = f2_mul(p[1], p[1]);
        if (ORDER > 3) p[3] = f2_mul(p[2], p[1]);
    };
    powers(dx, px);
    powers(dy, py);
    powers(dz, pz);
    f2_t tx = zero, ty = zero, tz = zero;   // sum_n t_n / r^(n-2), Horner in 1/r from the top rank
#pragma unroll
    for (int n = ORDER; n >= 2; --n) {
        const f2_t *T = nd + node_off(n);
        f2_t vx = zero, vy = zero, vz = zero;   // T_n . u^(n-1)
#pragma unroll
        for (int fa = n - 1; fa >= 0; --fa)
#pragma unroll
            for (int fb = n - 1 - fa; fb >= 0; --fb) {
                const int fc = n - 1 - fa - fb;
                const float wt = factf(n - 1) / (factf(fa) * factf(fb) * factf(fc));
                f2_t w = fa == 0 ? (fb == 0 ? pz[fc] : fc == 0 ? py[fb] : f2_mul(py[fb], pz[fc]))
                         : fb == 0 ? (fc == 0 ? px[fa] : f2_mul(px[fa], pz[fc]))
                         : fc == 0 ? f2_mul(px[fa], py[fb]) : f2_mul(px[fa], f2_mul(py[fb], pz[fc]));
                if (wt != 1.f) w = f2_mul(w, f2_dup(wt));
                vx = f2_fma(w, T[mono_idx(fa + 1, fb, fc)], vx);
                vy = f2_fma(w, T[mono_idx(fa, fb + 1, fc)], vy);
                vz = f2_fma(w, T[mono_idx(fa, fb, fc + 1)], vz);
            }
        const f2_t sn = f2_fma(vz, pz[1], f2_fma(vy, py[1], f2_mul(vx, px[1])));   // T_n . u^n
        const f2_t k1 = f2_dup((float)n), k2 = f2_mul(sn, f2_dup(-(float)(2 * n + 1)));
        tx = f2_fma(k1, vx, f2_fma(k2, px[1], f2_mul(tx, inv)));
        ty = f2_fma(k1, vy, f2_fma(k2, py[1], f2_mul(ty, inv)));
        tz = f2_fma(k1, vz, f2_fma(k2, pz[1], f2_mul(tz, inv)));
    }
    const f2_t inv2 = f2_mul(inv, inv), M = f2_mul(nd[3], f2_dup(-1.f));
    ax = f2_fma(inv2, f2_fma(tx, inv2, f2_mul(M, px[1])), ax);
    ay = f2_fma(inv2, f2_fma(ty, inv2, f2_mul(M, py[1])), ay);
    az = f2_fma(inv2, f2_fma(tz, inv2, f2_mul(M, pz[1])), az);
}

// One warp walks the tree for a group of 32 consecutive spheres in leaf
// order.  Each round takes up to 4 opened cells off the warp's stack and tests
// their children, one per lane, against the group's bounding box: a cell is
// accepted when the box is farther from its COM than its opening radius (so
// the test holds for every sphere of the group), an opened leaf is summed
// directly, any other opened cell goes on the stack.  Every lane then adds its
// own sphere's interaction with the round's accepted cells, two at a time (the
// lanes that accepted them stage them in shared memory as packed pairs), and
// with the spheres of its opened leaves, also two at a time, so the arithmetic
// has no divergence and the loads of a round overlap.
// Groups are 32 consecutive spheres of one pile in leaf order, counted from
// the pile's first sphere, so a pile's result does not depend on the other
// piles of the batch.  The walk of each group is split over kTreeParts
// warps (grid dimension y), each writing its partial sum, which k_tree_combine
// adds in order.
//
// Latency-bound (the rounds depend on one another; 42% of the issue slots,
// 28 warps an SM by registers).  A stack of cells still to be tested (4 KB)
// held 22 warps an SM and a cell at a time took twice the instructions: the
// 100,000-sphere cloud at theta 0.7 went from 758 to 427 us (ncu), its whole
// step with the lighter build around the walk from 1,041 to 508 us.
template <int ORDER>
__global__ void __launch_bounds__(32) k_tree_force(Arrays a, Sizes z)
{
    pdl_enter();
    // one warp per block: walks of very different lengths do not hold one
    // another's block resident
    constexpr int kNC = ORDER > 2 ? 36 : 11;       // a cell's components in use
    constexpr int kPairF2 = ORDER > 2 ? 38 : 14;   // components of a staged pair and padding (16-byte rows)
    constexpr int kLeafStage = 192;                // spheres of opened leaves staged at a time
    constexpr int kStageBytes = 16 * kPairF2 * 8 > kLeafStage * 20 ? 16 * kPairF2 * 8 : kLeafStage * 20;
    __shared__ int st[kTreeStack];
    __shared__ __align__(16) unsigned char stage[kStageBytes];
    __shared__ int lbase[32], lfirst[32];
    f2_t *cells = (f2_t *)stage;                   // [16][kPairF2]
    ulonglong2 *lxy = (ulonglong2 *)stage, *lzm = lxy + kLeafStage / 2;
    int2 *lag = (int2 *)(lzm + kLeafStage / 2);
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const int sub = blockIdx.y;      // subtree
    const int64_t wg = blockIdx.x;   // group
    if (wg >= z.TG) return;
    int lo = 0, hi = (int)z.P - 1;   // pile of the group
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.ps[mid].tg0 <= wg) lo = mid; else hi = mid - 1;
    }
    const int pp = lo;
    if (!tree_pile(a, pp)) return;   // uniform over the warp
    const PileStatic &S = a.ps[pp];
    const int64_t s0 = S.s0;
    const int ti = (int)(32 * (wg - S.tg0)) + lane;   // leaf-order position in the pile
    const bool mine = ti < S.ns;
    const int64_t k = s0 + ti;
    const float4 xi = mine ? a.tpos[k] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int ai = mine ? a.tagg[k] : -2;
    // group box (lanes past the pile's end take lane 0's position)
    const float lx = __shfl_sync(FULL, xi.x, 0), ly = __shfl_sync(FULL, xi.y, 0),
                lz = __shfl_sync(FULL, xi.z, 0);
    float bx0 = mine ? xi.x : lx, by0 = mine ? xi.y : ly, bz0 = mine ? xi.z : lz;
    float bx1 = bx0, by1 = by0, bz1 = bz0;
    for (int o = 16; o > 0; o >>= 1) {
        bx0 = fminf(bx0, __shfl_xor_sync(FULL, bx0, o));
        by0 = fminf(by0, __shfl_xor_sync(FULL, by0, o));
        bz0 = fminf(bz0, __shfl_xor_sync(FULL, bz0, o));
        bx1 = fmaxf(bx1, __shfl_xor_sync(FULL, bx1, o));
        by1 = fmaxf(by1, __shfl_xor_sync(FULL, by1, o));
        bz1 = fmaxf(bz1, __shfl_xor_sync(FULL, bz1, o));
    }
    const f2_t e2 = f2_dup((float)S.eps2);
    const f2_t xx = f2_dup(xi.x), xy = f2_dup(xi.y), xz = f2_dup(xi.z);
    const int D = S.tD;
    const float4 *nodes = a.tnode + kNodeF4 * S.tnode0;
    const int2 *leaves = a.tleaf + S.tleaf0;
    const float4 *tp = a.tpos + s0;
    const int32_t *tg = a.tagg + s0;
    f2_t ax = f2_dup(0.f), ay = ax, az = ax;
    int sp = 0;
    // first round: this warp's cells of level kSplitL
    int n = lane * kTreeParts < 64 ? (int)lvl_off(kSplitL) + sub + lane * kTreeParts : -1, L = kSplitL;
    for (;;) {
        // test this lane's cell
        float4 A = make_float4(0.f, 0.f, 0.f, 0.f), B = A;
        bool acc = false, leaf = false, open = false;
        int2 lf = make_int2(0, 0);
        if (n >= 0) {
            A = nodes[kNodeF4 * n];
            B = nodes[kNodeF4 * n + 1];   // opening radius^2, T2
            if (A.w != 0.f) {
                const float gx = fmaxf(fmaxf(bx0 - A.x, A.x - bx1), 0.f);
                const float gy = fmaxf(fmaxf(by0 - A.y, A.y - by1), 0.f);
                const float gz = fmaxf(fmaxf(bz0 - A.z, A.z - bz1), 0.f);
                acc = gx * gx + gy * gy + gz * gz > B.x;
                leaf = !acc && L == D;
                open = !acc && L < D;
                if (leaf) lf = leaves[n - lvl_off(D)];
            }
        }
        // opened cells go on the stack
        const unsigned om = __ballot_sync(FULL, open);
        if (open) st[sp + __popc(om & below)] = (n << 3) | L;
        sp += __popc(om);
        // accepted cells: staged in pairs (a last odd one with a massless cell
        // far away), then every lane adds each pair
        const unsigned am = __ballot_sync(FULL, acc);
        const int na = __popc(am);
        if (acc || (lane == 0 && (na & 1))) {
            if (acc) {
                const int s = __popc(am & below);
                float *c = (float *)(cells + (s >> 1) * kPairF2) + (s & 1);
                const float4 *nd = nodes + kNodeF4 * n;
                float v[36] = {A.x, A.y, A.z, A.w, B.x, B.y, B.z, B.w};
#pragma unroll
                for (int q = 2; q < (kNC + 3) / 4; ++q) {
                    const float4 t = nd[q];
                    v[4 * q] = t.x; v[4 * q + 1] = t.y; v[4 * q + 2] = t.z; v[4 * q + 3] = t.w;
                }
#pragma unroll
                for (int q = 0; q < kNC; ++q) c[2 * q] = v[q];
            }
            if (lane == 0 && (na & 1)) {
                float *c = (float *)(cells + (na >> 1) * kPairF2) + 1;
                for (int q = 0; q < kNC; ++q) c[2 * q] = q < 3 ? 1.0e18f : 0.f;
            }
        }
        __syncwarp();
        for (int p2 = 0; 2 * p2 < na; ++p2) node_force2<ORDER>(cells + p2 * kPairF2, xx, xy, xz, ax, ay, az);
        __syncwarp();
        // opened leaves: the spheres of all of them (leaves in lane order,
        // spheres in leaf order) are staged in pairs, kLeafStage at a time, one
        // round of loads for the whole round's leaves, then every lane adds
        // each pair.  A sphere's own aggregate is skipped, and with it the
        // sphere itself.
        const int lcnt = leaf ? lf.y : 0;
        if (__ballot_sync(FULL, lcnt > 0)) {
            int incl = lcnt;
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += v;
            }
            const int total = __shfl_sync(FULL, incl, 31);
            lbase[lane] = incl - lcnt;   // first staged position of this lane's leaf
            lfirst[lane] = lf.x;         // first sphere of the leaf (leaf order)
            __syncwarp();
            for (int c0 = 0; c0 < total; c0 += kLeafStage) {
                const int nb = min(kLeafStage, total - c0);
                for (int t = lane; t < ((nb + 1) & ~1); t += 32) {
                    float4 v = make_float4(1.0e18f, 1.0e18f, 1.0e18f, 0.f);
                    int g = -1;
                    if (t < nb) {
                        // the leaf holding staged position c0 + t: the last lane
                        // whose first staged position is not after it
                        int lo2 = 0, hi2 = 31;
                        while (lo2 < hi2) {
                            const int mid = (lo2 + hi2 + 1) >> 1;
                            if (lbase[mid] <= c0 + t) lo2 = mid; else hi2 = mid - 1;
                        }
                        const int idx = lfirst[lo2] + (c0 + t - lbase[lo2]);
                        v = tp[idx];
                        g = tg[idx];
                    }
                    float *q = (float *)(lxy + (t >> 1)) + (t & 1), *r = (float *)(lzm + (t >> 1)) + (t & 1);
                    q[0] = v.x; q[2] = v.y; r[0] = v.z; r[2] = v.w;
                    ((int *)(lag + (t >> 1)))[t & 1] = g;
                }
                __syncwarp();
#pragma unroll 2
                for (int u = 0; 2 * u < nb; ++u) {
                    const ulonglong2 ja = lxy[u], jb = lzm[u];
                    const int2 g = lag[u];
                    const f2_t ex = f2_sub(ja.x, xx), ey = f2_sub(ja.y, xy), ez = f2_sub(jb.x, xz);
                    float ra, rb, sa, sb;
                    f2_unpack(f2_fma(ez, ez, f2_fma(ey, ey, f2_fma(ex, ex, e2))), ra, rb);
                    const f2_t iv = f2_pack(rsqrtf(ra), rsqrtf(rb));
                    f2_unpack(f2_mul(f2_mul(jb.y, iv), f2_mul(iv, iv)), sa, sb);
                    const f2_t sj = f2_pack(g.x == ai ? 0.f : sa, g.y == ai ? 0.f : sb);
                    ax = f2_fma(ex, sj, ax);
                    ay = f2_fma(ey, sj, ay);
                    az = f2_fma(ez, sj, az);
                }
                __syncwarp();
            }
        }
        // next round: the children of up to 4 opened cells
        if (sp == 0) break;
        const int cnt = min(sp, 4);
        n = -1;
        if ((lane >> 3) < cnt) {
            const int e = st[sp - 1 - (lane >> 3)];
            L = (e & 7) + 1;
            n = (int)(lvl_off(L) + 8 * ((e >> 3) - lvl_off(L - 1))) + (lane & 7);
        }
        sp -= cnt;
        __syncwarp();
    }
    float x0, x1, y0, y1, z0, z1;
    f2_unpack(ax, x0, x1);
    f2_unpack(ay, y0, y1);
    f2_unpack(az, z0, z1);
    if (mine) a.tpart[(int64_t)sub * z.N + k] = make_float4(x0 + x1, y0 + y1, z0 + z1, 0.f);
}

// Sum the subtree partials of each sphere (float-float, fixed order).
__global__ void k_tree_combine(Arrays a, Sizes z)
{
    pdl_enter();
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= z.N) return;
    const int p = a.sph_pile[k];
    if (!tree_pile(a, p)) return;
    const PileStatic &S = a.ps[p];
    FFSum sx, sy, sz;
#pragma unroll 8
    for (int s = 0; s < kTreeParts; ++s) {
        const float4 v = a.tpart[(int64_t)s * z.N + k];
        sx.add(v.x); sy.add(v.y); sz.add(v.z);
    }
    const int i = a.tsorted[k];
    const double gm = S.G * a.m64[S.s0 + i];
    a.fg[S.s0 + i] = make_dbl4(gm * sx.value(), gm * sy.value(), gm * sz.value(), 0.0);
}

void launch_tree_gravity(const Arrays &a, const Sizes &z, int max_depth, int order, cudaStream_t st)
{
    if (z.N == 0 || z.TN == 0) return;
    const unsigned nb = (unsigned)((z.N + 255) / 256);
    const int64_t ni = z.TL > 6 * z.P ? z.TL : 6 * z.P;
    launch_pdl(k_tree_init, (unsigned)((ni + 255) / 256), 256, 0, st, a, z);
    launch_pdl(k_tree_box, (unsigned)((z.N + kBoxThreads - 1) / kBoxThreads), kBoxThreads, 0, st, a, z);
    launch_pdl(k_tree_keys, nb, 256, 0, st, a, z);
    const int64_t nl = (int64_t)1 << (3 * max_depth);
    const dim3 tiles((unsigned)z.P, (unsigned)((nl + kLeafTile - 1) / kLeafTile));
    if (tiles.y > 1) launch_pdl(k_tree_sums, tiles, kScanThreads, 0, st, a, z);
    launch_pdl(k_tree_scan, tiles, kScanThreads, 0, st, a, z);
    launch_pdl(k_tree_scatter, nb, 256, 0, st, a, z);
    launch_pdl(k_tree_gather, nb, 256, 0, st, a, z);
    launch_pdl(k_tree_leaves, (unsigned)((z.TL + 127) / 128), 128, 0, st, a, z);
    for (int L = max_depth - 1; L >= kSplitL; --L)
        launch_pdl(k_tree_up, dim3((unsigned)z.P, (unsigned)((((int64_t)8 << (3 * L)) + 127) / 128)), 128, 0,
                   st, a, z, L);
    if (order == 2) launch_pdl(k_tree_force<2>, dim3((unsigned)z.TG, kTreeParts), 32, 0, st, a, z);
    else launch_pdl(k_tree_force<4>, dim3((unsigned)z.TG, kTreeParts), 32, 0, st, a, z);
    launch_pdl(k_tree_combine, nb, 256, 0, st, a, z);
}

}  // namespace dem
