// kernels_contact.cu -- the contact pass: uniform cells of a wrapped grid,
// pairs inside one aggregate skipped (Sec. 2.2: members are rigidly bonded),
// linear spring-dashpot normal force, tangential spring with history and
// Coulomb cap, rolling and twisting couples (Sec. 2.1, Sec. 2.2.5), applied at
// the contact point at the centre of the intersection circle (Sec. 2.2.4,
// Eq. lever_arm).
//
// Candidate lists (built in kernels_lists.cu): at a rebuild every sphere lists
// the spheres of other aggregates whose centres are closer than the radii sum
// plus the skin, in the order of their home indices, in compressed rows per
// sorted sphere; every entry has the position of the same pair in the
// partner's list and whether its sphere owns the pair (the lower home index).
// The lists stay complete until some aggregate may have moved half the skin
// (checked at the drift).
//
// Shares of a pair.  Both spheres' shares come from one evaluation with the
// owner as sphere a:
//   a:  F,  tau_a = (l_a n) x F + M;   b:  -F,  tau_b = (l_b n) x F - M.
// The law is written with every operation's rounding pinned, and each of its
// steps maps exactly onto its negative or onto itself when the two spheres
// swap, so an evaluation with b as sphere a gives b's share bit for bit.
// Two forms of the pass, with bitwise the same results:
//   k_contact_sphere (the default): one thread per sorted sphere evaluates
//     every entry of its list with itself as sphere a (each pair twice, once
//     per sphere), sums its shares in list order and writes its own history;
//   k_contact (contact_mode 1): tiles of kCTile consecutive sorted spheres,
//     which fill compact blocks of space (cells are numbered brick by brick);
//     a pair inside a tile is evaluated once, by the thread that drew it from
//     the tile's work queue, and both shares go to the spheres' slots in a
//     shared-memory inbox; a pair that crosses tiles is evaluated by both
//     tiles, each keeping its own sphere's share.
// Every sphere sums its shares in list order, i.e. in the order of its
// partners' home indices, so forces, torques and history are bitwise the same
// whatever the form, the tiles, the cell size, the skin or the steps at which
// the lists were rebuilt.  Nothing is written with atomics except error flags.
//
// History (Sec. 2.1: the tangential displacement is tracked while the two
// spheres stay in contact) lives at each sphere's own list entry, from its own
// side, with .w = 1 while in contact: the two sides' evaluations give exactly
// opposite displacements, so the copies never differ but in sign, and every
// access is to consecutive entries of a warp and known ahead.  (Kept once, at
// the owner's entry, the partner's side read it out of order, often a second
// time from HBM: 272 us on the 1M lattice, 197 so.)  A rebuild carries it over
// to the new lists by partner index.
//
// Mixed precision positions.  The overlap x = s_a + s_b - |d| of two nearby
// spheres needs more than FP32's 24 bits of |d|.  Each sphere's position
// relative to the pile frame is held as the low 32 bits of round(r / q) per
// axis, q = 2^qexp with 2^31 q >= 10.5 x the largest radius (so that a
// candidate pair's difference fits in int32 after any allowed motion), its
// radius as round(s / q), and the four rounding remainders in FP32.  The
// integer difference is exact and the large cancellation in
// (s_a + s_b)^2 - |d|^2 happens exactly in int64; the remainders add small
// FP32 corrections, so x = ((s_a + s_b)^2 - |d|^2) / (s_a + s_b + |d|) keeps
// FP32 relative accuracy; the rest of the law is FP32.
//
// Force law (the paper defers the constants and form to earlier work):
//   d = r_b - r_a, n = d/|d|, x = s_a + s_b - |d| > 0 (overlap),
//   l_a = (s_a^2 - s_b^2 + |d|^2) / (2|d|), l_b = |d| - l_a,
//   u = (v_b + w_b x (-l_b n)) - (v_a + w_a x (l_a n)), u_n = (u.n) n, u_t = u - u_n,
//   F_N = -kn x n + cn u_n,
//   S = (S_prev projected on the tangent plane, rescaled to |S_prev|) + u_t h,
//   F_T = kt S + ct u_t, capped at mu_s |F_N| (then S = (F_T - ct u_t)/kt),
//   M = -mu_r |F_N| R w_r / max(|w_r|, w0) - mu_t |F_N| R w_t / max(|w_t|, w0),
//     w = w_a - w_b, w_t = (w.n) n, w_r = w - w_t, R = s_a s_b / (s_a + s_b).
#include "dem_internal.h"
#include "devmath.cuh"
#include "launch.cuh"
#include "reduce.cuh"

namespace dem {

struct ParamsF {
    float kn, kt, cn, ct, mu_s, mu_r, mu_t, w0, h;
};
struct ParamsD {
    double kn, kt, cn, ct, mu_s, mu_r, mu_t, w0, h;
};

template <typename T, typename V>
struct PairOut {
    V F, M, S, n;
    T la, lb, x, rmin;
};

// Division and square root of the force law: fast hardware approximations in
// FP32 (relative error ~1e-7, far inside the FP32 path's tolerance), IEEE in FP64.
__device__ __forceinline__ float qdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double qdiv(double a, double b) { return a / b; }
__device__ __forceinline__ float qsqrt(float x) { return x > 0.f ? x * rsqrtf(x) : 0.f; }
__device__ __forceinline__ double qsqrt(double x) { return sqrt(x); }

// Correctly rounded operations for the force law: every product, sum and
// fused multiply-add is written out, so the compiler neither contracts nor
// reassociates anything and the law gives the same bits in every kernel
// that inlines it (the pair kernels rely on that for bitwise results).
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double rsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }
template <typename T, typename V> __device__ __forceinline__ V vmk(T x, T y, T z);
template <> __device__ __forceinline__ float3 vmk<float, float3>(float x, float y, float z) { return f3(x, y, z); }
template <> __device__ __forceinline__ double3 vmk<double, double3>(double x, double y, double z) { return d3(x, y, z); }
template <typename T, typename V> __device__ __forceinline__ V vscale(T s, V a)
{ return vmk<T, V>(rmul(s, a.x), rmul(s, a.y), rmul(s, a.z)); }
template <typename T, typename V> __device__ __forceinline__ V vadd(V a, V b)
{ return vmk<T, V>(radd(a.x, b.x), radd(a.y, b.y), radd(a.z, b.z)); }
template <typename T, typename V> __device__ __forceinline__ V vsub(V a, V b)
{ return vmk<T, V>(rsub(a.x, b.x), rsub(a.y, b.y), rsub(a.z, b.z)); }
template <typename T, typename V> __device__ __forceinline__ V vaxpy(T s, V a, V b)   // s a + b
{ return vmk<T, V>(rfma(s, a.x, b.x), rfma(s, a.y, b.y), rfma(s, a.z, b.z)); }
template <typename T, typename V> __device__ __forceinline__ T vdot(V a, V b)
{ return rfma(a.z, b.z, rfma(a.y, b.y, rmul(a.x, b.x))); }
template <typename T, typename V> __device__ __forceinline__ V vcross(V a, V b)
{
    return vmk<T, V>(rfma(a.y, b.z, -rmul(a.z, b.y)), rfma(a.z, b.x, -rmul(a.x, b.z)),
                     rfma(a.x, b.y, -rmul(a.y, b.x)));
}
__device__ __forceinline__ float rdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double rdiv(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ float rnorm(float x) { return x > 0.f ? rmul(x, rsqrtf(x)) : 0.f; }
__device__ __forceinline__ double rnorm(double x) { return __dsqrt_rn(x); }

// Tangential spring, Coulomb cap and rolling/twisting couples, shared by
// both precisions (T = float or double).
template <typename T, typename V, typename P>
__device__ __forceinline__ void force_law(V n, T x, T la, T lb, V va, V wa, V vb, V wb, T sa,
                                          T sb, V Sprev, const P &prm, PairOut<T, V> &o)
{
    // relative velocity of b's contact point with respect to a's
    const V ca = vscale<T, V>(la, n), cb = vscale<T, V>(-lb, n);
    const V u = vsub<T, V>(vadd<T, V>(vb, vcross<T, V>(wb, cb)), vadd<T, V>(va, vcross<T, V>(wa, ca)));
    const T uns = vdot<T, V>(u, n);
    const V ut = vaxpy<T, V>(-uns, n, u);                 // u - (u.n) n
    // F_N is along n: its signed magnitude is -kn x + cn (u.n)
    const T fn = rfma(prm.cn, uns, -rmul(prm.kn, x));
    const T FNm = fabs(fn);
    // tangential spring: S_prev on the new tangent plane, rescaled to |S_prev|
    V Sp = vaxpy<T, V>(-vdot<T, V>(Sprev, n), n, Sprev);
    const T Spm = rnorm(vdot<T, V>(Sp, Sp)), Sprevm = rnorm(vdot<T, V>(Sprev, Sprev));
    Sp = Spm > T(0) ? vscale<T, V>(rdiv(Sprevm, Spm), Sp) : vmk<T, V>(T(0), T(0), T(0));
    V S = vaxpy<T, V>(prm.h, ut, Sp);
    V FT = vaxpy<T, V>(prm.ct, ut, vscale<T, V>(prm.kt, S));
    const T FTm = rnorm(vdot<T, V>(FT, FT)), cap = rmul(prm.mu_s, FNm);
    if (FTm > cap) {
        FT = vscale<T, V>(rdiv(cap, FTm), FT);
        S = prm.kt > T(0) ? vscale<T, V>(rdiv(T(1), prm.kt), vaxpy<T, V>(-prm.ct, ut, FT))
                          : vmk<T, V>(T(0), T(0), T(0));
    }
    // rolling and twisting couples
    const V w = vsub<T, V>(wa, wb);
    const T wn = vdot<T, V>(w, n);
    const V wt = vscale<T, V>(wn, n);
    const V wr = vsub<T, V>(w, wt);
    const T Rred = rdiv(rmul(sa, sb), radd(sa, sb));
    V M = vmk<T, V>(T(0), T(0), T(0));
    if (prm.mu_r > T(0)) {
        const T wrm = rnorm(vdot<T, V>(wr, wr));
        if (wrm > T(0)) M = vscale<T, V>(rdiv(-rmul(rmul(prm.mu_r, FNm), Rred), fmax(wrm, prm.w0)), wr);
    }
    if (prm.mu_t > T(0)) {
        const T wtm = rnorm(vdot<T, V>(wt, wt));
        if (wtm > T(0)) M = vaxpy<T, V>(rdiv(-rmul(rmul(prm.mu_t, FNm), Rred), fmax(wtm, prm.w0)), wt, M);
    }
    o.F = vaxpy<T, V>(fn, n, FT);                         // F_N + F_T
    o.M = M;
    o.S = S;
    o.n = n;
    o.la = la;
    o.lb = lb;
    o.x = x;
}

// Mixed-precision pair from fixed-point positions (see the file comment).
// A, B: (x, y, z low 32 bits, radius) in quanta q; RA, RB: the remainders of
// those roundings (in quanta).  In quanta, with d = D_i + dd_i per axis (D_i
// the exact integer difference, |dd_i| <= 1) and s = S + rho (S the integer
// radii sum):
//   (s_a + s_b)^2 - |d|^2 = (S^2 - sum D_i^2) + 2 S rho + rho^2
//                           - 2 sum D_i dd_i - sum dd_i^2,
// the first bracket exact in int64 (the large cancellation), the small terms
// in FP32; x = that / (s + |d|).
__device__ __forceinline__ bool pair_mixed(int4 A, float4 RA, int4 B, float4 RB, float q, float4 av,
                                           float4 aw, float4 bv, float4 bw, float3 Sprev,
                                           const ParamsF &prm, PairOut<float, float3> &o)
{
    const int dx = (int)((unsigned)B.x - (unsigned)A.x);
    const int dy = (int)((unsigned)B.y - (unsigned)A.y);
    const int dz = (int)((unsigned)B.z - (unsigned)A.z);
    const long long D = (long long)dx * dx + (long long)dy * dy + (long long)dz * dz;
    const int Ss = A.w + B.w;
    const long long num_i = (long long)Ss * Ss - D;
    const float ex = __fsub_rn(RB.x, RA.x), ey = __fsub_rn(RB.y, RA.y), ez = __fsub_rn(RB.z, RA.z);
    const float rho = __fadd_rn(RA.w, RB.w);
    const float fx = __int2float_rn(dx), fy = __int2float_rn(dy), fz = __int2float_rn(dz);
    const float Ssf = __int2float_rn(Ss);
    const float cr = __fmaf_rn(fz, ez, __fmaf_rn(fy, ey, __fmul_rn(fx, ex)));
    const float ee = __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmul_rn(ex, ex)));
    const float corr = __fsub_rn(__fsub_rn(__fmaf_rn(__fmul_rn(2.0f, Ssf), rho, __fmul_rn(rho, rho)),
                                           __fmul_rn(2.0f, cr)), ee);
    // the int64 bracket to FP32 from its 32-bit halves (two 32-bit conversions
    // and one FMA, off the FP64 unit that a 64-bit conversion would use;
    // within 2 ulp of the correctly rounded value and symmetric in a, b)
    const float numi = __fmaf_rn(__int2float_rn((int)(num_i >> 32)), 4294967296.0f,
                                 __uint2float_rn((unsigned)(num_i & 0xffffffffll)));
    const float num = __fadd_rn(numi, corr);
    if (!(num > 0.0f)) return false;
    const float3 d = f3(__fadd_rn(fx, ex), __fadd_rn(fy, ey), __fadd_rn(fz, ez));
    const float Df = __fmaf_rn(d.z, d.z, __fmaf_rn(d.y, d.y, __fmul_rn(d.x, d.x)));
    if (!(Df > 0.0f)) return false;
    const float inv = rsqrtf(Df);
    const float dist = __fmul_rn(Df, inv);
    const float3 n = f3(__fmul_rn(d.x, inv), __fmul_rn(d.y, inv), __fmul_rn(d.z, inv));
    const float sqa = __fadd_rn(__int2float_rn(A.w), RA.w), sqb = __fadd_rn(__int2float_rn(B.w), RB.w);
    const float ssum = __fadd_rn(sqa, sqb);
    const float x = __fmul_rn(__fdividef(num, __fadd_rn(ssum, dist)), q);
    // l_a, l_b = |d|/2 +- (s_a - s_b)(s_a + s_b)/(2|d|)
    const float hd = __fmul_rn(0.5f, dist);
    const float g = __fmul_rn(__fmul_rn(0.5f, __fsub_rn(sqa, sqb)), __fmul_rn(ssum, inv));
    const float la = __fmul_rn(__fadd_rn(hd, g), q);
    const float lb = __fmul_rn(__fsub_rn(hd, g), q);
    const float sa = __fmul_rn(sqa, q), sb = __fmul_rn(sqb, q);
    o.rmin = fminf(sa, sb);
    force_law<float, float3, ParamsF>(n, x, la, lb, f3(av.x, av.y, av.z), f3(aw.x, aw.y, aw.z),
                                      f3(bv.x, bv.y, bv.z), f3(bw.x, bw.y, bw.z), sa, sb, Sprev, prm, o);
    return true;
}

__device__ __forceinline__ bool pair_64(dbl4 ap, dbl4 av, dbl4 aw, dbl4 bp, dbl4 bv, dbl4 bw,
                                        double3 Sprev, const ParamsD &prm, PairOut<double, double3> &o)
{
    const double3 d = d3(__dsub_rn(bp.x, ap.x), __dsub_rn(bp.y, ap.y), __dsub_rn(bp.z, ap.z));
    const double dist = __dsqrt_rn(vdot<double, double3>(d, d));
    const double x = __dsub_rn(__dadd_rn(ap.w, bp.w), dist);
    if (!(x > 0.0) || !(dist > 0.0)) return false;
    const double inv = __ddiv_rn(1.0, dist);
    const double3 n = vscale<double, double3>(inv, d);
    const double hd = __dmul_rn(0.5, dist);
    const double g = __dmul_rn(__dmul_rn(__dsub_rn(ap.w, bp.w), __dadd_rn(ap.w, bp.w)), __dmul_rn(0.5, inv));
    double la = __dadd_rn(hd, g);
    double lb = __dsub_rn(hd, g);
    o.rmin = fmin(ap.w, bp.w);
    force_law<double, double3, ParamsD>(n, x, la, lb, d3(av.x, av.y, av.z), d3(aw.x, aw.y, aw.z),
                                        d3(bv.x, bv.y, bv.z), d3(bw.x, bw.y, bw.z), ap.w, bp.w, Sprev, prm, o);
    return true;
}

// The two spheres' shares of one evaluation, every operation pinned to its
// rounding (no contraction), so a share is the same bits wherever it is formed.
__device__ __forceinline__ float3 lever_x_force(float l, float3 n, float3 F)
{
    const float3 c = f3(__fmul_rn(l, n.x), __fmul_rn(l, n.y), __fmul_rn(l, n.z));
    return f3(__fmaf_rn(c.y, F.z, __fmul_rn(-c.z, F.y)), __fmaf_rn(c.z, F.x, __fmul_rn(-c.x, F.z)),
              __fmaf_rn(c.x, F.y, __fmul_rn(-c.y, F.x)));
}
__device__ __forceinline__ double3 lever_x_force(double l, double3 n, double3 F)
{
    const double3 c = d3(__dmul_rn(l, n.x), __dmul_rn(l, n.y), __dmul_rn(l, n.z));
    return d3(__fma_rn(c.y, F.z, __dmul_rn(-c.z, F.y)), __fma_rn(c.z, F.x, __dmul_rn(-c.x, F.z)),
              __fma_rn(c.x, F.y, __dmul_rn(-c.y, F.x)));
}
__device__ __forceinline__ float addr(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double addr(double a, double b) { return __dadd_rn(a, b); }

// One sphere's share of an evaluation: sphere a (side_a) gets F and
// (l_a n) x F + M, sphere b gets -F and (l_b n) x F - M.
template <typename T, typename V>
__device__ __forceinline__ void share(const PairOut<T, V> &o, bool side_a, V &F, V &Tq)
{
    const T sg = side_a ? T(1) : T(-1);
    const V c = lever_x_force(side_a ? o.la : o.lb, o.n, o.F);
    F = vmk<T, V>(sg * o.F.x, sg * o.F.y, sg * o.F.z);
    Tq = vmk<T, V>(addr(c.x, sg * o.M.x), addr(c.y, sg * o.M.y), addr(c.z, sg * o.M.z));
}

template <bool FP64> struct CT;
template <> struct CT<false> {
    typedef float T;
    typedef float3 V;
    typedef ParamsF Prm;
    typedef float4 H;                      // history record
    typedef int4 P;                        // position record
    typedef float4 VR;                     // velocity / spin record
    static constexpr int kCap = kInboxCap; // inbox entries per block
};
template <> struct CT<true> {
    typedef double T;
    typedef double3 V;
    typedef ParamsD Prm;
    typedef dbl4 H;
    typedef dbl4 P;
    typedef dbl4 VR;
    static constexpr int kCap = kInboxCap / 2;
};

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }
__device__ __forceinline__ float4 as_f4(int4 v)
{
    return make_float4(__int_as_float(v.x), __int_as_float(v.y), __int_as_float(v.z), __int_as_float(v.w));
}

// ---------------------------------------------------------------- step
// One sorted sphere k: every entry of its list is evaluated with the sphere as
// sphere a (see the file comment); it keeps its own share, summed in list order,
// and its own history.  Each pair is evaluated twice (once per sphere), with
// exactly opposite results, so the forces equal the tile form's bit for bit.
// s_x / s_v: the sorted spheres [kb0, kb0 + 128) staged in shared memory
// (mixed path), or null.
template <bool FP64>
__device__ __forceinline__ void sphere_contacts(const Arrays &a, const PileStatic &S, int lp,
                                                const typename CT<FP64>::H *hread,
                                                typename CT<FP64>::H *hwrite,
                                                const typename CT<FP64>::Prm &prm, float q, int64_t k,
                                                int64_t kb0, const int4 *s_x, const float4 *s_v, int &flags)
{
    typedef typename CT<FP64>::T T;
    typedef typename CT<FP64>::V V;
    typedef typename CT<FP64>::H H;
    const int64_t s0 = S.s0, e0 = S.e0;
    const int2 *cand = a.cand[lp] + e0;
    const int off = a.coff[lp][k], n = a.ccnt[lp][k];
    // own data
    typename CT<FP64>::P mp;
    float4 mr;
    typename CT<FP64>::VR mv, mw;
    if constexpr (FP64) { mp = a.dp_[k]; mv = a.dv_[k]; mw = a.dw_[k]; }
    else if (s_x) {
        const int64_t lk = k - kb0;
        mp = s_x[2 * lk]; mr = as_f4(s_x[2 * lk + 1]);
        mv = s_v[2 * lk]; mw = s_v[2 * lk + 1];
    } else {
        mp = a.xqr[2 * k]; mr = as_f4(a.xqr[2 * k + 1]);
        mv = a.svw[2 * k]; mw = a.svw[2 * k + 1];
    }
    V F, Tq;
    if constexpr (FP64) { F = d3(0, 0, 0); Tq = d3(0, 0, 0); }
    else { F = f3(0.f, 0.f, 0.f); Tq = f3(0.f, 0.f, 0.f); }
    int nc = 0;
    // One entry: this sphere as sphere a.  Every step of the law maps exactly
    // onto its negative or onto itself when the spheres swap (differences and
    // products of negated operands round to the negated or the same value),
    // so this evaluation's share a is bit for bit the share of this side of
    // the owner's evaluation, and S the owner's with its sign.
    auto entry = [&](int f, bool ok, const H &hp, const typename CT<FP64>::P &pp,
                     const float4 &pr, const typename CT<FP64>::VR &pv, const typename CT<FP64>::VR &pw) {
        PairOut<T, V> o;
        bool hit = false;
        if (ok) {
            if constexpr (FP64) {
                const double3 Sprev = hp.w != 0 ? d3(hp.x, hp.y, hp.z) : d3(0, 0, 0);
                hit = pair_64(mp, mv, mw, pp, pv, pw, Sprev, prm, o);
            } else {
                const float3 Sprev = hp.w != 0.f ? f3(hp.x, hp.y, hp.z) : f3(0.f, 0.f, 0.f);
                hit = pair_mixed(mp, mr, pp, pr, q, mv, mw, pv, pw, Sprev, prm, o);
            }
        }
        if (ok) {
            H h;
            if constexpr (FP64) h = hit ? make_dbl4(o.S.x, o.S.y, o.S.z, 1.0) : make_dbl4(0, 0, 0, 0);
            else h = hit ? make_float4(o.S.x, o.S.y, o.S.z, 1.f) : make_float4(0.f, 0.f, 0.f, 0.f);
            hwrite[f] = h;
        }
        if (!hit) return;
        if (o.x > T(0.1) * o.rmin) flags |= DEM_FLAG_OVERLAP;
        V sF, sT;
        share<T, V>(o, true, sF, sT);
        F.x = addr(F.x, sF.x); F.y = addr(F.y, sF.y); F.z = addr(F.z, sF.z);
        Tq.x = addr(Tq.x, sT.x); Tq.y = addr(Tq.y, sT.y); Tq.z = addr(Tq.z, sT.z);
        ++nc;
    };
    // an entry's partner (clamped: the check never fails)
    auto where = [&](int2 c, int64_t &g, bool &ok) {
        const int kk = c.x & 0x7fffffff;
        ok = (unsigned)kk < (unsigned)S.ns;
        g = s0 + (ok ? kk : 0);
    };
    if constexpr (FP64) {
        for (int e = 0; e < n; ++e) {
            const int f = off + 32 * e;
            int64_t g;
            bool ok;
            where(cand[f], g, ok);
            entry(f, ok, hread[f], a.dp_[g], make_float4(0.f, 0.f, 0.f, 0.f), a.dv_[g], a.dw_[g]);
        }
    } else {
        // partner data from the staged block when it is there, else from global memory
        auto fetch = [&](int64_t g, int4 &x, int4 &r, float4 &v, float4 &w) {
            const int64_t lk = g - kb0;
            if (s_x && (uint64_t)lk < 128) {
                x = s_x[2 * lk]; r = s_x[2 * lk + 1]; v = s_v[2 * lk]; w = s_v[2 * lk + 1];
            } else {
                x = a.xqr[2 * g]; r = a.xqr[2 * g + 1]; v = a.svw[2 * g]; w = a.svw[2 * g + 1];
            }
        };
        // the list entry and the history two ahead are in flight while an entry
        // is evaluated (both are consecutive for the warp, so no address waits
        // for a load); the partner's data is fetched where it is used, which
        // leaves room for a fifth block per SM (96 registers): 201 us on the 1M
        // lattice, 252 with it one entry ahead and four blocks, 210 with it
        // prefetched to L2 (197 without the pile lookup, see sphere_pile)
        const int last = off + 32 * (n - 1);   // (n > 0 where it is used)
        auto at = [&](int e) { return min(off + 32 * e, last); };
        int2 c0 = make_int2(0, 0), c1 = c0;
        H hp = make_float4(0.f, 0.f, 0.f, 0.f), h1 = hp;
        if (n > 0) {
            c0 = cand[off];
            c1 = cand[at(1)];
            hp = hread[off];
            h1 = hread[at(1)];
        }
        for (int e = 0; e < n; ++e) {
            int64_t g;
            bool ok;
            int4 px, pr;
            float4 pv, pw;
            where(c0, g, ok);
            fetch(g, px, pr, pv, pw);
            const int2 c2 = cand[at(e + 2)];
            const H h2 = hread[at(e + 2)];
            entry(off + 32 * e, ok, hp, px, as_f4(pr), pv, pw);
            c0 = c1; c1 = c2;
            hp = h1; h1 = h2;
        }
    }
    // stored at the sphere's home index (its aggregate's members are then
    // contiguous for k_agg_end); the gathered spin record carries that index
    // (checked against the pile's range: the check never fails)
    if constexpr (FP64) {
        const int hl = (int)mw.w;
        if ((unsigned)hl < (unsigned)S.ns) {
            a.ftc64[2 * (s0 + hl)] = make_dbl4(F.x, F.y, F.z, 0.0);
            a.ftc64[2 * (s0 + hl) + 1] = make_dbl4(Tq.x, Tq.y, Tq.z, 0.0);
        }
    } else {
        const int hl = __float_as_int(mw.w);
        if ((unsigned)hl < (unsigned)S.ns)
            st_f4x2(a.ftc32 + 2 * (s0 + hl), make_float4(F.x, F.y, F.z, 0.f), make_float4(Tq.x, Tq.y, Tq.z, 0.f));
    }
    if (nc > S.K) flags |= DEM_FLAG_SLOTS;
}

// Shared memory of k_contact (dynamic): list offsets and lengths of the
// tile's spheres and its slice bases, staged sphere data, the inbox (each
// entry's share: F and tau as six arrays, and a contact flag) and the work
// queue.
template <bool FP64>
struct Smem {
    typedef typename CT<FP64>::T T;
    static constexpr int kCap = CT<FP64>::kCap;
    static constexpr size_t off_bytes = sizeof(int) * (2 * kCTile + 32);   // keeps what follows 32-byte aligned
    static constexpr size_t stage_bytes = (FP64 ? 3 * sizeof(dbl4) : 4 * sizeof(float4)) * kCTile;
    static constexpr size_t inbox_bytes = 6 * sizeof(T) * kCap;
    static constexpr size_t flag_bytes = kCap;
    static constexpr size_t queue_bytes = sizeof(int) * kCap;
    static constexpr size_t scan_bytes = sizeof(int) * (kCTile / 32 + 8);
    static constexpr size_t total = off_bytes + stage_bytes + inbox_bytes + flag_bytes + queue_bytes + scan_bytes;
};

// Exclusive prefix sum over the block (kCTile threads); *total gets the sum.
__device__ __forceinline__ int block_exclusive_scan(int v, int *ws, int *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int t = lane < kCTile / 32 ? ws[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < kCTile / 32) ws[lane] = t;
        if (lane == kCTile / 32 - 1) ws[kCTile / 32] = t;
    }
    __syncthreads();
    const int r = (wid ? ws[wid - 1] : 0) + x - v;
    *total = ws[kCTile / 32];
    __syncthreads();
    return r;
}

template <bool FP64>
__global__ void __launch_bounds__(kCTile, FP64 ? 2 : 4) k_contact(Arrays a, Sizes z)
{
    pdl_enter();
    typedef typename CT<FP64>::T T;
    typedef typename CT<FP64>::V V;
    typedef typename CT<FP64>::H H;
    typedef Smem<FP64> SM;
    const int kCap = min(SM::kCap, max(32, z.icap));
    extern __shared__ __align__(32) unsigned char smem[];
    int *s_off = (int *)smem;                 // [kCTile] list offsets (pile-local entries)
    int *s_cnt = s_off + kCTile;              // [kCTile] list lengths
    int *s_sb = s_cnt + kCTile;               // [kSl + 1] slice bases, then the tile's end
    unsigned char *stage = smem + SM::off_bytes;
    T *inbox = (T *)(stage + SM::stage_bytes);   // [6][SM::kCap]
    unsigned char *flag = (unsigned char *)(inbox + 6 * SM::kCap);
    int *queue = (int *)(flag + SM::kCap);
    int *ws = (int *)((unsigned char *)queue + SM::queue_bytes);
    __shared__ int pile_flags;

    // the first blocks finish the piles' opening reductions
    if (blockIdx.x < z.P) {
        open_pile<kCTile>(a, blockIdx.x);
        return;
    }
    const int4 tl = a.ctile[blockIdx.x - z.P];
    const int p = tl.x;
    if (!pile_active(a, p)) return;
    const PileStatic &S = a.ps[p];
    const PileDyn &D = a.pd[p];
    if (D.flags & DEM_FLAG_SLOTS) return;          // lists could not be built: frozen this step
    const bool rb = D.rebuild != 0;
    const int lp = rb ? D.cpar ^ 1 : D.cpar, par = D.parity;
    const int64_t s0 = S.s0, e0 = S.e0;
    const int first = tl.y, nt = tl.z;
    const int K = S.K;
    typename CT<FP64>::Prm prm;
    const H *hread;
    H *hwrite;
    if constexpr (FP64) {
        prm = {S.kn, S.kt, S.cn, S.ct, S.mu_s, S.mu_r, S.mu_t, S.w0, S.h};
        hread = (rb ? a.hist64_rm : a.hist64[par]) + e0;
        hwrite = a.hist64[par ^ 1] + e0;
    } else {
        prm = {S.lawf[0], S.lawf[1], S.lawf[2], S.lawf[3], S.lawf[4], S.lawf[5], S.lawf[6], S.lawf[7],
               S.lawf[8]};
        hread = (rb ? a.hist32_rm : a.hist32[par]) + e0;
        hwrite = a.hist32[par ^ 1] + e0;
    }
    const float q = pow2f(S.qexp);
    const int2 *cand = a.cand[lp] + e0;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nsl = (nt + 31) >> 5;
    if (tid == 0) pile_flags = 0;
    {
        int off = 0, n = 0;
        if (tid < nt) {
            const int64_t k = s0 + first + tid;
            off = a.coff[lp][k];
            n = a.ccnt[lp][k];
            if constexpr (FP64) {
                dbl4 *st = (dbl4 *)stage;
                st[tid] = a.dp_[k];
                st[kCTile + tid] = a.dv_[k];
                st[2 * kCTile + tid] = a.dw_[k];
            } else {
                int4 *sx = (int4 *)stage;
                float4 *sv = (float4 *)(sx + kCTile);
                const int4 xr = a.xqr[2 * k + 1];
                sx[tid] = a.xqr[2 * k];
                sv[tid] = a.svw[2 * k];
                sv[kCTile + tid] = a.svw[2 * k + 1];
                sv[2 * kCTile + tid] = make_float4(__int_as_float(xr.x), __int_as_float(xr.y),
                                                   __int_as_float(xr.z), __int_as_float(xr.w));
            }
        }
        s_off[tid] = off;
        s_cnt[tid] = n;
        const int wmax = __reduce_max_sync(0xffffffffu, n);
        if (lane == 0 && wid < nsl) s_sb[wid] = off;               // lane 0 sits at its slice's base
        if (lane == 0 && wid == nsl - 1) s_sb[nsl] = off + 32 * wmax;
    }
    __syncthreads();
    int myflags = 0;
    // slice ranges [r0, r1) of the tile whose list entries fit the inbox
    for (int r0 = 0; r0 < nsl;) {
        int r1 = nsl;
        while (s_sb[r1] - s_sb[r0] > kCap && r1 - r0 > 1) r1 = r0 + (r1 - r0 + 1) / 2;
        const int E0 = s_sb[r0], nE = s_sb[r1] - E0;
        if (nE > SM::kCap) {
            // one slice with more list entries than the inbox holds: its
            // spheres evaluate their own lists (bitwise the same results)
            if (tid >= 32 * r0 && tid < min(32 * r1, nt))
                sphere_contacts<FP64>(a, S, lp, hread, hwrite, prm, q, s0 + first + tid, 0, nullptr, nullptr,
                                      myflags);
            r0 = r1;
            continue;
        }
        const int i0 = 32 * r0, i1 = min(32 * r1, nt);
        // work queue in (sphere, entry) order: pairs this range owns, and
        // pairs that leave the range (from this sphere's side)
        const unsigned lo = (unsigned)(first + i0), span = (unsigned)(i1 - i0);
        const bool inr = tid >= i0 && tid < i1;
        const int off = s_off[tid], n = inr ? s_cnt[tid] : 0;
        int cnt = 0;
        for (int e = 0; e < n; ++e) {
            const int2 c = cand[off + 32 * e];
            const unsigned kk = (unsigned)c.x & 0x7fffffffu;
            cnt += (c.x < 0 || kk - lo >= span) ? 1 : 0;
        }
        int nq;
        int pos = block_exclusive_scan(cnt, ws, &nq);
        for (int e = 0; e < n; ++e) {
            const int2 c = cand[off + 32 * e];
            const unsigned kk = (unsigned)c.x & 0x7fffffffu;
            if (c.x < 0 || kk - lo >= span) queue[pos++] = (tid << 12) | e;
        }
        __syncthreads();
        for (int r = tid; r < nq; r += kCTile) {
            const int rec = queue[r];
            const int i = rec >> 12, e = rec & 0xfff;
            const int f = s_off[i] + 32 * e;
            const int2 c = cand[f];
            const int kk = c.x & 0x7fffffff;
            const bool owned = c.x < 0;
            const bool inner = (unsigned)kk - lo < span;
            // sphere a is the owner
            const int ia = owned ? i : kk - first, ib = owned ? kk - first : i;
            const bool a_loc = owned || inner, b_loc = !owned || inner;
            if ((unsigned)kk >= (unsigned)S.ns || (unsigned)c.y >= (unsigned)S.ne) continue;   // (never taken)
            const H hp = hread[f];        // from this sphere's side; the evaluation takes the owner's
            const T sgn = owned ? T(1) : T(-1);
            PairOut<T, V> o;
            bool hit;
            if constexpr (FP64) {
                const dbl4 *st = (const dbl4 *)stage;
                const int64_t ga = s0 + (owned ? first + i : kk), gb = s0 + (owned ? kk : first + i);
                const dbl4 ap = a_loc ? st[ia] : a.dp_[ga], av = a_loc ? st[kCTile + ia] : a.dv_[ga],
                           aw = a_loc ? st[2 * kCTile + ia] : a.dw_[ga];
                const dbl4 bp = b_loc ? st[ib] : a.dp_[gb], bv = b_loc ? st[kCTile + ib] : a.dv_[gb],
                           bw = b_loc ? st[2 * kCTile + ib] : a.dw_[gb];
                const double3 Sprev = hp.w != 0 ? d3(sgn * hp.x, sgn * hp.y, sgn * hp.z) : d3(0, 0, 0);
                hit = pair_64(ap, av, aw, bp, bv, bw, Sprev, prm, o);
            } else {
                const int4 *sx = (const int4 *)stage;
                const float4 *sv = (const float4 *)(sx + kCTile);
                const int64_t ga = s0 + (owned ? first + i : kk), gb = s0 + (owned ? kk : first + i);
                const int4 A = a_loc ? sx[ia] : a.xqr[2 * ga], B = b_loc ? sx[ib] : a.xqr[2 * gb];
                const float4 RA = a_loc ? sv[2 * kCTile + ia] : as_f4(a.xqr[2 * ga + 1]);
                const float4 RB = b_loc ? sv[2 * kCTile + ib] : as_f4(a.xqr[2 * gb + 1]);
                const float4 av = a_loc ? sv[ia] : a.svw[2 * ga], aw = a_loc ? sv[kCTile + ia] : a.svw[2 * ga + 1];
                const float4 bv = b_loc ? sv[ib] : a.svw[2 * gb], bw = b_loc ? sv[kCTile + ib] : a.svw[2 * gb + 1];
                const float3 Sprev = hp.w != 0.f ? f3(sgn * hp.x, sgn * hp.y, sgn * hp.z) : f3(0.f, 0.f, 0.f);
                hit = pair_mixed(A, RA, B, RB, q, av, aw, bv, bw, Sprev, prm, o);
            }
            // this sphere's entry, and the partner's of an inner pair, each
            // from its own side
            auto keep = [&](int at, T sg) {
                H h;
                if constexpr (FP64) h = hit ? make_dbl4(sg * o.S.x, sg * o.S.y, sg * o.S.z, 1.0) : make_dbl4(0, 0, 0, 0);
                else h = hit ? make_float4(sg * o.S.x, sg * o.S.y, sg * o.S.z, 1.f) : make_float4(0.f, 0.f, 0.f, 0.f);
                hwrite[at] = h;
            };
            keep(f, sgn);
            if (inner) keep(c.y, -sgn);
            if (hit && o.x > T(0.1) * o.rmin) myflags |= DEM_FLAG_OVERLAP;
            V F, Tq;
            if (a_loc) {
                const int slot = (owned ? f : c.y) - E0;
                if ((unsigned)slot >= (unsigned)nE) continue;   // (lists are symmetric: never taken)
                if (hit) {
                    share<T, V>(o, true, F, Tq);
                    inbox[slot] = F.x; inbox[SM::kCap + slot] = F.y; inbox[2 * SM::kCap + slot] = F.z;
                    inbox[3 * SM::kCap + slot] = Tq.x; inbox[4 * SM::kCap + slot] = Tq.y;
                    inbox[5 * SM::kCap + slot] = Tq.z;
                }
                flag[slot] = hit ? 1 : 0;
            }
            if (b_loc) {
                const int slot = (owned ? c.y : f) - E0;
                if ((unsigned)slot >= (unsigned)nE) continue;
                if (hit) {
                    share<T, V>(o, false, F, Tq);
                    inbox[slot] = F.x; inbox[SM::kCap + slot] = F.y; inbox[2 * SM::kCap + slot] = F.z;
                    inbox[3 * SM::kCap + slot] = Tq.x; inbox[4 * SM::kCap + slot] = Tq.y;
                    inbox[5 * SM::kCap + slot] = Tq.z;
                }
                flag[slot] = hit ? 1 : 0;
            }
        }
        __syncthreads();
        // every sphere of the range sums its slots in list order
        if (inr) {
            V F, Tq;
            if constexpr (FP64) { F = d3(0, 0, 0); Tq = d3(0, 0, 0); }
            else { F = f3(0.f, 0.f, 0.f); Tq = f3(0.f, 0.f, 0.f); }
            int nc = 0;
            for (int e = 0; e < n; ++e) {
                const int slot = off - E0 + 32 * e;
                if (!flag[slot]) continue;
                F.x = addr(F.x, inbox[slot]); F.y = addr(F.y, inbox[SM::kCap + slot]);
                F.z = addr(F.z, inbox[2 * SM::kCap + slot]);
                Tq.x = addr(Tq.x, inbox[3 * SM::kCap + slot]); Tq.y = addr(Tq.y, inbox[4 * SM::kCap + slot]);
                Tq.z = addr(Tq.z, inbox[5 * SM::kCap + slot]);
                ++nc;
            }
            // at the sphere's home index (from the staged spin record; checked
            // against the pile's range, which it never leaves)
            if constexpr (FP64) {
                const int hl = (int)((const dbl4 *)stage)[2 * kCTile + tid].w;
                if ((unsigned)hl < (unsigned)S.ns) {
                    a.ftc64[2 * (s0 + hl)] = make_dbl4(F.x, F.y, F.z, 0.0);
                    a.ftc64[2 * (s0 + hl) + 1] = make_dbl4(Tq.x, Tq.y, Tq.z, 0.0);
                }
            } else {
                const float4 *sv = (const float4 *)((const int4 *)stage + kCTile);
                const int hl = __float_as_int(sv[kCTile + tid].w);
                if ((unsigned)hl < (unsigned)S.ns)
                    st_f4x2(a.ftc32 + 2 * (s0 + hl), make_float4(F.x, F.y, F.z, 0.f),
                            make_float4(Tq.x, Tq.y, Tq.z, 0.f));
            }
            if (nc > K) myflags |= DEM_FLAG_SLOTS;
        }
        __syncthreads();
        r0 = r1;
    }
    if (myflags) atomicOr(&pile_flags, myflags);
    __syncthreads();
    if (tid == 0 && pile_flags) atomicOr(&a.pd[p].flags, pile_flags);
}

// One thread per sorted sphere (sphere_contacts); the block's own 128 sorted
// spheres are staged in shared memory in the mixed path (consecutive sorted
// spheres fill a compact block of space, so most partners are among them).
template <bool FP64>
__global__ void __launch_bounds__(128, FP64 ? 1 : 5) k_contact_sphere(Arrays a, Sizes z)
{
    pdl_enter();
    typedef typename CT<FP64>::H H;
    if (blockIdx.x < z.P) {   // the first blocks finish the piles' opening reductions
        open_pile<128>(a, blockIdx.x);
        return;
    }
    const int64_t kb0 = (int64_t)(blockIdx.x - z.P) * 128;
    const int64_t k = kb0 + threadIdx.x;
    __shared__ int4 s_x[FP64 ? 1 : 2 * 128];
    __shared__ float4 s_v[FP64 ? 1 : 2 * 128];
    if constexpr (!FP64) {
        if (k < z.N) {
            s_x[2 * threadIdx.x] = a.xqr[2 * k];
            s_x[2 * threadIdx.x + 1] = a.xqr[2 * k + 1];
            s_v[2 * threadIdx.x] = a.svw[2 * k];
            s_v[2 * threadIdx.x + 1] = a.svw[2 * k + 1];
        }
        __syncthreads();
    }
    if (k >= z.N) return;
    const int p = sphere_pile(a, z, k);
    if (!pile_active(a, p)) return;
    const PileStatic &S = a.ps[p];
    const PileDyn &D = a.pd[p];
    if (D.flags & DEM_FLAG_SLOTS) return;
    const bool rb = D.rebuild != 0;
    const int lp = rb ? D.cpar ^ 1 : D.cpar, par = D.parity;
    typename CT<FP64>::Prm prm;
    const H *hread;
    H *hwrite;
    if constexpr (FP64) {
        prm = {S.kn, S.kt, S.cn, S.ct, S.mu_s, S.mu_r, S.mu_t, S.w0, S.h};
        hread = (rb ? a.hist64_rm : a.hist64[par]) + S.e0;
        hwrite = a.hist64[par ^ 1] + S.e0;
    } else {
        prm = {S.lawf[0], S.lawf[1], S.lawf[2], S.lawf[3], S.lawf[4], S.lawf[5], S.lawf[6], S.lawf[7],
               S.lawf[8]};
        hread = (rb ? a.hist32_rm : a.hist32[par]) + S.e0;
        hwrite = a.hist32[par ^ 1] + S.e0;
    }
    int flags = 0;
    sphere_contacts<FP64>(a, S, lp, hread, hwrite, prm, pow2f(S.qexp), k, kb0, FP64 ? nullptr : s_x,
                          FP64 ? nullptr : s_v, flags);
    if (flags) atomicOr(&a.pd[p].flags, flags);
}

cudaError_t contact_setup(bool fp64, int)
{
    if (fp64)
        return cudaFuncSetAttribute(k_contact<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)Smem<true>::total);
    return cudaFuncSetAttribute(k_contact<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)Smem<false>::total);
}

void launch_contact(const Arrays &a, const Sizes &z, bool fp64, int, cudaStream_t st)
{
    if (z.N == 0 || z.CT == 0) return;
    const unsigned nt = (unsigned)(z.CT + z.P), ns = (unsigned)((z.N + 127) / 128 + z.P);
    if (fp64) {
        if (z.cmode == 1) launch_pdl(k_contact<true>, nt, kCTile, Smem<true>::total, st, a, z);
        else launch_pdl(k_contact_sphere<true>, ns, 128, 0, st, a, z);
    } else {
        if (z.cmode == 1) launch_pdl(k_contact<false>, nt, kCTile, Smem<false>::total, st, a, z);
        else launch_pdl(k_contact_sphere<false>, ns, 128, 0, st, a, z);
    }
}

}  // namespace dem
