// kernels_step.cu -- the aggregate kernels that open and close a step:
// rigid-body kick/drift/rotation, and the reduction of sphere forces onto
// aggregates with the closing kick and the end of the piles' step.
//
// Paper references: leapfrog with predicted velocities (Sec. 2.1), aggregate
// mass and COM (Sec. 2.2.1, Eq. agg_mass, Eq. agg_position), Euler's equations
// for spin (Sec. 2.2.1), predicted sphere velocity (Sec. 2.2.2, Eq. pred-vel),
// aggregate force and torque sums (Sec. 2.2.3-2.2.4, Eq. agg_gravity,
// Eq. gravity_torque, Eq. agg_contact_accel, contact torque at the contact
// point), YORP increment (Sec. 4.1), point-mass planet (Sec. 4.2).
#include <type_traits>

#include "dem_internal.h"
#include "devmath.cuh"
#include "expand.cuh"
#include "launch.cuh"
#include "reduce.cuh"

namespace dem {

// ---------------------------------------------------------------- ids
__device__ int find_slot(const PileStatic *ps, int P, int64_t idx, int which)
{
    int lo = 0, hi = P - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        int64_t b = which == 0 ? ps[mid].s0 : which == 1 ? ps[mid].a0 : which == 2 ? ps[mid].t0 : ps[mid].ch0;
        if (b <= idx) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void k_fill_ids(Arrays a, Sizes z)
{
    pdl_enter();
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int P = (int)z.P;
    if (t < z.N) a.sph_pile[t] = find_slot(a.ps, P, t, 0);
    if (t < z.A) a.agg_pile[t] = find_slot(a.ps, P, t, 1);
    if (t < z.CH) a.chunk_pile[t] = find_slot(a.ps, P, t, 3);
}

void launch_fill_ids(const Arrays &a, const Sizes &z, cudaStream_t st)
{
    int64_t n = z.N > z.A ? z.N : z.A;
    if (z.CH > n) n = z.CH;
    if (n == 0 || z.P == 0) return;
    launch_pdl(k_fill_ids, (unsigned)((n + 255) / 256), 256, 0, st, a, z);
}

// ---------------------------------------------------------------- rotation
// Torque-free Euler equations in the body frame (Sec. 2.2.1):
//   dq/dt = 1/2 q (x) (0, w),  dw/dt = I^-1 (-w x (I w)).
__device__ __forceinline__ void rot_rhs(const double *y, const double *I, const double *Iinv,
                                        double *dy)
{
    const double *q = y, *w = y + 4;
    dy[0] = -0.5 * (q[1] * w[0] + q[2] * w[1] + q[3] * w[2]);
    dy[1] = 0.5 * (q[0] * w[0] + q[2] * w[2] - q[3] * w[1]);
    dy[2] = 0.5 * (q[0] * w[1] + q[3] * w[0] - q[1] * w[2]);
    dy[3] = 0.5 * (q[0] * w[2] + q[1] * w[1] - q[2] * w[0]);
    double3 wv = d3(w[0], w[1], w[2]);
    double3 Iw = mat_mul(I, wv);
    double3 g = -cross(wv, Iw);
    double3 dw = mat_mul(Iinv, g);
    dy[4] = dw.x; dy[5] = dw.y; dy[6] = dw.z;
}

// One classical RK4 step of the free rotor over h, q renormalised.
__device__ void free_rotate(double *q, double3 &wb, const double *I, const double *Iinv, double h)
{
    double y[7] = {q[0], q[1], q[2], q[3], wb.x, wb.y, wb.z};
    double k1[7], k2[7], k3[7], k4[7], t[7];
    rot_rhs(y, I, Iinv, k1);
    for (int c = 0; c < 7; ++c) t[c] = y[c] + 0.5 * h * k1[c];
    rot_rhs(t, I, Iinv, k2);
    for (int c = 0; c < 7; ++c) t[c] = y[c] + 0.5 * h * k2[c];
    rot_rhs(t, I, Iinv, k3);
    for (int c = 0; c < 7; ++c) t[c] = y[c] + h * k3[c];
    rot_rhs(t, I, Iinv, k4);
    for (int c = 0; c < 7; ++c) y[c] += h / 6.0 * (k1[c] + 2.0 * k2[c] + 2.0 * k3[c] + k4[c]);
    double n = sqrt(y[0] * y[0] + y[1] * y[1] + y[2] * y[2] + y[3] * y[3]);
    q[0] = y[0] / n; q[1] = y[1] / n; q[2] = y[2] / n; q[3] = y[3] / n;
    wb = d3(y[4], y[5], y[6]);
}

// Stage derivatives of the torque-free rotor in FP32 (mixed path).
__device__ __forceinline__ void rot_rhs_f(const float *y, const float *I, const float *Iinv, float *dy)
{
    const float *q = y, *w = y + 4;
    dy[0] = -0.5f * (q[1] * w[0] + q[2] * w[1] + q[3] * w[2]);
    dy[1] = 0.5f * (q[0] * w[0] + q[2] * w[2] - q[3] * w[1]);
    dy[2] = 0.5f * (q[0] * w[1] + q[3] * w[0] - q[1] * w[2]);
    dy[3] = 0.5f * (q[0] * w[2] + q[1] * w[1] - q[2] * w[0]);
    const float3 wv = f3(w[0], w[1], w[2]);
    const float3 dw = mat_mulf(Iinv, -cross(wv, mat_mulf(I, wv)));
    dy[4] = dw.x; dy[5] = dw.y; dy[6] = dw.z;
}

// The paper's rotation integrator (Sec. 2.2.1): time-adaptive fifth-order
// Runge-Kutta.  The torque-free rotation over h is taken in substeps of the
// embedded Cash-Karp RK5(4) pair; a substep is accepted when the difference
// of its fifth- and fourth-order results (q absolute, w relative to |w|) is
// within tol, the next one is scaled by 0.9 (tol/err)^(1/5) (at most x5), a
// rejected one retried at 0.9 (tol/err)^(1/4) of it (at least x0.1); the first
// trial is the whole step, and a substep below h / 2^20 is accepted whatever
// its error, so the loop ends.  FP64 in both precisions; q renormalised at the
// end as after RK4.
__device__ void free_rotate_adaptive(double *q, double3 &wb, const double *I, const double *Iinv,
                                     double h, double tol)
{
    // Cash-Karp coefficients
    const double A21 = 1.0 / 5.0;
    const double A31 = 3.0 / 40.0, A32 = 9.0 / 40.0;
    const double A41 = 3.0 / 10.0, A42 = -9.0 / 10.0, A43 = 6.0 / 5.0;
    const double A51 = -11.0 / 54.0, A52 = 5.0 / 2.0, A53 = -70.0 / 27.0, A54 = 35.0 / 27.0;
    const double A61 = 1631.0 / 55296.0, A62 = 175.0 / 512.0, A63 = 575.0 / 13824.0,
                 A64 = 44275.0 / 110592.0, A65 = 253.0 / 4096.0;
    const double B1 = 37.0 / 378.0, B3 = 250.0 / 621.0, B4 = 125.0 / 594.0, B6 = 512.0 / 1771.0;
    const double E1 = B1 - 2825.0 / 27648.0, E3 = B3 - 18575.0 / 48384.0,
                 E4 = B4 - 13525.0 / 55296.0, E5 = -277.0 / 14336.0, E6 = B6 - 1.0 / 4.0;
    double y[7] = {q[0], q[1], q[2], q[3], wb.x, wb.y, wb.z};
    double t = 0.0, dt = h;
    const double dt_min = h * 0x1p-20;
    while (t < h) {
        if (t + dt > h) dt = h - t;
        double k1[7], k2[7], k3[7], k4[7], k5[7], k6[7], z[7];
        rot_rhs(y, I, Iinv, k1);
        for (int c = 0; c < 7; ++c) z[c] = y[c] + dt * (A21 * k1[c]);
        rot_rhs(z, I, Iinv, k2);
        for (int c = 0; c < 7; ++c) z[c] = y[c] + dt * (A31 * k1[c] + A32 * k2[c]);
        rot_rhs(z, I, Iinv, k3);
        for (int c = 0; c < 7; ++c) z[c] = y[c] + dt * (A41 * k1[c] + A42 * k2[c] + A43 * k3[c]);
        rot_rhs(z, I, Iinv, k4);
        for (int c = 0; c < 7; ++c)
            z[c] = y[c] + dt * (A51 * k1[c] + A52 * k2[c] + A53 * k3[c] + A54 * k4[c]);
        rot_rhs(z, I, Iinv, k5);
        for (int c = 0; c < 7; ++c)
            z[c] = y[c] + dt * (A61 * k1[c] + A62 * k2[c] + A63 * k3[c] + A64 * k4[c] + A65 * k5[c]);
        rot_rhs(z, I, Iinv, k6);
        const double wn = sqrt(y[4] * y[4] + y[5] * y[5] + y[6] * y[6]);
        double err = 0.0;
        for (int c = 0; c < 7; ++c) {
            double e = fabs(dt * (E1 * k1[c] + E3 * k3[c] + E4 * k4[c] + E5 * k5[c] + E6 * k6[c]));
            if (c >= 4 && wn > 0.0) e /= wn;
            err = fmax(err, e);
        }
        const double ratio = err / tol;
        if (ratio <= 1.0 || dt <= dt_min) {
            for (int c = 0; c < 7; ++c)
                y[c] += dt * (B1 * k1[c] + B3 * k3[c] + B4 * k4[c] + B6 * k6[c]);
            t += dt;
            dt *= ratio > 0.0 ? fmin(5.0, 0.9 * pow(ratio, -0.2)) : 5.0;
        } else {
            dt *= fmax(0.1, 0.9 * pow(ratio, -0.25));
        }
    }
    double n = sqrt(y[0] * y[0] + y[1] * y[1] + y[2] * y[2] + y[3] * y[3]);
    q[0] = y[0] / n; q[1] = y[1] / n; q[2] = y[2] / n; q[3] = y[3] / n;
    wb = d3(y[4], y[5], y[6]);
}

// ---------------------------------------------------------------- step begin
// Neighbour-list validity.  Every sphere of the aggregate moved, relative to
// the pile frame extrapolated by one step (O + h V), by at most
// |c' - c'_ref| + |(R - R_ref) b| <= |c' - c'_ref| + 2 |b|max min|q -+ q_ref|
// since the last rebuild.  The candidate lists hold every pair closer than the
// radii sum plus the skin at the rebuild, so they stay complete while no
// sphere has moved more than half the skin.  The bound is taken in FP32
// (positions relative to the pile frame, reference stored in FP32) with a
// margin of a few units in the last place of the positions and 1e-4
// relative, far above its rounding.  c: COM relative to the frame (hi parts),
// qn: the new orientation in FP32.
__device__ __forceinline__ void rebuild_test(const Arrays &a, int p, int64_t g, const float (&c)[3],
                                             const float (&qn)[4])
{
    const double skin = a.ps[p].skin;
    if (!(skin > 0.0)) return;
    const float *ar = a.aref + 8 * g;
    const float *hv = a.pd[p].hVf;
    const float3 dcf = f3(c[0] - hv[0] - ar[0], c[1] - hv[1] - ar[1], c[2] - hv[2] - ar[2]);
    float dm = 0.f, dp = 0.f;
    for (int k = 0; k < 4; ++k) {
        const float m = qn[k] - ar[3 + k], s_ = qn[k] + ar[3 + k];
        dm = fmaf(m, m, dm);
        dp = fmaf(s_, s_, dp);
    }
    const float big = fmaxf(fabsf(c[0]), fmaxf(fabsf(c[1]), fabsf(c[2]))) +
                      fmaxf(fabsf(ar[0]), fmaxf(fabsf(ar[1]), fabsf(ar[2])));
    const float disp = sqrtf(dot(dcf, dcf)) + 2.0f * ar[7] * sqrtf(fminf(dm, dp)) + 1e-6f * (big + ar[7]);
    if (!(disp * 1.0001f <= 0.5f * (float)skin)) atomicOr(&a.pd[p].rebuild, 1);
}

// FP64 path.  Per aggregate: half kick of COM and spin with the stored
// a_A,n / N_A,n, drift, torque-free rotation, then the record the sphere
// kernels read: rotation, COM relative to the pile frame, predicted COM
// velocity v_A,n+1/2 + h/2 a_A,n (Eq. pred-vel) and predicted spin w_A,n+1
// (the drifted spin plus the second half kick of the old torque).
template <bool ADAPT>
__device__ __forceinline__ void agg_begin_64(const Arrays &a, int64_t g, int p)
{
    const double h = a.ps[p].h;
    const double *I = a.I + 9 * g, *Iinv = a.Iinv + 9 * g;
    double q[4] = {a.q[4 * g], a.q[4 * g + 1], a.q[4 * g + 2], a.q[4 * g + 3]};
    double3 r = ld3(a.r + 3 * g), v = ld3(a.v + 3 * g), wb = ld3(a.wb + 3 * g);
    const double3 acc = ld3(a.acc + 3 * g), N = ld3(a.torque + 3 * g);
    double R[9];
    quat_to_R(q, R);
    v = v + (0.5 * h) * acc;
    wb = wb + (0.5 * h) * mat_mul(Iinv, mat_tmul(R, N));
    r = r + h * v;
    if (ADAPT && a.ps[p].rot_tol > 0.0) free_rotate_adaptive(q, wb, I, Iinv, h, a.ps[p].rot_tol);
    else free_rotate(q, wb, I, Iinv, h);
    quat_to_R(q, R);
    const double3 wpred_b = wb + (0.5 * h) * mat_mul(Iinv, mat_tmul(R, N));
    const double3 ws = mat_mul(R, wpred_b);
    st3(a.r + 3 * g, r);
    st3(a.v + 3 * g, v);
    st3(a.wb + 3 * g, wb);
    a.q[4 * g] = q[0]; a.q[4 * g + 1] = q[1]; a.q[4 * g + 2] = q[2]; a.q[4 * g + 3] = q[3];
    const PileDyn &D = a.pd[p];
    const double3 c = r - ld3(D.O);
    const double3 vb = v + (0.5 * h) * acc - ld3(D.V);
    const float cf[3] = {(float)c.x, (float)c.y, (float)c.z};
    const float qn[4] = {(float)q[0], (float)q[1], (float)q[2], (float)q[3]};
    rebuild_test(a, p, g, cf, qn);
    AggRec64 rec;
    for (int k = 0; k < 9; ++k) rec.R[k] = R[k];
    st3(rec.c, c);
    st3(rec.vb, vb);
    st3(rec.w, ws);
    a.rec64[g] = rec;
}

// Mixed path: the torque-free RK4 step with the stage derivatives evaluated
// in FP32 (from FP32 copies of q, w and the inertia tensor) and the step's
// increment added to the float-float state; q is then renormalised in
// float-float by the series 1/|q| = 1 - e/2 + 3e^2/8 - ..., e = |q|^2 - 1
// ~ |increment|^2 (the increment is tangent to the unit sphere; the dropped
// terms are O(e^3)).  The increment is O(h |w|), so its FP32 rounding is
// ~1e-7 of the change per step, far below the FP32 error of the forces that
// drive it.
__device__ __forceinline__ void free_rotate_ff(ff (&q)[4], ff (&wb)[3], const float *qf, const float *I,
                                               const float *Iinv, float h)
{
    float y[7] = {qf[0], qf[1], qf[2], qf[3], wb[0].hi, wb[1].hi, wb[2].hi};
    float k1[7], k2[7], k3[7], k4[7], t[7];
    rot_rhs_f(y, I, Iinv, k1);
    for (int c = 0; c < 7; ++c) t[c] = y[c] + 0.5f * h * k1[c];
    rot_rhs_f(t, I, Iinv, k2);
    for (int c = 0; c < 7; ++c) t[c] = y[c] + 0.5f * h * k2[c];
    rot_rhs_f(t, I, Iinv, k3);
    for (int c = 0; c < 7; ++c) t[c] = y[c] + h * k3[c];
    rot_rhs_f(t, I, Iinv, k4);
    float d[7];
    for (int c = 0; c < 7; ++c) d[c] = (h / 6.0f) * (k1[c] + 2.0f * k2[c] + 2.0f * k3[c] + k4[c]);
    for (int c = 0; c < 4; ++c) q[c] = ff_addf(q[c], d[c]);
    ff n2 = ff_mul(q[0], q[0]);
    for (int c = 1; c < 4; ++c) n2 = ff_add(n2, ff_mul(q[c], q[c]));
    const ff em = ff_addf(n2, -1.0f);
    const float e = __fadd_rn(em.hi, em.lo);
    const ff inv = {1.0f, e * (-0.5f + 0.375f * e)};
    for (int c = 0; c < 4; ++c) q[c] = ff_mul(q[c], inv);
    for (int c = 0; c < 3; ++c) wb[c] = ff_addf(wb[c], d[4 + c]);
}

// Mixed path: the same step with the aggregate state in float-float pairs
// and every operation on the FP32 units (no FP64 instruction on this path
// unless the pile asks for the adaptive rotor, which runs in FP64).
template <bool ADAPT>
__device__ __forceinline__ void agg_begin_mixed(const Arrays &a, int64_t g, int p)
{
    const PileStatic &S = a.ps[p];
    const PileDyn &D = a.pd[p];
    const float hf = S.lawf[8];
    const ff hh = {0.5f * S.hff[0], 0.5f * S.hff[1]}, hfull = {S.hff[0], S.hff[1]};
    ff q[4], r[3], v[3], wb[3], acc[3];
    float3 Nf;
    for (int c = 0; c < 4; ++c) q[c] = ldff(a.q + 4 * g + c);
    for (int c = 0; c < 3; ++c) {
        r[c] = ldff(a.r + 3 * g + c);
        v[c] = ldff(a.v + 3 * g + c);
        wb[c] = ldff(a.wb + 3 * g + c);
        acc[c] = ldff(a.acc + 3 * g + c);
    }
    Nf = f3(ldff(a.torque + 3 * g).hi, ldff(a.torque + 3 * g + 1).hi, ldff(a.torque + 3 * g + 2).hi);
    // spin kicks and the rotor's stage derivatives are increments: FP32
    const float *I32 = a.I32 + 9 * g, *Iinv32 = a.Iinv32 + 9 * g;
    float qf[4] = {q[0].hi, q[1].hi, q[2].hi, q[3].hi};
    float Rf[9], Rlo[9];
    quat_to_Rf(qf, Rf);
    const float3 dw = (0.5f * hf) * mat_mulf(Iinv32, mat_tmulf(Rf, Nf));
    for (int c = 0; c < 3; ++c) v[c] = ff_add(v[c], ff_mul(hh, acc[c]));
    wb[0] = ff_addf(wb[0], dw.x); wb[1] = ff_addf(wb[1], dw.y); wb[2] = ff_addf(wb[2], dw.z);
    for (int c = 0; c < 3; ++c) r[c] = ff_add(r[c], ff_mul(hfull, v[c]));
    if (ADAPT && S.rot_tol > 0.0) {
        double qd[4] = {ff_value(q[0]), ff_value(q[1]), ff_value(q[2]), ff_value(q[3])};
        double3 wd = d3(ff_value(wb[0]), ff_value(wb[1]), ff_value(wb[2]));
        free_rotate_adaptive(qd, wd, a.I + 9 * g, a.Iinv + 9 * g, S.h, S.rot_tol);
        for (int c = 0; c < 4; ++c) q[c] = ff_of(qd[c]);
        wb[0] = ff_of(wd.x); wb[1] = ff_of(wd.y); wb[2] = ff_of(wd.z);
    } else {
        free_rotate_ff(q, wb, qf, I32, Iinv32, hf);
    }
    // rotation matrix in float-float from the float-float quaternion
    quat_ff_to_R_ff(q, Rf, Rlo);
    for (int c = 0; c < 4; ++c) qf[c] = q[c].hi;
    const float3 wpred = f3(wb[0].hi, wb[1].hi, wb[2].hi) + (0.5f * hf) * mat_mulf(Iinv32, mat_tmulf(Rf, Nf));
    const float3 wsf = mat_mulf(Rf, wpred);
    for (int c = 0; c < 4; ++c) stff(a.q + 4 * g + c, q[c]);
    for (int c = 0; c < 3; ++c) {
        stff(a.r + 3 * g + c, r[c]);
        stff(a.v + 3 * g + c, v[c]);
        stff(a.wb + 3 * g + c, wb[c]);
    }
    if (!(isfinite(r[0].hi) && isfinite(r[1].hi) && isfinite(r[2].hi)))
        atomicOr(&a.pd[p].flags, DEM_FLAG_NONFINITE);
    ff cc[3];
    float vb[3];
    for (int c = 0; c < 3; ++c) {
        cc[c] = ff_sub(r[c], ff_of2(D.Of[c]));
        vb[c] = ff_sub(ff_add(v[c], ff_mul(hh, acc[c])), ff_of2(D.Vf[c])).hi;
    }
    const float cf[3] = {cc[0].hi, cc[1].hi, cc[2].hi};
    rebuild_test(a, p, g, cf, qf);
    AggRecMixed rec;
    for (int k = 0; k < 9; ++k) { rec.Rh[k] = Rf[k]; rec.Rl[k] = Rlo[k]; }
    for (int c = 0; c < 3; ++c) { rec.ch[c] = cc[c].hi; rec.cl[c] = cc[c].lo; rec.vb[c] = vb[c]; }
    rec.w[0] = wsf.x; rec.w[1] = wsf.y; rec.w[2] = wsf.z;
    rec.pad[0] = rec.pad[1] = 0.f;
    a.rec32[g] = rec;
}

constexpr int kAggThreads = 128;   // threads per block of the aggregate kernels, an aggregate each

template <bool FP64, bool ADAPT>
__global__ void __launch_bounds__(kAggThreads) k_agg_begin(Arrays a, Sizes z)
{
    pdl_enter();
    int64_t g = (int64_t)blockIdx.x * kAggThreads + threadIdx.x;
    if (g >= z.A) return;
    int p = aggregate_pile(a, z, g);
    if (!pile_active(a, p)) return;
    if constexpr (FP64) agg_begin_64<ADAPT>(a, g, p);
    else agg_begin_mixed<ADAPT>(a, g, p);
}

void launch_agg_begin(const Arrays &a, const Sizes &z, bool fp64, cudaStream_t st)
{
    if (z.A == 0) return;
    const unsigned nb = (unsigned)((z.A + kAggThreads - 1) / kAggThreads);
    // the adaptive rotor needs many more registers: its variant runs only when
    // some pile asks for it
    if (z.adapt) {
        if (fp64) launch_pdl(k_agg_begin<true, true>, nb, kAggThreads, 0, st, a, z);
        else launch_pdl(k_agg_begin<false, true>, nb, kAggThreads, 0, st, a, z);
    } else {
        if (fp64) launch_pdl(k_agg_begin<true, false>, nb, kAggThreads, 0, st, a, z);
        else launch_pdl(k_agg_begin<false, false>, nb, kAggThreads, 0, st, a, z);
    }
}

// ---------------------------------------------------------------- host requests
// Host request (after a state write or a new layout): the next step rebuilds
// the cell list and hit lists of pile `slot` (all piles for slot < 0).
__global__ void k_force_rebuild(Arrays a, Sizes z, int slot)
{
    pdl_enter();
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= z.P || (slot >= 0 && p != slot)) return;
    a.pd[p].rebuild = 1;
}

// State slots for the read-out.
__global__ void k_state_values(const double *src, int64_t n, bool fp64, double *out)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[k] = fp64 ? src[k] : ff_value(ldff(src + k));
}

void launch_state_values(const double *src, int64_t n, bool fp64, double *out, cudaStream_t st)
{
    if (n > 0) k_state_values<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(src, n, fp64, out);
}

// Space-frame spin for the read-out, in FP64 in both precisions (a thread per
// aggregate; on the host it was 3.2 of 3.8 ms at 315,000 aggregates and half
// of the 36 us of a small pile's read).
__global__ void k_space_spin(Arrays a, int64_t a0, int64_t na, bool fp64, double *out)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= na) return;
    const int64_t g = a0 + k;
    double q[4], w[3], R[9];
    for (int c = 0; c < 4; ++c) q[c] = fp64 ? a.q[4 * g + c] : ff_value(ldff(a.q + 4 * g + c));
    for (int c = 0; c < 3; ++c) w[c] = fp64 ? a.wb[3 * g + c] : ff_value(ldff(a.wb + 3 * g + c));
    quat_to_R(q, R);
    st3(out + 3 * k, mat_mul(R, d3(w[0], w[1], w[2])));
}

void launch_space_spin(const Arrays &a, int64_t a0, int64_t na, bool fp64, double *out, cudaStream_t st)
{
    if (na > 0) k_space_spin<<<(unsigned)((na + 127) / 128), 128, 0, st>>>(a, a0, na, fp64, out);
}

void set_launch_pdl(int64_t n_spheres) { tl_pdl = n_spheres <= kPdlMaxSpheres; }

void launch_force_rebuild(const Arrays &a, const Sizes &z, int slot, cudaStream_t st)
{
    if (z.P == 0) return;
    launch_pdl(k_force_rebuild, (unsigned)((z.P + 127) / 128), 128, 0, st, a, z, slot);
}

// ---------------------------------------------------------------- step end
// Per aggregate: F_A = sum_i (F_c,i + F_g,i + F_e,i) and
// N_A = sum_i [(r_i - r_A) x F_i + tau_i], kept separately for contact,
// gravity and planet; a_A = F_A / M; closing half kick of COM and spin; YORP
// increment dw: v_A += dw x (r_A - R_pile), w_A += dw (rigid rotation of the
// whole pile).  Members are contiguous (spheres stored in aggregate order).
// GRAV = 0: no pile of the world has self-gravity (the gravity sums are left
// out, and with them their registers); 2: the sphere gravity of piles with
// more than one tile is still in the integer accumulators (Sizes::gacc_on).
// Fsum: the planet's force on the aggregate.
template <bool FP64, int GRAV, typename T>
__device__ __forceinline__ void agg_end(const Arrays &a, int64_t g, int p, T (&Fsum)[3])
{
    const PileStatic &S = a.ps[p];
    const PileDyn &D = a.pd[p];
    const double h = S.h;
    int64_t i0 = S.s0 + a.agg_first[g];
    int n = a.agg_count[g];
    double3 Fc, Nc, Fg, Ng;
    double3 Fe = d3(0, 0, 0), Ne = d3(0, 0, 0);
    const bool planet = S.ext_mass > 0;
    if constexpr (FP64) {
        Fc = Nc = Fg = Ng = d3(0, 0, 0);
        const AggRec64 &rec = a.rec64[g];
        for (int t = 0; t < n; ++t) {
            int64_t i = i0 + t;
            const double *b = a.b64 + 3 * i;
            const double3 lever = mat_mul(rec.R, d3(b[0], b[1], b[2]));
            const dbl4 f = a.ftc64[2 * i], tq = a.ftc64[2 * i + 1];
            const double3 fc = d3(f.x, f.y, f.z), tc = d3(tq.x, tq.y, tq.z);
            const dbl4 gg = GRAV ? a.fg[i] : make_dbl4(0.0, 0.0, 0.0, 0.0);
            const double3 fg = d3(gg.x, gg.y, gg.z);
            Fc = Fc + fc;
            Nc = Nc + cross(lever, fc) + tc;
            Fg = Fg + fg;
            Ng = Ng + cross(lever, fg);
            if (planet) {
                const double3 fe = planet_force(S.G * S.ext_mass, a.m64[i], ld3(D.P_pos), ld3(D.O) + expand_64(rec, b));
                Fe = Fe + fe;
                Ne = Ne + cross(lever, fe);
            }
        }
    } else {
        // per-sphere terms in FP32 (their inputs are FP32), sums float-float
        FFSum s[12];
        const AggRecMixed &rec = a.rec32[g];
        float Rh[9];
        for (int k = 0; k < 9; ++k) Rh[k] = rec.Rh[k];
        // members in order (without self-gravity the gravity sums stay zero)
        auto term = [&](float4 bh, float4 f, float4 tq, dbl4 gg) {
            const float3 lever = mat_mulf(Rh, f3(bh.x, bh.y, bh.z));
            const float3 fc = f3(f.x, f.y, f.z);
            const float3 nc = cross(lever, fc) + f3(tq.x, tq.y, tq.z);
            s[0].add(fc.x); s[1].add(fc.y); s[2].add(fc.z);
            s[3].add(nc.x); s[4].add(nc.y); s[5].add(nc.z);
            if (GRAV) {
                const float3 fg = f3((float)gg.x, (float)gg.y, (float)gg.z);
                const float3 ng = cross(lever, fg);
                s[6].add(fg.x); s[7].add(fg.y); s[8].add(fg.z);
                s[9].add(ng.x); s[10].add(ng.y); s[11].add(ng.z);
            }
        };
        // a pile without self-gravity has zero sphere gravity: not read
        const bool grav = GRAV && S.G != 0.0;
        const dbl4 g0 = make_dbl4(0.0, 0.0, 0.0, 0.0);
        const bool sums = GRAV == 2 && grav && a.gnchunk[p] > 1;
        auto gravity_of = [&](int64_t i) -> dbl4 {
            if (sums) {
                const dbl4 f = gacc_force(a, S, i, gacc_load(a, i));
                a.fg[i] = f;
                return f;
            }
            return grav ? a.fg[i] : g0;
        };
        auto gravity_of2 = [&](int64_t i, dbl4 &ga, dbl4 &gb) {
            if (sums) {   // both spheres' sums loaded before either is cleared
                const GaccSums x = gacc_load(a, i), y = gacc_load(a, i + 1);
                a.fg[i] = ga = gacc_force(a, S, i, x);
                a.fg[i + 1] = gb = gacc_force(a, S, i + 1, y);
                return;
            }
            ga = gravity_of(i);
            gb = gravity_of(i + 1);
        };
        auto planet_term = [&](float4 bh, dbl4 e) {
            const float3 lever = mat_mulf(Rh, f3(bh.x, bh.y, bh.z));
            const double3 fe = d3(e.x, e.y, e.z);
            Fe = Fe + fe;
            Ne = Ne + cross(d3(lever.x, lever.y, lever.z), fe);
        };
        auto planet_of = [&](int64_t i) -> dbl4 { return planet ? a.fe[i] : g0; };
        int t = 0;
        for (; t + 1 < n; t += 2) {   // the loads of two members issued together
            const int64_t i = i0 + t;
            const float4 bha = a.bh[i], bhb = a.bh[i + 1];
            float4 fa, ta, fb, tb;
            ld_f4x2(a.ftc32 + 2 * i, fa, ta);
            ld_f4x2(a.ftc32 + 2 * i + 2, fb, tb);
            const dbl4 ea = planet_of(i), eb = planet_of(i + 1);
            dbl4 ga, gb;
            gravity_of2(i, ga, gb);
            term(bha, fa, ta, ga);
            term(bhb, fb, tb, gb);
            if (planet) {
                planet_term(bha, ea);
                planet_term(bhb, eb);
            }
        }
        if (t < n) {
            const int64_t i = i0 + t;
            const float4 bh = a.bh[i];
            float4 fc, tc;
            ld_f4x2(a.ftc32 + 2 * i, fc, tc);
            const dbl4 e = planet_of(i);
            term(bh, fc, tc, gravity_of(i));
            if (planet) planet_term(bh, e);
        }
        // the parts as float-float pairs (readout only), the totals formed in
        // float-float and converted once (FP64 instructions are ~60 times
        // slower than FP32 ones here)
        ff part[18];
        for (int k = 0; k < 12; ++k) part[k] = ff{s[k].hi, s[k].lo};
        if (planet) {
            part[12] = ff_of(Fe.x); part[13] = ff_of(Fe.y); part[14] = ff_of(Fe.z);
            part[15] = ff_of(Ne.x); part[16] = ff_of(Ne.y); part[17] = ff_of(Ne.z);
            if constexpr (!FP64)
                for (int c = 0; c < 3; ++c) Fsum[c] = part[12 + c];
        } else {
            for (int k = 12; k < 18; ++k) part[k] = ff{0.f, 0.f};
        }
        // the gravity and planet parts of a pile without them stay zero (as
        // set when the pile was added): not rewritten
        for (int k = 0; k < 18; ++k)
            if (k < 6 || (k < 12 && grav) || (k >= 12 && planet))
                reinterpret_cast<float2 *>(a.out[k / 6] + 6 * g)[k % 6] = make_float2(part[k].hi, part[k].lo);
        // totals, a_A = F_A / M and the closing kick in float-float (the
        // state is float-float pairs: no FP64 instruction here)
        const ff hh = {0.5f * S.hff[0], 0.5f * S.hff[1]};
        const ff iM = ldff(a.invM + g);
        ff Ft[3], Nt[3], accf[3], v[3], wb[3];
        for (int c = 0; c < 3; ++c) {
            Ft[c] = ff_add(ff_add(part[c], part[6 + c]), part[12 + c]);
            Nt[c] = ff_add(ff_add(part[3 + c], part[9 + c]), part[15 + c]);
            accf[c] = ff_mul(Ft[c], iM);
            v[c] = ff_add(ldff(a.v + 3 * g + c), ff_mul(hh, accf[c]));
            wb[c] = ldff(a.wb + 3 * g + c);
        }
        // closing spin kick: an increment, FP32, with the step's rotation
        // matrix (the record's FP32 part)
        const float3 Nf = f3(Nt[0].hi, Nt[1].hi, Nt[2].hi);
        const float3 dw = (0.5f * S.lawf[8]) * mat_mulf(a.Iinv32 + 9 * g, mat_tmulf(Rh, Nf));
        wb[0] = ff_addf(wb[0], dw.x); wb[1] = ff_addf(wb[1], dw.y); wb[2] = ff_addf(wb[2], dw.z);
        if (S.yorp) {   // rigid-rotation increment of the whole pile: increments in FP32
            const float3 dwy = f3(S.spin_f[0], S.spin_f[1], S.spin_f[2]);
            const float3 lev = f3(ff_sub(ldff(a.r + 3 * g), ff_of2(D.Rcf[0])).hi,
                                  ff_sub(ldff(a.r + 3 * g + 1), ff_of2(D.Rcf[1])).hi,
                                  ff_sub(ldff(a.r + 3 * g + 2), ff_of2(D.Rcf[2])).hi);
            const float3 dv = cross(dwy, lev), dwb = mat_tmulf(Rh, dwy);
            v[0] = ff_addf(v[0], dv.x); v[1] = ff_addf(v[1], dv.y); v[2] = ff_addf(v[2], dv.z);
            wb[0] = ff_addf(wb[0], dwb.x); wb[1] = ff_addf(wb[1], dwb.y); wb[2] = ff_addf(wb[2], dwb.z);
        }
        bool fin = true;
        for (int c = 0; c < 3; ++c) {
            stff(a.acc + 3 * g + c, accf[c]);
            stff(a.torque + 3 * g + c, Nt[c]);
            stff(a.v + 3 * g + c, v[c]);
            stff(a.wb + 3 * g + c, wb[c]);
            fin = fin && isfinite(v[c].hi) && isfinite(wb[c].hi) && isfinite(Nt[c].hi);
        }
        if (!fin) {
            atomicOr(&a.pd[p].flags, DEM_FLAG_NONFINITE);
            __threadfence();   // before the pile's last block reads the flags
        }
    }
    if constexpr (FP64) {
        st3(Fsum, Fe);
        st3(a.out[0] + 6 * g, Fc); st3(a.out[0] + 6 * g + 3, Nc);
        st3(a.out[1] + 6 * g, Fg); st3(a.out[1] + 6 * g + 3, Ng);
        st3(a.out[2] + 6 * g, Fe); st3(a.out[2] + 6 * g + 3, Ne);
        const double3 F = Fc + Fg + Fe, N = Nc + Ng + Ne;
        const double3 acc = a.invM[g] * F;
        const double q[4] = {a.q[4 * g], a.q[4 * g + 1], a.q[4 * g + 2], a.q[4 * g + 3]};
        double3 v = ld3(a.v + 3 * g) + (0.5 * h) * acc;
        double3 wb = ld3(a.wb + 3 * g);
        const double3 dwy = ld3(S.spin_inc);
        double R[9];
        quat_to_R(q, R);
        wb = wb + (0.5 * h) * mat_mul(a.Iinv + 9 * g, mat_tmul(R, N));
        if (dwy.x != 0.0 || dwy.y != 0.0 || dwy.z != 0.0) {
            v = v + cross(dwy, ld3(a.r + 3 * g) - ld3(D.Rc));
            wb = wb + mat_tmul(R, dwy);
        }
        st3(a.acc + 3 * g, acc);
        st3(a.torque + 3 * g, N);
        st3(a.v + 3 * g, v);
        st3(a.wb + 3 * g, wb);
        if (!finite3(v) || !finite3(wb) || !finite3(N) || !finite3(ld3(a.r + 3 * g))) {
            atomicOr(&a.pd[p].flags, DEM_FLAG_NONFINITE);
            __threadfence();   // before the pile's last block reads the flags
        }
    }
}

// One block per kAggThreads aggregates of a chunk of a pile.
template <bool FP64, int GRAV>
__global__ void __launch_bounds__(kAggThreads) k_agg_end(Arrays a, Sizes z)
{
    pdl_enter();
    constexpr int kCtas = kAggChunk / kAggThreads;
    const int64_t ch = blockIdx.x / kCtas;
    const int p = z.P == 1 ? 0 : a.chunk_pile[ch];
    int64_t beg, end;
    chunk_range(a, ch, p, beg, end);
    beg += (int64_t)(blockIdx.x % kCtas) * kAggThreads;
    if (beg >= end || !pile_active(a, p)) return;
    const int64_t g = beg + threadIdx.x;
    typename std::conditional<FP64, double, ff>::type Fe[3] = {};
    if (g < end) agg_end<FP64, GRAV>(a, g, p, Fe);
    close_pile<kAggThreads>(a, ch, p, Fe);
}

void launch_agg_end(const Arrays &a, const Sizes &z, bool fp64, cudaStream_t st)
{
    if (z.CH == 0) return;
    const unsigned nb = (unsigned)z.CH * (kAggChunk / kAggThreads);
    if (fp64) {
        if (z.grav) launch_pdl(k_agg_end<true, 1>, nb, kAggThreads, 0, st, a, z);
        else launch_pdl(k_agg_end<true, 0>, nb, kAggThreads, 0, st, a, z);
    } else {
        if (z.grav && z.gacc_on == 2) launch_pdl(k_agg_end<false, 2>, nb, kAggThreads, 0, st, a, z);
        else if (z.grav) launch_pdl(k_agg_end<false, 1>, nb, kAggThreads, 0, st, a, z);
        else launch_pdl(k_agg_end<false, 0>, nb, kAggThreads, 0, st, a, z);
    }
}

}  // namespace dem
