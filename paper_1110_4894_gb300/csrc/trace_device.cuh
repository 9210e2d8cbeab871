// trace_device.cuh -- device functions of one trace shared by the per-stage
// kernels and the batched persistent kernel: background cosmology and the
// step table, bundle initialiser, field gather with mean subtraction, the
// geodesic right-hand side, one RK4 stage of one ray, and the bundle reducer.
#pragma once
#include <math_constants.h>

#include "rt3d_internal.cuh"

namespace rt3d {

// ---------------------------------------------------------------------------
// background cosmology on the device (Sec. 3.5, Eq. raytracedistance)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double hubble_E(const Cosmo &c, double z)
{
    double u = 1.0 + z;
    return sqrt(c.om * u * u * u + c.ol);
}

// The integrals below are evaluated by groups of kGroup lanes.  A redshift is
// five or six Newton iterations on chi(z), each 25 panels (z = 0.5) of five
// square roots and divisions in FP64, and an affine step needs 17 of them: in one
// thread that chain took 6-7 ms per trace, whatever the number of steps, and 54
// ms for 48 cones.  The panels are independent, so the lanes of a group take
// one each and only the sum stays serial: it is taken in panel order with the
// operations written out, and gives the same bits as one thread does.  Eight
// lanes waste few of them on the short integrals of nearby nodes; the two FP64
// lanes per SM are then the bound: 0.2 ms for 200 steps to z = 0.5, 2 ms for the
// 48 cones.  Whole warps call these functions (the
// groups of a warp may hold different arguments).
constexpr int kGroup = 8;

// chi(z) = (1/H0) int_0^z dz'/E(z') by composite Boole's rule (5-point
// Newton-Cotes, error O(h^7)), panels no wider than 0.02 in z.
__device__ __forceinline__ double inv_hubble_E(const Cosmo &c, double z)
{
    const double u = 1.0 + z;
    return 1.0 / sqrt(fma(__dmul_rn(__dmul_rn(c.om, u), u), u, c.ol));
}

static __device__ double comoving_distance(const Cosmo &c, double z)
{
    const int lane = threadIdx.x & (kGroup - 1);
    const int panels = z > 0.0 ? max(1, (int)ceil(z / 0.02)) : 0;
    const double w = panels ? z / panels : 0.0, h = 0.25 * w;
    const double coef = 2.0 * h / 45.0;
    const int most = __reduce_max_sync(0xffffffffu, panels);
    double acc = 0.0;
    for (int p0 = 0; p0 < most; p0 += kGroup) {
        double t = 0.0;
        if (p0 + lane < panels) {
            const double z0 = __dmul_rn((double)(p0 + lane), w);
            const double f0 = inv_hubble_E(c, z0), f1 = inv_hubble_E(c, __dadd_rn(z0, h)),
                         f2 = inv_hubble_E(c, __dadd_rn(z0, 2.0 * h)), f3 = inv_hubble_E(c, fma(3.0, h, z0)),
                         f4 = inv_hubble_E(c, __dadd_rn(z0, w));
            t = fma(12.0, f2, fma(7.0, __dadd_rn(f0, f4), __dmul_rn(32.0, __dadd_rn(f1, f3))));
        }
#pragma unroll
        for (int q = 0; q < kGroup; ++q) {
            const double v = __shfl_sync(0xffffffffu, t, q, kGroup);
            if (p0 + q < panels) acc = fma(v, coef, acc);
        }
    }
    return panels ? acc / c.H0 : 0.0;
}

// redshift at comoving distance chi (Newton on chi(z), d chi/dz = 1/(H0 E))
static __device__ double redshift_at(const Cosmo &c, double chi)
{
    double z = chi > 0.0 ? chi * c.H0 : 0.0;
    bool run = chi > 0.0;
    for (int it = 0; it < 40 && __any_sync(0xffffffffu, run); ++it) {
        const double x = __dmul_rn(comoving_distance(c, z) - chi, c.H0), E = hubble_E(c, z);
        if (run) {
            const double dz = __dmul_rn(x, E);
            z = __dadd_rn(z, -dz);
            run = !(fabs(dz) <= 2e-16 * (1.0 + z));
        }
    }
    return z;
}

__device__ __forceinline__ double sched_node(int kind, int n, int k, double chi_s, double chi_l, double s)
{
    if (k == 0) return 0.0;
    if (k == n) return chi_s;
    if (kind == RT3D_SCHED_UNIFORM) return chi_s * (double)k / (double)n;
    const double u0 = asinh((0.0 - chi_l) / s), u1 = asinh((chi_s - chi_l) / s);
    return chi_l + s * sinh(u0 + (u1 - u0) * (double)k / (double)n);
}


// Affine steps of the unperturbed ray: dlam[k] = int a^2 dchi over [x_k,
// x_{k+1}] by composite Boole's rule with 4 panels of 5 points.  One block of
// kSchedThreads takes a step at a time, one lane group per quadrature point.
constexpr int kSchedThreads = 160;  // 17 points of kGroup lanes, whole warps
__device__ __forceinline__ void schedule_steps(const Cosmo &c, int kind, int n, double chi_s, double chi_l, double s,
                                               double *__restrict__ dlam)
{
    __shared__ double s_a[kSchedThreads / kGroup];
    const int q = threadIdx.x / kGroup;  // point: 0 the step's start, then 4 per panel
    for (int k = blockIdx.x; k < n; k += gridDim.x) {
        const double x0 = sched_node(kind, n, k, chi_s, chi_l, s), x1 = sched_node(kind, n, k + 1, chi_s, chi_l, s);
        const double w = __dmul_rn(__dadd_rn(x1, -x0), 0.25), h = 0.25 * w;
        const int i = (q - 1) & 3;
        const double xa = fma((double)((q - 1) >> 2), w, x0);
        double x = i == 0 ? xa + h : (i == 1 ? fma(2.0, h, xa) : (i == 2 ? fma(3.0, h, xa) : xa + w));
        if (q == 0) x = x0;
        if (q == 16) x = x1;
        if (q > 16) x = 0.0;
        const double a = 1.0 / (1.0 + redshift_at(c, x));
        if ((threadIdx.x & (kGroup - 1)) == 0) s_a[q] = a;
        __syncthreads();
        if (threadIdx.x == 0) {
            const double coef = 2.0 * h / 45.0;
            double acc = 0.0;
            for (int p = 0; p < 4; ++p) {
                const double *g = s_a + 4 * p;
                const double s04 = __dadd_rn(__dmul_rn(g[0], g[0]), __dmul_rn(g[4], g[4]));
                const double s13 = fma(g[1], g[1], __dmul_rn(g[3], g[3]));
                acc = fma(fma(12.0, __dmul_rn(g[2], g[2]), fma(32.0, s13, __dmul_rn(7.0, s04))), coef, acc);
            }
            dlam[k] = acc;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// bundle initialiser (Sec. 3.1, ray bundle; initial state of Sec. 3.4)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void ray_theta(const TraceParams &tp, const double *theta, int64_t b, int k,
                                          double &tx, double &ty)
{
    tx = theta[2 * b];
    ty = theta[2 * b + 1];
    if (k > 0) {
        const double ang = tp.phase + 2.0 * CUDART_PI * (double)(k - 1) / (double)tp.n_ring;
        double sn, cs;
        sincos(ang, &sn, &cs);
        tx += tp.theta_r * cs;
        ty += tp.theta_r * sn;
    }
}


// bundle initialiser for ray i (Sec. 3.1; initial state of Sec. 3.4)
__device__ __forceinline__ void init_ray(const TraceParams &tp, const DevField &f, const double *__restrict__ theta,
                                         const RayState &rs, int64_t i)
{
    const int64_t b = i / rs.nr;
    const int k = (int)(i % rs.nr);
    double tx, ty;
    ray_theta(tp, theta, b, k, tx, ty);
    // observer: t = 0 (lookback), x = 0, direction (theta_x, theta_y, 1) with
    // dx3/dl = 1; dt/dl is set from the null condition at the first stage
    const double v[8] = {0.0, 0.0, 0.0, 0.0, sqrt(tx * tx + ty * ty + 1.0), tx, ty, 1.0};
    const int64_t n = rs.stride;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        rs.y[q * n + i] = v[q];
        rs.ys[q * n + i] = v[q];
        rs.ks[q * n + i] = 0.0;
        rs.fin[q * n + i] = 0.0;
    }
    rs.done[i] = 0;
    rs.steps[i] = -1;
    if (k == 0) rs.rep[b] = replica_of(f, 0.0);  // stage parity 0
}

// ---------------------------------------------------------------------------
// integrator stage (Eq. geodesiceqn with the App. A symbols, classical RK4,
// termination on x3 with linear interpolation: Sec. 3.4)
// ---------------------------------------------------------------------------
// phi and grad phi from the reduced pair sums, plus the mean subtraction.
// The sums hold sum m'' / |d| and sum m'' d / |d|^3 (Mpc) with d = particle -
// point and m'' = mu_G m 2^ms (or the same sums without m'' for a uniform-mass
// field, mfac = m''): phi = -S0 mfac / 2^ms, grad phi = -S mfac / 2^ms.
// Bundle prism record (kPrismRec doubles per bundle): the central ray's stage
// position, and the replica prism's I, grad I and Hessian there.
// A ray whose offset e from its bundle's central ray is below 1/kPrismNear of
// the central ray's distance to every face of the prism takes I and grad I
// from the second-order Taylor expansion about the central ray; the
// remainder is O(|e|^3 / d) in I and O(|e|^2 / d) in grad I, d the face
// distance (the prism's third derivatives fall off as 1/d inside), i.e. a
// relative 1/(2 kPrismNear) of the tidal term H e.  Other rays use the
// closed form.
constexpr double kPrismNear = 1000.0;

__device__ __forceinline__ void prism_of_ray(const DevField &f, int rep, const double p[3],
                                             const double *__restrict__ rec, double I[4])
{
    const double lo[3] = {-0.5 * f.L, -0.5 * f.L, (double)rep * f.L};
    const double hi[3] = {0.5 * f.L, 0.5 * f.L, (double)(rep + 1) * f.L};
    if (rec) {
        const double e[3] = {p[0] - rec[0], p[1] - rec[1], p[2] - rec[2]};
        const double en = sqrt(e[0] * e[0] + e[1] * e[1] + e[2] * e[2]);
        double d = rec[0] - lo[0];
        d = fmin(d, hi[0] - rec[0]);
        d = fmin(d, rec[1] - lo[1]);
        d = fmin(d, hi[1] - rec[1]);
        d = fmin(d, rec[2] - lo[2]);
        d = fmin(d, hi[2] - rec[2]);
        if (d > kPrismNear * en) {
            const double *g = rec + 3, *h = rec + 7;  // g = (I, grad I)
            const double he[3] = {h[0] * e[0] + h[1] * e[1] + h[2] * e[2], h[1] * e[0] + h[3] * e[1] + h[4] * e[2],
                                  h[2] * e[0] + h[4] * e[1] + h[5] * e[2]};
            I[0] = g[0] + (g[1] * e[0] + g[2] * e[1] + g[3] * e[2]) +
                   0.5 * (e[0] * he[0] + e[1] * he[1] + e[2] * he[2]);
            I[1] = g[1] + he[0];
            I[2] = g[2] + he[1];
            I[3] = g[3] + he[2];
            return;
        }
    }
    prism_field<double>(lo, hi, p, I);
}

// rec: the bundle's prism record, or null (closed form at p)
__device__ __forceinline__ void field_from_sums(const DevField &f, const double acc[4], int rep, const double p[3],
                                                double mfac, double F[4], const double *rec = nullptr)
{
    const double sp = f.mscale_inv * mfac, sg = sp;
    F[0] = -acc[0] * sp;
    F[1] = -acc[1] * sg;
    F[2] = -acc[2] * sg;
    F[3] = -acc[3] * sg;
    if (f.replicated && f.mean_subtract) {
        // remove the field of the replica's uniform mean density (Sec. 3.3)
        double I[4];
        prism_of_ray(f, rep, p, rec, I);
        F[0] += f.rho_term * I[0];
        F[1] += f.rho_term * I[1];
        F[2] += f.rho_term * I[2];
        F[3] += f.rho_term * I[3];
    }
}

// The prism record of bundle b at its central ray's stage position, by kCorners
// lanes: each takes one corner of the prism (three logarithms, three
// arctangents and a square root: some 440 FP64 operations), then lane q adds up
// quantity q of the record over the corners, in the order of
// prism_field_hess.  One thread per bundle kept all eight corners of 128
// bundles on one SM's two FP64 lanes: 105 us a stage, 16 us now.  s_q: 80 doubles of shared
// memory per group of lanes; whole warps call this (b < 0: nothing to do).
constexpr int kCorners = 8;
__device__ __forceinline__ void bundle_prism(const DevField &f, const RayState &rs, int g, int64_t b,
                                             double *__restrict__ rec, double *s_q)
{
    const int c = threadIdx.x & (kCorners - 1);
    if (b >= 0) {
        const int64_t ic = b * rs.nr, st = rs.stride;
        const int rep = rs.rep[(g & 1) * rs.n_b + b];
        const double p[3] = {rs.ys[st + ic], rs.ys[2 * st + ic], rs.ys[3 * st + ic]};
        const double lo[3] = {-0.5 * f.L, -0.5 * f.L, (double)rep * f.L};
        const double hi[3] = {0.5 * f.L, 0.5 * f.L, (double)(rep + 1) * f.L};
        const double x = ((c & 1) ? hi[0] : lo[0]) - p[0];
        const double y = ((c & 2) ? hi[1] : lo[1]) - p[1];
        const double z = ((c & 4) ? hi[2] : lo[2]) - p[2];
        double v[10];
        prism_corner_hess(x, y, z, v);
#pragma unroll
        for (int q = 0; q < 10; ++q) s_q[kCorners * q + c] = v[q];
        if (c < 3) rec[kPrismRec * b + c] = p[c];
    }
    __syncwarp();
    if (b >= 0)
        for (int q = c; q < 10; q += kCorners) {
            double acc = 0.0;
#pragma unroll
            for (int k = 0; k < kCorners; ++k) {
                const bool minus = ((3 - __popc(k)) & 1) != 0;  // inclusion-exclusion over the corners
                // I and the mixed derivatives add a corner's term, the gradient and the pure ones take it off
                const bool add = minus != (q == 0 || q >= 7);
                acc = add ? acc + s_q[kCorners * q + k] : acc - s_q[kCorners * q + k];
            }
            // record: position, I, grad I, then xx, xy, xz, yy, yz, zz
            const int slot = q < 4 ? 3 + q : (q == 4 ? 7 : q == 5 ? 10 : q == 6 ? 12 : q == 7 ? 8 : q == 8 ? 9 : 11);
            rec[kPrismRec * b + slot] = acc;
        }
    __syncwarp();
}

// One more split's (hi, lo) in a double-float sum in FP32 (TwoSum on the high
// parts, low parts carried)
__device__ __forceinline__ void reduce_step(float &hi, float &lo, float2 v)
{
    const float t = hi + v.x;
    const float bb = t - hi;
    const float err = (hi - (t - bb)) + (v.x - bb);
    hi = t;
    lo += err + v.y;
}

// One output of one ray's split partials, converted once to FP64.
__device__ __forceinline__ double reduce_partials_mixed(const float2 *__restrict__ pm, int S, int64_t n, int64_t i,
                                                        int o)
{
    float hi = 0.0f, lo = 0.0f;
#pragma unroll 8  // loads in flight ahead of the serial sum
    for (int s = 0; s < S; ++s) reduce_step(hi, lo, pm[((int64_t)s * 4 + o) * n + i]);
    return (double)hi + (double)lo;
}

// Reduce the pair-sum partials of one ray and add the mean subtraction:
// F = (phi, dphi/dx1, dphi/dx2, dphi/dx3) at the ray's stage position.
__device__ __forceinline__ void gather_field(const DevField &f, int S, bool fp64, const void *partials, int64_t n,
                                             int64_t i, int rep, const double p[3], double mfac, double F[4],
                                             const double *rec = nullptr)
{
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (fp64) {
        const double *pd = (const double *)partials;
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int o = 0; o < 4; ++o) acc[o] += pd[((int64_t)s * 4 + o) * n + i];
    } else {
        // the (hi, lo) FP32 pairs are added as double-float numbers (TwoSum on
        // hi, lo carried separately): ~48-bit sums on the FP32 pipe, converted
        // to FP64 once, instead of 2S conversions and adds on the FP64 pipe
        const float2 *pm = (const float2 *)partials;
        float hi[4] = {0.0f, 0.0f, 0.0f, 0.0f}, lo[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                const float2 v = pm[((int64_t)s * 4 + o) * n + i];
                const float t = hi[o] + v.x;
                const float bb = t - hi[o];
                const float err = (hi[o] - (t - bb)) + (v.x - bb);
                hi[o] = t;
                lo[o] += err + v.y;
            }
#pragma unroll
        for (int o = 0; o < 4; ++o) acc[o] = (double)hi[o] + (double)lo[o];
    }
    field_from_sums(f, acc, rep, p, mfac, F, rec);
}

// d y / d lambda for y = (t, x1, x2, x3, dt/dl, dx1/dl, dx2/dl, dx3/dl):
// d^2 x^a / dl^2 = -Gamma^a_bc u^b u^c with App. A's first-order symbols
//   Gamma^t_tt = -a' phi / a^2,  Gamma^t_ti = phi_i / a,  Gamma^t_ii = a' (a + phi)
//   Gamma^i_tt = phi_i / a^3,    Gamma^i_ti = a' (a + phi) / a^2,
//   Gamma^i_jk = (-phi_k d_ij - phi_j d_ik + phi_i d_jk) / a
// (christoffel = DERIVED replaces Gamma^t_ii by a' (a - 3 phi)).
__device__ __forceinline__ void geodesic_rhs(const double y[8], const double F[4], double a, double ia, double ad,
                                             int christoffel, double k[8])
{
    const double T = y[4], vx = y[5], vy = y[6], vz = y[7];
    const double phi = F[0], gx = F[1], gy = F[2], gz = F[3];
    const double gv = gx * vx + gy * vy + gz * vz;
    const double v2 = vx * vx + vy * vy + vz * vz;
    const double gtii = christoffel == RT3D_CHRISTOFFEL_DERIVED ? ad * (a - 3.0 * phi) : ad * (a + phi);
    const double gitj = ad * (a + phi) * ia * ia;
    k[0] = T;
    k[1] = vx;
    k[2] = vy;
    k[3] = vz;
    k[4] = ad * phi * ia * ia * T * T - 2.0 * ia * gv * T - gtii * v2;
    const double tt = T * T * ia * ia * ia;
    const double drag = 2.0 * gitj * T;
    k[5] = -gx * tt - drag * vx - ia * (gx * v2 - 2.0 * vx * gv);
    k[6] = -gy * tt - drag * vy - ia * (gy * v2 - 2.0 * vy * gv);
    k[7] = -gz * tt - drag * vz - ia * (gz * v2 - 2.0 * vz * gv);
}

// d y / d lambda at stage state ys with the field F; at the observer (first)
// dt/dl of ys and of the step's state y is set from the null condition.
__device__ __forceinline__ void ray_slope(const TraceParams &tp, double ys[8], const double F[4], bool first,
                                          double y[8], double k[8])
{
    const double a = cosmo_a(tp.cosmo, ys[0]);
    const double ia = 1.0 / a;
    const double ad = cosmo_adot_ia(tp.cosmo, a, ia);
    if (first) {
        // null condition of Eq. expandingmetric with psi = phi / a
        const double vn = sqrt(ys[5] * ys[5] + ys[6] * ys[6] + ys[7] * ys[7]);
        const double T = a * vn * sqrt((1.0 - 2.0 * F[0] / a) / (1.0 + 2.0 * F[0] / a));
        ys[4] = T;
        y[4] = T;
    }
    geodesic_rhs(ys, F, a, ia, ad, tp.christoffel, k);
}

// One ray's RK4 stage: gather phi and grad phi, set dt/dl from the null
// condition at the observer, evaluate the geodesic right-hand side, update the
// stage state or (stage 3) combine, terminate and interpolate.  rs is a view:
// ray i of this trace lives at index i with component stride rs.stride, and
// its partials at ((s * 4 + o) * rs.n_rays + i).  Returns whether the ray was
// still in flight (counts towards interactions).
__device__ __forceinline__ bool stage_ray(const TraceParams &tp, const DevField &f, const RayState &rs, int S,
                                          bool fp64, double mfac, const void *__restrict__ partials,
                                          const double *__restrict__ dlam, double chi_s, int step, int stage,
                                          unsigned long long *cnt, int64_t i, const double *pre = nullptr,
                                          const double *prism = nullptr)
{
    const int64_t st = rs.stride;
    const int64_t b = i / rs.nr;
    const int g = step * 4 + stage;  // global stage index: replica buffers alternate on its parity
    const int rep = rs.rep[(g & 1) * rs.n_b + b];
    double ys[8], y[8], k[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        ys[q] = rs.ys[q * st + i];
        y[q] = rs.y[q * st + i];
    }
    double F[4];
    const double *rec = prism ? prism + kPrismRec * b : nullptr;
    if (pre) field_from_sums(f, pre, rep, ys + 1, mfac, F, rec);
    else gather_field(f, S, fp64, partials, rs.n_rays, i, rep, ys + 1, mfac, F, rec);
    ray_slope(tp, ys, F, step == 0 && stage == 0, y, k);
    if (step == 0 && stage == 0) rs.y[4 * st + i] = y[4];
    const double dl = dlam[step < tp.n_steps ? step : tp.n_steps - 1];
    const int done = rs.done[i];
    double nx[8];
    if (stage < 3) {
        const double c = stage == 2 ? dl : 0.5 * dl;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const double acc = stage == 0 ? k[q] : rs.ks[q * st + i] + 2.0 * k[q];
            rs.ks[q * st + i] = acc;
            nx[q] = y[q] + c * k[q];
            rs.ys[q * st + i] = nx[q];
        }
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) nx[q] = y[q] + dl * (1.0 / 6.0) * (rs.ks[q * st + i] + k[q]);
        if (!done && nx[3] >= chi_s) {
            const double s = (chi_s - y[3]) / (nx[3] - y[3]);
#pragma unroll
            for (int q = 0; q < 8; ++q) rs.fin[q * st + i] = y[q] + s * (nx[q] - y[q]);
            rs.done[i] = 1;
            rs.steps[i] = step + 1;
        } else if (!done) {
            atomicAdd(&cnt[step & 1], 1ull);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            rs.y[q * st + i] = nx[q];
            rs.ys[q * st + i] = nx[q];
        }
    }
    if (i % rs.nr == 0) rs.rep[((g + 1) & 1) * rs.n_b + b] = replica_of(f, nx[3]);
    return !done;
}

// RK4 stages [g0, g1) of every ray, for a field that each ray evaluates for
// itself: eval(r, x3, F) gives phi and grad phi at r, x3 the central ray's.
// Nothing but that x3 then couples the rays, so a warp takes whole bundles (6 of
// 5 rays, 3 of 9), keeps their states in registers and runs through all the
// stages in one launch; x3 comes by shuffle.  The bound is FP64: about 150
// operations per ray and stage on two lanes per SM, in a chain of some sixty.
// A bundle whose rays are all across stops: results are taken at the crossing,
// and the stages after it only served other bundles.  Blocks are one warp
// (kTraceRaysNT), which spreads a few hundred warps evenly over the SMs.

template <class Eval>
__device__ __forceinline__ void trace_rays(const TraceParams &tp, const RayState &rs, int g0, int g1,
                                           const double *__restrict__ dlam, const double *__restrict__ misc,
                                           unsigned long long *cnt, const Eval &eval)
{
    const int lane = threadIdx.x & 31, per_warp = 32 / rs.nr;
    const int64_t b = (int64_t)blockIdx.x * per_warp + lane / rs.nr;
    const bool valid = lane < per_warp * rs.nr && b < rs.n_b;
    const int64_t i = valid ? b * rs.nr + lane % rs.nr : 0, st = rs.stride;
    const int src = valid ? lane - lane % rs.nr : lane;  // the central ray's lane
    double y[8], ys[8], ks[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        y[q] = rs.y[q * st + i];
        ys[q] = rs.ys[q * st + i];
        ks[q] = rs.ks[q * st + i];
    }
    bool done = !valid || rs.done[i] != 0;
    const double chi_s = misc[0];
    unsigned active = 0;
    for (int s = g0; s < g1; ++s) {
        const int step = s >> 2, stage = s & 3;
        if ((stage == 0 || s == g0) && !__any_sync(0xffffffffu, !done)) break;
        const double dl = dlam[step < tp.n_steps ? step : tp.n_steps - 1];
        double F[4], k[8];
        eval(ys + 1, __shfl_sync(0xffffffffu, ys[3], src), F);
        ray_slope(tp, ys, F, s == 0, y, k);
        active += done ? 0u : 1u;
        if (stage < 3) {
            const double c = stage == 2 ? dl : 0.5 * dl;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                ks[q] = stage == 0 ? k[q] : ks[q] + 2.0 * k[q];
                ys[q] = y[q] + c * k[q];
            }
        } else {
            double nx[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) nx[q] = y[q] + dl * (1.0 / 6.0) * (ks[q] + k[q]);
            if (!done && nx[3] >= chi_s) {
                const double f = (chi_s - y[3]) / (nx[3] - y[3]);
#pragma unroll
                for (int q = 0; q < 8; ++q) rs.fin[q * st + i] = y[q] + f * (nx[q] - y[q]);
                rs.done[i] = 1;
                rs.steps[i] = step + 1;
                done = true;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) y[q] = ys[q] = nx[q];
        }
    }
    if (valid) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            rs.y[q * st + i] = y[q];
            rs.ys[q * st + i] = ys[q];
            rs.ks[q * st + i] = ks[q];
        }
    }
    const unsigned sum = __reduce_add_sync(0xffffffffu, valid ? active : 0u);
    if (lane == 0 && sum) atomicAdd(&cnt[2], (unsigned long long)sum);
}

// One bundle's lens-map Jacobian from its rays' states at x3 = chi_s; writes
// (mu, kappa, gamma1, gamma2, omega, flags) to o[0..5] and, when rout is
// given, each ray's final state to rout[(b * nr + k) * 8 + q].
__device__ __forceinline__ void reduce_bundle(const TraceParams &tp, const double *__restrict__ theta,
                                              const RayState &rs, double chi_s, int64_t b, double *__restrict__ o,
                                              double *__restrict__ rout)
{
    const int64_t n = rs.stride;
    int flags = 0;
    double x0 = 0, y0 = 0, tx0 = 0, ty0 = 0;
    double M00 = 0, M01 = 0, M10 = 0, M11 = 0, N00 = 0, N01 = 0, N10 = 0, N11 = 0;
    for (int k = 0; k < rs.nr; ++k) {
        const int64_t i = b * rs.nr + k;
        const int done = rs.done[i];
        const double *src = done ? rs.fin : rs.y;
        if (!done) flags |= RT3D_F_NOCROSS;
        double st[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            st[q] = src[q * n + i];
            if (!isfinite(st[q])) flags |= RT3D_F_NONFINITE;
        }
        if (rout)
#pragma unroll
            for (int q = 0; q < 8; ++q) rout[i * 8 + q] = st[q];
        double tx, ty;
        ray_theta(tp, theta, b, k, tx, ty);
        if (k == 0) {
            x0 = st[1];
            y0 = st[2];
            tx0 = tx;
            ty0 = ty;
        } else {
            const double dbx = (st[1] - x0) / chi_s, dby = (st[2] - y0) / chi_s;
            const double dtx = tx - tx0, dty = ty - ty0;
            M00 += dbx * dtx;
            M01 += dbx * dty;
            M10 += dby * dtx;
            M11 += dby * dty;
            N00 += dtx * dtx;
            N01 += dtx * dty;
            N10 += dty * dtx;
            N11 += dty * dty;
        }
    }
    const double dn = N00 * N11 - N01 * N10;
    const double i00 = N11 / dn, i01 = -N01 / dn, i10 = -N10 / dn, i11 = N00 / dn;
    const double A00 = M00 * i00 + M01 * i10, A01 = M00 * i01 + M01 * i11;
    const double A10 = M10 * i00 + M11 * i10, A11 = M10 * i01 + M11 * i11;
    const double det = A00 * A11 - A01 * A10;
    const double mu = 1.0 / det;
    if (!isfinite(mu)) flags |= RT3D_F_NONFINITE;
    if (mu < 0.0) flags |= RT3D_F_NEGPARITY;
    o[0] = mu;
    o[1] = 1.0 - 0.5 * (A00 + A11);
    o[2] = 0.5 * (A11 - A00);
    o[3] = -0.5 * (A01 + A10);
    o[4] = 0.5 * (A01 - A10);
    o[5] = (double)flags;
}

}  // namespace rt3d
