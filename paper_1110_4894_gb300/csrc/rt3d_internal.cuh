// rt3d_internal.cuh -- shared definitions of the sm_103a ray-bundle library.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/rt3d.h"

namespace rt3d {

// ---------------------------------------------------------------------------
// physical constants (IAU nominal G Msun, SI c, Mpc)
// ---------------------------------------------------------------------------
constexpr double kGMsun = 1.32712440018e20;          // m^3 s^-2
constexpr double kC = 299792458.0;                   // m s^-1
constexpr double kMpc = 3.0856775814913673e22;       // m
constexpr double kMuG = kGMsun / (kC * kC) / kMpc;   // G Msun / c^2 in Mpc
constexpr double kCkms = 299792.458;                 // c in km s^-1

struct Cosmo {
    double om, ol, h;
    double H0;  // H0 / c in 1/Mpc
    double t0;  // lookback time of the big bang (Mpc)
    double k;   // 1.5 sqrt(OL) H0
    double r;   // OM / OL
    // a(t) and atab_h da/dt at t = j atab_h, j < atab_n (interleaved), or
    // null: the closed form is then evaluated at every call
    const double *atab = nullptr;
    int atab_n = 0;
    double atab_h = 0.0, atab_ih = 0.0;  // node spacing and its inverse
};

// Eq. scalefac2: a(t) for t the lookback time, closed form.
__device__ __forceinline__ double cosmo_a_exact(const Cosmo &c, double t)
{
    double s = sinh(c.k * (c.t0 - t));
    return cbrt(c.r * s * s);
}

// a(t) by cubic Hermite interpolation of the table (a and da/dt at the
// nodes): the remainder h^4 max|d^4a/dt^4| / 384 is below 1e-13 of a up to
// z = 5 for the 4096-node table, against the closed form's FP64 rounding of a
// few 1e-16; outside the table, the closed form.  It replaces an FP64 sinh
// and cbrt per ray and stage on a GPU whose FP64 rate is 1/64 of FP32.
__device__ __forceinline__ double cosmo_a(const Cosmo &c, double t)
{
    if (c.atab) {
        const double u = t * c.atab_ih;
        if (u >= 0.0 && u < (double)(c.atab_n - 1)) {
            const int j = (int)u;
            const double s = u - (double)j;
            const double a0 = c.atab[2 * j], d0 = c.atab[2 * j + 1];
            const double a1 = c.atab[2 * j + 2], d1 = c.atab[2 * j + 3];
            // the cubic through (a0, d0) at s = 0 and (a1, d1) at s = 1, in powers of s
            const double D = a1 - a0;
            const double c2 = 3.0 * D - 2.0 * d0 - d1, c3 = d0 + d1 - 2.0 * D;
            return a0 + s * (d0 + s * (c2 + s * c3));
        }
    }
    return cosmo_a_exact(c, t);
}

// d a / d t (lookback): -a H(a) for the same flat Lemaitre model.
__device__ __forceinline__ double cosmo_adot(const Cosmo &c, double a)
{
    return -a * c.H0 * sqrt(c.om / (a * a * a) + c.ol);
}

// the same with ia = 1 / a already at hand
__device__ __forceinline__ double cosmo_adot_ia(const Cosmo &c, double a, double ia)
{
    return -a * c.H0 * sqrt(c.om * (ia * ia * ia) + c.ol);
}

// ---------------------------------------------------------------------------
// field of a uniform rectangular prism (mean subtraction, Sec. 3.3):
// I = int dV / |r - r'| and dI/dr, from the closed-form antiderivative.
// ---------------------------------------------------------------------------
// log(u + rho) with rho = |(u, v, w)|, q = v^2 + w^2; stable for u < 0.
template <typename T>
__device__ __forceinline__ T prism_log(T u, T rho, T q)
{
    if (u >= T(0)) return log(u + rho);
    if (q == T(0)) return T(0);  // only ever multiplied by a zero coefficient
    return log(q / (rho - u));
}

template <typename T>
__device__ __forceinline__ void prism_corner(T x, T y, T z, T &F, T &Hx, T &Hy, T &Hz)
{
    T xx = x * x, yy = y * y, zz = z * z;
    T rho = sqrt(xx + yy + zz);
    T lx = prism_log(x, rho, yy + zz), ly = prism_log(y, rho, xx + zz), lz = prism_log(z, rho, xx + yy);
    T tx = (x != T(0)) ? atan(y * z / (x * rho)) : T(0);
    T ty = (y != T(0)) ? atan(z * x / (y * rho)) : T(0);
    T tz = (z != T(0)) ? atan(x * y / (z * rho)) : T(0);
    F = x * y * lz + y * z * lx + z * x * ly - T(0.5) * (xx * tx + yy * ty + zz * tz);
    Hx = y * lz + z * ly - x * tx;
    Hy = z * lx + x * lz - y * ty;
    Hz = x * ly + y * lx - z * tz;
}

// out = (I, dI/dx1, dI/dx2, dI/dx3) for the prism [lo, hi] at point p.
template <typename T>
__device__ __forceinline__ void prism_field(const T lo[3], const T hi[3], const T p[3], T out[4])
{
    T I = 0, gx = 0, gy = 0, gz = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const T x = ((c & 1) ? hi[0] : lo[0]) - p[0];
        const T y = ((c & 2) ? hi[1] : lo[1]) - p[1];
        const T z = ((c & 4) ? hi[2] : lo[2]) - p[2];
        T F, Hx, Hy, Hz;
        prism_corner(x, y, z, F, Hx, Hy, Hz);
        // inclusion-exclusion over the corners: (-1)^(number of lower limits)
        const T sg = ((3 - __popc(c)) & 1) ? T(-1) : T(1);
        I += sg * F;
        gx -= sg * Hx;
        gy -= sg * Hy;
        gz -= sg * Hz;
    }
    out[0] = I;
    out[1] = gx;
    out[2] = gy;
    out[3] = gz;
}

// One corner's terms, unsigned: F and its first derivatives as prism_corner,
// the pure second derivatives tx, ty, tz, then the mixed xy, xz, yz
__device__ __forceinline__ void prism_corner_hess(double x, double y, double z, double v[10])
{
    const double xx = x * x, yy = y * y, zz = z * z;
    const double rho = sqrt(xx + yy + zz);
    const double lx = prism_log(x, rho, yy + zz), ly = prism_log(y, rho, xx + zz), lz = prism_log(z, rho, xx + yy);
    const double tx = (x != 0.0) ? atan(y * z / (x * rho)) : 0.0;
    const double ty = (y != 0.0) ? atan(z * x / (y * rho)) : 0.0;
    const double tz = (z != 0.0) ? atan(x * y / (z * rho)) : 0.0;
    v[0] = x * y * lz + y * z * lx + z * x * ly - 0.5 * (xx * tx + yy * ty + zz * tz);
    v[1] = y * lz + z * ly - x * tx;
    v[2] = z * lx + x * lz - y * ty;
    v[3] = x * ly + y * lx - z * tz;
    v[4] = tx;
    v[5] = ty;
    v[6] = tz;
    v[7] = lz;
    v[8] = ly;
    v[9] = lx;
}

// As prism_field, plus the Hessian d2I/dp_i dp_j (h = xx, xy, xz, yy, yz,
// zz) from the same logarithms and arctangents: for the corner function,
// d2F/dx2 = -atan(yz / (x rho)) and d2F/dx dy = log(z + rho) (cyclically).
template <typename T>
__device__ __forceinline__ void prism_field_hess(const T lo[3], const T hi[3], const T p[3], T out[4], T h[6])
{
    T I = 0, gx = 0, gy = 0, gz = 0, hxx = 0, hxy = 0, hxz = 0, hyy = 0, hyz = 0, hzz = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const T x = ((c & 1) ? hi[0] : lo[0]) - p[0];
        const T y = ((c & 2) ? hi[1] : lo[1]) - p[1];
        const T z = ((c & 4) ? hi[2] : lo[2]) - p[2];
        const T xx = x * x, yy = y * y, zz = z * z;
        const T rho = sqrt(xx + yy + zz);
        const T lx = prism_log(x, rho, yy + zz), ly = prism_log(y, rho, xx + zz), lz = prism_log(z, rho, xx + yy);
        const T tx = (x != T(0)) ? atan(y * z / (x * rho)) : T(0);
        const T ty = (y != T(0)) ? atan(z * x / (y * rho)) : T(0);
        const T tz = (z != T(0)) ? atan(x * y / (z * rho)) : T(0);
        const T sg = ((3 - __popc(c)) & 1) ? T(-1) : T(1);
        I += sg * (x * y * lz + y * z * lx + z * x * ly - T(0.5) * (xx * tx + yy * ty + zz * tz));
        gx -= sg * (y * lz + z * ly - x * tx);
        gy -= sg * (z * lx + x * lz - y * ty);
        gz -= sg * (x * ly + y * lx - z * tz);
        hxx -= sg * tx;
        hyy -= sg * ty;
        hzz -= sg * tz;
        hxy += sg * lz;
        hyz += sg * lx;
        hxz += sg * ly;
    }
    out[0] = I;
    out[1] = gx;
    out[2] = gy;
    out[3] = gz;
    h[0] = hxx;
    h[1] = hxy;
    h[2] = hxz;
    h[3] = hyy;
    h[4] = hyz;
    h[5] = hzz;
}

// ---------------------------------------------------------------------------
// overlapped launches
// ---------------------------------------------------------------------------
// The short kernels of a trace follow one another some thousand times, and the
// gap between two of them (2.7 us, against 4 to 8 us of work in a small trace)
// is launch latency (4 bundles through 5000 particles, 200 steps: 18.1 -> 12.6
// ms).  Launched this way, a kernel's blocks may start as soon as every block of
// the kernel before it in the stream has ended, or has called let_next_start; it
// must call wait_for_previous before it reads what an earlier kernel of the stream
// wrote, or writes anything.  The wait returns when the kernel before is complete
// and its writes are visible; as that one waited too, so is every earlier kernel.
// In a kernel launched the ordinary way both calls do nothing.
//
// Blocks that wait beside the running ones are packed several to an SM, and the
// FP64 stage of a mid-size trace then runs on part of the SMs.  So the stage
// kernels and k_force_fp64 never let the next one in, k_force_bundle1 does where
// its blocks leave every SM room (and no prism kernel comes in between), and the
// short k_prism and k_merge do.  30 steps with all of them letting the next one in
// / launched the ordinary way / as here: 66 bundles through 20,000 particles 3.85 /
// 3.85 / 2.85 ms, 512 through 2000 4.4 / 3.7 / 2.75, 2048 through 300 5.1 / 3.6 / 2.6;
// mean-subtracted boxes: 256 through 5000 13.2 / 7.2 / 5.8, 1024 of 8 rays through
// 500 20.5 / 7.4 / 6.0; FP64, 66 through 300 3.56 / 3.85 / 2.73.  Larger traces: the
// same.  4 bundles through 5000 particles, 200 steps, with / here / none letting the
// next one in: 13.3 / 12.6 / 13.0.
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_overlapped(void (*kern)(P...), dim3 grid, int threads, cudaStream_t st, const A &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// ---------------------------------------------------------------------------
// device-side particle field
// ---------------------------------------------------------------------------
struct DevField {
    const int4 *part;      // (qx, qy, qz, m32 bits): integer grid position, scaled mass (FP32)
    const float *eps2;     // per-particle eps^2 (Mpc^2), or nullptr
    const double *m64;     // scaled masses (FP64 path)
    const double *eps2_64; // per-particle eps^2 (FP64 path) or nullptr
    const int *rot;        // n_rep * 9
    const int *shift;      // n_rep * 3, grid units
    int64_t n;
    float eps2u;           // uniform eps^2 (Mpc^2)
    double eps2u64;
    int replicated, mean_subtract, n_rep;
    int Lq;                // box length in grid units (replicated)
    double delta, inv_delta;  // grid spacing 2^-e (Mpc) and its inverse
    double O[3];           // world position of grid origin (isolated fields)
    double L;              // box length (Mpc)
    double mscale_inv;     // 1 / 2^ms (masses are stored as mu_G m 2^ms)
    double rho_term;       // mu_G * mean density (mean subtraction), Mpc^-2
    int uniform_mass;      // every particle has the same mass
    double m_uniform;      // that mass, scaled as stored (mu_G m 2^ms)
};

// world position of the grid origin of replica j (replicated) or the field origin
__device__ __forceinline__ void frame_origin(const DevField &f, int j, double o[3])
{
    if (f.replicated) {
        o[0] = -0.5 * f.L;
        o[1] = -0.5 * f.L;
        o[2] = (double)j * f.L;
    } else {
        o[0] = f.O[0];
        o[1] = f.O[1];
        o[2] = f.O[2];
    }
}

// Replica transform of a box-frame grid position, q' = wrap(R (q - c) + c + s),
// c = Lq / 2, exactly and in 32 bits: R is a signed permutation and Lq even, so
// a component is q or Lq - q of one axis, plus the shift, minus Lq where that
// reaches it (both below 2 Lq <= 2^32).  Staging reads the map once per tile.
// Nine 64-bit products per particle, with R and s read for each, took 1.8 % of
// the pair sum of the 2^21-particle box (768 bundles: 2.692 -> 2.642 ms) and 1 %
// of the lens planes.
struct ReplicaMap {
    int axis[3];       // the axis a component comes from
    bool flip[3];      // Lq - q instead of q
    unsigned s[3], L;  // shift, box length
};

__device__ __forceinline__ ReplicaMap replica_map(const DevField &f, int j)
{
    ReplicaMap m;
    const int *R = f.rot + 9 * j, *S = f.shift + 3 * j;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const int a = R[3 * r], b = R[3 * r + 1], c = R[3 * r + 2];
        m.axis[r] = a ? 0 : (b ? 1 : 2);
        m.flip[r] = a + b + c < 0;
        m.s[r] = (unsigned)S[r];
    }
    m.L = (unsigned)f.Lq;
    return m;
}

__device__ __forceinline__ void replica_q(const ReplicaMap &m, int qx, int qy, int qz, int out[3])
{
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const unsigned q = (unsigned)(m.axis[r] == 0 ? qx : (m.axis[r] == 1 ? qy : qz));
        const unsigned v = (m.flip[r] ? m.L - q : q) + m.s[r];
        out[r] = (int)min(v, v - m.L);  // (v - L wraps to a larger number below L)
    }
}

// q - a in FP32, rounded once: through a 32-bit conversion where the difference
// fits one (a 64-bit one is several instructions)
__device__ __forceinline__ float grid_offset(int q, long long a)
{
    const long long d = (long long)q - a;
    const int lo = (int)d;
    return (long long)lo == d ? (float)lo : (float)d;
}

__device__ __forceinline__ int replica_of(const DevField &f, double x3)
{
    if (!f.replicated) return 0;
    double q = floor(x3 / f.L);
    if (q < 0.0) return 0;
    if (q > (double)(f.n_rep - 1)) return f.n_rep - 1;
    return (int)q;
}

// 1 / sqrt(x) of a positive FP64 number: the hardware's approximation y
// (rsqrt.approx.ftz.f64, relative error 2^-20 or better, its low word zero, so
// y^2 is exact), corrected by the binomial series (1 - e)^(-1/2) = 1 + e / 2 + 3
// e^2 / 8 + ... for e = 1 - x y^2; |e| <= 2^-19, so the term left out, 5 e^3 / 16,
// is below 2^-58.  Five FP64 operations, where x and y^2 are normal numbers.
// Subnormal numbers and those from 2^1022 on are scaled by a power of two first;
// zero gives infinity, infinity zero and NaN NaN, as rsqrt does.
__device__ __forceinline__ double rsqrt_estimate(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}

__device__ __forceinline__ double rsqrt_corrected(double x, double y)
{
    const double e = fma(-x, y * y, 1.0);
    return fma(y, e * fma(e, 0.375, 0.5), y);
}

__device__ __forceinline__ double rsqrt_series(double x)
{
    if ((unsigned)__double2hiint(x) - 0x00100000u >= 0x7fc00000u) {
        const bool small = __double2hiint(x) < 0x00100000;
        x *= small ? 0x1p108 : 0x1p-108;
        const double y = rsqrt_estimate(x);
        return y > 0.0 && y < 0x1p1000 ? rsqrt_corrected(x, y) * (small ? 0x1p54 : 0x1p-54) : y;
    }
    return rsqrt_corrected(x, rsqrt_estimate(x));
}

// one particle of mass m at offset d: adds m / r and m d / r^3, r^2 = |d|^2 + e2
__device__ __forceinline__ void pair_fp64(double dx, double dy, double dz, double m, double e2, double acc[4])
{
    const double inv = rsqrt_series(fma(dx, dx, fma(dy, dy, fma(dz, dz, e2))));
    const double mi = m * inv, mi3 = mi * (inv * inv);
    acc[0] += mi;
    acc[1] = fma(dx, mi3, acc[1]);
    acc[2] = fma(dy, mi3, acc[2]);
    acc[3] = fma(dz, mi3, acc[3]);
}

// ---------------------------------------------------------------------------
// ray state (SoA, FP64): index [component * n_rays + ray]
// ---------------------------------------------------------------------------
struct RayState {
    double *y;     // 8 x nr  current state
    double *ys;    // 8 x nr  stage state (positions read by the pair sum)
    double *ks;    // 8 x nr  RK4 accumulator
    double *fin;   // 8 x nr  state interpolated to x3 = chi_s
    int *done;     // nr
    int *steps;    // nr
    int *rep;      // 2 x n_bundles: replica of each bundle for even / odd stages
    int64_t n_rays, n_b;
    int nr;        // rays per bundle (1 + n_ring)
    int64_t stride;  // component stride of y, ys, ks, fin (n_rays for a single trace)
};

struct TraceParams {
    Cosmo cosmo;
    double chi_s;
    int n_ring;
    double theta_r, phase;
    int christoffel;
    int n_steps, max_extra;
};

// force launch shape
struct ForceShape {
    int R;        // rays per thread
    int NT;       // threads per block
    int splits;   // particle splits (blocks along y)
    int variant;  // 0 packed FP32x2, 1 scalar FP32, 2 FP64, 3-5 bundle-centric, 6 grid path
    int umass;    // packed kernel without per-particle masses (uniform-mass field)
    int cl = 1;   // thread-block cluster size along the splits: the cluster adds its
                  // CTAs' partials in distributed shared memory, one partial per cluster
    int lanes = 0;  // variant 5: one ray per lane (k_force_bundle1), one tile per split
};
// threads of a block of k_force_bundle1: one warp while it holds all the bundles,
// else four warps, which share the staging of a tile
inline int lanes_threads(const ForceShape &sh, int64_t n_rays) { return n_rays / sh.R <= 32 / sh.R ? 32 : 128; }
constexpr int kTraceRaysNT = 32;  // threads of a block of the one-launch traces (trace_rays)
// split partials a shape leaves for the integrator stage
inline int partial_splits(const ForceShape &sh) { return sh.splits / sh.cl; }

// device scratch of a trace (grow-only, owned by the context)
struct Scratch {
    void *partials = nullptr;      // splits * 4 * n_rays (float2 or double)
    size_t partials_bytes = 0;
    double *dlam = nullptr;        // n_steps
    size_t dlam_n = 0;
    double *misc = nullptr;        // [0] chi_s, [1..] spare
    unsigned long long *counters = nullptr; // [0] active-after slot 0, [1] slot 1, [2] active ray-stages
    double *state = nullptr;       // 32 * n_rays
    size_t state_rays = 0;
    int *ints = nullptr;           // 2 * n_rays + n_b
    size_t ints_n = 0;
    double *theta = nullptr;       // n_b * 2
    size_t theta_n = 0;
    double *bout = nullptr;        // n_b * 6
    size_t bout_n = 0;
    double *rout = nullptr;        // n_rays * 8
    size_t rout_n = 0;
    double *prism = nullptr;       // n_b * 13 bundle prism records
    size_t prism_n = 0;
    char *planes = nullptr;        // lens-plane table of the multi-plane system
    size_t planes_bytes = 0;
};

// streaming multiprocessors of the current device (queried once per device;
// 152 on GB300), for grid sizes counted in waves of resident blocks
int device_sm_count();

// kernels (launch wrappers; return cudaError_t of the launch)
// fill the a(t) table of c (n nodes, spacing h) at d_tab
cudaError_t launch_atab(const Cosmo &c, int n, double h, double *d_tab, cudaStream_t st);
cudaError_t launch_schedule(const Cosmo &c, double z_s, int kind, int n, double chi_l, double s,
                            double *d_dlam, double *d_misc, cudaStream_t st);
cudaError_t launch_init(const TraceParams &tp, const DevField &f, const double *d_theta, RayState rs,
                        unsigned long long *d_counters, cudaStream_t st);
cudaError_t launch_force(const DevField &f, const RayState &rs, const ForceShape &sh, bool fp64,
                         void *d_partials, const unsigned long long *d_active, int gate, cudaStream_t st);
cudaError_t launch_stage(const TraceParams &tp, const DevField &f, RayState rs, const ForceShape &sh,
                         bool fp64, void *d_partials, const double *d_dlam, const double *d_misc,
                         int step, int stage, unsigned long long *d_counters, cudaStream_t st,
                         const double *d_prism = nullptr);
// whether launch_stage adds the split partials up in a kernel of its own first
bool stage_merges(const ForceShape &sh, bool fp64, int64_t n_rays);
// per-bundle prism records (value, gradient, Hessian at the central ray) of a
// mean-subtracted replicated field, for launch_stage: kPrismRec doubles each
constexpr int kPrismRec = 13;
cudaError_t launch_prism(const TraceParams &tp, const DevField &f, RayState rs, int step, int stage,
                         const unsigned long long *d_counters, double *d_prism, cudaStream_t st);
// factor the integrator stage applies to the pair-sum partials of shape sh
inline double partial_mass_factor(const DevField &f, const ForceShape &sh)
{
    return sh.umass ? f.m_uniform : 1.0;
}
// RK4 stages [g0, g1) of an FP64 trace through an isolated field of few particles
constexpr int kFewParticles = 64, kFewAlways = 22;
bool few_in_one_launch(int64_t n_particles, int64_t n_rays);
cudaError_t launch_few_trace(const TraceParams &tp, const DevField &f, const RayState &rs, int g0, int g1,
                             const double *d_dlam, const double *d_misc, unsigned long long *d_counters,
                             cudaStream_t st);
cudaError_t launch_reduce(const TraceParams &tp, const double *d_theta, RayState rs, const double *d_misc,
                          double *d_bout, double *d_rout, cudaStream_t st);
// words of d_scal: five counters, a ticket, three doubles per block
constexpr int kHistBlocks = 1024;
constexpr int kHistScal = 6 + 3 * kHistBlocks;
cudaError_t launch_histogram(int64_t n, const double *d_mu, int mu_stride, const int *d_flags,
                             const double *d_flagsd, int bins, double mu_min, double mu_max,
                             unsigned long long *d_counts, unsigned long long *d_wfix,
                             unsigned long long *d_scal, double *d_out8, cudaStream_t st,
                             const double *d_g1 = nullptr, const double *d_g2 = nullptr);
cudaError_t launch_potential(const DevField &f, bool fp64, const double *d_pts, const int *d_rep,
                             int64_t n, const ForceShape &sh, void *d_partials, double *d_out,
                             cudaStream_t st);
cudaError_t launch_stage_field(const DevField &f, const ForceShape &sh, bool fp64, const void *d_partials,
                               const double *d_pts, const int *d_rep, int64_t n, double *d_out,
                               cudaStream_t st);

// gridded field (Sec. 3.3 grid path, App. B): node values and x3 spline
// second derivatives, 4 n^3 doubles each, [f][i1][i2][i3] with i3 fastest
// doubles per grid node in the node table: phi, dphi/dx1, dphi/dx2, dphi/dx3,
// then their natural-spline second derivatives along x3 (App. B)
constexpr int kGridRec = 8;
struct GridDev {
    int n = 0, n_int = 0;
    double lo[3] = {0.0, 0.0, 0.0};
    double h = 0.0, inv_h = 0.0;  // node spacing and its inverse
    // one of the two: [i1][i2][i3][kGridRec], i3 fastest, in FP64 (FP64
    // contexts) or rounded to FP32 (mixed contexts)
    double *tab = nullptr;
    float *tab32 = nullptr;
    // cube-tiled replicated box (cubes > 0): n_rep * cubes node tables stored
    // one after the other (stride kGridRec n^3), replica-major; cube c of
    // replica j has lo = (-W/2, -W/2, j L + c W) and spacing W / (n - 1)
    int cubes = 0, n_rep = 1;
    double L = 0.0, W = 0.0;
    // points up to margin node spacings outside the node range take the end
    // intervals' cubics (box cubes: 1, for the rays of a bundle near a cube
    // face); farther out the field is zero
    double margin = 0.0;
};
// build g.tab (fp64) or g.tab32 (allocated here) from host particles; returns
// an rt3d status and sets err on failure
int grid_build(GridDev &g, int64_t np, const double *pos, const double *mass, double soft, int mean_subtract,
               bool fp64, cudaStream_t st, std::string &err);
// build the n_rep * cubes node tables of a cube-tiled replicated box (g.n,
// n_rep, cubes, L, W, h set by the caller; g.tab allocated here) from the
// box's host particles, each replica placed by rot[9 j] and shift[3 j]
int grid_build_box(GridDev &g, int64_t np, const double *pos, const double *mass, double soft,
                   const int32_t *rot, const double *shift, int mean_subtract, bool fp64, cudaStream_t st,
                   std::string &err);
void grid_free(GridDev &g);
// App. B evaluation at n points (SoA px, py, pz) from the grid's table.  mode
// 0 (mixed path, FP32 table): -F as (hi, 0) pairs in the pair-sum partial
// layout (one split); 1 (FP64 table): -F as FP64 partials; 2: F at
// out[4 i + f] as FP64 numbers
cudaError_t launch_grid_eval(const GridDev &g, const double *px, const double *py, const double *pz, int64_t n,
                             int mode, void *out, const unsigned long long *gate, cudaStream_t st,
                             int group = 1);

// RK4 stages [g0, g1) of a trace on a grid in one launch
cudaError_t launch_grid_trace(const TraceParams &tp, const GridDev &g, const RayState &rs, bool fp64, int g0, int g1,
                              const double *dlam, const double *misc, unsigned long long *cnt, cudaStream_t st);

// Born approximation (born.cu): scratch size and the run over node chunks of
// K nodes with the Hessian pair sum split `splits` ways; d_out = n_b x 3
size_t born_scratch_bytes(int64_t n_b, int n_steps, int K, int splits);
cudaError_t born_run(const Cosmo &c, const DevField &f, int64_t n_particles, double z_s, int64_t n_b,
                     const double *d_theta, int kind, int n_steps, double chi_l, double s, int K, int splits,
                     void *scratch, double *d_out, cudaStream_t st);

int force_max_splits(const ForceShape &sh, int64_t n_particles);
size_t partials_bytes(const ForceShape &sh, int64_t n_rays, bool fp64);

// multiple lens-plane comparison system (multiplane.cu)
size_t mp_plane_bytes();
size_t mp_partials_bytes(int n_ring, int64_t n_b, int splits, bool fp64);
cudaError_t mp_run(const Cosmo &c, const DevField &f, double z_s, int slices, double x3_lo, double x3_hi,
                   const TraceParams &tp, const double *d_theta, RayState rs, void *d_planes, int n_pl, void *partials,
                   int splits, bool fp64, bool umass, double *misc, unsigned long long *count, double *d_bout,
                   double *d_rout, cudaStream_t st);

}  // namespace rt3d
