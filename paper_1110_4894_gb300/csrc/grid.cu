// grid.cu -- the paper's grid force path (Sec. 3.3 and App. B).
//
// Build, once per mass distribution:
//   1. cloud-in-cell assignment of the particle masses to n^3 nodes, summed in
//      64-bit fixed point with integer atomics (order-independent, so the
//      node masses are bit-reproducible);
//   2. optional subtraction of the mean node mass (Sec. 3.3 removes the mean
//      density);
//   3. phi and grad phi on the nodes: the zero-padded (2n)^3 FFT convolution
//      of the node masses with the Plummer kernels (Eqs. psi, derivs with
//      phi = a psi), by cuFFT (double precision, real-to-complex);
//   4. the natural-spline second derivatives of every node line along x3
//      (App. B: computed once).
// Per RK4 stage, App. B's interpolation at every ray: along x3 from the
// global line splines, then natural splines through the 2 n_int nodes around
// the ray along x1 and along x2.  A natural spline through unit-spaced values
// is linear in them, so the x1 and x2 splines are applied as weight vectors
// (computed once per point) to the four fields at once.  One thread per point;
// the node table keeps, per node, the four field values and their x3-spline
// second derivatives side by side (64 bytes), so the two nodes a point reads on
// each x3 line are one contiguous 128-byte span.
#include <cufft.h>

#include <algorithm>
#include <new>
#include <thread>
#include <vector>

#include "grid_device.cuh"
#include "rt3d_internal.cuh"
#include "trace_device.cuh"

namespace rt3d {

constexpr int kMaxGridN = 1024;

// ---------------------------------------------------------------------------
// build kernels
// ---------------------------------------------------------------------------
__global__ void k_cic(int64_t np, const double *__restrict__ pos, const double *__restrict__ mass, double lo0,
                      double lo1, double lo2, double inv_h, int n, double qscale,
                      unsigned long long *__restrict__ node_q)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    const double u[3] = {(pos[3 * p] - lo0) * inv_h, (pos[3 * p + 1] - lo1) * inv_h, (pos[3 * p + 2] - lo2) * inv_h};
    int64_t i0[3];
    double f[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double fl = floor(u[d]);
        i0[d] = (int64_t)fl;
        f[d] = u[d] - fl;
    }
    const double m = mass[p] * qscale;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int64_t a = i0[0] + (c & 1), b = i0[1] + ((c >> 1) & 1), z = i0[2] + ((c >> 2) & 1);
        if (a < 0 || a >= n || b < 0 || b >= n || z < 0 || z >= n) continue;
        const double w = ((c & 1) ? f[0] : 1.0 - f[0]) * (((c >> 1) & 1) ? f[1] : 1.0 - f[1]) *
                         (((c >> 2) & 1) ? f[2] : 1.0 - f[2]);
        const unsigned long long q = (unsigned long long)__double2ll_rn(m * w);
        atomicAdd(&node_q[(a * n + b) * n + z], q);
    }
}

__global__ void k_sum_q(int64_t m, const unsigned long long *__restrict__ q, unsigned long long *__restrict__ total)
{
    __shared__ unsigned long long s[256];
    unsigned long long acc = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        acc += q[i];
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if ((int)threadIdx.x < k) s[threadIdx.x] += s[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(total, s[0]);
}

// padded (P = 2n)^3 real array: node masses (minus the mean) in the first n^3 corner
__global__ void k_fill_mass(int n, const unsigned long long *__restrict__ q, const unsigned long long *__restrict__ total,
                            double qinv, int mean_subtract, double *__restrict__ buf)
{
    const int P = 2 * n;
    const int64_t m = (int64_t)P * P * P;
    const double mean = mean_subtract ? (double)*total * qinv / ((double)n * n * n) : 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int k3 = (int)(i % P), k2 = (int)((i / P) % P), k1 = (int)(i / ((int64_t)P * P));
        double v = 0.0;
        if (k1 < n && k2 < n && k3 < n) v = (double)q[((int64_t)k1 * n + k2) * n + k3] * qinv - mean;
        buf[i] = v;
    }
}

// the convolution kernels for node displacements 0..n-1 per axis (phi, then
// grad phi where nf = 4 or its x1 component where nf = 2), kernel-major: each
// square root and division (some forty FP64 operations) once, for all the
// octants and kernels that share it
__global__ void k_kernel_octant(int n, int nf, double h, double eps2, double *__restrict__ oct)
{
    const int64_t m = (int64_t)n * n * n;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int k[3] = {(int)(i / ((int64_t)n * n)), (int)((i / n) % n), (int)(i % n)};
        double d[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) d[c] = (double)k[c] * h;
        const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps2;
        const double inv = r2 > 0.0 ? 1.0 / sqrt(r2) : 0.0;
        oct[i] = -kMuG * inv;
        for (int f = 1; f < nf; ++f) oct[f * m + i] = kMuG * d[f - 1] * inv * inv * inv;
    }
}

// kernel f on the padded (P = 2n)^3 grid from its octant, indexed by node
// displacement (k < n: +k, k > n: k - 2n, k = n: unused, zero); a gradient
// kernel is odd along its axis
__global__ void k_unfold(int n, int f, const double *__restrict__ oct, double *__restrict__ buf)
{
    const int P = 2 * n;
    const int64_t m = (int64_t)P * P * P;
    oct += f * ((int64_t)n * n * n);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int k[3] = {(int)(i / ((int64_t)P * P)), (int)((i / P) % P), (int)(i % P)};
        double v = 0.0;
        if (k[0] != n && k[1] != n && k[2] != n) {
            const int q[3] = {k[0] < n ? k[0] : P - k[0], k[1] < n ? k[1] : P - k[1], k[2] < n ? k[2] : P - k[2]};
            v = oct[((int64_t)q[0] * n + q[1]) * n + q[2]];
            if (f > 0 && k[f - 1] > n) v = -v;
        }
        buf[i] = v;
    }
}

__device__ __forceinline__ cufftDoubleComplex cmul_scaled(cufftDoubleComplex x, cufftDoubleComplex y, double scale)
{
    return make_cuDoubleComplex((x.x * y.x - x.y * y.y) * scale, (x.x * y.y + x.y * y.x) * scale);
}

// out = a b scale (out may be b)
__global__ void k_cmul(int64_t m, const cufftDoubleComplex *__restrict__ a, const cufftDoubleComplex *b,
                       cufftDoubleComplex *out, double scale)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = cmul_scaled(a[i], b[i], scale);
}

// The grid is a cube, so the x2 and x3 gradient kernels are the x1 kernel with
// two axes exchanged, and so are their spectra (half spectra [k1][k2][k3 <= n]):
// out = a b' scale with b'(k1, k2, k3) = b(k2, k1, k3), or b(k3, k2, k1), where
// the x1 kernel is even along x3, b(., ., P - k) = b(., ., k).  That saves two
// of the five forward transforms.
__global__ void k_cmul_x2(int n, const cufftDoubleComplex *__restrict__ a, const cufftDoubleComplex *__restrict__ b,
                          cufftDoubleComplex *__restrict__ out, double scale)
{
    const int P = 2 * n, H = n + 1;
    const int64_t m = (int64_t)P * P * H;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k3 = i % H, k2 = (i / H) % P, k1 = i / ((int64_t)P * H);
        out[i] = cmul_scaled(a[i], b[(k2 * P + k1) * H + k3], scale);
    }
}

constexpr int kCmulTile = 16;  // k1 x k3 tile, transposed through shared memory
__global__ void __launch_bounds__(kCmulTile *kCmulTile) k_cmul_x3(int n, const cufftDoubleComplex *__restrict__ a,
                                                                const cufftDoubleComplex *__restrict__ b,
                                                                cufftDoubleComplex *__restrict__ out, double scale)
{
    __shared__ cufftDoubleComplex s[kCmulTile][kCmulTile + 1];
    const int P = 2 * n, H = n + 1;
    const int c0 = blockIdx.x * kCmulTile, a0 = blockIdx.y * kCmulTile, k2 = blockIdx.z;
    const int x = threadIdx.x, y = threadIdx.y;
    if (c0 + y < H && a0 + x < P) {
        const int k = a0 + x <= n ? a0 + x : P - (a0 + x);
        s[y][x] = b[((int64_t)(c0 + y) * P + k2) * H + k];
    }
    __syncthreads();
    if (c0 + x < H && a0 + y < P) {
        const int64_t i = ((int64_t)(a0 + y) * P + k2) * H + c0 + x;
        out[i] = cmul_scaled(a[i], s[x][y], scale);
    }
}

__global__ void k_extract(int n, const double *__restrict__ buf, double *__restrict__ out)
{
    const int P = 2 * n;
    const int64_t m = (int64_t)n * n * n;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k3 = i % n, k2 = (i / n) % n, k1 = i / ((int64_t)n * n);
        out[i] = buf[(k1 * P + k2) * P + k3];
    }
}

// natural cubic spline along each x3 line (unit spacing):
// y2[i-1] + 4 y2[i] + y2[i+1] = 6 (y[i+1] - 2 y[i] + y[i-1]), y2 = 0 at the ends.
// The elimination factors depend on n only and are shared by all lines.
__global__ void k_spline_lines(int n, int64_t lines, const double *__restrict__ val, double *__restrict__ y2)
{
    __shared__ double s_inv[kMaxGridN];  // 1 / the elimination's pivots
    if (threadIdx.x == 0) {
        double cp = 0.0;
        for (int i = 1; i <= n - 2; ++i) s_inv[i] = cp = 1.0 / (4.0 - cp);
    }
    __syncthreads();
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= lines) return;
    const double *y = val + l * n;
    double *z = y2 + l * n;
    z[0] = 0.0;
    z[n - 1] = 0.0;
    if (n < 3) return;
    double dp = 0.0;
    for (int i = 1; i <= n - 2; ++i) {
        dp = (6.0 * (y[i + 1] - 2.0 * y[i] + y[i - 1]) - dp) * s_inv[i];
        z[i] = dp;
    }
    for (int i = n - 3; i >= 1; --i) z[i] = z[i] - z[i + 1] * s_inv[i];
}

// node table: per node the four values, then the four x3-spline second
// derivatives (kGridRec doubles); tab32 holds the same numbers rounded to FP32
// (either may be null)
__global__ void k_interleave(int64_t n3, const double *__restrict__ val, const double *__restrict__ y2,
                             double *__restrict__ tab, float *__restrict__ tab32)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n3; i += (int64_t)gridDim.x * blockDim.x) {
        const double r[kGridRec] = {val[i], val[n3 + i], val[2 * n3 + i], val[3 * n3 + i],
                                    y2[i],  y2[n3 + i],  y2[2 * n3 + i],  y2[3 * n3 + i]};
        if (tab) {
            double2 *t = reinterpret_cast<double2 *>(tab + kGridRec * i);
            t[0] = make_double2(r[0], r[1]);
            t[1] = make_double2(r[2], r[3]);
            t[2] = make_double2(r[4], r[5]);
            t[3] = make_double2(r[6], r[7]);
        }
        if (tab32) {
            float4 *t32 = reinterpret_cast<float4 *>(tab32 + kGridRec * i);
            t32[0] = make_float4((float)r[0], (float)r[1], (float)r[2], (float)r[3]);
            t32[1] = make_float4((float)r[4], (float)r[5], (float)r[6], (float)r[7]);
        }
    }
}

// ---------------------------------------------------------------------------
// App. B evaluation
// ---------------------------------------------------------------------------
// Weights c of the natural cubic spline through W unit-spaced values y,
// evaluated at u in [0, W-1]: S(u) = sum_j c[j] y[j].  The second derivatives
// z of the spline through the unit vector e_j solve the same tridiagonal
// system as any data (z[i-1] + 4 z[i] + z[i+1] = 6 (e[i+1] - 2 e[i] + e[i-1]),
// z = 0 at the ends); they are constants of W.
template <int W>
__device__ __forceinline__ void spline_weights(double u, double (&c)[W])
{
    int k = (int)floor(u);
    k = k > W - 2 ? W - 2 : k;
    k = k < 0 ? 0 : k;
    const double A = (double)(k + 1) - u, B = u - (double)k;
    const double cA = (A * A * A - A) / 6.0, cB = (B * B * B - B) / 6.0;
#pragma unroll
    for (int j = 0; j < W; ++j) {
        double z[W];
        z[0] = 0.0;
        z[W - 1] = 0.0;
        if (W >= 3) {
            double den[W], dp = 0.0, cp = 0.0;
#pragma unroll
            for (int i = 1; i <= W - 2; ++i) {
                const double e = (i + 1 == j ? 1.0 : 0.0) - 2.0 * (i == j ? 1.0 : 0.0) + (i - 1 == j ? 1.0 : 0.0);
                den[i] = 4.0 - cp;
                cp = 1.0 / den[i];
                dp = (6.0 * e - dp) / den[i];
                z[i] = dp;
            }
#pragma unroll
            for (int i = W - 3; i >= 1; --i) z[i] = z[i] - z[i + 1] / den[i];
        }
        double zk = z[0], zk1 = z[1];
#pragma unroll
        for (int i = 1; i < W - 1; ++i)
            if (k == i) {
                zk = z[i];
                zk1 = z[i + 1];
            }
        c[j] = (j == k ? A : 0.0) + (j == k + 1 ? B : 0.0) + (cA * zk + cB * zk1);
    }
}

// phi and grad phi at position r from the FP64 node table (the cube of a box:
// the one holding x3, the central ray's)
template <int NI>
__device__ __forceinline__ void grid_eval64_at(const GridDev &g, const double r[3], double x3, double F[4])
{
    constexpr int W = 2 * NI;
    const int n = g.n;
    double lo[3] = {g.lo[0], g.lo[1], g.lo[2]};
    const double *tab = g.tab + grid_cube(g, x3, lo) * (kGridRec * (int64_t)n * n * n);
    double u[3];
    int s[3];
    bool inside = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        u[d] = grid_coord(r[d] - lo[d], g.h, g.inv_h);
        inside = inside && (u[d] >= -g.margin && u[d] <= (double)(n - 1) + g.margin);
        int sd = inside ? (int)floor(u[d]) - NI + 1 : 0;
        sd = sd > n - W ? n - W : sd;
        s[d] = sd < 0 ? 0 : sd;
    }
    F[0] = F[1] = F[2] = F[3] = 0.0;
    if (inside) {
        int k3 = (int)floor(u[2]);
        k3 = k3 > n - 2 ? n - 2 : k3;
        k3 = k3 < 0 ? 0 : k3;
        const double A = (double)(k3 + 1) - u[2], B = u[2] - (double)k3;
        const double cA = (A * A * A - A) / 6.0, cB = (B * B * B - B) / 6.0;
        double c1[W], c2[W];
        spline_weights<W>(u[0] - (double)s[0], c1);
        spline_weights<W>(u[1] - (double)s[1], c2);
#pragma unroll
        for (int b = 0; b < W; ++b) {
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
            for (int a = 0; a < W; ++a) {
                // along x3 on node line (s1 + a, s2 + b): the global spline
                // from nodes k3 and k3 + 1 (values, then second derivatives)
                const int64_t node = ((int64_t)(s[0] + a) * n + (s[1] + b)) * n + k3;
                const double2 *p = reinterpret_cast<const double2 *>(tab + kGridRec * node);
                const double2 v01 = __ldg(p), v23 = __ldg(p + 1), y01 = __ldg(p + 2), y23 = __ldg(p + 3);
                const double2 w01 = __ldg(p + 4), w23 = __ldg(p + 5), z01 = __ldg(p + 6), z23 = __ldg(p + 7);
                const double t0 = A * v01.x + B * w01.x + (cA * y01.x + cB * z01.x);
                const double t1 = A * v01.y + B * w01.y + (cA * y01.y + cB * z01.y);
                const double t2 = A * v23.x + B * w23.x + (cA * y23.x + cB * z23.x);
                const double t3 = A * v23.y + B * w23.y + (cA * y23.y + cB * z23.y);
                // along x1
                acc[0] += c1[a] * t0;
                acc[1] += c1[a] * t1;
                acc[2] += c1[a] * t2;
                acc[3] += c1[a] * t3;
            }
            // along x2
#pragma unroll
            for (int f = 0; f < 4; ++f) F[f] += c2[b] * acc[f];
        }
    }
}

// group: points per bundle; a cube-tiled box takes the cube holding the x3
// of the group's first point (the bundle's central ray), as the direct sum
// takes its replica
template <int NI>
__global__ void __launch_bounds__(128) k_grid_eval(GridDev g, const double *__restrict__ px,
                                                   const double *__restrict__ py, const double *__restrict__ pz,
                                                   int64_t n_pts, int mode, void *__restrict__ out,
                                                   const unsigned long long *__restrict__ gate, int group)
{
    if (gate && *gate == 0ull) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_pts) return;
    const double r[3] = {px[i], py[i], pz[i]};
    double F[4];
    grid_eval64_at<NI>(g, r, g.cubes > 0 ? pz[(i / group) * group] : 0.0, F);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        if (mode == 2) {
            ((double *)out)[4 * i + f] = F[f];
        } else if (mode == 1) {
            ((double *)out)[(int64_t)f * n_pts + i] = -F[f];
        } else {
            const float hi = (float)(-F[f]);
            const float lo2 = (float)(-F[f] - (double)hi);
            ((float2 *)out)[(int64_t)f * n_pts + i] = make_float2(hi, lo2);
        }
    }
}

// The mixed path's evaluation (grid_device.cuh): output modes 0 (hi = -F,
// lo = 0) and 2.
template <int NI>
__global__ void __launch_bounds__(128) k_grid_eval32(GridDev g, const double *__restrict__ px,
                                                     const double *__restrict__ py, const double *__restrict__ pz,
                                                     int64_t n_pts, int mode, void *__restrict__ out,
                                                     const unsigned long long *__restrict__ gate, int group)
{
    if (gate && *gate == 0ull) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_pts) return;
    float F[4];
    grid_eval32_point<NI>(g, px, py, pz, i, group, F);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        if (mode == 2)
            ((double *)out)[4 * i + f] = (double)F[f];
        else
            ((float2 *)out)[(int64_t)f * n_pts + i] = make_float2(-F[f], 0.0f);
    }
}

cudaError_t launch_grid_eval(const GridDev &g, const double *px, const double *py, const double *pz, int64_t n,
                             int mode, void *out, const unsigned long long *gate, cudaStream_t st, int group)
{
    if (n <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)((n + 127) / 128);
    // the FP32 table serves the mixed path (mode 0) and, where it is the only
    // table, point evaluation (mode 2)
    if (g.tab32 && (mode == 0 || !g.tab)) {
        if (mode == 1) return cudaErrorInvalidValue;
        switch (g.n_int) {
        case 1: k_grid_eval32<1><<<grid, 128, 0, st>>>(g, px, py, pz, n, mode, out, gate, group); break;
        case 2: k_grid_eval32<2><<<grid, 128, 0, st>>>(g, px, py, pz, n, mode, out, gate, group); break;
        case 3: k_grid_eval32<3><<<grid, 128, 0, st>>>(g, px, py, pz, n, mode, out, gate, group); break;
        case 4: k_grid_eval32<4><<<grid, 128, 0, st>>>(g, px, py, pz, n, mode, out, gate, group); break;
        default: return cudaErrorInvalidValue;
        }
        return cudaGetLastError();
    }
    if (!g.tab) return cudaErrorInvalidValue;
    switch (g.n_int) {
    case 1: k_grid_eval<1><<<grid, 128, 0, st>>>(g, px, py, pz, n, mode, out, gate, group); break;
    case 2: k_grid_eval<2><<<grid, 128, 0, st>>>(g, px, py, pz, n, mode, out, gate, group); break;
    case 3: k_grid_eval<3><<<grid, 128, 0, st>>>(g, px, py, pz, n, mode, out, gate, group); break;
    case 4: k_grid_eval<4><<<grid, 128, 0, st>>>(g, px, py, pz, n, mode, out, gate, group); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// traces on a grid
// ---------------------------------------------------------------------------
// trace_rays with the grid's interpolation.  Stage by stage, a trace was an
// evaluation and an update kernel per stage with the state, the field and their
// launches between them: 11.5 + 5.9 us for 20,480 rays and a 128^3 grid; grid
// and trace of 500 steps together 75.6 -> 36.4 ms (the grid was 20 ms of both).
// What is left is each stage's FP64 behind the latency of its node gather.
template <int NI, bool FP64>
__global__ void __launch_bounds__(kTraceRaysNT) k_grid_trace(TraceParams tp, GridDev g, RayState rs, int g0, int g1,
                                                            const double *__restrict__ dlam,
                                                            const double *__restrict__ misc, unsigned long long *cnt)
{
    trace_rays(tp, rs, g0, g1, dlam, misc, cnt, [&](const double r[3], double x3, double F[4]) {
        if constexpr (FP64) {
            grid_eval64_at<NI>(g, r, x3, F);
        } else {
            float f[4];
            grid_eval32_at<NI>(g, r, x3, f);
#pragma unroll
            for (int q = 0; q < 4; ++q) F[q] = (double)f[q];
        }
    });
}

template <bool FP64>
static cudaError_t go_grid_trace(const TraceParams &tp, const GridDev &g, const RayState &rs, int g0, int g1,
                                 const double *dlam, const double *misc, unsigned long long *cnt, cudaStream_t st)
{
    const int per_warp = 32 / rs.nr;
    const unsigned grid = (unsigned)((rs.n_b + per_warp - 1) / per_warp);
    switch (g.n_int) {
    case 1: k_grid_trace<1, FP64><<<grid, kTraceRaysNT, 0, st>>>(tp, g, rs, g0, g1, dlam, misc, cnt); break;
    case 2: k_grid_trace<2, FP64><<<grid, kTraceRaysNT, 0, st>>>(tp, g, rs, g0, g1, dlam, misc, cnt); break;
    case 3: k_grid_trace<3, FP64><<<grid, kTraceRaysNT, 0, st>>>(tp, g, rs, g0, g1, dlam, misc, cnt); break;
    case 4: k_grid_trace<4, FP64><<<grid, kTraceRaysNT, 0, st>>>(tp, g, rs, g0, g1, dlam, misc, cnt); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_grid_trace(const TraceParams &tp, const GridDev &g, const RayState &rs, bool fp64, int g0, int g1,
                              const double *dlam, const double *misc, unsigned long long *cnt, cudaStream_t st)
{
    if (fp64 ? !g.tab : !g.tab32) return cudaErrorInvalidValue;
    return fp64 ? go_grid_trace<true>(tp, g, rs, g0, g1, dlam, misc, cnt, st)
                : go_grid_trace<false>(tp, g, rs, g0, g1, dlam, misc, cnt, st);
}

// ---------------------------------------------------------------------------
// build orchestration
// ---------------------------------------------------------------------------
void grid_free(GridDev &g)
{
    cudaFree(g.tab);
    cudaFree(g.tab32);
    g.tab = nullptr;
    g.tab32 = nullptr;
}

static unsigned blocks_for(int64_t m)
{
    const int64_t b = (m + 255) / 256, cap = (int64_t)device_sm_count() * 64;
    return (unsigned)(b < cap ? (b > 0 ? b : 1) : cap);
}

namespace {
// Device state for building grids of one shape (n nodes per side, spacing h,
// softening eps): FFT buffers and plans, node-mass and value temporaries, and
// (keep: where they fit) the spectra of the phi and x1 kernels, which give all
// four, depend on the shape only and so serve every cube of a replicated box.
// Freed on every exit.
//
// A 3D transform is one over the (x2, x3) planes and one along x1: the node
// masses fill, and the node values need, only the first half of the planes, so
// the plane transforms of the other half are left out (the FP64 of the
// transforms bounds the build; 128^3 nodes: 15.8 -> 9.1 ms of them, and 3.4 ->
// 0.3 ms for the kernels they transform).
struct Builder {
    int n = 0;
    double h = 0.0, eps2 = 0.0;
    bool keep = false, have_k = false;
    double *pos = nullptr, *mass = nullptr, *buf = nullptr, *val = nullptr, *y2 = nullptr;
    unsigned long long *q = nullptr, *total = nullptr;
    cufftDoubleComplex *fm = nullptr, *fk = nullptr, *kspec = nullptr;
    cufftHandle r2c = 0, c2r = 0, c2c = 0;  // half the planes, both ways; along x1
    bool have_r2c = false, have_c2r = false, have_c2c = false;
    std::string *err = nullptr;
    ~Builder()
    {
        cudaFree(pos);
        cudaFree(mass);
        cudaFree(buf);
        cudaFree(val);
        cudaFree(y2);
        cudaFree(q);
        cudaFree(total);
        cudaFree(fm);
        cudaFree(fk);
        cudaFree(kspec);
        if (have_r2c) cufftDestroy(r2c);
        if (have_c2r) cufftDestroy(c2r);
        if (have_c2c) cufftDestroy(c2c);
    }
    int cuda_fail(cudaError_t e, const char *what)
    {
        *err = std::string(what) + ": " + cudaGetErrorString(e);
        return e == cudaErrorMemoryAllocation ? RT3D_ENOMEM : RT3D_ECUDA;
    }
    int fft_fail(cufftResult r, const char *what)
    {
        *err = std::string(what) + ": cuFFT error " + std::to_string((int)r);
        return r == CUFFT_ALLOC_FAILED ? RT3D_ENOMEM : RT3D_ECUDA;
    }
    int64_t P3() const { return 8 * (int64_t)n * n * n; }
    int64_t Pc() const { return 4 * (int64_t)n * n * (n + 1); }
    int64_t n3() const { return (int64_t)n * n * n; }
};
}  // namespace

#define GCK(x, what)                                        \
    do {                                                    \
        cudaError_t e_ = (x);                               \
        if (e_ != cudaSuccess) return B.cuda_fail(e_, what); \
    } while (0)
#define FCK(x, what)                                        \
    do {                                                    \
        cufftResult r_ = (x);                               \
        if (r_ != CUFFT_SUCCESS) return B.fft_fail(r_, what); \
    } while (0)

// np_most: the most particles of any grid to be built
static int builder_init(Builder &B, int n, double h, double soft, int64_t np_most, cudaStream_t st, std::string &err)
{
    B.n = n;
    B.h = h;
    B.eps2 = soft * soft;
    B.err = &err;
    const int P = 2 * n;
    GCK(cudaMalloc(&B.q, sizeof(unsigned long long) * (size_t)B.n3()), "grid node buffer");
    GCK(cudaMalloc(&B.total, sizeof(unsigned long long)), "grid total");
    GCK(cudaMalloc(&B.buf, sizeof(double) * (size_t)B.P3()), "grid FFT buffer");
    GCK(cudaMalloc(&B.fm, sizeof(cufftDoubleComplex) * (size_t)B.Pc()), "grid FFT buffer");
    GCK(cudaMalloc(&B.fk, sizeof(cufftDoubleComplex) * (size_t)B.Pc()), "grid FFT buffer");
    GCK(cudaMalloc(&B.val, sizeof(double) * 4 * (size_t)B.n3()), "grid values");
    GCK(cudaMalloc(&B.y2, sizeof(double) * 4 * (size_t)B.n3()), "grid spline table");
    if (np_most > 0) {
        GCK(cudaMalloc(&B.pos, sizeof(double) * 3 * (size_t)np_most), "particle upload");
        GCK(cudaMalloc(&B.mass, sizeof(double) * (size_t)np_most), "particle upload");
    }
    // (64-bit sizes: from 813 nodes on the transforms cover more than 2^31 elements)
    long long plane[2] = {P, P}, half[2] = {P, n + 1}, line[1] = {P};
    const long long pd = (long long)P * P, pc = (long long)P * (n + 1);
    size_t work = 0;
    FCK(cufftCreate(&B.r2c), "cufftCreate");
    B.have_r2c = true;
    FCK(cufftMakePlanMany64(B.r2c, 2, plane, plane, 1, pd, half, 1, pc, CUFFT_D2Z, n, &work), "cuFFT plan D2Z");
    FCK(cufftCreate(&B.c2r), "cufftCreate");
    B.have_c2r = true;
    FCK(cufftMakePlanMany64(B.c2r, 2, plane, half, 1, pc, plane, 1, pd, CUFFT_Z2D, n, &work), "cuFFT plan Z2D");
    FCK(cufftCreate(&B.c2c), "cufftCreate");
    B.have_c2c = true;
    FCK(cufftMakePlanMany64(B.c2c, 1, line, line, pc, 1, line, pc, 1, CUFFT_Z2Z, pc, &work), "cuFFT plan Z2Z");
    FCK(cufftSetStream(B.r2c, st), "cufftSetStream");
    FCK(cufftSetStream(B.c2r, st), "cufftSetStream");
    FCK(cufftSetStream(B.c2c, st), "cufftSetStream");
    return RT3D_OK;
}

// The two kernel spectra stay resident where they are small and fit.  Called
// after everything that a build cannot do without has its memory.
static void builder_keep_spectra(Builder &B)
{
    const size_t bytes = 2 * (size_t)B.Pc() * sizeof(cufftDoubleComplex);
    B.keep = bytes <= ((size_t)8 << 30);
    if (B.keep && cudaMalloc(&B.kspec, bytes) != cudaSuccess) {
        cudaGetLastError();
        B.kspec = nullptr;
        B.keep = false;
    }
}

// one grid: the particles' CIC node masses on the nodes lo + h i, optionally
// minus their mean, convolved with the four Plummer kernels; the node table
// (kGridRec n^3 doubles) goes to dest, its FP32 copy to dest32
static int builder_run(Builder &B, int64_t np, const double *pos, const double *mass, const double lo[3],
                       int mean_subtract, double *dest, float *dest32, cudaStream_t st)
{
    const int n = B.n;
    const int64_t n3 = B.n3(), P3 = B.P3(), Pc = B.Pc();
    // fixed-point scale: the node sums stay below 2^62 for any assignment
    double msum = 0.0;
    for (int64_t i = 0; i < np; ++i) msum += mass[i];
    const int e = msum > 0.0 ? 61 - (int)ceil(log2(msum)) : 0;
    const double qscale = ldexp(1.0, e), qinv = ldexp(1.0, -e);
    GCK(cudaMemsetAsync(B.q, 0, sizeof(unsigned long long) * (size_t)n3, st), "memset");
    GCK(cudaMemsetAsync(B.total, 0, sizeof(unsigned long long), st), "memset");
    if (np > 0) {
        GCK(cudaMemcpyAsync(B.pos, pos, sizeof(double) * 3 * (size_t)np, cudaMemcpyHostToDevice, st), "upload");
        GCK(cudaMemcpyAsync(B.mass, mass, sizeof(double) * (size_t)np, cudaMemcpyHostToDevice, st), "upload");
        k_cic<<<(unsigned)((np + 255) / 256), 256, 0, st>>>(np, B.pos, B.mass, lo[0], lo[1], lo[2], 1.0 / B.h, n,
                                                             qscale, B.q);
        GCK(cudaGetLastError(), "k_cic");
    }
    k_sum_q<<<blocks_for(n3), 256, 0, st>>>(n3, B.q, B.total);
    GCK(cudaGetLastError(), "k_sum_q");
    k_fill_mass<<<blocks_for(P3), 256, 0, st>>>(n, B.q, B.total, qinv, mean_subtract, B.buf);
    GCK(cudaGetLastError(), "k_fill_mass");
    const int P = 2 * n;
    const int64_t half_d = P3 / 2, half_c = Pc / 2;
    FCK(cufftExecD2Z(B.r2c, B.buf, B.fm), "cufftExecD2Z");  // the masses' planes; the others are zero
    GCK(cudaMemsetAsync(B.fm + half_c, 0, sizeof(cufftDoubleComplex) * (size_t)half_c, st), "memset");
    FCK(cufftExecZ2Z(B.c2c, B.fm, B.fm, CUFFT_FORWARD), "cufftExecZ2Z");
    const auto kernel_spectrum = [&](int f, cufftDoubleComplex *ks) -> int {
        k_unfold<<<blocks_for(P3), 256, 0, st>>>(n, f, B.y2, B.buf);
        GCK(cudaGetLastError(), "k_unfold");
        FCK(cufftExecD2Z(B.r2c, B.buf, ks), "cufftExecD2Z");
        FCK(cufftExecD2Z(B.r2c, B.buf + half_d, ks + half_c), "cufftExecD2Z");
        FCK(cufftExecZ2Z(B.c2c, ks, ks, CUFFT_FORWARD), "cufftExecZ2Z");
        return RT3D_OK;
    };
    if (!B.have_k) {  // (the octants wait where the splines will be)
        k_kernel_octant<<<blocks_for(n3), 256, 0, st>>>(n, B.keep ? 2 : 4, B.h, B.eps2, B.y2);
        GCK(cudaGetLastError(), "k_kernel_octant");
        for (int f = 0; f < 2 && B.keep; ++f)
            if (const int rc = kernel_spectrum(f, B.kspec + f * Pc)) return rc;
        B.have_k = B.keep;
    }
    const double scale = 1.0 / (double)P3;
    for (int f = 0; f < 4; ++f) {
        if (!B.keep) {
            if (const int rc = kernel_spectrum(f, B.fk)) return rc;
            k_cmul<<<blocks_for(Pc), 256, 0, st>>>(Pc, B.fm, B.fk, B.fk, scale);
        } else if (f < 2) {
            k_cmul<<<blocks_for(Pc), 256, 0, st>>>(Pc, B.fm, B.kspec + f * Pc, B.fk, scale);
        } else if (f == 2) {
            k_cmul_x2<<<blocks_for(Pc), 256, 0, st>>>(n, B.fm, B.kspec + Pc, B.fk, scale);
        } else {
            const dim3 tiles((unsigned)((n + kCmulTile) / kCmulTile), (unsigned)((P + kCmulTile - 1) / kCmulTile),
                             (unsigned)P);
            k_cmul_x3<<<tiles, dim3(kCmulTile, kCmulTile), 0, st>>>(n, B.fm, B.kspec + Pc, B.fk, scale);
        }
        GCK(cudaGetLastError(), "k_cmul");
        FCK(cufftExecZ2Z(B.c2c, B.fk, B.fk, CUFFT_INVERSE), "cufftExecZ2Z");
        FCK(cufftExecZ2D(B.c2r, B.fk, B.buf), "cufftExecZ2D");
        k_extract<<<blocks_for(n3), 256, 0, st>>>(n, B.buf, B.val + f * n3);
        GCK(cudaGetLastError(), "k_extract");
    }
    const int64_t lines = 4 * (int64_t)n * n;
    k_spline_lines<<<(unsigned)((lines + 127) / 128), 128, 0, st>>>(n, lines, B.val, B.y2);
    GCK(cudaGetLastError(), "k_spline_lines");
    k_interleave<<<blocks_for(n3), 256, 0, st>>>(n3, B.val, B.y2, dest, dest32);
    GCK(cudaGetLastError(), "k_interleave");
    return RT3D_OK;
}

int grid_build(GridDev &g, int64_t np, const double *pos, const double *mass, double soft, int mean_subtract,
               bool fp64, cudaStream_t st, std::string &err)
{
    Builder B;
    int rc = builder_init(B, g.n, g.h, soft, np, st, err);
    if (rc != RT3D_OK) return rc;
    if (fp64)
        GCK(cudaMalloc(&g.tab, sizeof(double) * kGridRec * (size_t)B.n3()), "grid node table");
    else
        GCK(cudaMalloc(&g.tab32, sizeof(float) * kGridRec * (size_t)B.n3()), "grid node table");
    builder_keep_spectra(B);
    rc = builder_run(B, np, pos, mass, g.lo, mean_subtract, g.tab, g.tab32, st);
    if (rc != RT3D_OK) return rc;
    GCK(cudaStreamSynchronize(st), "grid build");
    return RT3D_OK;
}

int grid_build_box(GridDev &g, int64_t np, const double *pos, const double *mass, double soft,
                   const int32_t *rot, const double *shift, int mean_subtract, bool fp64, cudaStream_t st,
                   std::string &err)
{
    const int R = g.n_rep, C = g.cubes;
    const double L = g.L, W = g.W, c = 0.5 * L;
    // every replica's prism particles, cube by cube (host threads over replicas)
    std::vector<std::vector<double>> cp((size_t)R * C), cm((size_t)R * C);
    auto select = [&](int j) {
        const int32_t *Rm = rot + 9 * j;
        const double *sh = shift + 3 * j;
        for (int64_t i = 0; i < np; ++i) {
            const double *p = pos + 3 * i;
            double w[3];
            for (int r = 0; r < 3; ++r) {
                double v = 0.0;
                for (int k = 0; k < 3; ++k) v += (double)Rm[3 * r + k] * (p[k] - c);
                v = v + c + sh[r];
                while (v >= L) v -= L;
                while (v < 0.0) v += L;
                w[r] = v;
            }
            w[0] -= c;
            w[1] -= c;
            w[2] += (double)j * L;
            if (!(w[0] >= -0.5 * W && w[0] < 0.5 * W && w[1] >= -0.5 * W && w[1] < 0.5 * W)) continue;
            for (int q = 0; q < C; ++q) {
                const double z0 = (double)j * L + (double)q * W;
                if (w[2] >= z0 && w[2] < z0 + W) {
                    std::vector<double> &P = cp[(size_t)j * C + q];
                    P.insert(P.end(), w, w + 3);
                    cm[(size_t)j * C + q].push_back(mass[i]);
                    break;
                }
            }
        }
    };
    {
        const int nt = std::max(1, std::min(R, (int)std::thread::hardware_concurrency()));
        std::vector<std::thread> th;
        std::vector<char> oom((size_t)nt, 0);
        for (int t = 0; t < nt; ++t)
            th.emplace_back([&, t] {
                try {
                    for (int j = t; j < R; j += nt) select(j);
                } catch (const std::bad_alloc &) {
                    oom[(size_t)t] = 1;
                }
            });
        for (auto &x : th) x.join();
        for (char o : oom)
            if (o) {
                err = "host memory for the prism particles";
                return RT3D_ENOMEM;
            }
    }
    Builder B;
    size_t most = 0;
    for (const auto &m : cm) most = std::max(most, m.size());
    int rc = builder_init(B, g.n, g.h, soft, (int64_t)most, st, err);
    if (rc != RT3D_OK) return rc;
    const size_t stride = kGridRec * (size_t)B.n3();
    if (fp64)
        GCK(cudaMalloc(&g.tab, sizeof(double) * stride * (size_t)R * C), "grid node tables");
    else
        GCK(cudaMalloc(&g.tab32, sizeof(float) * stride * (size_t)R * C), "grid node tables");
    builder_keep_spectra(B);
    for (int j = 0; j < R; ++j)
        for (int q = 0; q < C; ++q) {
            const size_t cell = (size_t)j * C + q;
            const double lo[3] = {-0.5 * W, -0.5 * W, (double)j * L + (double)q * W};
            rc = builder_run(B, (int64_t)cm[cell].size(), cp[cell].data(), cm[cell].data(), lo, mean_subtract,
                             g.tab ? g.tab + cell * stride : nullptr, g.tab32 ? g.tab32 + cell * stride : nullptr,
                             st);
            if (rc != RT3D_OK) return rc;
            // the host lists of this cube must outlive its asynchronous upload
            GCK(cudaStreamSynchronize(st), "grid build");
        }
    return RT3D_OK;
}
#undef GCK
#undef FCK

}  // namespace rt3d
