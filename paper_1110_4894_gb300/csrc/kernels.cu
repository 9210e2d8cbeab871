// kernels.cu -- FP64 kernels of the trace: step schedule (cosmology
// precompute), bundle initialiser, RK4 integrator stage, bundle reducer,
// muPDF histogram and particle staging.
#include <algorithm>

#include "trace_device.cuh"

namespace rt3d {

// ---------------------------------------------------------------------------
// background cosmology on the device (Sec. 3.5, Eq. raytracedistance)
// ---------------------------------------------------------------------------
// a(t) and h da/dt at t = j h (the closed forms of Eq. scalefac2)
__global__ void k_atab(Cosmo c, int n, double h, double *__restrict__ tab)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double a = cosmo_a_exact(c, (double)j * h);
    tab[2 * j] = a;
    tab[2 * j + 1] = h * cosmo_adot(c, a);
}

cudaError_t launch_atab(const Cosmo &c, int n, double h, double *d_tab, cudaStream_t st)
{
    k_atab<<<(n + 255) / 256, 256, 0, st>>>(c, n, h, d_tab);
    return cudaGetLastError();
}

// chi_s to misc[0] and the affine steps
__global__ void __launch_bounds__(kSchedThreads) k_schedule(Cosmo c, double z_s, int kind, int n, double chi_l,
                                                            double s, double *dlam, double *misc)
{
    const double chi_s = comoving_distance(c, z_s);
    if (blockIdx.x == 0 && threadIdx.x == 0) misc[0] = chi_s;
    schedule_steps(c, kind, n, chi_s, chi_l, s, dlam);
}

cudaError_t launch_schedule(const Cosmo &c, double z_s, int kind, int n, double chi_l, double s, double *d_dlam,
                            double *d_misc, cudaStream_t st)
{
    k_schedule<<<std::min(n, 16 * device_sm_count()), kSchedThreads, 0, st>>>(c, z_s, kind, n, chi_l, s, d_dlam,
                                                                              d_misc);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// bundle initialiser (Sec. 3.1, ray bundle; initial state of Sec. 3.4)
// ---------------------------------------------------------------------------
__global__ void k_init(TraceParams tp, DevField f, const double *__restrict__ theta, RayState rs,
                       unsigned long long *cnt)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        cnt[0] = cnt[1] = cnt[2] = 0ull;
    }
    if (i >= rs.n_rays) return;
    init_ray(tp, f, theta, rs, i);
}

cudaError_t launch_init(const TraceParams &tp, const DevField &f, const double *d_theta, RayState rs,
                        unsigned long long *d_counters, cudaStream_t st)
{
    const int64_t blocks = (rs.n_rays + 255) / 256;
    k_init<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, st>>>(tp, f, d_theta, rs, d_counters);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// integrator stage (Eq. geodesiceqn with the App. A symbols, classical RK4,
// termination on x3 with linear interpolation: Sec. 3.4)
// ---------------------------------------------------------------------------
// Rays with many split partials: a block of four warps serves 32 rays.  Each
// warp adds up one output of its rays, a serial double-float sum in split order
// (reduce_step), then one warp runs the FP64 stage update of the 32 rays.  The
// sum is a chain of thousands of steps in few warps where few bundles meet many
// particles (4096 splits of 640 rays: 281 us a stage while its loads waited for
// one another), so AHEAD rows of partials are kept in flight in registers: 84 us
// with 64 rows.  96 rows leave an SM two blocks instead of three and pay off over
// many splits where the launch gives no SM two (a whole stage of 256 bundles in
// the 1,048,576-particle box, 2048 splits: 744 -> 734 us; but 200 bundles and 118
// splits 47.7 -> 48.4, 4096 bundles and 196 splits 848 -> 861).
constexpr int kStageRays = 32, kStageThreads = 4 * kStageRays;
constexpr int kRows = 16;  // rows per load group
// from this many rays on (four blocks of 256 per SM), one ray per thread
// still gives every SM several blocks
static int64_t stage_wide_rays() { return (int64_t)device_sm_count() * 4 * 256; }

int device_sm_count()
{
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 152;
    if (dev >= 0 && dev < 64 && cache[dev] > 0) return cache[dev];
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 152;
    if (dev >= 0 && dev < 64) cache[dev] = sms;
    return sms;
}

// (The kernels below are launched overlapped: no pointer of theirs is declared
// __restrict__, which would let its loads move ahead of the wait.)
// the bundles' prism records of this stage (mean-subtracted boxes), read by
// every ray of the bundle in k_stage: one warp per block, four bundles of eight
// lanes, so that few bundles still use the FP64 lanes of many SMs
constexpr int kPrismBundles = 32 / kCorners;
__global__ void __launch_bounds__(32) k_prism(TraceParams tp, DevField f, RayState rs, int step, int stage,
                                              const unsigned long long *cnt, double *prism)
{
    __shared__ double s_q[kPrismBundles][10 * kCorners];
    let_next_start();
    wait_for_previous();
    if (step >= tp.n_steps && cnt[(step - 1) & 1] == 0ull) return;  // every ray is across
    const int k = threadIdx.x / kCorners;
    const int64_t b = (int64_t)blockIdx.x * kPrismBundles + k;
    bundle_prism(f, rs, step * 4 + stage, b < rs.n_b ? b : -1, prism, s_q[k]);
}

cudaError_t launch_prism(const TraceParams &tp, const DevField &f, RayState rs, int step, int stage,
                         const unsigned long long *d_counters, double *d_prism, cudaStream_t st)
{
    const int64_t blocks = (rs.n_b + kPrismBundles - 1) / kPrismBundles;
    return launch_overlapped(k_prism, dim3((unsigned)(blocks > 0 ? blocks : 1)), 32, st, tp, f, rs, step, stage,
                             d_counters, d_prism);
}

// The sum of many split partials ahead of the stage, in place: row 0 of the
// partials becomes the double-float sum of all rows, the same bits as k_stage's
// own sum.  There a warp issues some twelve instructions a row, and few rays make
// few warps (640 rays x 4096 splits: 80 warps on 20 SMs, 72 us).  Only the
// additions hi + x and lo + w are chains: here one warp runs both (lanes 0-15 the
// high sums of tile k of kMergeRows rows, lanes 16-31 the low sums of tile
// k - 2), and the other warps do what is not serial in between: the TwoSum errors
// w of tile k - 1, and the copies of later tiles into shared memory.  16 rays of
// one output a block (a row is then a 128-byte line), so 640 rays use every SM:
// 38 us.  What is left is the chain, 16 cycles a row with a tile's barrier; more
// tiles in flight, longer ones, or more helper warps change nothing.
constexpr int kMergeRays = 16, kMergeRows = 48, kMergeTiles = 6, kMergeHelpers = 192, kMergeThreads = 32 + kMergeHelpers;
constexpr int kMergeAhead = kMergeTiles - 3;  // tiles on their way; three are in use
constexpr int kMergeGroup = 16;               // rows that the chains read ahead of their additions
// Many splits: from 256 rows on.  k_merge up to two of its blocks an SM; a whole
// stage (k_stage alone -> with k_merge, us): 64 bundles and 65,536 particles (256
// splits) 171 -> 141, 64 bundles and 1,048,576 particles 551 -> 526, 128 of 5 rays
// 449 -> 429, 128 of 9 rays (288 blocks) 835 -> 807; but 256 of 5 rays (320
// blocks, and warps enough for k_stage) 737 -> 746, 768 of 5 3692 -> 3714, and 200
// bundles with 118 splits 50 -> 53.
constexpr int kMergeFrom = 256;
static int64_t merge_blocks(int64_t n_rays) { return (n_rays + kMergeRays - 1) / kMergeRays; }
bool stage_merges(const ForceShape &sh, bool fp64, int64_t n_rays)
{
    return !fp64 && partial_splits(sh) >= kMergeFrom && 4 * merge_blocks(n_rays) <= 2 * (int64_t)device_sm_count();
}

__device__ __forceinline__ void copy_async8(void *dst, const void *src, bool valid)  // zeros if not valid
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(valid ? 8 : 0)
                 : "memory");
}

__global__ void __launch_bounds__(kMergeThreads) k_merge(float2 *partials, int S, int64_t n_rays, int n_steps, int step,
                                                         const unsigned long long *cnt)
{
    __shared__ float2 s_v[kMergeTiles][kMergeRows][kMergeRays];  // (x, y) of a row; y becomes w
    __shared__ float s_t[2][kMergeRows + 1][kMergeRays];         // high sums before each row, and after the last
    let_next_start();
    wait_for_previous();
    if (step >= n_steps && cnt[(step - 1) & 1] == 0ull) return;  // every ray is across
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, o = blockIdx.y;
    const int64_t i0 = (int64_t)blockIdx.x * kMergeRays;
    const int n_tiles = (S + kMergeRows - 1) / kMergeRows;
    const int r = lane % kMergeRays;
    // a helper thread has ray r of every kStep-th row, from row0 on
    constexpr int kStep = kMergeHelpers / kMergeRays, kEach = kMergeRows / kStep;
    static_assert(kEach * kStep == kMergeRows, "whole rows per helper thread");
    const int row0 = ((int)threadIdx.x - 32) / kMergeRays;
    const float2 *src = partials + ((int64_t)row0 * 4 + o) * n_rays + i0 + r;
    const int64_t pitch = (int64_t)kStep * 4 * n_rays;
    int stage_in = 0, left = i0 + r < n_rays ? S - row0 : 0;  // slot of the next tile; rows of this thread's from here
    const auto load = [&]() {
#pragma unroll
        for (int j = 0; j < kEach; ++j, left -= kStep, src += pitch)
            copy_async8(&s_v[stage_in][row0 + j * kStep][r], left > 0 ? src : partials, left > 0);
        stage_in = stage_in + 1 == kMergeTiles ? 0 : stage_in + 1;
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (warp > 0)
        for (int t = 0; t < kMergeAhead; ++t) load();
    const bool high = lane < kMergeRays;
    float acc = 0.0f;  // of this lane's chain
    for (int k = 0; k < n_tiles + 2; ++k) {
        if (warp > 0) asm volatile("cp.async.wait_group %0;" ::"n"(kMergeAhead - 1) : "memory");  // tile k is there
        __syncthreads();
        if (warp == 0) {
            const int t = high ? k : k - 2;
            if (t >= 0 && t < n_tiles) {
                const float *src = high ? &s_v[t % kMergeTiles][0][r].x : &s_v[t % kMergeTiles][0][r].y;
                float *dst = &s_t[t & 1][0][r];
                float v[2][kMergeGroup];
#pragma unroll
                for (int q = 0; q < kMergeGroup; ++q) v[0][q] = src[q * 2 * kMergeRays];
#pragma unroll
                for (int g = 0; g < kMergeRows / kMergeGroup; ++g) {
                    if (g + 1 < kMergeRows / kMergeGroup) {
#pragma unroll
                        for (int q = 0; q < kMergeGroup; ++q)
                            v[(g + 1) & 1][q] = src[((g + 1) * kMergeGroup + q) * 2 * kMergeRays];
                    }
#pragma unroll
                    for (int q = 0; q < kMergeGroup; ++q) {
                        if (high) dst[(g * kMergeGroup + q) * kMergeRays] = acc;
                        acc += v[g & 1][q];
                    }
                }
                if (high) dst[kMergeRows * kMergeRays] = acc;
            }
        } else {
            load();
            if (k >= 1 && k <= n_tiles) {
                const int t = k - 1;
                float2(*tile)[kMergeRays] = s_v[t % kMergeTiles];
                float(*sums)[kMergeRays] = s_t[t & 1];
#pragma unroll
                for (int j = 0; j < kEach; ++j) {
                    const int row = row0 + j * kStep;
                    const float hi = sums[row][r], sum = sums[row + 1][r];
                    const float2 v = tile[row][r];
                    const float bb = sum - hi;
                    tile[row][r].y = (hi - (sum - bb)) + (v.x - bb) + v.y;
                }
            }
        }
    }
    if (warp > 0) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        return;
    }
    const float lo = __shfl_down_sync(0xffffffffu, acc, kMergeRays);
    if (high && i0 + r < n_rays) partials[o * n_rays + i0 + r] = make_float2(acc, lo);
}

template <int AHEAD>
__global__ void __launch_bounds__(kStageThreads) k_stage(TraceParams tp, DevField f, RayState rs, int S, int fp64,
                                                        double mfac, const float2 *partials,
                                                        const double *dlam,
                                                        const double *misc, int step, int stage,
                                                        unsigned long long *cnt, const double *prism)
{
    wait_for_previous();
    if (stage == 0 && blockIdx.x == 0 && threadIdx.x == 0) cnt[step & 1] = 0ull;
    if (step >= tp.n_steps && cnt[(step - 1) & 1] == 0ull) return;  // every ray is across
    __shared__ double s_acc[kStageRays][4];
    const int o = threadIdx.x / kStageRays, lane = threadIdx.x % kStageRays;
    const int64_t i = (int64_t)blockIdx.x * kStageRays + lane;
    if (i < rs.n_rays) {
        constexpr int G = AHEAD / kRows;
        const float2 *src = partials + (int64_t)o * rs.n_rays + i;
        const int64_t pitch = 4 * rs.n_rays;
        float2 buf[G][kRows];
        // (rows past the last split are zeros, which leave the sum as it is; read
        // from L2: this block may have started while k_merge, on the same SM, had
        // the lines of row 0 in L1)
        const auto load = [&](int g, int s0) {
#pragma unroll
            for (int r = 0; r < kRows; ++r, src += pitch)
                buf[g][r] = s0 + r < S ? __ldcg(src) : make_float2(0.0f, 0.0f);
        };
#pragma unroll
        for (int g = 0; g < G; ++g) load(g, g * kRows);
        float hi = 0.0f, lo = 0.0f;
        double acc = 0.0;
        for (int s0 = 0; s0 < S; s0 += AHEAD) {
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if (s0 + g * kRows >= S) break;
                if (fp64) {
#pragma unroll
                    for (int r = 0; r < kRows; ++r)
                        acc += __hiloint2double(__float_as_int(buf[g][r].y), __float_as_int(buf[g][r].x));
                } else {
#pragma unroll
                    for (int r = 0; r < kRows; ++r) reduce_step(hi, lo, buf[g][r]);
                }
                load(g, s0 + AHEAD + g * kRows);
            }
        }
        s_acc[lane][o] = fp64 ? acc : (double)hi + (double)lo;
    }
    __syncthreads();
    if (threadIdx.x >= kStageRays) return;
    const bool act = i < rs.n_rays && stage_ray(tp, f, rs, S, fp64 != 0, mfac, partials, dlam, misc[0], step, stage, cnt, i,
                                                s_acc[lane], prism);
    const unsigned m = __ballot_sync(0xffffffffu, act);
    if (lane == 0 && m) atomicAdd(&cnt[2], (unsigned long long)__popc(m));
}

// One ray per thread, its four outputs reduced by the same thread: for few
// splits (the grid path) or enough rays to fill the GPU, where the FP64
// stage, not the reduction, needs the threads.
__global__ void __launch_bounds__(256) k_stage_wide(TraceParams tp, DevField f, RayState rs, int S, int fp64,
                                                   double mfac, const void *partials,
                                                   const double *dlam,
                                                   const double *misc, int step, int stage,
                                                   unsigned long long *cnt, const double *prism)
{
    wait_for_previous();
    if (stage == 0 && blockIdx.x == 0 && threadIdx.x == 0) cnt[step & 1] = 0ull;
    if (step >= tp.n_steps && cnt[(step - 1) & 1] == 0ull) return;  // every ray is across
    __shared__ unsigned s_active;
    if (threadIdx.x == 0) s_active = 0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < rs.n_rays) {
        double acc[4];
        if (!fp64) {
#pragma unroll
            for (int o = 0; o < 4; ++o) acc[o] = reduce_partials_mixed((const float2 *)partials, S, rs.n_rays, i, o);
        }
        if (stage_ray(tp, f, rs, S, fp64 != 0, mfac, partials, dlam, misc[0], step, stage, cnt, i,
                      fp64 ? nullptr : acc, prism))
            atomicAdd(&s_active, 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_active) atomicAdd(&cnt[2], (unsigned long long)s_active);
}

cudaError_t launch_stage(const TraceParams &tp, const DevField &f, RayState rs, const ForceShape &sh, bool fp64,
                         void *d_partials, const double *d_dlam, const double *d_misc, int step, int stage,
                         unsigned long long *d_counters, cudaStream_t st, const double *d_prism)
{
    const int S = partial_splits(sh);
    const double mfac = partial_mass_factor(f, sh);
    if (S <= 8 || rs.n_rays >= stage_wide_rays()) {
        // the two FP64 lanes of an SM serve all its warps: few rays go one warp
        // per block, to as many SMs as there are
        int nt = 256;
        while (nt > 32 && rs.n_rays < 2 * (int64_t)device_sm_count() * nt) nt /= 2;
        const int64_t blocks = (rs.n_rays + nt - 1) / nt;
        return launch_overlapped(k_stage_wide, dim3((unsigned)blocks), nt, st, tp, f, rs, S, fp64 ? 1 : 0, mfac,
                                 d_partials, d_dlam, d_misc, step, stage, d_counters, d_prism);
    } else {
        const int64_t blocks = (rs.n_rays + kStageRays - 1) / kStageRays;
        if (stage_merges(sh, fp64, rs.n_rays)) {
            const cudaError_t e = launch_overlapped(k_merge, dim3((unsigned)merge_blocks(rs.n_rays), 4), kMergeThreads,
                                                    st, (float2 *)d_partials, S, rs.n_rays, tp.n_steps, step,
                                                    d_counters);
            if (e != cudaSuccess) return e;
            return launch_overlapped(k_stage<16>, dim3((unsigned)blocks), kStageThreads, st, tp, f, rs, 1, 0, mfac,
                                     (const float2 *)d_partials, d_dlam, d_misc, step, stage, d_counters, d_prism);
        }
        return launch_overlapped(S >= kMergeFrom && blocks <= device_sm_count() ? k_stage<96> : k_stage<64>,
                                 dim3((unsigned)blocks), kStageThreads, st, tp, f, rs, S, fp64 ? 1 : 0, mfac,
                                 (const float2 *)d_partials, d_dlam, d_misc, step, stage, d_counters, d_prism);
    }
}

// trace_rays in FP64 through an isolated field of at most kFewParticles
// particles (the point lenses of Sec. 4.1), each ray summing them up itself.  A
// stage of those is all launches and latency otherwise: a point mass, 66
// bundles, 1000 steps, took 87.3 ms stage by stage, and takes 17.5 (4.3 us a
// stage, most of it the issue of some 200 FP64 instructions at 16 cycles each).
//
// One launch costs each ray its particles in turn (4.4 + 0.65 us a particle and
// stage while the warps have a scheduler each), the two kernels of a stage 18 us
// and more from a few thousand rays on.  ms for 50 steps in one launch / by
// stages: 66 bundles of 5: 8 particles 1.9 / 3.6, 22 3.6 / 3.9, 32 4.9 / 3.9, 64
// 8.8 / 3.8; 1024 bundles: 22 3.6 / 3.8, 32 4.9 / 5.0, 64 8.8 / 6.3; 2048: 22 3.6 /
// 5.0, 32 4.9 / 6.3, 64 8.8 / 9.0; 4096: 64 11.9 / 14.4; 32,768: 22 33 / 39, 64 81 /
// 85.  So the stages run by themselves from 23 particles on where there are fewer
// than 64 rays an SM.
bool few_in_one_launch(int64_t n_particles, int64_t n_rays)
{
    return n_particles <= kFewAlways ||
           (n_particles <= kFewParticles && n_rays >= 64 * (int64_t)device_sm_count());
}

template <bool PEPS>
__global__ void __launch_bounds__(kTraceRaysNT) k_few_trace(TraceParams tp, DevField f, RayState rs, int g0, int g1,
                                                           const double *__restrict__ dlam,
                                                           const double *__restrict__ misc, unsigned long long *cnt)
{
    __shared__ double4_16a s_p[kFewParticles];
    __shared__ double s_e[PEPS ? kFewParticles : 1];
    const int n = (int)f.n;
    for (int q = threadIdx.x; q < n; q += kTraceRaysNT) {
        const int4 pr = f.part[q];
        s_p[q] = make_double4_16a((double)pr.x * f.delta, (double)pr.y * f.delta, (double)pr.z * f.delta, f.m64[q]);
        if (PEPS) s_e[q] = f.eps2_64[q];
    }
    __syncwarp();
    trace_rays(tp, rs, g0, g1, dlam, misc, cnt, [&](const double r[3], double, double F[4]) {
        const double x = r[0] - f.O[0], y = r[1] - f.O[1], z = r[2] - f.O[2];
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        for (int q = 0; q < n; ++q) {
            const double4_16a p = s_p[q];
            pair_fp64(p.x - x, p.y - y, p.z - z, p.w, PEPS ? s_e[q] : f.eps2u64, acc);
        }
        field_from_sums(f, acc, 0, r, 1.0, F);
    });
}

cudaError_t launch_few_trace(const TraceParams &tp, const DevField &f, const RayState &rs, int g0, int g1,
                             const double *d_dlam, const double *d_misc, unsigned long long *d_counters,
                             cudaStream_t st)
{
    const int per_warp = 32 / rs.nr;
    const unsigned grid = (unsigned)((rs.n_b + per_warp - 1) / per_warp);
    const auto kern = f.eps2_64 ? k_few_trace<true> : k_few_trace<false>;
    kern<<<grid, kTraceRaysNT, 0, st>>>(tp, f, rs, g0, g1, d_dlam, d_misc, d_counters);
    return cudaGetLastError();
}

// field at arbitrary points (rt3d_potential): reduce partials + mean subtraction
__global__ void k_field_points(DevField f, int S, int fp64, double mfac, const void *__restrict__ partials,
                               const double *__restrict__ pts, const int *__restrict__ rep, int64_t n,
                               double *__restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double p[3] = {pts[i], pts[n + i], pts[2 * n + i]};
    const int r = rep ? rep[i] : 0;
    double F[4];
    if (r < 0 || r >= f.n_rep || !isfinite(p[0]) || !isfinite(p[1]) || !isfinite(p[2])) {
        // a replica index outside [0, n_rep) or a non-finite point: the pair
        // sum skipped it, and its result is NaN rather than a silent value
#pragma unroll
        for (int o = 0; o < 4; ++o) out[4 * i + o] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    gather_field(f, S, fp64 != 0, partials, n, i, r, p, mfac, F);
#pragma unroll
    for (int o = 0; o < 4; ++o) out[4 * i + o] = F[o];
}

cudaError_t launch_stage_field(const DevField &f, const ForceShape &sh, bool fp64, const void *d_partials,
                               const double *d_pts, const int *d_rep, int64_t n, double *d_out, cudaStream_t st)
{
    const int64_t blocks = (n + 255) / 256;
    k_field_points<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, st>>>(
        f, partial_splits(sh), fp64 ? 1 : 0, partial_mass_factor(f, sh), d_partials, d_pts, d_rep, n, d_out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// bundle reducer: least-squares lens-map Jacobian of the polygon offsets
// (Sec. 3.1; Eqs. lensmap, magnification), in FP64
// ---------------------------------------------------------------------------
__global__ void k_reduce(TraceParams tp, const double *__restrict__ theta, RayState rs,
                         const double *__restrict__ misc, double *__restrict__ bout, double *__restrict__ rout)
{
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= rs.n_b) return;
    reduce_bundle(tp, theta, rs, misc[0], b, bout + 6 * b, rout);
}

cudaError_t launch_reduce(const TraceParams &tp, const double *d_theta, RayState rs, const double *d_misc,
                          double *d_bout, double *d_rout, cudaStream_t st)
{
    const int64_t blocks = (rs.n_b + 127) / 128;
    k_reduce<<<(unsigned)(blocks > 0 ? blocks : 1), 128, 0, st>>>(tp, d_theta, rs, d_misc, d_bout, d_rout);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// muPDF (Sec. 5.3, Eq. weighthisto): integer counts and fixed-point weights
// by atomics (order-independent, so bit-reproducible), moments in a fixed
// order.
// ---------------------------------------------------------------------------
// value binned and weight base of entry i: v = |mu| (muPDF) or, with a shear
// pair, v = |gamma| = sqrt(g1^2 + g2^2) (shear PDF, Sec. 5.4, products and sum
// rounded separately as in the FP64 definition); the weight is 1/|mu| in both
struct HistIn {
    const double *mu;
    int stride;
    const int *fl;
    const double *fld;
    const double *g1, *g2;  // shear PDF; null for the muPDF
};

__device__ __forceinline__ bool hist_take(const HistIn &h, int64_t i, double &m, double &v)
{
    m = h.mu[i * h.stride];
    int f = h.fl ? h.fl[i] : (h.fld ? (int)h.fld[i * h.stride] : 0);
    if ((f & (RT3D_F_NOCROSS | RT3D_F_NONFINITE)) || !isfinite(m) || m == 0.0) return false;
    if (h.g1) {
        const double a = h.g1[i], b = h.g2[i];
        v = sqrt(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)));
        if (!isfinite(v)) return false;
    } else {
        v = fabs(m);
    }
    return true;
}

// Bin of |value| v, floor((log10 v - lmin) / dl) in FP64.  GB300 has two FP64
// lanes per SM and log10 is some sixty of their operations, so the bin is first
// estimated in FP32 (1 ulp log2f); only where the estimate lies within its
// error bound of a bin edge is the FP64 formula evaluated.  The bin is the
// formula's in either case.
struct HistBins {
    int bins;
    double lmin, dl;
    float lminf, inv_dl;
};

__device__ __forceinline__ double hist_bin(const HistBins &hb, double v)
{
    const float vf = (float)v;
    if (vf > 1e-30f && vf < 1e30f) {
        const float l = 0.30102999566f * log2f(vf);
        const float e = (l - hb.lminf) * hb.inv_dl, fl = floorf(e), fr = e - fl;
        // rounding of v, log2f, the products and the difference, in log10, then in bins
        const float err = 4e-7f * (fabsf(l) + fabsf(hb.lminf) + 1.0f) * hb.inv_dl + 4e-7f * fabsf(e);
        if (fr > err && fr < 1.0f - err) return (double)fl;
    }
    return floor((log10(v) - hb.lmin) / hb.dl);
}

// sums of w, w v and w (v - mean)^2 of a set of values, mean = wv / w, and of
// the union of two disjoint sets
struct HistPart {
    double W, S, M2;
};

__device__ __forceinline__ HistPart hist_join(const HistPart &a, const HistPart &b)
{
    if (!(b.W > 0.0)) return a;
    if (!(a.W > 0.0)) return b;
    HistPart r;
    r.W = a.W + b.W;
    r.S = a.S + b.S;
    const double d = b.S / b.W - a.S / a.W;
    r.M2 = a.M2 + b.M2 + d * d * a.W * (b.W / r.W);
    return r;
}

// One pass over the values: a block takes chunks of kHistChunk values, keeps
// them in registers, bins them into shared memory and forms the chunk's
// weighted mean and spread about that mean; the chunks are joined by the
// union formula, the blocks by the last one to finish (fixed order, so the
// result does not depend on timing).  The bound is FP64: about 25 operations
// per value.  The first version binned with global atomics (224 us for 2^20
// values) and took the moments in one block of 1024 threads, two passes
// (6311 us); now 102 us for the same call.
constexpr int kHistThreads = 256, kHistPer = 4, kHistChunk = kHistThreads * kHistPer;
constexpr int kHistSharedBins = 1024;  // more bins go to global atomics

template <int Q>
__device__ __forceinline__ void hist_block_sum(double (&x)[Q], double (*s_w)[Q])
{
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) x[q] += __shfl_xor_sync(0xffffffffu, x[q], d);
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int q = 0; q < Q; ++q) s_w[threadIdx.x >> 5][q] = x[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        x[q] = 0.0;
#pragma unroll
        for (int w = 0; w < kHistThreads / 32; ++w) x[q] += s_w[w][q];
    }
}

__global__ void k_hist_clear(int bins, unsigned long long *counts, unsigned long long *wfix, unsigned long long *scal)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < bins) counts[i] = wfix[i] = 0ull;
    if (i < 6) scal[i] = 0ull;  // five counters and the ticket
}

__global__ void __launch_bounds__(kHistThreads) k_hist(int64_t n, HistIn h, HistBins hb, unsigned long long *counts,
                                                      unsigned long long *wfix, unsigned long long *scal,
                                                      HistPart *parts, double *out8)
{
    __shared__ unsigned s_n[kHistSharedBins], s_lo[kHistSharedBins], s_hi[kHistSharedBins];
    __shared__ double s_w[kHistThreads / 32][2];
    __shared__ unsigned s_scal[5];
    __shared__ HistPart s_part[kHistThreads];
    __shared__ int s_last;
    const int tid = threadIdx.x;
    const bool local = hb.bins <= kHistSharedBins;
    if (local)
        for (int k = tid; k < hb.bins; k += kHistThreads) s_n[k] = s_lo[k] = s_hi[k] = 0u;
    if (tid < 5) s_scal[tid] = 0u;
    __syncthreads();
    HistPart mine = {0.0, 0.0, 0.0};
    unsigned cnt[5] = {0u, 0u, 0u, 0u, 0u};
    for (int64_t c0 = (int64_t)blockIdx.x * kHistChunk; c0 < n; c0 += (int64_t)gridDim.x * kHistChunk) {
        double v[kHistPer], w[kHistPer], sum[2] = {0.0, 0.0};
#pragma unroll
        for (int q = 0; q < kHistPer; ++q) {
            const int64_t i = c0 + q * kHistThreads + tid;
            double m = 0.0;
            v[q] = w[q] = 0.0;
            if (i >= n) continue;
            if (!hist_take(h, i, m, v[q])) {
                v[q] = 0.0;
                ++cnt[4];
                continue;
            }
            ++cnt[0];
            if (m < 0.0) ++cnt[3];
            w[q] = __drcp_rn(fabs(m));
            sum[0] += w[q];
            sum[1] += w[q] * v[q];
            const double bb = hist_bin(hb, v[q]);
            if (bb < 0.0) {
                ++cnt[1];
            } else if (bb >= (double)hb.bins) {
                ++cnt[2];
            } else {
                const int k = (int)bb;
                const unsigned long long x = (unsigned long long)__double2ll_rn(w[q] * 4294967296.0);
                if (local) {  // 64-bit sum as two 32-bit atomics with the carry
                    const unsigned xl = (unsigned)x, old = atomicAdd(&s_lo[k], xl);
                    atomicAdd(&s_n[k], 1u);
                    const unsigned xh = (unsigned)(x >> 32) + (old + xl < old ? 1u : 0u);
                    if (xh) atomicAdd(&s_hi[k], xh);
                } else {
                    atomicAdd(&counts[k], 1ull);
                    atomicAdd(&wfix[k], x);
                }
            }
        }
        hist_block_sum<2>(sum, s_w);
        const double mean = sum[0] > 0.0 ? sum[1] / sum[0] : 0.0;
        double m2[1] = {0.0};
#pragma unroll
        for (int q = 0; q < kHistPer; ++q) m2[0] += w[q] * (v[q] - mean) * (v[q] - mean);
        hist_block_sum<1>(m2, reinterpret_cast<double(*)[1]>(s_w));
        mine = hist_join(mine, HistPart{sum[0], sum[1], m2[0]});
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const unsigned t = __reduce_add_sync(0xffffffffu, cnt[q]);
        if ((tid & 31) == 0 && t) atomicAdd(&s_scal[q], t);
    }
    __syncthreads();
    if (local)
        for (int k = tid; k < hb.bins; k += kHistThreads)
            if (s_n[k]) {
                atomicAdd(&counts[k], (unsigned long long)s_n[k]);
                atomicAdd(&wfix[k], ((unsigned long long)s_hi[k] << 32) | s_lo[k]);
            }
    if (tid < 5 && s_scal[tid]) atomicAdd(&scal[tid], (unsigned long long)s_scal[tid]);
    if (tid == 0) parts[blockIdx.x] = mine;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&scal[5], 1ull) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    HistPart t = {0.0, 0.0, 0.0};
    for (int k = tid; k < gridDim.x; k += kHistThreads) {
        const volatile HistPart *q = parts + k;
        const HistPart x = {q->W, q->S, q->M2};
        t = hist_join(t, x);
    }
    s_part[tid] = t;
    for (int d = kHistThreads / 2; d > 0; d >>= 1) {
        __syncthreads();
        if (tid < d) s_part[tid] = hist_join(s_part[tid], s_part[tid + d]);
    }
    if (tid == 0) {
        const volatile unsigned long long *sc = scal;
        for (int q = 0; q < 5; ++q) out8[q] = (double)sc[q];  // used, under, over, negative, excluded
        const HistPart r = s_part[0];
        out8[5] = r.W;
        out8[6] = r.W > 0.0 ? r.S / r.W : 0.0;
        out8[7] = r.W > 0.0 ? sqrt(r.M2 / r.W) : 0.0;
    }
}

// d_scal: kHistScal words, the five counters, the ticket and the blocks' parts
cudaError_t launch_histogram(int64_t n, const double *d_mu, int mu_stride, const int *d_flags, const double *d_flagsd,
                             int bins, double mu_min, double mu_max, unsigned long long *d_counts,
                             unsigned long long *d_wfix, unsigned long long *d_scal, double *d_out8,
                             cudaStream_t st, const double *d_g1, const double *d_g2)
{
    const double lmin = log10(mu_min);
    const double dl = (log10(mu_max) - lmin) / (double)bins;
    HistIn h{d_mu, mu_stride, d_flags, d_flagsd, d_g1, d_g2};
    HistBins hb{bins, lmin, dl, (float)lmin, (float)(1.0 / dl)};
    k_hist_clear<<<(bins + 255) / 256, 256, 0, st>>>(bins, d_counts, d_wfix, d_scal);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t chunks = std::max<int64_t>(1, (n + kHistChunk - 1) / kHistChunk);
    k_hist<<<(unsigned)std::min<int64_t>(chunks, kHistBlocks), kHistThreads, 0, st>>>(
        n, h, hb, d_counts, d_wfix, d_scal, reinterpret_cast<HistPart *>(d_scal + 6), d_out8);
    return cudaGetLastError();
}

}  // namespace rt3d
