// project.cu -- ray-driven cone-beam forward projector A (Sec. 4.1
// "Projection operator"), its angular sub-sample loop (Sec. 3.4, Sec. 4.2.2),
// the per-sample motion warp (Sec. 3.1.1, Sec. 4.2.1) and the fused
// detector-space correction R (p - A x) with residual norms (Sec. 4.1
// "Correction kernel", Eq. (1) terms 1-2).
//
// Launch shape: one thread per detector pixel, 32 x 4 pixels per CTA so that
// a warp covers 32 neighbouring pixels of one detector row (neighbouring rays
// sample neighbouring voxels at every step).  Grid = (u tiles, views, v
// tiles): the CTAs resident at one time cover a band of detector rows across
// many views, whose rays all cross the same z-slab of the volume, so that
// slab stays in L2 while it is being sampled.
#include <cooperative_groups.h>

#include "atlas.cuh"
#include "cylinder.cuh"
#include "dyrect.cuh"
#include "fwd_common.cuh"
#include "joseph.cuh"
#include "ray.cuh"
#include "roi.cuh"

namespace ctrex {

// Samples per spline cell from which the deformation goes by runs (ray.cuh).
// 60 views at 80^3 / 96^3 / 112^3 / 128^3 (32 / 38 / 45 / 51 samples), by
// pairs: 1.30 / 2.07 / 3.14 / 4.52 ms, by runs: 1.49 / 2.20 / 3.15 / 4.31 ms.
constexpr float FWD_RUN_MIN = 45.0f;

template <typename TV>
__device__ __forceinline__ float LinearSampler<TV>::operator()(float gx, float gy, float gz, float &wsum) const
{
    return trilinear(vol, nx, ny, nz, gx, gy, gz, wsum);
}

template <typename TV>
__device__ __forceinline__ float LinearSampler<TV>::interior(float gx, float gy, float gz) const
{
    float ws;
    return trilinear(vol, nx, ny, nz, gx, gy, gz, ws);
}

// How a motion projector forms its samples' positions: not at all, by the
// pose alone, with the spline two samples at a time, or run by run (SplineRun).
enum FwdMotion { MOTION_NONE, MOTION_POSE, MOTION_PAIRS, MOTION_RUNS };

// The samples of a ray (positions relative to the grid centre `cen`) displaced
// by the pose alone, linear in the sample index.  In a kernel without the
// spline's registers (60 views of 128^3, pixels of a voxel, 1.18 ms; as pairs
// in the spline's kernel 2.04; unrolled by 2 or 4, 1.23).
template <typename Sampler>
__device__ __forceinline__ void pose_samples(const Grid &G, const Ray &R, const float d0[3], const float ds[3],
                                             const float cen[3], const Sampler &vol, float &a, float &ars)
{
    auto sample = [&](float kap, float &ws) {
        float q[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) q[r] = fmaf(kap, R.sg[r], R.g0[r]) + fmaf(kap, ds[r], d0[r]) + cen[r];
        return vol(q[0], q[1], q[2], ws);
    };
    float ws;
#pragma unroll 1
    for (int k = 0; k < R.K - 1; ++k) {
        a += sample((float)k, ws);
        ars += ws;
    }
    a *= G.step_mm;
    ars *= G.step_mm;
    if (R.w_last > 0.0f) {
        a = fmaf(R.w_last, sample(last_kappa(G, R), ws), a);
        ars = fmaf(R.w_last, ws, ars);
    }
}

// One ray's integral and row sum under motion, by the pose alone or run by run.
template <typename Sampler, bool RUNS>
__device__ __forceinline__ void motion_line_integral(const Grid &G, const ViewGPU &V, const MotionGPU &mo,
                                                     const float4 *spline, const Sampler &vol, float u, float v,
                                                     float &a, float &ars)
{
    a = 0.0f;
    ars = 0.0f;
    float cen[3];
    grid_centre(G, cen);
    Ray R;
    if (!setup_ray(G, V, u, v, R, cen)) return;
    float d0[3], ds[3];
    pose_line(mo, R, d0, ds);
    // (a view whose time scale is 0 sees no deformation, whatever the coefficients are)
    if (!RUNS || mo.s == 0.0f) {
        pose_samples(G, R, d0, ds, cen, vol, a, ars);
        return;
    }
    SplineLine L;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        L.x0[r] = fmaf(R.g0[r] + d0[r] + cen[r] + 0.5f, G.spl_scale[r], 1.0f);
        L.xs[r] = (R.sg[r] + ds[r]) * G.spl_scale[r];
    }
    const float kl = last_kappa(G, R);
    for (int k = 0; k < R.K;) {
        SplineRun run;
        const int end = run.find(L, k, R.K, kl);
        float2 axy[CHEB_N];
        float az[CHEB_N];
        run.fit(spline, L, axy, az);
        const float ih = 1.0f / run.half;
        float b = 0.0f, brs = 0.0f;  // the run's sums
#pragma unroll 1
        for (; k < end; ++k) {
            const bool last = k == R.K - 1;
            const float kap = last ? kl : (float)k, w = last ? fmaxf(R.w_last, 0.0f) : G.step_mm;
            float T[CHEB_N], u[3], q[3], ws;
            cheb_values((kap - run.mid) * ih, T);
            SplineRun::value(axy, az, T, u);
#pragma unroll
            for (int r = 0; r < 3; ++r)
                q[r] = fmaf(kap, R.sg[r], R.g0[r]) + fmaf(mo.s, u[r], fmaf(kap, ds[r], d0[r])) + cen[r];
            b = fmaf(w, vol(q[0], q[1], q[2], ws), b);
            brs = fmaf(w, ws, brs);
        }
        a += b;
        ars += brs;
    }
}

// Integral of one pixel (mean over its sub-angle rays): value and row sum.
// On the cylindrical domain the ray is clipped to the bounding cylinder and
// every sample is mapped to (r, phi, z) by the sampler; the rest is shared.
template <typename Sampler, int MOTION>
__device__ __forceinline__ void pixel_integral(const Grid &G, const ViewGPU *__restrict__ views,
                                               const MotionGPU &mo, const float4 *spline,
                                               const Sampler &vol, int view, float u,
                                               float v, float &val, float &rs)
{
    float acc = 0.0f, acc_rs = 0.0f;
    for (int s = 0; s < G.n_sub; ++s) {
        const ViewGPU V = views[view * G.n_sub + s];
        if constexpr (Sampler::ROI) {
            float a, ars;
            roi_integral<false>(G, vol, V, u, v, a, ars);
            acc += a;
            acc_rs += ars;
            continue;
        }
        if constexpr (Sampler::JOSEPH) {
            float a, ars;
            joseph_integral(G, vol, V, u, v, a, ars);
            acc += a;
            acc_rs += ars;
            continue;
        }
        if constexpr (MOTION == MOTION_POSE || MOTION == MOTION_RUNS) {
            float a, ars;
            motion_line_integral<Sampler, MOTION == MOTION_RUNS>(G, V, mo, spline, vol, u, v, a, ars);
            acc += a;
            acc_rs += ars;
            continue;
        }
        Ray R;
        if constexpr (Sampler::CYLINDER) {
            if (!setup_ray_cyl(G, vol.C, V, u, v, R)) continue;
        } else {
            if (!setup_ray(G, V, u, v, R)) continue;
        }
        float a = 0.0f, ars = 0.0f;
        const int Km1 = R.K - 1;
        int ka = Km1, kb = Km1;
        if (!MOTION && !Sampler::CYLINDER) interior_range(G, R, ka, kb);
        if constexpr (MOTION == MOTION_PAIRS) {
            for (int k = 0; k < R.K; k += 2) {
                float g[2][3], w[2], y[2][3];
                sample_pair(G, R, k, g, w);
                warp_pair(G, mo, spline, g, y);
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    float ws;
                    a = fmaf(w[n], vol(y[n][0], y[n][1], y[n][2], ws), a);
                    ars = fmaf(w[n], ws, ars);
                }
            }
            acc += a;
            acc_rs += ars;
            continue;
        }
        auto general = [&](int k) {
            float ws;
            a += vol(fmaf((float)k, R.sg[0], R.g0[0]), fmaf((float)k, R.sg[1], R.g0[1]),
                     fmaf((float)k, R.sg[2], R.g0[2]), ws);
            ars += ws;
        };
        for (int k = 0; k < ka; ++k) general(k);
        for (int k = ka; k < kb; ++k)
            a += vol.interior(fmaf((float)k, R.sg[0], R.g0[0]), fmaf((float)k, R.sg[1], R.g0[1]),
                              fmaf((float)k, R.sg[2], R.g0[2]));
        ars += (float)(kb - ka);
        for (int k = kb; k < Km1; ++k) general(k);
        a *= G.step_mm;
        ars *= G.step_mm;
        if (R.w_last > 0.0f) {
            float ws;
            a = fmaf(R.w_last, vol(R.g_last[0], R.g_last[1], R.g_last[2], ws), a);
            ars = fmaf(R.w_last, ws, ars);
        }
        acc += a;
        acc_rs += ars;
    }
    val = acc * G.inv_sub;
    rs = acc_rs * G.inv_sub;
}

template <typename Sampler, typename TP, int MODE, int MOTION>
__device__ __forceinline__ void fwd_body(Grid G, const ViewGPU *__restrict__ views,
                                         const MotionGPU *__restrict__ motion, const float4 *spline,
                                         const Sampler &vol_in, const int *__restrict__ view_idx,
                                         TP *__restrict__ out, float *__restrict__ rowsum_out,
                                         const TP *__restrict__ p, float *__restrict__ partials, unsigned *devcheck,
                                         int p_by_view)
{
    __shared__ float s_red[2][FWD_TX * FWD_TY / 32];
    __shared__ float2 s_tile[Sampler::TILE_TABLE];
    Sampler vol = vol_in;
    vol.bind(s_tile, threadIdx.y * FWD_TX + threadIdx.x, FWD_TX * FWD_TY);
    const int k = blockIdx.y;
    int view = view_idx ? view_idx[k] : k;
    bool ok = true;
    if (view < 0 || view >= G.n_views) {
        if (threadIdx.x == 0 && threadIdx.y == 0) atomicOr(devcheck, (unsigned)DEVCHECK_OOB);
        ok = false;
        view = 0;
    }
    if constexpr (Sampler::DYRECT) vol.set_view(view);  // the view's acquisition time
    MotionGPU mo;
    constexpr bool SPLINE = MOTION == MOTION_PAIRS || MOTION == MOTION_RUNS;
    __shared__ float4 s_spline[SPLINE ? SPLINE_TABLE : 1];
    if (MOTION) mo = motion[view];
    if (SPLINE) {
        load_spline(s_spline, spline, threadIdx.y * FWD_TX + threadIdx.x, FWD_TX * FWD_TY);
        spline = s_spline;
    }
    if (MOTION) __syncthreads();
    int iu, iv;
    tile_pixel<MOTION != MOTION_NONE>(blockIdx.x * FWD_TX, blockIdx.z * FWD_TY, iu, iv);
    const bool in_pix = iu < G.nu && iv < G.nv;
    const bool inside = ok && in_pix;
    float val = 0.0f, rs = 0.0f;
    if (inside) pixel_integral<Sampler, MOTION>(G, views, mo, spline, vol, view, (float)iu, (float)iv, val, rs);
    fwd_epilogue<TP, MODE>(G, k, view, ok, in_pix, iu, iv, val, rs, out, rowsum_out, p, partials, p_by_view,
                           s_red);
}

template <typename Sampler, typename TP, int MODE, int MOTION>
__global__ void __launch_bounds__(FWD_TX *FWD_TY)
    fwd_kernel(Grid G, const ViewGPU *__restrict__ views, const MotionGPU *__restrict__ motion,
               const float4 *spline, const Sampler vol_in, const int *__restrict__ view_idx,
               TP *__restrict__ out, float *__restrict__ rowsum_out, const TP *__restrict__ p,
               float *__restrict__ partials, unsigned *devcheck, int p_by_view)
{
    fwd_body<Sampler, TP, MODE, MOTION>(G, views, motion, spline, vol_in, view_idx, out, rowsum_out, p, partials,
                                        devcheck, p_by_view);
}

// The motion projector with the deformation run by run (ray.cuh): 45 views of
// the 256^3 motion workload 18.4 ms (by pairs 23.8), and half the error of the
// pairs against 64 bits (positions relative to the grid centre, a sum per
// run).  Four CTAs per SM (128^3, 60 views: 4.31 ms; 3: 4.55, 5: 4.74).
template <typename Sampler, typename TP, int MODE>
__global__ void __launch_bounds__(FWD_TX *FWD_TY, 4)
    fwd_run_kernel(Grid G, const ViewGPU *__restrict__ views, const MotionGPU *__restrict__ motion,
                   const float4 *spline, const Sampler vol_in, const int *__restrict__ view_idx,
                   TP *__restrict__ out, float *__restrict__ rowsum_out, const TP *__restrict__ p,
                   float *__restrict__ partials, unsigned *devcheck, int p_by_view)
{
    fwd_body<Sampler, TP, MODE, MOTION_RUNS>(G, views, motion, spline, vol_in, view_idx, out, rowsum_out, p, partials,
                                             devcheck, p_by_view);
}

// Projectors whose sampler declares MIN_BLOCKS > 0 (the event model and
// the multi-resolution ROI) run through this entry, compiled for that many
// resident CTAs per SM; the others keep fwd_kernel's bounds.  Event model:
// 72 registers and 7 CTAs gave 1128 ms on the 512^3 event workload, 56
// registers and 9 CTAs 1058 ms.
template <typename Sampler, typename TP, int MODE>
__global__ void __launch_bounds__(FWD_TX *FWD_TY, Sampler::MIN_BLOCKS > 0 ? Sampler::MIN_BLOCKS : 1)
    fwd_kernel_mb(Grid G, const ViewGPU *__restrict__ views, const Sampler vol_in, const int *__restrict__ view_idx,
                  TP *__restrict__ out, float *__restrict__ rowsum_out, const TP *__restrict__ p,
                  float *__restrict__ partials, unsigned *devcheck, int p_by_view)
{
    fwd_body<Sampler, TP, MODE, MOTION_NONE>(G, views, nullptr, nullptr, vol_in, view_idx, out, rowsum_out, p,
                                             partials, devcheck, p_by_view);
}

// Second pass of the residual reduction, FP64 from the first add in a fixed
// order: CTA b sums a contiguous part of the n pairs, a cluster of CTAs adds
// its parts in order and writes one pair (several clusters leave theirs for a
// last launch).  FP64 adds and conversions run at two per clock and SM, so the
// single CTA that a 64^3 iteration's 6480 pairs would fill is bound by them:
// FINISH_TIMES.
constexpr int FINISH_CLUSTER = 8;

template <typename T>
__global__ void __cluster_dims__(FINISH_CLUSTER, 1, 1) __launch_bounds__(512)
    finish_sums_kernel(const T *__restrict__ pairs, size_t n, double *__restrict__ out, size_t second = 0, size_t n2 = 0)
{
    namespace cg = cooperative_groups;
    __shared__ double s[2][16], part[2];
    const size_t per = (n + gridDim.x - 1) / gridDim.x, i0 = per * blockIdx.x, i1 = min(i0 + per, n);
    double a = 0.0, b = 0.0;
#pragma unroll 4
    for (size_t i = i0 + threadIdx.x; i < i1; i += 512) {
        a += (double)pairs[2 * i];
        if (n2 == 0) b += (double)pairs[2 * i + 1];
    }
    // n2: the second sum is that of the n2 pairs from `second` on
    const size_t per2 = (n2 + gridDim.x - 1) / gridDim.x, j0 = second + per2 * blockIdx.x,
                 j1 = min(j0 + per2, second + n2);
#pragma unroll 4
    for (size_t i = j0 + threadIdx.x; i < j1; i += 512) b += (double)pairs[2 * i + 1];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, off);
        b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if ((threadIdx.x & 31) == 0) {
        s[0][threadIdx.x >> 5] = a;
        s[1][threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (int w = 0; w < 16; ++w) t += s[threadIdx.x][w];
        part[threadIdx.x] = t;
    }
    const cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (cluster.block_rank() == 0 && threadIdx.x < 2) {
        double t = 0.0;
        for (int r = 0; r < FINISH_CLUSTER; ++r) t += *cluster.map_shared_rank(part + threadIdx.x, r);
        out[2 * (blockIdx.x / FINISH_CLUSTER) + threadIdx.x] = t;
    }
    cluster.sync();  // the parts are read before their CTAs end
}

// |p|^2 in the texture kernel's tiles of 32 x 4 pixels and its order of
// additions (a warp per tile), for ctrex_fwd_correct from the column kernels,
// whose CTAs hold other pixels: the norm that it reports in FP64 is then the
// same number whichever kernel projects (their FP32 partials differ by up to
// 4e-9 of it).  One read of p: 0.1 ms for 360 images of 384^2, beside a Joseph
// projection of 7.1.
template <typename TP>
__global__ void __launch_bounds__(256) norm_tiles_kernel(Grid G, const int *__restrict__ view_idx, dim3 tiles,
                                                         const TP *__restrict__ p, float *__restrict__ partials)
{
    const size_t bid = (size_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (bid >= (size_t)tiles.x * tiles.y * tiles.z) return;
    const int tu = (int)(bid % tiles.x), k = (int)(bid / tiles.x % tiles.y), tv = (int)(bid / ((size_t)tiles.x * tiles.y));
    const int view = view_idx ? view_idx[k] : k, lane = threadIdx.x & 31, iu = tu * FWD_TX + lane;
    const bool ok = view >= 0 && view < G.n_views && iu < G.nu;
    float p2[FWD_TY], b = 0.0f;
#pragma unroll
    for (int r = 0; r < FWD_TY; ++r) {
        const int iv = tv * FWD_TY + r;
        const float pm = ok && iv < G.nv ? Storage<TP>::load(p + ((size_t)k * G.nv + iv) * G.nu + iu) : 0.0f;
        p2[r] = pm * pm;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int r = 0; r < FWD_TY; ++r) p2[r] += __shfl_xor_sync(0xffffffffu, p2[r], off);
#pragma unroll
    for (int r = 0; r < FWD_TY; ++r) b += p2[r];
    if (lane == 0) partials[2 * bid + 1] = b;
}

// Exact sample count (same set-up arithmetic as the projector): ray
// segments, or for the Joseph projector slice crossings with a tap inside.
enum CountKind { COUNT_BOX = 0, COUNT_CYL = 1, COUNT_JOSEPH = 2, COUNT_ROI = 3 };
template <int KIND>
__global__ void __launch_bounds__(FWD_TX *FWD_TY)
    count_kernel(Grid G, CylGPU C, RoiGPU Q, const ViewGPU *__restrict__ views, const int *__restrict__ view_idx,
                 unsigned long long *out)
{
    const int k = blockIdx.y;
    const int view = view_idx ? view_idx[k] : k;
    if (view < 0 || view >= G.n_views) return;
    const int iu = blockIdx.x * FWD_TX + threadIdx.x;
    const int iv = blockIdx.z * FWD_TY + threadIdx.y;
    unsigned long long n = 0;
    if (iu < G.nu && iv < G.nv) {
        for (int s = 0; s < G.n_sub; ++s) {
            Ray R;
            const ViewGPU &V = views[view * G.n_sub + s];
            if (KIND == COUNT_ROI) {
                RoiSampler rs{};
                rs.R = Q;
                float a, b;
                n += (unsigned long long)roi_integral<true>(G, rs, V, (float)iu, (float)iv, a, b);
                continue;
            }
            if (KIND == COUNT_JOSEPH) {
                JRay J;
                if (joseph_setup(G, V, (float)iu, (float)iv, J)) n += (unsigned long long)(J.khi - J.klo + 1);
                continue;
            }
            const bool hit = KIND == COUNT_CYL ? setup_ray_cyl(G, C, V, (float)iu, (float)iv, R)
                                               : setup_ray(G, V, (float)iu, (float)iv, R);
            if (hit) n += (unsigned long long)R.K;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) n += __shfl_xor_sync(0xffffffffu, n, off);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(out, n);
}

// Pairs up to which one cluster sums alone (one launch / two: 25,600 pairs 9.3 /
// 12.8 us, 51,200 12.8 / 13.1, 102,400 20.7 / 14.6), and the CTAs beyond.
constexpr int FINISH_ONE = 49152, FINISH_CTAS = 152;
static_assert(FINISH_CTAS % FINISH_CLUSTER == 0, "whole clusters");

static dim3 fwd_grid(const Grid &G, int n_idx)
{
    return dim3((G.nu + FWD_TX - 1) / FWD_TX, n_idx, (G.nv + FWD_TY - 1) / FWD_TY);
}

int forward_partials_needed(const Grid &G, int n_idx)
{
    const dim3 g = fwd_grid(G, n_idx);
    const int col = column_partials_needed(G, n_idx), n = (int)(g.x * g.y * g.z);
    // either launch shape, and room for the second pass
    return n + col + 2 * FINISH_CTAS;
}

template <typename Sampler, typename TP, int MODE>
static cudaError_t fwd_launch(const FwdArgs &a, const Sampler &smp, TP *out, float *rowsum, const TP *p,
                              float *partials)
{
    const Grid &G = *a.grid;
    const dim3 grid = fwd_grid(G, a.n_idx), block(FWD_TX, FWD_TY);
    if constexpr (!Sampler::CYLINDER && !Sampler::JOSEPH && !Sampler::ROI && !Sampler::DYRECT) {
        if (a.motion && a.spline && spline_runs(G, FWD_RUN_MIN)) {
            fwd_run_kernel<Sampler, TP, MODE><<<grid, block, 0, a.stream>>>(
                G, a.views, a.motion, a.spline, smp, a.view_idx, out, rowsum, p, partials, a.devcheck, a.p_by_view);
            return cudaGetLastError();
        }
        if (a.motion) {
            auto *kernel = a.spline ? fwd_kernel<Sampler, TP, MODE, MOTION_PAIRS>
                                    : fwd_kernel<Sampler, TP, MODE, MOTION_POSE>;
            kernel<<<grid, block, 0, a.stream>>>(G, a.views, a.motion, a.spline, smp, a.view_idx, out, rowsum, p,
                                                 partials, a.devcheck, a.p_by_view);
            return cudaGetLastError();
        }
    } else if (a.motion) {
        return cudaErrorNotSupported;  // the motion warp is defined for the trilinear Cartesian projector only
    }
    if constexpr (Sampler::MIN_BLOCKS > 0)
        fwd_kernel_mb<Sampler, TP, MODE><<<grid, block, 0, a.stream>>>(G, a.views, smp, a.view_idx, out, rowsum, p,
                                                                      partials, a.devcheck, a.p_by_view);
    else
        fwd_kernel<Sampler, TP, MODE, MOTION_NONE><<<grid, block, 0, a.stream>>>(
            G, a.views, nullptr, nullptr, smp, a.view_idx, out, rowsum, p, partials, a.devcheck, a.p_by_view);
    return cudaGetLastError();
}

// Texture-atlas sampling when the context has uploaded the volume into one;
// row-major loads otherwise (volumes beyond the 2D texture limits).
template <typename TP, int MODE>
static cudaError_t fwd_dispatch_sampler(const FwdArgs &a, TP *out, float *rowsum, const TP *p, float *partials)
{
    if (a.roi) {  // context and ROI grids, each from its own atlas
        if (!a.atlas || !a.roi_atlas || a.cyl || a.joseph) return cudaErrorInvalidValue;
        RoiSampler rs{RoiAtlasSampler{*a.atlas}, RoiAtlasSampler{*a.roi_atlas}, *a.roi};
        return fwd_launch<RoiSampler, TP, MODE>(a, rs, out, rowsum, p, partials);
    }
    if (a.dyr) {  // mu0 from the volume atlas, mu1 and tau from their own
        if (!a.atlas || !a.dyr->mu1 || !a.dyr->tau_atlas || a.cyl || a.joseph) return cudaErrorInvalidValue;
        DyrectSampler ds{*a.atlas, *a.dyr->mu1, *a.dyr->tau_atlas, a.dyr->t_view, a.dyr->tau_brick, a.dyr->bnx,
                         a.dyr->bny};
        return fwd_launch<DyrectSampler, TP, MODE>(a, ds, out, rowsum, p, partials);
    }
    if (a.joseph) {  // the Joseph projector reads its three-stack atlas only
        if (!a.atlas || a.cyl) return cudaErrorInvalidValue;
        const Grid &G = *a.grid;
        JosephSampler js{AtlasSampler{*a.atlas}, {G.nx, G.ny, G.nz}, {0, G.nx, G.nx + G.ny}};
        return fwd_launch<JosephSampler, TP, MODE>(a, js, out, rowsum, p, partials);
    }
    if (a.cyl) {  // the cylindrical domain is sampled from its atlas only
        if (!a.atlas) return cudaErrorInvalidValue;
        return fwd_launch<CylSampler, TP, MODE>(a, CylSampler{AtlasSampler{*a.atlas}, *a.cyl}, out, rowsum, p,
                                               partials);
    }
    if (a.atlas) return fwd_launch<AtlasSampler, TP, MODE>(a, AtlasSampler{*a.atlas}, out, rowsum, p, partials);
    const Grid &G = *a.grid;
    if (a.vol_dtype == CTREX_F32)
        return fwd_launch<LinearSampler<float>, TP, MODE>(
            a, LinearSampler<float>{static_cast<const float *>(a.vol), G.nx, G.ny, G.nz}, out, rowsum, p, partials);
    return fwd_launch<LinearSampler<__nv_bfloat16>, TP, MODE>(
        a, LinearSampler<__nv_bfloat16>{static_cast<const __nv_bfloat16 *>(a.vol), G.nx, G.ny, G.nz}, out, rowsum,
        p, partials);
}

template <int MODE>
static cudaError_t fwd_dispatch(const FwdArgs &a, int pdt, void *out, float *rowsum, const void *p,
                                float *partials)
{
    if (a.column) return launch_forward_column(a, MODE == MODE_CORRECT, pdt, out, rowsum, p, partials);
    if (pdt == CTREX_F32)
        return fwd_dispatch_sampler<float, MODE>(a, (float *)out, rowsum, (const float *)p, partials);
    return fwd_dispatch_sampler<__nv_bfloat16, MODE>(a, (__nv_bfloat16 *)out, rowsum, (const __nv_bfloat16 *)p,
                                                     partials);
}

cudaError_t launch_forward(const FwdArgs &a, void *proj, int proj_dtype, float *rowsum)
{
    if (a.n_idx == 0) return cudaSuccess;
    return fwd_dispatch<MODE_PROJECT>(a, proj_dtype, proj, rowsum, nullptr, nullptr);
}

cudaError_t launch_forward_correct(const FwdArgs &a, const void *p, int p_dtype, void *r, int r_dtype,
                                   float *partials, int n_partials_cap, double *sums)
{
    if (p_dtype != r_dtype) return cudaErrorInvalidValue;
    if (a.n_idx == 0) {
        if (sums) return cudaMemsetAsync(sums, 0, 2 * sizeof(double), a.stream);
        return cudaSuccess;
    }
    const dim3 fg = fwd_grid(*a.grid, a.n_idx);
    const int n = a.column ? column_partials_needed(*a.grid, a.n_idx) : (int)(fg.x * fg.y * fg.z);
    const bool norm = a.column && a.norm_tiles && sums;
    const size_t nt = norm ? (size_t)fg.x * fg.y * fg.z : 0;
    if (n + nt + 2 * FINISH_CTAS > (size_t)n_partials_cap) return cudaErrorInvalidValue;
    if (norm) {  // first: r may be p itself
        const unsigned ctas = (unsigned)((nt + 7) / 8);
        if (p_dtype == CTREX_F32)
            norm_tiles_kernel<<<ctas, 256, 0, a.stream>>>(*a.grid, a.view_idx, fg,
                                                          static_cast<const float *>(p), partials + 2 * (size_t)n);
        else
            norm_tiles_kernel<<<ctas, 256, 0, a.stream>>>(*a.grid, a.view_idx, fg,
                                                          static_cast<const __nv_bfloat16 *>(p), partials + 2 * (size_t)n);
    }
    cudaError_t e = fwd_dispatch<MODE_CORRECT>(a, p_dtype, r, nullptr, p, partials);
    if (e != cudaSuccess || sums == nullptr) return e;
    if (n <= FINISH_ONE) {
        finish_sums_kernel<<<FINISH_CLUSTER, 512, 0, a.stream>>>(partials, (size_t)n, sums, (size_t)n, nt);
    } else {  // the intermediate sums lie behind the partials
        double *mid = reinterpret_cast<double *>(partials + 2 * ((size_t)n_partials_cap - 2 * FINISH_CTAS));
        finish_sums_kernel<<<FINISH_CTAS, 512, 0, a.stream>>>(partials, (size_t)n, mid, (size_t)n, nt);
        finish_sums_kernel<<<FINISH_CLUSTER, 512, 0, a.stream>>>(mid, (size_t)(FINISH_CTAS / FINISH_CLUSTER), sums);
    }
    return cudaGetLastError();
}

cudaError_t launch_count_samples(const FwdArgs &a, unsigned long long *out)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), a.stream);
    if (e != cudaSuccess || a.n_idx == 0) return e;
    const dim3 grid = fwd_grid(*a.grid, a.n_idx), block(FWD_TX, FWD_TY);
    if (a.cyl)
        count_kernel<COUNT_CYL><<<grid, block, 0, a.stream>>>(*a.grid, *a.cyl, RoiGPU{}, a.views, a.view_idx, out);
    else if (a.joseph)
        count_kernel<COUNT_JOSEPH><<<grid, block, 0, a.stream>>>(*a.grid, CylGPU{}, RoiGPU{}, a.views, a.view_idx,
                                                                 out);
    else if (a.roi)
        count_kernel<COUNT_ROI><<<grid, block, 0, a.stream>>>(*a.grid, CylGPU{}, *a.roi, a.views, a.view_idx, out);
    else
        count_kernel<COUNT_BOX><<<grid, block, 0, a.stream>>>(*a.grid, CylGPU{}, RoiGPU{}, a.views, a.view_idx,
                                                              out);
    return cudaGetLastError();
}

// (min, max) transition times of parts of the volume, computed once by
// ctrex_set_dyrect.  A NaN transition time sends its tap to mu1 (t < NaN is
// false): a part with one never takes the mu0 shortcut, and the mu1 one only
// for t = +inf.
//
// Cells of 4^3 voxels: a warp takes 8 of them along x, a lane 4 x 4 values.
__global__ void __launch_bounds__(128) tau_cell_kernel(const float *__restrict__ tau, int nx, int ny, int nz, int cnx,
                                                       int cny, int cnz, float2 *__restrict__ cell)
{
    const int per = (cnx + 7) / 8, lane = threadIdx.x & 31;
    const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= (long long)per * cny * cnz) return;
    const int gx = (int)(w % per), cy = (int)((w / per) % cny), cz = (int)(w / ((long long)per * cny));
    const int x = gx * 32 + lane;
    float lo = INFINITY, hi = -INFINITY;
    bool nan = false;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int y = 4 * cy + (i & 3), z = 4 * cz + (i >> 2);
        if (x < nx && y < ny && z < nz) {
            const float v = __ldg(tau + ((size_t)z * ny + y) * nx + x);
            nan |= v != v;
            lo = fminf(lo, v);
            hi = fmaxf(hi, v);
        }
    }
    if (nan) {
        lo = -INFINITY;
        hi = INFINITY;
    }
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
    }
    const int cx = gx * 8 + lane / 4;
    if ((lane & 3) == 0 && cx < cnx) cell[((size_t)cz * cny + cy) * cnx + cx] = make_float2(lo, hi);
}

// brick: the 8^3 brick b and the voxel past each of its upper faces; block:
// voxels 8 b - 4 .. 8 b + 15.  One warp per brick.
__global__ void __launch_bounds__(128) tau_brick_kernel(const float *__restrict__ tau, const float2 *__restrict__ cell,
                                                        int nx, int ny, int nz, int bnx, int bny, int bnz, int cnx,
                                                        int cny, int cnz, float2 *__restrict__ brick,
                                                        float2 *__restrict__ block)
{
    const long long b = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= (long long)bnx * bny * bnz) return;
    const int lane = threadIdx.x & 31;
    const int bx = (int)(b % bnx), by = (int)((b / bnx) % bny), bz = (int)(b / ((long long)bnx * bny));
    float lo = INFINITY, hi = -INFINITY, blo = INFINITY, bhi = -INFINITY;
    bool nan = false;
    for (int i = lane; i < 729; i += 32) {
        const int x = min(8 * bx + i % 9, nx - 1), y = min(8 * by + i / 9 % 9, ny - 1), z = min(8 * bz + i / 81, nz - 1);
        const float v = __ldg(tau + ((size_t)z * ny + y) * nx + x);
        nan |= v != v;
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
    for (int i = lane; i < 125; i += 32) {
        const int x = min(max(2 * bx - 1 + i % 5, 0), cnx - 1), y = min(max(2 * by - 1 + i / 5 % 5, 0), cny - 1),
                  z = min(max(2 * bz - 1 + i / 25, 0), cnz - 1);
        const float2 c = __ldg(cell + ((size_t)z * cny + y) * cnx + x);
        blo = fminf(blo, c.x);
        bhi = fmaxf(bhi, c.y);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
        blo = fminf(blo, __shfl_xor_sync(0xffffffffu, blo, off));
        bhi = fmaxf(bhi, __shfl_xor_sync(0xffffffffu, bhi, off));
    }
    nan = __any_sync(0xffffffffu, nan);
    if (lane == 0) {
        brick[b] = nan ? make_float2(-INFINITY, INFINITY) : make_float2(lo, hi);
        block[b] = make_float2(blo, bhi);
    }
}

cudaError_t launch_tau_bricks(const float *tau, int nx, int ny, int nz, float2 *cell, float2 *brick, float2 *block,
                              cudaStream_t stream)
{
    const int bnx = (nx + 7) / 8, bny = (ny + 7) / 8, bnz = (nz + 7) / 8;
    const int cnx = (nx + 3) / 4, cny = (ny + 3) / 4, cnz = (nz + 3) / 4;
    const long long nb = (long long)bnx * bny * bnz, nw = (long long)((cnx + 7) / 8) * cny * cnz;
    tau_cell_kernel<<<(unsigned)((nw + 3) / 4), 128, 0, stream>>>(tau, nx, ny, nz, cnx, cny, cnz, cell);
    tau_brick_kernel<<<(unsigned)((nb + 3) / 4), 128, 0, stream>>>(tau, cell, nx, ny, nz, bnx, bny, bnz, cnx, cny, cnz,
                                                                  brick, block);
    return cudaGetLastError();
}

}  // namespace ctrex
