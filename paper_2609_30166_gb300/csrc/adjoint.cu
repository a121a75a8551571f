// adjoint.cu -- matched ray-driven adjoint A^T (exact transpose of the
// projector in project.cu, motion included) and the gradient of <g, A x> with
// respect to the motion parameters (chain rule through the pose and the
// B-spline warp; the deformation is recomputed per sample, never stored).
// The paper motivates geometry refinement and learned components (Sec. 5)
// but prints no such operator; both are the transpose / derivative of its
// Sec. 4.1 projector with the Sec. 2.2.2 / 3.1 warp.
#include "column.cuh"
#include "ray.cuh"

#include <type_traits>

namespace ctrex {

constexpr int ADJ_TX = 32, ADJ_TY = 4;
// Motion gradient CTA: four warps on 8 x 4 pixel patches side by side, which
// share the spline table and the CTA's partial sums; three CTAs per SM (168
// registers), by runs and sample by sample (45 views of the 256^3 motion
// workload: 40.4 and 94.7 ms; two warps, six CTAs: 50.5 and 106 ms).  The pose
// alone needs none of that: eight CTAs, sums in registers (60 views of 128^3
// 1.82 ms; in the spline's kernel with sums in shared memory 4.0).
constexpr int MG_WARPS = 4, MG_THREADS = 32 * MG_WARPS, MG_MIN_BLOCKS = 3, MG_POSE_BLOCKS = 8;
// Warps per CTA of the pose's kernels: a few views have too few CTAs of four
// (256 x 256 x 8, 12 views of 128 x 4 pixels, pose alone 0.38 -> 0.34 ms; 32^3, 60
// views, under a deformation 0.29 -> 0.25, by one 0.24 but 64^3 of half a voxel's
// pixels 3.66 for 3.49).
constexpr int MG_POSE_WARPS = 1, MG_WARPED_WARPS = 2;
// Samples per spline cell from which the gradient goes by runs.  60 views at
// 64^3 / 80^3 / 96^3 / 112^3 / 128^3 (26 / 32 / 38 / 45 / 51 samples), by
// samples: 4.8 / 7.7 / 11.1 / 16.3 / 22.1 ms, by runs: 4.9 / 6.8 / 8.8 / 11.8 /
// 14.5 ms; the pose's alone: 1.18 / 2.09 / 3.30 / 5.02 / 7.20 and 1.81 / 2.76 /
// 3.87 / 5.34 / 7.01 ms.
constexpr float MG_RUN_MIN = 30.0f, MG_RUN_MIN_POSE = 50.0f;
constexpr int NCOEF = 8 * 8 * 8 * 3;

// ---------------------------------------------------------------------------
// Adjoint: scatter y_i * w_k * trilinear weight into the 8 taps (FP32 atomics)
// ---------------------------------------------------------------------------

// Trilinear scatter of val at the point with centred index coordinates gc
// (index coordinates minus the integer grid centre c: floor and fraction are
// exact in them).  Each (y, z) row of the 2 x 2 x 2 footprint adds w0, w1 to
// the neighbours x0, x0 + 1, consecutive floats.  When both lie in one
// 16-byte-aligned quad of the volume (x0 % 4 != 3 in element terms; 3 cases
// in 4), one vector reduction adds (.., w0, w1, ..) with zeros in the other
// two lanes, so a footprint issues about 5 reductions instead of 8 (the
// reductions' L1/TEX path bounds the kernel).  The zero lanes belong to
// neighbouring voxels (possibly of the adjacent row) inside the volume;
// adding +0 leaves them unchanged.  vec: the volume is 16-byte aligned;
// nvox: its element count.
// A footprint waiting to be scattered: the lower corner (ix, iy, iz) in
// voxel indices and the summed weight of each of its eight taps.  A ray's
// samples lie half a voxel apart, so consecutive ones often share the
// corner: their weights are added here and reduced into the volume once,
// when the corner moves or the ray ends.
struct Footprint {
    int ix = 0, iy = 0, iz = 0;
    bool live = false;
    float w[2][2][2] = {{{0.f, 0.f}, {0.f, 0.f}}, {{0.f, 0.f}, {0.f, 0.f}}};
};

__device__ __forceinline__ void scatter_footprint(float *__restrict__ vol, int nx, int ny, int nz,
                                                  const Footprint &F, bool vec, long long nvox)
{
    const int ix = F.ix, iy = F.iy, iz = F.iz;
    const bool in0 = (unsigned)ix < (unsigned)nx, in1 = (unsigned)(ix + 1) < (unsigned)nx;
#pragma unroll
    for (int dz = 0; dz < 2; ++dz) {
        const int z = iz + dz;
        if ((unsigned)z >= (unsigned)nz) continue;
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const int y = iy + dy;
            if ((unsigned)y >= (unsigned)ny) continue;
            const long long e = ((long long)z * ny + y) * nx + ix;  // element of tap x0 (x0 may be -1)
            const float w0 = in0 ? F.w[dz][dy][0] : 0.0f, w1 = in1 ? F.w[dz][dy][1] : 0.0f;
            const int lane = (int)(e & 3);
            if (vec && lane != 3 && e >= 0 && (e | 3) < nvox) {
                float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (lane == 0) {
                    q.x = w0;
                    q.y = w1;
                } else if (lane == 1) {
                    q.y = w0;
                    q.z = w1;
                } else {
                    q.z = w0;
                    q.w = w1;
                }
                atomicAdd(reinterpret_cast<float4 *>(vol + (e - lane)), q);
            } else {
                if (in0) atomicAdd(vol + e, w0);
                if (in1) atomicAdd(vol + e + 1, w1);
            }
        }
    }
}

// Event-based 4D model (Sec. 3.3): the transpose sends each tap's share to
// mu0 (vol[j]) if the view's time t precedes the voxel's transition time
// tau_j, else to mu1 (vol[nvox + j]); scalar reductions.  The choice is the
// voxel's for the whole view, so merged weights route as their samples'.
__device__ __forceinline__ void scatter_footprint_dyrect(float *__restrict__ vol, int nx, int ny, int nz,
                                                         const Footprint &F, const float *__restrict__ tau, float t,
                                                         long long nvox)
{
#pragma unroll
    for (int dz = 0; dz < 2; ++dz) {
        const int z = F.iz + dz;
        if ((unsigned)z >= (unsigned)nz) continue;
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const int y = F.iy + dy;
            if ((unsigned)y >= (unsigned)ny) continue;
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) {
                const int x = F.ix + dx;
                if ((unsigned)x >= (unsigned)nx) continue;
                const long long j = ((long long)z * ny + y) * nx + x;
                atomicAdd(vol + (t < __ldg(tau + j) ? j : nvox + j), F.w[dz][dy][dx]);
            }
        }
    }
}

// Adds val at the point with centred index coordinates gc to the pending
// footprint F, first scattering F if the point's corner differs (DYR: into
// the event model's two fields, by tau and the view's time t).
template <bool DYR>
__device__ __forceinline__ void scatter_trilinear(float *__restrict__ vol, int nx, int ny, int nz, const float c[3],
                                                  const float gc[3], float val, bool vec, long long nvox,
                                                  Footprint &F, const float *__restrict__ tau, float t)
{
    const float fx = floorf(gc[0]), fy = floorf(gc[1]), fz = floorf(gc[2]);
    const int ix = (int)fx + (int)c[0], iy = (int)fy + (int)c[1], iz = (int)fz + (int)c[2];
    const float ax = gc[0] - fx, ay = gc[1] - fy, az = gc[2] - fz;
    const float wx[2] = {1.0f - ax, ax}, wy[2] = {1.0f - ay, ay}, wz[2] = {1.0f - az, az};
    if (F.live && (ix != F.ix || iy != F.iy || iz != F.iz)) {
        if (DYR)
            scatter_footprint_dyrect(vol, nx, ny, nz, F, tau, t, nvox);
        else
            scatter_footprint(vol, nx, ny, nz, F, vec, nvox);
        F.live = false;
    }
    if (!F.live) {
        F.ix = ix;
        F.iy = iy;
        F.iz = iz;
        F.live = true;
#pragma unroll
        for (int dz = 0; dz < 2; ++dz)
#pragma unroll
            for (int dy = 0; dy < 2; ++dy)
#pragma unroll
                for (int dx = 0; dx < 2; ++dx) F.w[dz][dy][dx] = 0.0f;
    }
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            const float wzy = val * wz[dz] * wy[dy];
            F.w[dz][dy][0] = fmaf(wzy, wx[0], F.w[dz][dy][0]);
            F.w[dz][dy][1] = fmaf(wzy, wx[1], F.w[dz][dy][1]);
        }
}

// SPLINE: motion with a deformation; MOTION alone: by the pose.
template <bool MOTION, bool SPLINE, bool DYR>
__global__ void __launch_bounds__(ADJ_TX *ADJ_TY)
    adjoint_kernel(Grid G, const ViewGPU *__restrict__ views, const MotionGPU *__restrict__ motion,
                   const float4 *spline, const int *__restrict__ view_idx,
                   const float *__restrict__ proj, float *__restrict__ vol, unsigned *devcheck,
                   const float *__restrict__ tau, const float *__restrict__ t_view)
{
    const int k = blockIdx.y;
    const int view = view_idx ? view_idx[k] : k;
    if (view < 0 || view >= G.n_views) {
        if (threadIdx.x == 0 && threadIdx.y == 0) atomicOr(devcheck, (unsigned)DEVCHECK_OOB);
        return;
    }
    MotionGPU mo;
    __shared__ float4 s_spline[SPLINE ? SPLINE_TABLE : 1];
    if (MOTION) mo = motion[view];
    if (SPLINE) {
        load_spline(s_spline, spline, threadIdx.y * ADJ_TX + threadIdx.x, ADJ_TX * ADJ_TY);
        spline = s_spline;
        __syncthreads();
    }
    int iu, iv;
    tile_pixel<MOTION>(blockIdx.x * ADJ_TX, blockIdx.z * ADJ_TY, iu, iv);
    if (iu >= G.nu || iv >= G.nv) return;
    const float y = proj[((size_t)k * G.nv + iv) * G.nu + iu] * G.inv_sub;
    if (y == 0.0f) return;
    const bool vec = (reinterpret_cast<uintptr_t>(vol) & 15) == 0;
    const long long nvox = (long long)G.nx * G.ny * G.nz;
    const float t = DYR ? __ldg(t_view + view) : 0.0f;
    float cen[3];
    grid_centre(G, cen);
    Footprint F;  // the pending footprint of this thread's samples
    for (int s = 0; s < G.n_sub; ++s) {
        Ray R;  // sample positions relative to the grid centre
        if (!setup_ray(G, views[view * G.n_sub + s], (float)iu, (float)iv, R, cen)) continue;
        float d0[3], ds[3];
        if (MOTION && !SPLINE) pose_line(mo, R, d0, ds);
        const float kl = last_kappa(G, R);
        for (int kk = 0; kk < R.K; kk += 2) {
            float g[2][3], w[2], gc[2][3];
            sample_pair(G, R, kk, g, w);
            if (SPLINE) {
                warp_pair_c(G, mo, spline, g, gc);
            } else if (MOTION) {
#pragma unroll
                for (int n = 0; n < 2; ++n)
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const float kap = kk + n >= R.K - 1 ? kl : (float)(kk + n);
                        gc[n][a] = g[n][a] + fmaf(kap, ds[a], d0[a]);
                    }
            }
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const float *q = MOTION ? gc[n] : g[n];
                if (w[n] > 0.0f && q[0] >= -1.0f - cen[0] && q[0] < (float)G.nx - cen[0] && q[1] >= -1.0f - cen[1] &&
                    q[1] < (float)G.ny - cen[1] && q[2] >= -1.0f - cen[2] && q[2] < (float)G.nz - cen[2])
                    scatter_trilinear<DYR>(vol, G.nx, G.ny, G.nz, cen, q, y * w[n], vec, nvox, F, tau, t);
            }
        }
    }
    if (F.live) {
        if (DYR)
            scatter_footprint_dyrect(vol, G.nx, G.ny, G.nz, F, tau, t, nvox);
        else
            scatter_footprint(vol, G.nx, G.ny, G.nz, F, vec, nvox);
    }
}

cudaError_t launch_adjoint(const FwdArgs &a, const float *proj, float *vol)
{
    if (a.n_idx == 0) return cudaSuccess;
    const Grid &G = *a.grid;
    const dim3 grid((G.nu + ADJ_TX - 1) / ADJ_TX, a.n_idx, (G.nv + ADJ_TY - 1) / ADJ_TY);
    const dim3 block(ADJ_TX, ADJ_TY);
    if (a.dyr && a.motion) return cudaErrorInvalidValue;  // the event model is defined without motion
    if (a.motion && !a.spline)
        adjoint_kernel<true, false, false><<<grid, block, 0, a.stream>>>(G, a.views, a.motion, nullptr, a.view_idx, proj,
                                                                        vol, a.devcheck, nullptr, nullptr);
    else if (a.motion)
        adjoint_kernel<true, true, false><<<grid, block, 0, a.stream>>>(G, a.views, a.motion, a.spline, a.view_idx,
                                                                 proj, vol, a.devcheck, nullptr, nullptr);
    else if (a.dyr)
        adjoint_kernel<false, false, true><<<grid, block, 0, a.stream>>>(G, a.views, nullptr, nullptr, a.view_idx, proj,
                                                                 vol, a.devcheck, a.dyr->tau, a.dyr->t_view);
    else
        adjoint_kernel<false, false, false><<<grid, block, 0, a.stream>>>(G, a.views, nullptr, nullptr, a.view_idx, proj,
                                                                  vol, a.devcheck, nullptr, nullptr);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Motion gradient
// ---------------------------------------------------------------------------
//
// dL/dtheta and dL/dcoef of L = <g, A x> (chain rule of the Sec. 4.1
// projector through the Sec. 2.2.2 pose and the Sec. 3.1 warp).  Per sample
// k of ray i, with y = g' + s u(g'), g' = M g + b:
//   dL/dy  = g_i w_k grad mu(y)                 (trilinear gradient, index units)
//   dL/dg' = dL/dy (I + s du/dg')               -> dL/db += dL/dg', dL/dM += dL/dg' g^T
//   dL/dc_ijk[c] += s dL/dy[c] beta(xi - i) beta(eta - j) beta(zeta - k)
// Sample positions, the warp and the pose sums are formed relative to the
// integer grid centre c (as in the adjoint): dL/dM = sum dL/dg' (g - c)^T +
// (sum dL/dg') c^T, the last term added in FP64 by the finish kernel.

// Zero-padded trilinear interpolant's gradient (index units) inside the cell
// floor(y), at the point with centred index coordinates yc = y - c (floor and
// fraction exact in them).
template <typename TV>
__device__ __forceinline__ void trilinear_grad_c(const TV *__restrict__ vol, int nx, int ny, int nz, const float c[3],
                                                 const float yc[3], float grad[3])
{
    const float fx = floorf(yc[0]), fy = floorf(yc[1]), fz = floorf(yc[2]);
    const int ix = (int)fx + (int)c[0], iy = (int)fy + (int)c[1], iz = (int)fz + (int)c[2];
    const float ax = yc[0] - fx, ay = yc[1] - fy, az = yc[2] - fz;
    float v[2][2][2];
#pragma unroll
    for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int dy = 0; dy < 2; ++dy)
#pragma unroll
            for (int dx = 0; dx < 2; ++dx) {
                const int x = ix + dx, y = iy + dy, z = iz + dz;
                const bool in = (unsigned)x < (unsigned)nx && (unsigned)y < (unsigned)ny && (unsigned)z < (unsigned)nz;
                v[dz][dy][dx] = in ? Storage<TV>::load(vol + ((long long)z * ny + y) * nx + x) : 0.0f;
            }
    const float by0 = 1.0f - ay, bz0 = 1.0f - az, bx0 = 1.0f - ax;
    grad[0] = bz0 * (by0 * (v[0][0][1] - v[0][0][0]) + ay * (v[0][1][1] - v[0][1][0])) +
              az * (by0 * (v[1][0][1] - v[1][0][0]) + ay * (v[1][1][1] - v[1][1][0]));
    grad[1] = bz0 * (bx0 * (v[0][1][0] - v[0][0][0]) + ax * (v[0][1][1] - v[0][0][1])) +
              az * (bx0 * (v[1][1][0] - v[1][0][0]) + ax * (v[1][1][1] - v[1][0][1]));
    grad[2] = by0 * (bx0 * (v[1][0][0] - v[0][0][0]) + ax * (v[1][0][1] - v[0][0][1])) +
              ay * (bx0 * (v[1][1][0] - v[0][1][0]) + ax * (v[1][1][1] - v[0][1][1]));
}

// Displacement u and its derivatives with respect to the three spline
// coordinates at fractions f of the cell at `c`: the x polynomials and their
// derivatives, then the weighted sums over y and z.
__device__ __forceinline__ void spline_value_jacobian(const float4 *c, const float f[3], float u[3], float Jx[3],
                                                      float Jy[3], float Jz[3])
{
    float wy[4], wz[4], ey[4], ez[4];
    bspline_weights(f[1], wy);
    bspline_weights(f[2], wz);
    bspline_dweights(f[1], ey);
    bspline_dweights(f[2], ez);
    // the x and y components packed, z beside them
    float2 U = two(0.f), X = two(0.f), Y = two(0.f), Z = two(0.f);
    float uz = 0.f, xz = 0.f, yz = 0.f, zz = 0.f;
    const float2 fx = two(f[0]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float wk = wz[k], ek = ez[k];
        float2 v = two(0.f), dx = two(0.f), dy = two(0.f);
        float vz = 0.f, dxz = 0.f, dyz = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 *row = c + k * SPL_PLANE + j * SPL_ROW;
            const float4 c3 = row[3], c2 = row[2], c1 = row[1], c0 = row[0];
            // q0: the polynomial, d: its derivative
            const float2 p3 = make_float2(c3.x, c3.y);
            const float2 q2 = __ffma2_rn(fx, p3, make_float2(c2.x, c2.y));
            const float2 q1 = __ffma2_rn(fx, q2, make_float2(c1.x, c1.y));
            const float2 q0 = __ffma2_rn(fx, q1, make_float2(c0.x, c0.y));
            const float2 d = __ffma2_rn(fx, __ffma2_rn(fx, p3, q2), q1);
            v = __ffma2_rn(two(wy[j]), q0, v);
            dx = __ffma2_rn(two(wy[j]), d, dx);
            dy = __ffma2_rn(two(ey[j]), q0, dy);
            const float z2 = fmaf(f[0], c3.z, c2.z), z1 = fmaf(f[0], z2, c1.z), z0 = fmaf(f[0], z1, c0.z);
            const float dz = fmaf(f[0], fmaf(f[0], c3.z, z2), z1);
            vz = fmaf(wy[j], z0, vz);
            dxz = fmaf(wy[j], dz, dxz);
            dyz = fmaf(ey[j], z0, dyz);
        }
        U = __ffma2_rn(two(wk), v, U);
        X = __ffma2_rn(two(wk), dx, X);
        Y = __ffma2_rn(two(wk), dy, Y);
        Z = __ffma2_rn(two(ek), v, Z);
        uz = fmaf(wk, vz, uz);
        xz = fmaf(wk, dxz, xz);
        yz = fmaf(wk, dyz, yz);
        zz = fmaf(ek, vz, zz);
    }
    u[0] = U.x, u[1] = U.y, u[2] = uz;
    Jx[0] = X.x, Jx[1] = X.y, Jx[2] = xz;
    Jy[0] = Y.x, Jy[1] = Y.y, Jy[2] = yz;
    Jz[0] = Z.x, Jz[1] = Z.y, Jz[2] = zz;
}

// --- coefficient gradient on the tensor cores --------------------------------
//
// Over the samples s of a warp that share one spline cell, the coefficient
// gradient of that cell is an outer-product sum
//   G[(c, kz)][(j, i)] = sum_s  (v_s[c] wz_s[kz]) (wy_s[j] wx_s[i]),
// v_s = s_view dL/dy_s: a 12 x 16 matrix = A (12 x samples) B (samples x 16),
// i.e. a GEMM with K = samples.  One warp step (32 samples) is 4 k-chunks of
// mma.m16n8k8 (TF32) per 8-column half of G, with rows 12..15 zero.  FP32
// accuracy comes from the 3-term split x = hi + lo (hi = tf32(x), lo =
// tf32(x - hi)): A B ~ Alo Bhi + Ahi Blo + Ahi Bhi, each product within about
// 3 * 2^-22 of the FP32 one.  A step's MMAs start from zero (a chain of 12
// k-steps), and its result is added to FP32 register sums of the warp's
// current cell; those go to the CTA's FP64 shared partials (atomics, once per
// change of cell) and, at the end, to FP64 global sums.
//
// Fragment layouts of mma.m16n8k8 .tf32 (g = lane / 4, t = lane % 4):
//   A (row-major 16 x 8): a0 (g, t), a1 (g + 8, t), a2 (g, t + 4), a3 (g + 8, t + 4)
//   B (col-major 8 x 8):  b0 (k = t, n = g), b1 (k = t + 4, n = g)
//   C/D (16 x 8):         d0 (g, 2t), d1 (g, 2t + 1), d2 (g + 8, 2t), d3 (g + 8, 2t + 1)
// With k = sample, lane (g, t) needs samples t and t + 4 of each chunk: it
// reads their spline fractions and v by shuffles and evaluates the B-spline
// basis functions its rows / columns need (kz = i = g % 4, j = g / 4 for the
// first half of G, 2 + g / 4 for the second) itself.

__device__ __forceinline__ unsigned tf32_bits(float x)
{
    unsigned r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// x = hi + lo as two TF32 values.
__device__ __forceinline__ void tf32_split(float x, unsigned &hi, unsigned &lo)
{
    hi = tf32_bits(x);
    lo = tf32_bits(x - __uint_as_float(hi));
}

__device__ __forceinline__ void mma_tf32_16x8x8(float d[4], const unsigned a[4], unsigned b0, unsigned b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float horner(const float4 p, float f)
{
    return fmaf(fmaf(fmaf(p.w, f, p.z), f, p.y), f, p.x);
}

// The warp's coefficient-gradient state: FP32 sums of the current cell's
// 12 x 16 block in fragment layout (two 8-column halves).
struct CoefAcc {
    float acc[2][4];
    int cell;  // packed i0 of the current cell, -1 for none (warp-uniform)
};

// Adds the sums of acc's cell to the CTA's FP64 partials and clears them.
__device__ __forceinline__ void coef_flush(CoefAcc &A, double *s_g64, int lane)
{
    if (A.cell >= 0) {
        const int i0x = A.cell & 7, i0y = (A.cell >> 3) & 7, i0z = A.cell >> 6;
        const int g = lane >> 2, t = lane & 3;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int row = g + 8 * (q >> 1), col = 8 * h + 2 * t + (q & 1);
                const float v = A.acc[h][q];
                A.acc[h][q] = 0.0f;
                if (row >= 12 || v == 0.0f) continue;
                const int comp = row >> 2, kz = row & 3, j = col >> 2, i = col & 3;
                const int cx = i0x + i, cy = i0y + j, cz = i0z + kz;
                atomicAdd(s_g64 + 3 * ((cz * 8 + cy) * 8 + cx) + comp, (double)v);
            }
    }
}

// One warp step of the coefficient gradient.  Per lane: cell = packed i0 of
// its sample, f = spline fractions, v = s_view dL/dy (zero when the lane has
// no contribution), live = whether it has one.  Warp-collective.
__device__ __forceinline__ void coef_step(CoefAcc &A, double *s_g64, int cell, const float f[3], const float v[3],
                                          bool live, const float4 *s_piece)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    // the B-spline pieces of this lane's rows and columns
    const float4 pz = s_piece[g & 3], px = pz, py0 = s_piece[g >> 2], py1 = s_piece[2 + (g >> 2)];
    unsigned pending = __ballot_sync(full, live);
    while (pending) {  // warp-uniform: one round per distinct cell of this step
        const int leader = __ffs(pending) - 1;
        const int lcell = __shfl_sync(full, cell, leader);
        const bool mine = ((pending >> lane) & 1u) && cell == lcell;
        const unsigned who = __ballot_sync(full, mine);
        if (lcell != A.cell) {
            coef_flush(A, s_g64, lane);
            A.cell = lcell;
        }
        const float pv0 = mine ? v[0] : 0.0f, pv1 = mine ? v[1] : 0.0f, pv2 = mine ? v[2] : 0.0f;
        const float pfx = mine ? f[0] : 0.0f, pfy = mine ? f[1] : 0.0f, pfz = mine ? f[2] : 0.0f;
        float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
            if (!((who >> (8 * q)) & 0xffu)) continue;  // warp-uniform: no sample of this chunk
            float a[4], b[2][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int src = 8 * q + t + 4 * h;
                const float fx = __shfl_sync(full, pfx, src), fy = __shfl_sync(full, pfy, src),
                            fz = __shfl_sync(full, pfz, src);
                const float x0 = __shfl_sync(full, pv0, src), x1 = __shfl_sync(full, pv1, src),
                            x2 = __shfl_sync(full, pv2, src);
                const float wz = horner(pz, fz), wx = horner(px, fx);
                a[2 * h] = (g < 4 ? x0 : x1) * wz;        // row g:     c = g / 4, kz = g % 4
                a[2 * h + 1] = g < 4 ? x2 * wz : 0.0f;    // row g + 8: c = 2 (rows 12..15 zero)
                b[0][h] = horner(py0, fy) * wx;           // column g of half 0: j = g / 4, i = g % 4
                b[1][h] = horner(py1, fy) * wx;           // column g of half 1: j = 2 + g / 4
            }
            unsigned ah[4], al[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) tf32_split(a[e], ah[e], al[e]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                unsigned bh0, bl0, bh1, bl1;
                tf32_split(b[h][0], bh0, bl0);
                tf32_split(b[h][1], bh1, bl1);
                mma_tf32_16x8x8(d[h], al, bh0, bh1);
                mma_tf32_16x8x8(d[h], ah, bl0, bl1);
                mma_tf32_16x8x8(d[h], ah, bh0, bh1);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 4; ++e) A.acc[h][e] += d[h][e];
        pending &= ~who;
    }
}

// The volume's trilinear gradient at centred index coordinates yc (zero
// outside the grid), from row-major memory or from a column store.
template <typename TV> struct RowVolume {
    const TV *p;
    __device__ __forceinline__ void gradient(const Grid &G, const float c[3], const float yc[3], float g[3]) const
    {
        trilinear_grad_c(p, G.nx, G.ny, G.nz, c, yc, g);
    }
};
struct ColumnVolume {
    ColVolume V;
    __device__ __forceinline__ void gradient(const Grid &, const float c[3], const float yc[3], float g[3]) const
    {
        const float fx = floorf(yc[0]), fy = floorf(yc[1]), fz = floorf(yc[2]);
        const ColTaps t = col_load(V, V.index((int)fx + (int)c[0] + 1, (int)fy + (int)c[1] + 1, (int)fz + (int)c[2] + 1));
        const float ax = yc[0] - fx, ay = yc[1] - fy, az = yc[2] - fz;
        const float a = col_value(t.q00, az), b = col_value(t.q10, az), d = col_value(t.q01, az),
                    e = col_value(t.q11, az);
        const float dx0 = b - a, dx1 = e - d;
        g[0] = lerp(dx0, dx1, ay);
        g[1] = fmaf(ax, dx1, d) - fmaf(ax, dx0, a);
        g[2] = lerp(lerp(t.q00.y, t.q10.y, ax), lerp(t.q01.y, t.q11.y, ax), ay);
    }
};

// Per ray, the samples of each run in one spline cell are reduced to 10: the
// coefficient gradient sums v(t) times polynomials of degree 9 over the run's
// samples, and so do the pose sums (J^T v times a linear position), so the
// Chebyshev moments C_j = sum v(t) T_j(t) of the samples' v = dL/dy determine
// them, and the run's samples may be replaced by the 10 nodes with
//   V_n = 1/10 (C_0 + 2 sum_{j > 0} T_j(tau_n) C_j).
// Only the displacement (by its Chebyshev form), the volume's gradient and
// the moments are left per sample; the spline's Jacobian and the tensor-core
// step run per node.  45 views of the 256^3 motion workload: sample by sample
// with the volume row-major 104.3 ms (spline loads and the tensor-core step's
// shuffles), from the columns 94.7, by runs 40.4 (pose only 60.3, 42.6, 25.1).
// What a launch has to form: MG_POSE: no deformation; MG_WARPED: the pose's
// gradient under a deformation; MG_SAMPLES: the coefficients' too, sample by
// sample (short runs, MG_RUN_MIN); MG_RUNS: either of the last two, as above.
enum MotionGradKind { MG_POSE, MG_WARPED, MG_SAMPLES, MG_RUNS };

template <typename Volume, int KIND, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, (KIND == MG_POSE ? MG_POSE_BLOCKS : MG_MIN_BLOCKS) * MG_WARPS / WARPS)
    motion_grad_kernel(Grid G, const ViewGPU *__restrict__ views, const MotionGPU *__restrict__ motion,
                       const float4 *table, const int *__restrict__ view_idx, const Volume vol,
                       const float *__restrict__ gproj, double *__restrict__ grad_M, double *__restrict__ grad_b,
                       double *__restrict__ grad_coef, unsigned *devcheck)
{
    constexpr int THREADS = 32 * WARPS;
    constexpr bool RUNS = KIND == MG_RUNS, COEF = KIND == MG_SAMPLES || RUNS;
    __shared__ float4 s_spline[KIND == MG_POSE ? 1 : SPLINE_TABLE];
    __shared__ double s_g64[COEF ? NCOEF : 1];  // the CTA's coefficient-gradient partials
    __shared__ double s_red[12][WARPS];
    __shared__ float4 s_piece[4];
    __shared__ float s_pose[COEF ? 12 : 1][THREADS];
    extern __shared__ float s_V[][MG_THREADS];  // RUNS: the nodes' dL/dy of each thread's run, 3 CHEB_N
    const int tid = threadIdx.y * 32 + threadIdx.x;
    const int lane = tid & 31;
    const int k = blockIdx.y;
    const int view = view_idx ? view_idx[k] : k;
    if (!(view >= 0 && view < G.n_views)) {
        if (tid == 0) atomicOr(devcheck, (unsigned)DEVCHECK_OOB);
        return;  // uniform over the CTA
    }
    const float mos = motion[view].s;
    const bool spline = KIND != MG_POSE && mos != 0.0f;
    const bool want_coef = COEF && spline && grad_coef != nullptr;
    if (spline) load_spline(s_spline, table, tid, THREADS);
    if (want_coef)
        for (int i = tid; i < NCOEF; i += THREADS) s_g64[i] = 0.0;
    if (COEF && tid < 4) s_piece[tid] = bspline_piece(tid);
    __syncthreads();
    float cen[3];
    grid_centre(G, cen);
    CoefAcc CA;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) CA.acc[h][e] = 0.0f;
    CA.cell = -1;
    // this thread's 12 pose sums (9 of dL/dM, 3 of dL/db): in registers, or in
    // shared memory beside the coefficients' sums
    float pose_reg[12];
#pragma unroll
    for (int q = 0; q < 12; ++q) {
        pose_reg[q] = 0.0f;
        if (COEF) s_pose[q][tid] = 0.0f;
    }
    auto pose_add = [&](int q, float a, float b) {
        if (COEF)
            s_pose[q][tid] = fmaf(a, b, s_pose[q][tid]);
        else
            pose_reg[q] = fmaf(a, b, pose_reg[q]);
    };
    int iu, iv;
    tile_pixel<true>(blockIdx.x * 8 * WARPS, blockIdx.z * 4, iu, iv);
    const bool pix_ok = iu < G.nu && iv < G.nv;
    const float y = pix_ok ? gproj[((size_t)k * G.nv + iv) * G.nu + iu] * G.inv_sub : 0.0f;
    for (int s = 0; s < G.n_sub; ++s) {
        Ray R;  // sample positions relative to the grid centre
        const bool hit = pix_ok && setup_ray(G, views[view * G.n_sub + s], (float)(pix_ok ? iu : 0),
                                             (float)(pix_ok ? iv : 0), R, cen);
        const int K = hit && y != 0.0f ? R.K : 0;
        // displacement by the pose at sample index kappa: d = D g + bc, linear
        float d0[3], ds[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float *D = motion[view].D + 3 * r;
            d0[r] = fmaf(D[0], R.g0[0], fmaf(D[1], R.g0[1], fmaf(D[2], R.g0[2], motion[view].bc[r])));
            ds[r] = fmaf(D[0], R.sg[0], fmaf(D[1], R.sg[1], D[2] * R.sg[2]));
        }
        const float kl = last_kappa(G, R);
        // dL/dy of one sample with spline displacement u (voxels)
        auto sample = [&](int kk, const float u[3], float g[3]) {
            const bool last = kk == K - 1;
            const float kap = last ? kl : (float)kk, w = last ? fmaxf(R.w_last, 0.0f) : G.step_mm;
            float yc[3];
#pragma unroll
            for (int r = 0; r < 3; ++r)
                yc[r] = fmaf(kap, R.sg[r], R.g0[r]) + fmaf(mos, u[r], fmaf(kap, ds[r], d0[r]));
            g[0] = g[1] = g[2] = 0.0f;
            if (w > 0.0f && yc[0] >= -1.0f - cen[0] && yc[0] < (float)G.nx - cen[0] && yc[1] >= -1.0f - cen[1] &&
                yc[1] < (float)G.ny - cen[1] && yc[2] >= -1.0f - cen[2] && yc[2] < (float)G.nz - cen[2])
                vol.gradient(G, cen, yc, g);
#pragma unroll
            for (int c = 0; c < 3; ++c) g[c] *= y * w;
        };
        auto pose = [&](float kap, const float gg[3]) {
            float gc[3];
#pragma unroll
            for (int r = 0; r < 3; ++r) gc[r] = fmaf(kap, R.sg[r], R.g0[r]);
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                pose_add(9 + r, gg[r], 1.0f);
#pragma unroll
                for (int c = 0; c < 3; ++c) pose_add(3 * r + c, gg[r], gc[c]);
            }
        };
        // pose sums of dL/dy = gy at kappa: dL/dg' = dL/dy (I + s J), J[c][a] =
        // du_c / dg'_a
        auto point = [&](float kap, const float gy[3], const bool on[3], const float Jx[3], const float Jy[3],
                         const float Jz[3]) {
            const float sx = on[0] ? mos * G.spl_scale[0] : 0.f, sy = on[1] ? mos * G.spl_scale[1] : 0.f,
                        sz = on[2] ? mos * G.spl_scale[2] : 0.f;
            const float gg[3] = {fmaf(sx, gy[0] * Jx[0] + gy[1] * Jx[1] + gy[2] * Jx[2], gy[0]),
                                 fmaf(sy, gy[0] * Jy[0] + gy[1] * Jy[1] + gy[2] * Jy[2], gy[1]),
                                 fmaf(sz, gy[0] * Jz[0] + gy[1] * Jz[1] + gy[2] * Jz[2], gy[2])};
            pose(kap, gg);
        };
        if (!spline) {  // CTA-uniform: the pose alone
            // the ray's sums of dL/dy and of dL/dy (kappa - mid): the position
            // is linear in kappa
            const float u[3] = {0.f, 0.f, 0.f}, mid = 0.5f * kl;
            float S[3] = {0.f, 0.f, 0.f}, S1[3] = {0.f, 0.f, 0.f};
            for (int kk = 0; kk < K; ++kk) {
                float g[3];
                sample(kk, u, g);
                const float t = (kk == K - 1 ? kl : (float)kk) - mid;
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    S[r] += g[r];
                    S1[r] = fmaf(t, g[r], S1[r]);
                }
            }
            if (K > 0)
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    pose_add(9 + r, S[r], 1.0f);
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        pose_add(3 * r + c, S[r], fmaf(mid, R.sg[c], R.g0[c]));
                        pose_add(3 * r + c, S1[r], R.sg[c]);
                    }
                }
            continue;
        }
        if constexpr (KIND != MG_POSE) {
        SplineLine L;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            L.x0[a] = fmaf(R.g0[a] + d0[a] + cen[a] + 0.5f, G.spl_scale[a], 1.0f);
            L.xs[a] = (R.sg[a] + ds[a]) * G.spl_scale[a];
        }
        if constexpr (!RUNS) {
            // the coefficient step is collective: lanes without work run the
            // loop with zero weight up to the warp's longest ray
            int Kmax = K;
            if (COEF)
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) Kmax = max(Kmax, __shfl_xor_sync(0xffffffffu, Kmax, off));
            for (int kk = 0; kk < Kmax; ++kk) {
                const float kap = kk == K - 1 ? kl : (float)kk;
                int i0[3];
                float f[3], u[3], Jx[3], Jy[3], Jz[3], gy[3] = {0.f, 0.f, 0.f};
                bool on[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) spline_cell_of(fmaf(kap, L.xs[a], L.x0[a]), i0[a], f[a], on[a]);
                spline_value_jacobian(spline_cell(s_spline, i0), f, u, Jx, Jy, Jz);
                if (kk < K) {
                    sample(kk, u, gy);
                    point(kap, gy, on, Jx, Jy, Jz);
                }
                if (COEF && want_coef) {  // CTA-uniform
                    const float v[3] = {mos * gy[0], mos * gy[1], mos * gy[2]};
                    coef_step(CA, s_g64, (i0[2] * 8 + i0[1]) * 8 + i0[0], f, v,
                              kk < K && (v[0] != 0.0f || v[1] != 0.0f || v[2] != 0.0f), s_piece);
                }
            }
            continue;
        }
        // run after run, the warp together (the coefficient step is collective)
        int k = 0;
        while (__any_sync(0xffffffffu, k < K)) {
            SplineRun run;
            const bool act = k < K;
            const int end = run.find(L, act ? k : 0, act ? K : 1, kl);
            if (act) {
                float2 Cxy[CHEB_N], axy[CHEB_N];
                float Cz[CHEB_N], az[CHEB_N];
                run.fit(s_spline, L, axy, az);
#pragma unroll
                for (int j = 0; j < CHEB_N; ++j) {
                    Cxy[j] = two(0.0f);
                    Cz[j] = 0.0f;
                }
                const float ih = 1.0f / run.half;
                for (int kk = k; kk < end; ++kk) {
                    float T[CHEB_N], u[3], g[3];
                    cheb_values(((kk == K - 1 ? kl : (float)kk) - run.mid) * ih, T);
                    SplineRun::value(axy, az, T, u);
                    sample(kk, u, g);
                    const float2 gxy = make_float2(g[0], g[1]);
#pragma unroll
                    for (int j = 0; j < CHEB_N; ++j) {
                        Cxy[j] = __ffma2_rn(two(T[j]), gxy, Cxy[j]);
                        Cz[j] = fmaf(T[j], g[2], Cz[j]);
                    }
                }
                k = end;
                // the nodes' V: even moments count alike at +-tau, odd ones
                // with opposite signs
#pragma unroll
                for (int n = 0; n < CHEB_N / 2; ++n) {
                    float2 e = two(0.0f), o = two(0.0f);
                    float ez = 0.0f, oz = 0.0f;
#pragma unroll
                    for (int j = 0; j < CHEB_N; ++j) {
                        const float w = cheb_cos20(j * (2 * n + 1)) * (j == 0 ? 0.1f : 0.2f);
                        if (j & 1) {
                            o = __ffma2_rn(two(w), Cxy[j], o);
                            oz = fmaf(w, Cz[j], oz);
                        } else {
                            e = __ffma2_rn(two(w), Cxy[j], e);
                            ez = fmaf(w, Cz[j], ez);
                        }
                    }
                    s_V[3 * n][tid] = e.x + o.x;
                    s_V[3 * n + 1][tid] = e.y + o.y;
                    s_V[3 * n + 2][tid] = ez + oz;
                    s_V[3 * (CHEB_N - 1 - n)][tid] = e.x - o.x;
                    s_V[3 * (CHEB_N - 1 - n) + 1][tid] = e.y - o.y;
                    s_V[3 * (CHEB_N - 1 - n) + 2][tid] = ez - oz;
                }
            }
            const int cell = (run.cell[2] * 8 + run.cell[1]) * 8 + run.cell[0];
            const float4 *cc = spline_cell(s_spline, run.cell);
#pragma unroll 1
            for (int n = 0; n < CHEB_N; ++n) {
                const int m = n < CHEB_N / 2 ? n : CHEB_N - 1 - n;
                const float sign = n < CHEB_N / 2 ? 1.0f : -1.0f;
                float gy[3] = {0.f, 0.f, 0.f};
                if (act) {
                    gy[0] = s_V[3 * n][tid];
                    gy[1] = s_V[3 * n + 1][tid];
                    gy[2] = s_V[3 * n + 2][tid];
                }
                const float kap = fmaf(sign * c_cheb.t[m][1], run.half, run.mid);
                float f[3], u[3], Jx[3], Jy[3], Jz[3];
                run.fraction(L, kap, f);
                spline_value_jacobian(cc, f, u, Jx, Jy, Jz);
                if (act) point(kap, gy, run.on, Jx, Jy, Jz);
                if (want_coef) {  // CTA-uniform
                    const float v[3] = {mos * gy[0], mos * gy[1], mos * gy[2]};
                    coef_step(CA, s_g64, cell, f, v, act && (v[0] != 0.0f || v[1] != 0.0f || v[2] != 0.0f), s_piece);
                }
            }
        }
        }
    }
    if (want_coef) coef_flush(CA, s_g64, lane);
    // CTA reduction of the 12 pose-gradient entries: FP32 warp sums, FP64 over
    // the warps and across CTAs
#pragma unroll
    for (int q = 0; q < 12; ++q) {
        float v = COEF ? s_pose[q][tid] : pose_reg[q];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) s_red[q][tid >> 5] = (double)v;
    }
    __syncthreads();
    if (tid < 12) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) v += s_red[tid][w];
        if (grad_M && tid < 9) atomicAdd(grad_M + 9 * view + tid, v);
        if (grad_b && tid >= 9) atomicAdd(grad_b + 3 * view + (tid - 9), v);
    }
    if (want_coef) {
        for (int i = tid; i < NCOEF; i += THREADS) {
            const double v = s_g64[i];
            if (v != 0.0) atomicAdd(grad_coef + i, v);
        }
    }
}

cudaError_t launch_motion_grad(const FwdArgs &a, const float *gproj, double *grad_M, double *grad_b,
                               double *grad_coef_idx)
{
    if (a.n_idx == 0) return cudaSuccess;
    const Grid &G = *a.grid;
    const bool runs = a.spline && spline_runs(G, grad_coef_idx ? MG_RUN_MIN : MG_RUN_MIN_POSE);
    const int warps = !a.spline ? MG_POSE_WARPS : runs || grad_coef_idx ? MG_WARPS : MG_WARPED_WARPS;
    const dim3 grid((G.nu + 8 * warps - 1) / (8 * warps), a.n_idx, (G.nv + 3) / 4);
    const dim3 block(32, warps);
    cudaError_t err = cudaSuccess;
    auto launch = [&](const auto &vol) {
        typedef std::decay_t<decltype(vol)> V;
        auto *kernel = !a.spline       ? motion_grad_kernel<V, MG_POSE, MG_POSE_WARPS>
                       : runs          ? motion_grad_kernel<V, MG_RUNS, MG_WARPS>
                       : grad_coef_idx ? motion_grad_kernel<V, MG_SAMPLES, MG_WARPS>
                                       : motion_grad_kernel<V, MG_WARPED, MG_WARPED_WARPS>;
        const int nodes = runs ? 3 * CHEB_N * MG_THREADS * (int)sizeof(float) : 0;  // 53 KB with the static part
        if (runs) err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, nodes);
        if (err != cudaSuccess) return;
        kernel<<<grid, block, nodes, a.stream>>>(G, a.views, a.motion, a.spline, a.view_idx, vol, gproj, grad_M,
                                                 grad_b, grad_coef_idx, a.devcheck);
        err = cudaGetLastError();
    };
    if (a.column)
        launch(ColumnVolume{col_view(*a.column)});
    else if (a.vol_dtype == CTREX_F32)
        launch(RowVolume<float>{static_cast<const float *>(a.vol)});
    else
        launch(RowVolume<__nv_bfloat16>{static_cast<const __nv_bfloat16 *>(a.vol)});
    return err;
}

// ---------------------------------------------------------------------------
// Per-view motion set-up and the final chain rule to (omega, t, A, coef)
// ---------------------------------------------------------------------------

struct Frame {
    double vox[3];
    double origin[3];
    double cen[3];  // integer grid centre floor((n - 1) / 2) per axis (index coordinates)
};

// Rodrigues R = I + a K + b K^2 and dR/domega_i (FP64, one thread per view).
__device__ void rodrigues(const double w[3], double R[9], double dR[27])
{
    const double th = sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
    double a, b, dat, dbt;
    if (th < 1e-4) {
        const double t2 = th * th;
        a = 1.0 - t2 / 6.0 + t2 * t2 / 120.0;
        b = 0.5 - t2 / 24.0 + t2 * t2 / 720.0;
        dat = -1.0 / 3.0 + t2 / 30.0;
        dbt = -1.0 / 12.0 + t2 / 180.0;
    } else {
        const double s = sin(th), c = cos(th);
        a = s / th;
        b = (1.0 - c) / (th * th);
        dat = (th * c - s) / (th * th * th);
        dbt = (th * s - 2.0 * (1.0 - c)) / (th * th * th * th);
    }
    const double K[9] = {0, -w[2], w[1], w[2], 0, -w[0], -w[1], w[0], 0};
    double K2[9];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) K2[3 * r + c] = K[3 * r] * K[c] + K[3 * r + 1] * K[3 + c] + K[3 * r + 2] * K[6 + c];
    for (int q = 0; q < 9; ++q) R[q] = (q % 4 == 0 ? 1.0 : 0.0) + a * K[q] + b * K2[q];
    for (int i = 0; i < 3; ++i) {
        double E[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        if (i == 0) { E[5] = -1; E[7] = 1; }
        if (i == 1) { E[2] = 1; E[6] = -1; }
        if (i == 2) { E[1] = -1; E[3] = 1; }
        for (int r = 0; r < 3; ++r)
            for (int c = 0; c < 3; ++c) {
                double ek = 0.0, ke = 0.0;
                for (int q = 0; q < 3; ++q) {
                    ek += E[3 * r + q] * K[3 * q + c];
                    ke += K[3 * r + q] * E[3 * q + c];
                }
                dR[9 * i + 3 * r + c] = dat * w[i] * K[3 * r + c] + a * E[3 * r + c] +
                                        dbt * w[i] * K2[3 * r + c] + b * (ek + ke);
            }
    }
}

__global__ void motion_setup_kernel(const float *__restrict__ theta, const float *__restrict__ s_view,
                                    int n_views, Frame F, MotionGPU *__restrict__ motion,
                                    float *__restrict__ dRdw)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n_views) return;
    double R[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1}, dR[27] = {0}, A[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};
    double t[3] = {0, 0, 0};
    if (theta) {
        const double w[3] = {theta[15 * v], theta[15 * v + 1], theta[15 * v + 2]};
        rodrigues(w, R, dR);
        for (int q = 0; q < 3; ++q) t[q] = theta[15 * v + 3 + q];
        for (int q = 0; q < 9; ++q) A[q] = theta[15 * v + 6 + q];
    }
    // world map x' = Mw x + bw with Mw = A R, bw = A t
    double Mw[9], bw[3];
    for (int r = 0; r < 3; ++r) {
        for (int c = 0; c < 3; ++c) Mw[3 * r + c] = A[3 * r] * R[c] + A[3 * r + 1] * R[3 + c] + A[3 * r + 2] * R[6 + c];
        bw[r] = A[3 * r] * t[0] + A[3 * r + 1] * t[1] + A[3 * r + 2] * t[2];
    }
    // index map g' = M g + b: M = diag(1/vox) Mw diag(vox), b = (Mw o + bw - o) / vox
    MotionGPU m;
    for (int r = 0; r < 3; ++r) {
        double acc = bw[r] - F.origin[r];
        for (int c = 0; c < 3; ++c) {
            m.M[3 * r + c] = (float)(Mw[3 * r + c] * F.vox[c] / F.vox[r]);
            acc += Mw[3 * r + c] * F.origin[c];
        }
        const double b = acc / F.vox[r];
        m.b[r] = (float)b;
        double bc = b;
        for (int c = 0; c < 3; ++c) {
            const double Mrc = Mw[3 * r + c] * F.vox[c] / F.vox[r];
            const double Drc = Mrc - (r == c ? 1.0 : 0.0);
            m.D[3 * r + c] = (float)Drc;
            bc += Drc * F.cen[c];
        }
        m.bc[r] = (float)bc;
    }
    m.s = s_view ? s_view[v] : 0.0f;
    m.pad[0] = m.pad[1] = m.pad[2] = 0.0f;
    motion[v] = m;
    for (int q = 0; q < 27; ++q) dRdw[27 * v + q] = (float)dR[q];
}

// The spline's table (ray.cuh), FP64: thread = (z, y, cell, power).
__global__ void __launch_bounds__(160) spline_table_kernel(const float *__restrict__ coef, Frame F,
                                                                 float4 *__restrict__ table)
{
    // f^p coefficients of piece m (B-spline matrix times 6)
    const double B[4][4] = {{1, -3, 3, -1}, {4, 0, -6, 3}, {1, 3, 3, -3}, {0, 0, 0, 1}};
    const int p = threadIdx.x & 3, cell = threadIdx.x / 4 % 5, y = threadIdx.x / 20, z = blockIdx.x;
    double s[3] = {0.0, 0.0, 0.0};
    for (int m = 0; m < 4; ++m)
        for (int a = 0; a < 3; ++a) s[a] += B[m][p] / 6.0 * (double)coef[3 * ((z * 8 + y) * 8 + cell + m) + a];
    table[z * SPL_PLANE + y * SPL_ROW + cell * 4 + p] =
        make_float4((float)(s[0] / F.vox[0]), (float)(s[1] / F.vox[1]), (float)(s[2] / F.vox[2]), 0.f);
}

cudaError_t launch_motion_setup(const float *theta, const float *coef, const float *s_view, int n_views,
                                const Grid &G, const double vox[3], const double origin[3], MotionGPU *motion,
                                float4 *spline, float *dRdw, cudaStream_t stream)
{
    Frame F;
    const int n[3] = {G.nx, G.ny, G.nz};
    for (int a = 0; a < 3; ++a) {
        F.vox[a] = vox[a];
        F.origin[a] = origin[a];
        F.cen[a] = (double)((n[a] - 1) / 2);
    }
    motion_setup_kernel<<<(n_views + 127) / 128, 128, 0, stream>>>(theta, s_view, n_views, F, motion, dRdw);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (coef) {
        spline_table_kernel<<<8, 160, 0, stream>>>(coef, F, spline);
        e = cudaGetLastError();
    }
    return e;
}

// dL/d(omega, t, A) from dL/d(M, b) (index coordinates); one thread per view.
// gMc holds sum dL/dg' (g - c)^T, so dL/dM = gMc + gb c^T (c: integer grid
// centre).
__global__ void motion_finish_kernel(const float *__restrict__ theta, const float *__restrict__ dRdw,
                                     const double *__restrict__ gMc, const double *__restrict__ gb, int n_views,
                                     Frame F, float *__restrict__ grad_theta)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n_views) return;
    double R[9], dR[27], A[9], t[3];
    const double w[3] = {theta[15 * v], theta[15 * v + 1], theta[15 * v + 2]};
    rodrigues(w, R, dR);
    for (int q = 0; q < 3; ++q) t[q] = theta[15 * v + 3 + q];
    for (int q = 0; q < 9; ++q) A[q] = theta[15 * v + 6 + q];
    // dL/dMw[r][c] = gM[r][c] vox[c]/vox[r] + gb[r] origin[c]/vox[r];  dL/dbw[r] = gb[r]/vox[r]
    double gMw[9], gbw[3];
    for (int r = 0; r < 3; ++r) {
        gbw[r] = gb[3 * v + r] / F.vox[r];
        for (int c = 0; c < 3; ++c) {
            const double gM = gMc[9 * v + 3 * r + c] + gb[3 * v + r] * F.cen[c];
            gMw[3 * r + c] = gM * F.vox[c] / F.vox[r] + gb[3 * v + r] * F.origin[c] / F.vox[r];
        }
    }
    // Mw = A R, bw = A t
    double gA[9], gR[9], gt[3];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) {
            double s = 0.0;
            for (int q = 0; q < 3; ++q) s += gMw[3 * r + q] * R[3 * c + q];
            gA[3 * r + c] = s + gbw[r] * t[c];
            double s2 = 0.0;
            for (int q = 0; q < 3; ++q) s2 += A[3 * q + r] * gMw[3 * q + c];
            gR[3 * r + c] = s2;
        }
    for (int c = 0; c < 3; ++c) {
        double s = 0.0;
        for (int q = 0; q < 3; ++q) s += A[3 * q + c] * gbw[q];
        gt[c] = s;
    }
    for (int i = 0; i < 3; ++i) {
        double s = 0.0;
        for (int q = 0; q < 9; ++q) s += gR[q] * dR[9 * i + q];
        grad_theta[15 * v + i] += (float)s;
        grad_theta[15 * v + 3 + i] += (float)gt[i];
    }
    for (int q = 0; q < 9; ++q) grad_theta[15 * v + 6 + q] += (float)gA[q];
    (void)dRdw;
}

__global__ void coef_grad_finish_kernel(const double *__restrict__ g_idx, Frame F, float *__restrict__ grad_coef)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NCOEF) grad_coef[i] += (float)(g_idx[i] / F.vox[i % 3]);
}

cudaError_t launch_motion_grad_finish(const float *theta, const float *dRdw, const double *grad_M,
                                      const double *grad_b, const double *grad_coef_idx, int n_views,
                                      const Grid &G, const double vox[3], const double origin[3],
                                      float *grad_theta, float *grad_coef, cudaStream_t stream)
{
    Frame F;
    const int n[3] = {G.nx, G.ny, G.nz};
    for (int a = 0; a < 3; ++a) {
        F.vox[a] = vox[a];
        F.origin[a] = origin[a];
        F.cen[a] = (double)((n[a] - 1) / 2);
    }
    if (grad_theta && theta) {
        motion_finish_kernel<<<(n_views + 127) / 128, 128, 0, stream>>>(theta, dRdw, grad_M, grad_b, n_views, F,
                                                                        grad_theta);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (grad_coef && grad_coef_idx) {
        coef_grad_finish_kernel<<<(NCOEF + 255) / 256, 256, 0, stream>>>(grad_coef_idx, F, grad_coef);
        return cudaGetLastError();
    }
    return cudaSuccess;
}

}  // namespace ctrex
