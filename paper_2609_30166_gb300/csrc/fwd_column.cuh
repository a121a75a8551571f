// fwd_column.cuh -- what the column projectors share (fwd_column.cu: the
// static model; fwd_column_models.cu: event model, multi-resolution ROI,
// cylindrical domain, classical Joseph): launch shape, fixed-point runs of
// interior samples, edge samples.
#pragma once

#include "column.cuh"
#include "fwd_common.cuh"
#include "ray.cuh"

namespace ctrex {

// A CTA is 32 pixels along v by 4 columns (8 columns: the same within 1 %).
constexpr int COL_TU = 4;
constexpr int COL_MIN_BLOCKS = 8;  // CTAs per SM of the models' kernels (7 and 10: within 3 %)
constexpr int COL_UNROLL = 2;  // samples per step of the interior loop (1: +3 %; 3, 4: +1 %)
// CTAs are ordered in strips of 32 tiles (128 columns), then views, then
// strips and bands of 32 rows: the views resident together then cross one
// strip of the volume instead of all of it, and what they share stays in L2
// (DRAM reads of 16 views of the 512^3 scan: 2.0 GB, 10.3 GB with whole rows
// of tiles; strips of 8 to 64 tiles measured alike).
constexpr int COL_STRIP = 32;

// Whether an axis's fixed-point samples p, p + d, .., p + (n - 1) d lie in
// padded indices 1 .. h + 1 (the grid): they run evenly from end to end (sg
// is the step as a float: its bound keeps the products below 2^63).
__device__ __forceinline__ bool axis_inside(long long p, long long d, float sg, int n, float h)
{
    if (n < 1 || !(fabsf(sg) * (float)n < 1.0e9f)) return false;
    const long long q = p + (long long)(n - 1) * d, top = ((long long)h + 1) << 32;
    return p >= (1ll << 32) && p <= top && q >= (1ll << 32) && q <= top;
}

// Samples ka, ka + 1, .. of a ray, g0 + k sg, in 32.32 fixed point and padded
// index coordinates: a 64-bit add per axis and step, whose high word is the
// cell and whose low word the fraction; exact, where a float position rounds
// at the coordinate's magnitude.
struct ColRun {
    long long px, py, pz, dx, dy, dz;

    __device__ __forceinline__ void set(const float g0[3], const float sg[3])
    {
        const float F = 4294967296.0f;
        dx = __float2ll_rn(sg[0] * F);
        dy = __float2ll_rn(sg[1] * F);
        dz = __float2ll_rn(sg[2] * F);
        px = __float2ll_rn(g0[0] * F) + (1ll << 32);
        py = __float2ll_rn(g0[1] * F) + (1ll << 32);
        pz = __float2ll_rn(g0[2] * F) + (1ll << 32);
    }
    // From sample ka on.  False if one of the n samples is not inside the
    // grid (a ray with non-finite parameters): such a range is left to the
    // clamped path.
    __device__ __forceinline__ bool start(const ColVolume &V, const float g0[3], const float sg[3], int ka, int n)
    {
        set(g0, sg);
        px += ka * dx;
        py += ka * dy;
        pz += ka * dz;
        return axis_inside(px, dx, sg[0], n, V.hx) && axis_inside(py, dy, sg[1], n, V.hy) &&
               axis_inside(pz, dz, sg[2], n, V.hz);
    }
    // From sample 0 on.  False if one of the n samples comes within a quarter
    // of a voxel of the border's outer edge (the clip box ends half a voxel
    // inside it, so this too takes a ray with non-finite parameters): the two
    // end positions decide, in FP32, whose rounding is far smaller.
    __device__ __forceinline__ bool start_all(const ColVolume &V, const float g0[3], const float sg[3], int n)
    {
        const float h[3] = {V.hx, V.hy, V.hz}, k = (float)(n - 1);
        bool ok = n > 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float e = fmaf(k, sg[a], g0[a]);
            ok = ok && fminf(g0[a], e) >= -0.75f && fmaxf(g0[a], e) <= h[a] + 0.75f && h[a] < 4.0e6f;
        }
        set(g0, sg);
        return ok;
    }
    __device__ __forceinline__ unsigned index(const ColVolume &V) const
    {
        return V.index((unsigned)(px >> 32), (unsigned)(py >> 32), (unsigned)(pz >> 32));
    }
    template <typename Taps> __device__ __forceinline__ float interp(const Taps &t) const
    {
        return col_interp(t, fixed_fraction((unsigned)px), fixed_fraction((unsigned)py), fixed_fraction((unsigned)pz));
    }
    __device__ __forceinline__ void next()
    {
        px += dx;
        py += dy;
        pz += dz;
    }
    // a plus the next n samples
    template <bool PAIRS = false> __device__ __forceinline__ float sum(const ColVolume &V, int n, float a)
    {
#pragma unroll COL_UNROLL
        for (int left = n; left > 0; --left) {
            a += PAIRS ? interp(col_load_pairs(V, index(V))) : interp(col_load(V, index(V)));
            next();
        }
        return a;
    }
};

// A sample beside the interior range: inside the border by the clip box, and
// clamped for any input; ws: its summed weight of the taps inside the grid.
template <typename Taps>
__device__ __forceinline__ float col_edge(const ColVolume &V, float gx, float gy, float gz, float &ws, Taps taps)
{
    gx = fminf(fmaxf(gx, -1.0f), V.hx + 0.75f);
    gy = fminf(fmaxf(gy, -1.0f), V.hy + 0.75f);
    gz = fminf(fmaxf(gz, -1.0f), V.hz + 0.75f);
    const float fx = floorf(gx), fy = floorf(gy), fz = floorf(gz);
    const float ax = gx - fx, ay = gy - fy, az = gz - fz;
    ws = col_inside(gx, ax, V.hx) * col_inside(gy, ay, V.hy) * col_inside(gz, az, V.hz);
    return col_interp(taps((int)fx + 1, (int)fy + 1, (int)fz + 1), ax, ay, az);
}

// Samples ka .. kb - 1 of the n ones at g0 + k sg, all taps of which lie in the
// grid by a margin of 0.01 voxel (or a few less: the weights of the others
// come from col_weight, which is 1 there too).
__device__ __forceinline__ void col_interior(const ColVolume &V, const float g0[3], const float sg[3], int n, int &ka,
                                             int &kb)
{
    const float h[3] = {V.hx, V.hy, V.hz};
    float lo = 0.0f, hi = (float)(n - 1);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float inv = __frcp_rn(sg[a]), l = 0.01f - g0[a], u = h[a] - 0.01f - g0[a];
        const bool moves = fabsf(sg[a]) > 1.0e-9f;
        const float t0 = moves ? l * inv : (l <= 0.0f ? -1.0f : 1.0e9f), t1 = moves ? u * inv : (u >= 0.0f ? 1.0e9f : -1.0f);
        lo = fmaxf(lo, fminf(t0, t1));
        hi = fminf(hi, fmaxf(t0, t1));
        if (!(u >= l)) hi = -1.0f;  // one voxel along this axis
    }
    ka = min(max((int)ceilf(lo), 0), n);
    kb = max(min((int)floorf(hi) + 1, n), ka);
}

// Summed weight of a sample's taps inside the grid, from its position alone.
__device__ __forceinline__ float col_weight(const ColVolume &V, float gx, float gy, float gz)
{
    return __saturatef(fminf(gx + 1.0f, V.hx + 1.0f - gx)) * __saturatef(fminf(gy + 1.0f, V.hy + 1.0f - gy)) *
           __saturatef(fminf(gz + 1.0f, V.hz + 1.0f - gz));
}

// The kernel's frame: the CTA's pixels, one integral per thread by `pixel`
// (view, u, v, value, row sum), and the epilogue.
template <typename TP, int MODE, typename Pixel>
__device__ __forceinline__ void col_body(const Grid &G, const int *__restrict__ view_idx, TP *__restrict__ out,
                                         float *__restrict__ rowsum_out, const TP *__restrict__ p,
                                         float *__restrict__ partials, unsigned *devcheck, int p_by_view, int n_strips,
                                         Pixel pixel)
{
    __shared__ float s_red[2][COL_TU];
    const int k = blockIdx.y;
    int view = view_idx ? view_idx[k] : k;
    bool ok = true;
    if (view < 0 || view >= G.n_views) {
        if (threadIdx.x == 0 && threadIdx.y == 0) atomicOr(devcheck, (unsigned)DEVCHECK_OOB);
        ok = false;
        view = 0;
    }
    const int strip = blockIdx.z % n_strips, band = blockIdx.z / n_strips;
    const int iu = (strip * gridDim.x + blockIdx.x) * COL_TU + threadIdx.y, iv = band * 32 + threadIdx.x;
    const bool in_pix = iu < G.nu && iv < G.nv;
    float val = 0.0f, rs = 0.0f;
    if (ok && in_pix) pixel(view, (float)iu, (float)iv, val, rs);
    fwd_epilogue<TP, MODE, COL_TU>(G, k, view, ok, in_pix, iu, iv, val, rs, out, rowsum_out, p, partials, p_by_view,
                                   s_red);
}

// grid: tiles of a strip, views, strips x bands
inline dim3 col_grid(const Grid &G, int n_idx, int &n_strips)
{
    const int tiles = (G.nu + COL_TU - 1) / COL_TU, per = tiles < COL_STRIP ? tiles : COL_STRIP;
    n_strips = (tiles + per - 1) / per;
    return dim3(per, n_idx, n_strips * ((G.nv + 31) / 32));
}

}  // namespace ctrex
