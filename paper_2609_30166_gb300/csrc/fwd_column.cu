// fwd_column.cu -- the trilinear forward projector (and fused correction) of
// project.cu for scans whose detector columns run along z: one thread per
// pixel, a warp on 32 pixels of a detector column, the volume in column
// layout (column.cuh).
//
// What bounds it: L1's data path (82 % busy, 12.6 wavefronts per 32 samples,
// of which 8 are the taps themselves) and next to it issue (68 %, 39
// instructions per sample); the texture kernel's bound was the gathers'
// return path.  On 144 views of the 512^3 x 768^2 scan, FP32 / BF16 volume:
// 146.5 / 75.8 ms with texture gathers, 59.6 / 65.8 ms here.  What each part
// gave there (FP32): columns with floor by conversion-free adds 70.5 ms; the
// CTA order below 62.6; fixed-point positions, the x neighbour at an
// immediate offset and packed lerps 59.6.
#include "column.cuh"
#include "fwd_common.cuh"
#include "ray.cuh"

namespace ctrex {

// A CTA is 32 pixels along v by 4 columns (8 or 16 columns: the same within
// 1 %), 8 CTAs per SM (64 registers; capped at 48 for 10 CTAs: the same).
constexpr int COL_TU = 4;
constexpr int COL_MIN_BLOCKS = 8;
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
    if (!(fabsf(sg) * (float)n < 1.0e9f)) return false;
    const long long q = p + (long long)(n - 1) * d, top = ((long long)h + 1) << 32;
    return p >= (1ll << 32) && p <= top && q >= (1ll << 32) && q <= top;
}

// Integral and row sum of one pixel (mean over its sub-angle rays), as
// pixel_integral in project.cu.
__device__ __forceinline__ void col_pixel(const Grid &G, const ViewGPU *__restrict__ views, const ColVolume &vol, int view,
                                          float u, float v, float &val, float &rs)
{
    float acc = 0.0f, acc_rs = 0.0f;
    for (int s = 0; s < G.n_sub; ++s) {
        Ray R;
        if (!setup_ray(G, views[view * G.n_sub + s], u, v, R)) continue;
        const int Km1 = R.K - 1;
        int ka, kb;
        interior_range(G, R, ka, kb);
        // Interior positions in 32.32 fixed point, padded index coordinates:
        // a 64-bit add per axis and step, whose high word is the cell and
        // whose low word the fraction; exact, where a float position rounds
        // at the coordinate's magnitude.
        const float F = 4294967296.0f;
        const long long dx = __float2ll_rn(R.sg[0] * F), dy = __float2ll_rn(R.sg[1] * F),
                        dz = __float2ll_rn(R.sg[2] * F);
        long long px = __float2ll_rn(R.g0[0] * F) + (1ll << 32) + ka * dx,
                  py = __float2ll_rn(R.g0[1] * F) + (1ll << 32) + ka * dy,
                  pz = __float2ll_rn(R.g0[2] * F) + (1ll << 32) + ka * dz;
        // a range that is not inside (a ray with non-finite parameters) is
        // left to the clamped path
        const int n = kb - ka;
        if (n > 0 && !(axis_inside(px, dx, R.sg[0], n, vol.hx) && axis_inside(py, dy, R.sg[1], n, vol.hy) &&
                       axis_inside(pz, dz, R.sg[2], n, vol.hz)))
            kb = ka;
        auto edge = [&](float gx, float gy, float gz, float &ws) {
            // inside the border by the clip box; the clamp holds for any input
            gx = fminf(fmaxf(gx, -1.0f), vol.hx + 0.75f);
            gy = fminf(fmaxf(gy, -1.0f), vol.hy + 0.75f);
            gz = fminf(fmaxf(gz, -1.0f), vol.hz + 0.75f);
            float ax, ay, az;
            const float f = col_sample(vol, gx, gy, gz, ax, ay, az);
            ws = col_inside(gx, ax, vol.hx) * col_inside(gy, ay, vol.hy) * col_inside(gz, az, vol.hz);
            return f;
        };
        // the few samples beside the interior range first: the long loop then
        // holds little more than the ray itself in registers
        float a = 0.0f, ars = 0.0f, ws;
        for (int k = ka > 0 ? 0 : kb; k < Km1; k = k + 1 == ka ? kb : k + 1) {
            const float kf = (float)k;
            a += edge(fmaf(kf, R.sg[0], R.g0[0]), fmaf(kf, R.sg[1], R.g0[1]), fmaf(kf, R.sg[2], R.g0[2]), ws);
            ars += ws;
        }
        ars = (ars + (float)(kb - ka)) * G.step_mm;
        if (R.w_last > 0.0f) {
            acc = fmaf(R.w_last, edge(R.g_last[0], R.g_last[1], R.g_last[2], ws), acc);
            ars = fmaf(R.w_last, ws, ars);
        }
        acc_rs += ars;
#pragma unroll 2
        for (int left = kb - ka; left > 0; --left) {
            const ColTaps t =
                col_load(vol, vol.index((unsigned)(px >> 32), (unsigned)(py >> 32), (unsigned)(pz >> 32)));
            a += col_interp(t, fixed_fraction((unsigned)px), fixed_fraction((unsigned)py),
                            fixed_fraction((unsigned)pz));
            px += dx;
            py += dy;
            pz += dz;
        }
        acc = fmaf(a, G.step_mm, acc);
    }
    val = acc * G.inv_sub;
    rs = acc_rs * G.inv_sub;
}

template <typename TP, int MODE>
__global__ void __launch_bounds__(32 * COL_TU, COL_MIN_BLOCKS)
    fwd_column_kernel(Grid G, const ViewGPU *__restrict__ views, const ColVolume vol,
                      const int *__restrict__ view_idx, TP *__restrict__ out, float *__restrict__ rowsum_out,
                      const TP *__restrict__ p, float *__restrict__ partials, unsigned *devcheck, int p_by_view,
                      int n_strips)
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
    if (ok && in_pix) col_pixel(G, views, vol, view, (float)iu, (float)iv, val, rs);
    fwd_epilogue<TP, MODE, COL_TU>(G, k, view, ok, in_pix, iu, iv, val, rs, out, rowsum_out, p, partials, p_by_view,
                                   s_red);
}

// grid: tiles of a strip, views, strips x bands
static dim3 col_grid(const Grid &G, int n_idx, int &n_strips)
{
    const int tiles = (G.nu + COL_TU - 1) / COL_TU, per = tiles < COL_STRIP ? tiles : COL_STRIP;
    n_strips = (tiles + per - 1) / per;
    return dim3(per, n_idx, n_strips * ((G.nv + 31) / 32));
}

bool column_grid_fits(const Grid &G)
{
    int n_strips;
    return col_grid(G, 1, n_strips).z <= 65535;
}

int column_partials_needed(const Grid &G, int n_idx)
{
    int n_strips;
    const dim3 g = col_grid(G, n_idx, n_strips);
    return (int)(g.x * g.y * g.z);
}

template <typename TP, int MODE>
static cudaError_t col_launch(const FwdArgs &a, void *out, float *rowsum, const void *p, float *partials)
{
    int n_strips;
    const dim3 grid = col_grid(*a.grid, a.n_idx, n_strips);
    fwd_column_kernel<TP, MODE><<<grid, dim3(32, COL_TU), 0, a.stream>>>(
        *a.grid, a.views, col_view(*a.column), a.view_idx, static_cast<TP *>(out), rowsum, static_cast<const TP *>(p),
        partials, a.devcheck, a.p_by_view, n_strips);
    return cudaGetLastError();
}

cudaError_t launch_forward_column(const FwdArgs &a, bool correct, int pdt, void *out, float *rowsum, const void *p,
                                  float *partials)
{
    if (pdt == CTREX_F32)
        return correct ? col_launch<float, MODE_CORRECT>(a, out, rowsum, p, partials)
                       : col_launch<float, MODE_PROJECT>(a, out, rowsum, p, partials);
    return correct ? col_launch<__nv_bfloat16, MODE_CORRECT>(a, out, rowsum, p, partials)
                   : col_launch<__nv_bfloat16, MODE_PROJECT>(a, out, rowsum, p, partials);
}

}  // namespace ctrex
