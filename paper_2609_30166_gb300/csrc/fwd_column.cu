// fwd_column.cu -- the trilinear forward projector (and fused correction) of
// project.cu for scans whose detector columns run along z: one thread per
// pixel, a warp on 32 pixels of a detector column, the volume in column
// layout (column.cuh).
//
// What bounds it: L1's data path (12.6 wavefronts per 32 samples, of which 8
// are the taps themselves; 16-byte loads of x pairs too need as many; 86 % busy
// at 512^3, 49 to 67 % at 64^3 and 128^3) and next to it the issue ports (68 %
// busy at every size, and held longer by packed multiply-adds); the texture
// kernel's bound was the gathers' return path.  On 144 views of the 512^3 x
// 768^2 scan, FP32 / BF16 volume: 146.5 / 75.8 ms with texture gathers, 52.5 /
// 52.5 ms here.  What each part gave there (FP32): columns with floor by
// conversion-free adds 70.5 ms; the CTA order below 62.6; fixed-point
// positions, the x neighbour at an immediate offset and packed lerps 59.4;
// every sample in the fast loop, with only the weights of those beside the
// interior on the side, 55.5 (64^3 x 90 views: 0.164 -> 0.141 ms, sparse 128^3:
// 0.549 -> 0.490); differences instead of second values in the store 52.5 (0.137,
// 0.466).
#include "fwd_column.cuh"

namespace ctrex {

// Integral and row sum of one pixel (mean over its sub-angle rays), as
// pixel_integral in project.cu.
__device__ __forceinline__ void col_pixel(const Grid &G, const ViewGPU *__restrict__ views, const ColVolume &vol, int view,
                                          float u, float v, float &val, float &rs)
{
    float acc = 0.0f, acc_rs = 0.0f;
    auto taps = [&](unsigned i, unsigned j, unsigned k) { return col_load(vol, vol.index(i, j, k)); };
    for (int s = 0; s < G.n_sub; ++s) {
        Ray R;
        if (!setup_ray(G, views[view * G.n_sub + s], u, v, R)) continue;
        const int Km1 = R.K - 1;
        // The border makes every sample's value the fast loop's; the row sum
        // takes the weights of the few samples beside the interior range.
        ColRun run;
        int n = Km1;
        float a = 0.0f, ars = 0.0f, ws;
        if (run.start_all(vol, R.g0, R.sg, n)) {
            int ka, kb;
            col_interior(vol, R.g0, R.sg, n, ka, kb);
            for (int k = ka > 0 ? 0 : kb; k < Km1; k = k + 1 == ka ? kb : k + 1) {
                const float kf = (float)k;
                ars += col_weight(vol, fmaf(kf, R.sg[0], R.g0[0]), fmaf(kf, R.sg[1], R.g0[1]),
                                  fmaf(kf, R.sg[2], R.g0[2]));
            }
            ars += (float)(kb - ka);
        } else {
            n = 0;
            for (int k = 0; k < Km1; ++k) {
                const float kf = (float)k;
                a += col_edge(vol, fmaf(kf, R.sg[0], R.g0[0]), fmaf(kf, R.sg[1], R.g0[1]),
                              fmaf(kf, R.sg[2], R.g0[2]), ws, taps);
                ars += ws;
            }
        }
        ars *= G.step_mm;
        if (R.w_last > 0.0f) {
            acc = fmaf(R.w_last, col_edge(vol, R.g_last[0], R.g_last[1], R.g_last[2], ws, taps), acc);
            ars = fmaf(R.w_last, ws, ars);
        }
        acc_rs += ars;
        acc = fmaf(run.sum(vol, n, a), G.step_mm, acc);
    }
    val = acc * G.inv_sub;
    rs = acc_rs * G.inv_sub;
}

template <typename TP, int MODE>
__global__ void __launch_bounds__(32 * COL_TU, 9)  // 56 registers (8 CTAs: 53.8 ms, 9: 52.5, 10: 53.9)
    fwd_column_kernel(Grid G, const ViewGPU *__restrict__ views, const ColVolume vol,
                      const int *__restrict__ view_idx, TP *__restrict__ out, float *__restrict__ rowsum_out,
                      const TP *__restrict__ p, float *__restrict__ partials, unsigned *devcheck, int p_by_view,
                      int n_strips)
{
    col_body<TP, MODE>(G, view_idx, out, rowsum_out, p, partials, devcheck, p_by_view, n_strips,
                       [&](int view, float u, float v, float &val, float &rs) {
                           col_pixel(G, views, vol, view, u, v, val, rs);
                       });
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
    if (a.roi || a.dyr || a.cyl || a.joseph)
        return launch_forward_column_models(a, correct, pdt, out, rowsum, p, partials);
    if (pdt == CTREX_F32)
        return correct ? col_launch<float, MODE_CORRECT>(a, out, rowsum, p, partials)
                       : col_launch<float, MODE_PROJECT>(a, out, rowsum, p, partials);
    return correct ? col_launch<__nv_bfloat16, MODE_CORRECT>(a, out, rowsum, p, partials)
                   : col_launch<__nv_bfloat16, MODE_PROJECT>(a, out, rowsum, p, partials);
}

}  // namespace ctrex
