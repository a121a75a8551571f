// context.cu -- the C ABI of libctrex: context, geometry and motion set-up,
// operator entry points and the SIRT driver (the paper's Rex / Trajectory
// split, Sec. 2.1-2.3, as a native library).
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <string>
#include <vector>

#include "atlas.cuh"
#include "column.cuh"
#include "ctrex_internal.cuh"

using namespace ctrex;

struct ctrex_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    std::string err;
    // geometry
    bool has_geom = false;
    Grid grid{};
    double vox[3] = {1, 1, 1}, origin[3] = {0, 0, 0};
    double step_vox = 0.5;
    ViewGPU *d_views = nullptr;
    // motion
    bool has_motion = false;
    double margin = 0.0;
    MotionGPU *d_motion = nullptr;
    float *d_theta = nullptr;     // [n_views][15] copy (or null)
    float *d_coef = nullptr;      // [8][8][8][3] mm
    float4 *d_spline = nullptr;   // its table, voxels (ray.cuh)
    float *d_dRdw = nullptr;      // [n_views][27]
    double *d_gM = nullptr, *d_gb = nullptr, *d_gcoef = nullptr;  // gradient scratch (FP64 sums)
    bool coef_valid = false, theta_valid = false;
    // scratch
    float *d_partials = nullptr;
    int partials_cap = 0;
    double *d_sums = nullptr;
    double *h_sums = nullptr;         // the SIRT loop's residual on the host (pinned)
    cudaEvent_t sums_done = nullptr;  // and its arrival
    unsigned *d_devcheck = nullptr;
    unsigned long long *d_count = nullptr;
    void *d_r = nullptr;  // SIRT correction images
    size_t r_bytes = 0;
    // texture atlas of the volume read by the forward projector
    AtlasStore vol_atlas;
    Atlas vol_atlas_view;
    // the volume in column layout, where the scan's detector columns run along z
    double col_lean = 10.0, col_step = 1.0, col_pixel = 1.0;  // detector_column_step
    bool bp_flat = false, bp_flat_roi = false;  // backproject_flat (Cartesian grids)
    std::vector<ViewGPU> hviews;     // the views, and the windows, on the host
    std::vector<int4> hwindow;
    double bp_inside = 0.0;          // set_bp_inside
    ColStore vol_col;
    ColStore col1;     // the ROI grid, or the event model's final values
    ColStore tau_col;  // the event model's transition times
    bool tau_col_set = false;
    float *d_adj = nullptr;  // the adjoint's scatter volume
    size_t adj_elems = 0;
    ColStore img_col;  // the correction images
    // the last use of the stores and the scatter volume (ScratchUse)
    cudaEvent_t scratch_done = nullptr;
    unsigned long long scratch_stream = 0;  // its id (unique among all streams ever made)
    bool scratch_open = false;
    bool scratch_captured = false;  // a graph may hold the stores' addresses
    // texture atlas of the correction images read by the backprojector
    AtlasStore img_atlas;
    Atlas img_atlas_view;
    bool img_atlas_unfit = false;
    bool atlas_unfit = false;  // geometry exceeds the 2D texture limits: row-major sampling
    // backprojector detector windows (extended field of view), int4 per view
    int4 *d_window = nullptr;
    bool has_window = false;
    // sub-voxel backprojection points per axis (motion blur), 1 = off
    int bp_subvoxel = 1;
    // aligned cylindrical domain (set by ctrex_set_geometry_cylinder)
    bool cyl = false;
    CylGPU cylg{};
    // forward projector: CTREX_PROJ_TRILINEAR or CTREX_PROJ_JOSEPH (three-stack atlas)
    int projector = CTREX_PROJ_TRILINEAR;
    AtlasStore jos_atlas;
    Atlas jos_atlas_view;
    // multi-resolution ROI (set by ctrex_set_roi): a finer grid whose voxels
    // follow the context grid's in every volume buffer
    std::vector<double> hostP;  // world matrices of the current geometry
    double ctr[3] = {0, 0, 0};  // the centre P was sign-normalised with
    bool roi = false;
    Grid roi_grid{};
    ViewGPU *d_views_roi = nullptr;
    RoiGPU roig{};
    AtlasStore roi_atlas;
    Atlas roi_atlas_view;
    // event-based 4D model (set by ctrex_set_dyrect): volume buffers hold
    // the initial values followed by the final values
    bool dyr = false;
    float *d_tau = nullptr;     // [nz][ny][nx] transition times
    float *d_tview = nullptr;   // [n_views] acquisition times
    float2 *d_tau_brick = nullptr;  // (min, max) transition time per 8^3 brick
    float2 *d_tau_block = nullptr;  // the same around each brick (launch_tau_bricks)
    float2 *d_tau_cell = nullptr;   // its scratch
    AtlasStore dyr_atlas1;      // the final values (the volume atlas holds the initial ones)
    AtlasStore tau_atlas;
    Atlas dyr_atlas1_view, tau_atlas_view;
    DyrArgs dyra{};
    // ordered-subset SIRT: concatenated subset view lists, per-subset norms
    int *d_subset_views = nullptr;
    size_t subset_views_bytes = 0;
    double *d_subset_sums = nullptr;
    size_t subset_sums_bytes = 0;
    // host-buffer entry point scratch
    void *d_hvol = nullptr, *d_hp = nullptr;
    float *d_hw = nullptr;
    size_t hvol_bytes = 0, hp_bytes = 0, hw_bytes = 0;
    // its first iteration overlaps the projections' upload with the forward
    // projection: A x and the row sums (FP32), a copy stream, two events
    void *d_hq = nullptr;
    float *d_hrs = nullptr;
    double *d_hcs = nullptr;  // the correction's partial norms
    size_t hq_bytes = 0, hrs_bytes = 0, hcs_bytes = 0;
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_vol = nullptr, ev_p = nullptr;
};

namespace {

const char *g_static_err = "ctrex: invalid context";

int fail(ctrex_ctx *c, int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    if (c) c->err = buf;
    return code;
}

int cuda_fail(ctrex_ctx *c, cudaError_t e, const char *where)
{
    cudaGetLastError();  // not for the next call to find after its launches
    return fail(c, e == cudaErrorMemoryAllocation ? CTREX_E_NOMEM : CTREX_E_CUDA, "%s: %s (%s)", where,
                cudaGetErrorString(e), cudaGetErrorName(e));
}

#define CT_CUDA(c, call)                                  \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return cuda_fail(c, e_, #call); \
    } while (0)

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// The column stores and the adjoint's scatter volume belong to the context,
// while calls may run on different streams (ctrex_set_stream) with nothing
// that orders them: a call waits for the last one's use before its own
// (scratch_begin) and leaves an event behind it (ScratchUse, at the end of
// the entry point).  A capturing stream can wait for no event outside its
// graph, nor allocate: what read the caller's buffers alone before there were
// stores does so there, and work replayed from a graph is ordered by the caller.
bool capturing(const ctrex_ctx *c) { return stream_capturing(c->stream); }

cudaError_t scratch_begin(ctrex_ctx *c)
{
    if (c->scratch_open) return cudaSuccess;
    if (capturing(c)) {
        c->scratch_captured = true;
        return cudaSuccess;
    }
    c->scratch_open = true;
    unsigned long long id = 0;
    cudaError_t e = cudaStreamGetId(c->stream, &id);
    if (e == cudaSuccess && id != c->scratch_stream) e = cudaStreamWaitEvent(c->stream, c->scratch_done, 0);
    c->scratch_stream = id;
    return e;
}

struct ScratchUse {
    ctrex_ctx *c;
    explicit ScratchUse(ctrex_ctx *ctx) : c(ctx) {}
    ~ScratchUse()
    {
        if (!c->scratch_open) return;
        c->scratch_open = false;
        if (cudaEventRecord(c->scratch_done, c->stream) != cudaSuccess) {
            cudaGetLastError();
            cudaStreamSynchronize(c->stream);
        }
    }
};

template <typename T> void dfree(T *&p)
{
    if (p) cudaFree((void *)p);
    p = nullptr;
}

// Gives the column scratch back (laid out again by the next call that uses it).
void release_columns(ctrex_ctx *c)
{
    col_release(c->vol_col);
    col_release(c->col1);
    col_release(c->tau_col);
    c->tau_col_set = false;
    col_release(c->img_col);
    dfree(c->d_adj);
    c->adj_elems = 0;
}

// An allocation, with the column scratch given back if it fails at first:
// nothing that fits without the scratch is refused for it (unless a graph may
// hold its addresses).
template <typename Make> cudaError_t alloc_or_release(ctrex_ctx *c, Make make)
{
    cudaError_t e = make();
    if (e != cudaErrorMemoryAllocation || c->scratch_captured) return e;
    cudaGetLastError();
    release_columns(c);
    return make();
}

int ensure(ctrex_ctx *c, void **p, size_t *have, size_t need, const char *what)
{
    if (*have >= need && *p) return CTREX_OK;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *have = 0;
    cudaError_t e = alloc_or_release(c, [&] { return cudaMalloc(p, need); });
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(c, CTREX_E_NOMEM, "cannot allocate %zu bytes for %s: %s", need, what, cudaGetErrorString(e));
    }
    *have = need;
    return CTREX_OK;
}

size_t dtype_size(int dt) { return dt == CTREX_BF16 ? 2 : 4; }
bool dtype_ok(int dt) { return dt == CTREX_F32 || dt == CTREX_BF16; }

int check_ctx(ctrex_ctx *c)
{
    if (!c) return CTREX_E_ARG;
    return CTREX_OK;
}

int check_views(ctrex_ctx *c, const int *view_idx, int n_idx)
{
    if (!c->has_geom) return fail(c, CTREX_E_STATE, "set_geometry has not been called");
    if (n_idx < 0 || n_idx > 65535) return fail(c, CTREX_E_SHAPE, "n_idx %d outside [0, 65535]", n_idx);
    if (!view_idx && n_idx != 0 && n_idx != c->grid.n_views)
        return fail(c, CTREX_E_SHAPE, "view_idx is NULL but n_idx (%d) != n_views (%d)", n_idx, c->grid.n_views);
    return CTREX_OK;
}

FwdArgs fwd_args(ctrex_ctx *c, const void *vol, int vdt, const int *view_idx, int n_idx)
{
    FwdArgs a;
    a.grid = &c->grid;
    a.views = c->d_views;
    a.motion = c->has_motion ? c->d_motion : nullptr;
    a.spline = (c->has_motion && c->coef_valid) ? c->d_spline : nullptr;
    a.vol = vol;
    a.vol_dtype = vdt;
    a.view_idx = view_idx;
    a.n_idx = n_idx;
    a.stream = c->stream;
    a.devcheck = c->d_devcheck;
    a.cyl = c->cyl ? &c->cylg : nullptr;
    a.joseph = c->projector == CTREX_PROJ_JOSEPH ? 1 : 0;
    a.roi = c->roi ? &c->roig : nullptr;
    a.dyr = c->dyr ? &c->dyra : nullptr;
    return a;
}

size_t grid_voxels(const Grid &G) { return (size_t)G.nx * G.ny * G.nz; }

// Elements of a volume buffer: the grid, then the ROI grid if one is set;
// with the event-based model the grid's initial then final values.
size_t volume_elems(const ctrex_ctx *c)
{
    return grid_voxels(c->grid) * (c->dyr ? 2 : 1) + (c->roi ? grid_voxels(c->roi_grid) : 0);
}

void dyr_release(ctrex_ctx *c)
{
    c->dyr = false;
    if (c->d_tau) cudaFree(c->d_tau);
    if (c->d_tview) cudaFree(c->d_tview);
    if (c->d_tau_brick) cudaFree(c->d_tau_brick);
    c->d_tau = c->d_tview = nullptr;
    c->d_tau_brick = nullptr;
    dfree(c->d_tau_block);
    dfree(c->d_tau_cell);
    col_release(c->tau_col);
    col_release(c->col1);
    c->tau_col_set = false;
    atlas_release(c->dyr_atlas1);
    atlas_release(c->tau_atlas);
}

// Which scans take the column kernels (fwd_column.cu, bp_column.cu) and which
// stay with texture gathers, by measurement on a 512^3 volume:
// - the detector rotated in its plane (768^2 pixels, 72 views; ms column /
//   texture at 0, 20, 30, 45, 90 degrees): forward 30 / 73, 53 / 81, 65 / 92,
//   81 / 113, 231 / 183; backprojection 9.4 / 17.8, 12.9 / 17.8, 16.9 / 17.8,
//   24.2 / 17.8, 64 / 17.7;
// - coarse pixels spread a warp's rays (pixel steps of 2, 4, 8 voxels):
//   forward FP32 13.6 / 27.0, 11.7 / 22.3, 19.4 / 15.9 ms, BF16 13.6 / 14.4,
//   11.7 / 10.9, 19.4 / 7.8 ms;
// - fine pixels spread a warp's voxels (768^2 pixels, 90 views, voxel steps
//   of 2 and 4 pixels): backprojection 2.0 / 3.0 ms, 0.66 / 0.62 ms.
// The other models and BF16 volumes: see column_forward.
constexpr double COL_LEAN_FWD = 1.0, COL_STEP_FP32 = 6.0, COL_STEP_BF16 = 3.0;
constexpr double COL_STEP_BP_MIN = 0.3;  // (and see column_backproject)
// The adjoint's warps: 32 rows of a detector column up to this lean, 8 x 4
// patches beyond (45 views of 384^2 on 256^3, ms column / patch at 0, 6, 8, 45
// degrees: 5.7 / 7.8, 12.0 / 12.4, 13.8 / 13.4, 29 / 17; in place 16.6 .. 18.3).
constexpr double COL_LEAN_ADJ = 0.12;

// The forward projector: also the lanes that each kernel's tiles (4 x 32
// columns x rows here, 32 x 4 there) waste on a ragged detector, against what
// the columns gain over the gathers.  90 views of 256^3, 384^2 pixels, ms
// columns / gathers at 0, 5, 10, 15, 20, 30, 44 degrees:
//   static, FP32  6.3/16.6 7.6/16.7 9.2/16.8 10.7/16.9 12.0/17.0 14.0/17.8 16.5/20.3
//   static, BF16  6.3/8.6  7.7/8.8  9.3/9.0  10.7/9.0  12.0/9.1  14.0/9.2  16.5/9.7
//   event, FP32   8.3/24.4 9.2/25.0 10.7/25.7 12.3/26.4 13.8/27.1 16.6/28.3 19.9/30.1
//   ROI, FP32     9.1/20.3 11.1/20.6 12.9/21.0 14.7/21.3 16.4/21.8 19.2/23.3 22.3/26.5
//   cylinder      11.0/15.4 11.1/15.6 11.2/15.8 11.2/15.8 11.4/15.8 11.9/15.9 13.4/17.0
//   Joseph, FP32  2.7/3.8  2.8/3.9  3.2/3.9  3.6/3.9   3.9/3.9   4.4/3.9   5.1/3.9
//   Joseph, BF16  2.6/3.7  2.8/3.8  3.2/3.8  3.6/3.8   3.9/3.8   4.4/3.8   5.1/3.7
// (event and ROI in BF16 gain as in FP32).  Coarse pixels spread a leaning
// warp further.  Of 376 ragged detectors for each model and type (96^3 and
// 256^3, pixel steps of 1 to 4.5 voxels, 0 to 44 degrees) the choice below is
// slower than gathers by more than 3 % on 5 Joseph ones (8 % at most, 86 us for
// 79) and no other; with one limit per type for all models it was on 370.
bool column_forward(const ctrex_ctx *c, int vdt)
{
    if (!(c->col_lean <= COL_LEAN_FWD && column_grid_fits(c->grid))) return false;
    const double step = c->col_step * (c->roi ? fmax(1.0, c->roig.sc[2]) : 1.0);
    if (step > (vdt == CTREX_F32 ? COL_STEP_FP32 : COL_STEP_BF16)) return false;
    const double u4 = (c->grid.nu + 3) / 4 * 4.0, u32 = (c->grid.nu + 31) / 32 * 32.0;
    const double v4 = (c->grid.nv + 3) / 4 * 4.0, v32 = (c->grid.nv + 31) / 32 * 32.0;
    const double spread = c->col_lean * fmax(step, 1.0);
    double gain = vdt == CTREX_F32 ? 2.2 : 1.2;
    if (c->projector == CTREX_PROJ_JOSEPH)
        gain = fmin(gain, 2.1 - 0.1 * step - 3.0 * spread);
    else if (c->cyl)
        gain = fmin(gain, 1.6);
    else if (vdt == CTREX_BF16 && !c->dyr && !c->roi)
        gain = fmin(gain, 1.75 - 5.0 * spread);
    return u4 * v32 <= u32 * v4 * gain;
}

// The backprojector: time by columns over time by gathers, fitted to 12,700
// scans of all kinds and both image types (40^2 to 512^2 voxels in x and y, 8 to
// 512 slices, pixel steps of 0.3 to 3.5 voxels, 0 to 38 degrees of lean).
// - A pixel step of s voxels spreads a warp's 32 voxels over 32 / s rows and
//   lean * 32 / s columns, each one more line (256^3, 90 views, 0.8 voxels a
//   pixel, static FP32, ms columns / gathers at 0, 8, 15, 22 degrees: 1.6 / 2.9,
//   2.1 / 2.9, 2.5 / 2.9, 2.9 / 2.9).
// - Blocks of 64 or 128 slices repeat slices, which costs where the launch has
//   more than a wave or two of CTAs (`full`; 12 slices of 256 x 256 take 2.2 times
//   the gathers' time, of 72 x 72 0.77; 70 slices 1.15 and 0.94).
// - Terms of a block that reaches beyond the detector or a window, as the part
//   beyond a volume of less than 64 slices may, take the general path (28 slices
//   of 256 x 256: 1.4 -> 2.9; 96 behind a window that cuts them 0.9 -> 1.4).
// What is chosen takes more than 3 % longer than gathers on 583 of the scans,
// 10 % on 143; one lean limit for all, with a height rule for the static model
// alone, was slower on 3265 of 8638 of them, up to seven times.
double bp_column_cost(const ctrex_ctx *c, const Grid &G, int rdt, double step)
{
    struct {
        double base, rows, cols, bf16;
    } k = {0.49, 0.13, 0.63, 1.22};  // static, cylinder
    if (c->bp_subvoxel > 1)
        k = {0.56, 0.10, 0.24, 1.02};
    else if (c->dyr)
        k = {0.55, 0.07, 0.59, 1.12};
    else if (c->has_window)
        k = {0.60 + 0.35 * (1.0 - c->bp_inside), 0.06, 0.70, 1.12};
    const bool subv = c->bp_subvoxel > 1;
    const double slices = backproject_column_slices(G, c->dyr || subv);
    const double ctas = (G.nx + 7) / 8 * (double)G.ny * (slices / 64.0), wave = subv ? 1500.0 : 3000.0;
    const double full = c->col_lean > 0.1 ? 1.0 : ctas * ctas / (ctas * ctas + wave * wave);
    const double out = fmin(2.5 * (1.0 - c->bp_inside), 1.0);
    const double blocks = (1.0 - 0.2 * (1.0 - full) * (1.0 - out)) * (1.0 + (slices / G.nz - 1.0) * full) *
                          (1.0 + 0.9 * out * fmin(fmax((64 - G.nz) / 24.0, 0.0), 1.0));
    // what a turn moves the volume's sides along the detector's rows by, over its height
    const double width = c->cyl ? 2.0 * G.nx * c->cylg.dr / c->cylg.dz : (double)(G.nx > G.ny ? G.nx : G.ny);
    return blocks * (rdt == CTREX_BF16 ? k.bf16 : 1.0) *
           (k.base + k.rows / step + k.cols * fmin(c->col_lean / step, 0.35) +
            0.25 * fmin(c->col_lean * width / G.nz, 3.0));
}

bool column_backproject(const ctrex_ctx *c, int rdt)
{
    const Grid &G = c->grid;
    if (!(c->col_step >= COL_STEP_BP_MIN && backproject_column_fits(G))) return false;
    if (c->roi && !backproject_column_fits(c->roi_grid)) return false;
    double cost = bp_column_cost(c, G, rdt, c->col_step);
    if (c->roi) {
        const double v = (double)grid_voxels(G), w = (double)grid_voxels(c->roi_grid);
        cost = (cost * v + bp_column_cost(c, c->roi_grid, rdt, c->col_step * c->roig.sc[2]) * w) / (v + w);
    }
    return cost <= 1.0;
}

// Voxels that the rays of n_idx views pass, about.
double ray_voxels(const ctrex_ctx *c, int n_idx)
{
    const Grid &G = c->grid;
    return (double)n_idx * G.n_sub * G.nu * G.nv * fmax(G.nx, fmax(G.ny, G.nz));
}

// (By the pose and a few rows, patches: 192 x 12 pixels 0.23 ms, rows 0.28.)
bool adjoint_along_z(const ctrex_ctx *c)
{
    return c->col_lean <= COL_LEAN_ADJ && (!c->has_motion || c->grid.nv > 16);
}

// The adjoint through a scatter volume, if that can be had (and its launch: an
// 8192^2 detector with motion is beyond it).  The volume is zeroed and added
// once per call, so the call's rays have to outweigh it (one view of 64^2
// pixels on 512^3: 0.71 ms, 0.65 in place; 768^2: 1.7, 3.6 in place).
bool column_adjoint(ctrex_ctx *c, int n_idx)
{
    const Grid &G = c->grid;
    if (c->dyr || capturing(c)) return false;
    if (!adjoint_column_fits(G, c->has_motion && c->coef_valid, adjoint_along_z(c))) return false;
    const double rays = ray_voxels(c, n_idx), vox = (double)grid_voxels(G);
    if (rays < 0.03 * vox) return false;
    // Turned detectors (no deformation, enough rays to fill the GPU): the rays
    // of a warp drift apart in z, with fine pixels soonest, while in place they
    // share footprints; large volumes with coarse pixels lose too.  256^3, 16
    // views, ms here / in place at 10, 35, 60 degrees: 0.4 voxels a pixel 37.9 /
    // 41.1, 46.3 / 42.8, 53.1 / 42.5; 2 voxels 2.25 / 2.01, 2.67 / 2.01, 2.77 /
    // 2.00 (by the pose, whose patches keep to three CTAs per SM, fine pixels only).  Of 4872 scans (32^2 to 256^2 in x and
    // y, 8 to 256 slices, 1 to 60 views, 0 to 88 degrees) 157 take more than 3 %
    // longer than in place before there was a scatter volume; 330 with columns
    // throughout.
    const double pixel = c->col_pixel;
    if (!(c->has_motion && c->coef_valid) && G.nz >= 32 && rays >= 2e7) {
        if (pixel < 0.55 && c->col_lean > 0.45) return false;
        if (!c->has_motion && pixel < 1.0 && c->col_lean > 1.0) return false;
        if (!c->has_motion && pixel >= 1.6 && vox > 6e6 && rays >= 3e7 && c->col_lean > 0.1) return false;
    }
    const size_t n = adjoint_column_elems(G);
    if (n == 0) return false;
    if (n > c->adj_elems || n < c->adj_elems / 2) {
        size_t free = 0, total = 0;
        const bool fits = cudaMemGetInfo(&free, &total) == cudaSuccess &&
                          n * sizeof(float) <= (free + c->adj_elems * sizeof(float)) / 2;
        if (fits) {
            dfree(c->d_adj);
            c->adj_elems = 0;
        }
        if (!fits || cudaMalloc((void **)&c->d_adj, n * sizeof(float)) != cudaSuccess) {
            cudaGetLastError();
            if (fits) c->d_adj = nullptr;
            return false;
        }
        c->adj_elems = n;
    }
    return true;
}

// Uploads vol into the context's column stores and points a.column at them; a
// shape that the model's texture atlases refuse, and a store that does not
// fit, are left to the atlas path (a.column stays null).
int prepare_columns(ctrex_ctx *c, FwdArgs &a, const void *vol, int vdt)
{
    const int nx = c->grid.nx, ny = c->grid.ny, nz = c->grid.nz, d = c->device;
    const int rx = c->roi_grid.nx, ry = c->roi_grid.ny, rz = c->roi_grid.nz;
    if (c->projector == CTREX_PROJ_JOSEPH && !atlas_fits(nx > ny ? nx : ny, ny > nz ? ny : nz, nx + ny + nz, d))
        return CTREX_OK;
    if ((c->cyl && !atlas_fits(nx, ny + 1, nz, d)) || (c->dyr && !atlas_fits(nx, ny, nz, d)) ||
        (c->roi && !(atlas_fits(nx, ny, nz, d) && atlas_fits(rx, ry, rz, d))))
        return CTREX_OK;
    cudaError_t e = scratch_begin(c);
    if (e != cudaSuccess) return cuda_fail(c, e, "column scratch");
    e = col_ensure(c->vol_col, nx, ny, nz, c->stream, c->cyl);
    if (e == cudaSuccess && c->dyr) e = col_ensure(c->col1, nx, ny, nz, c->stream);
    if (e == cudaSuccess && c->roi) e = col_ensure(c->col1, rx, ry, rz, c->stream);
    if (e == cudaSuccess && c->dyr && !c->tau_col_set) {
        e = capturing(c) ? cudaErrorInvalidValue : col_ensure(c->tau_col, nx, ny, nz, c->stream);
        if (e == cudaSuccess) e = col_upload(c->tau_col, c->d_tau, CTREX_F32, c->stream, true);
        c->tau_col_set = e == cudaSuccess;
    }
    if (e == cudaErrorInvalidValue) {
        // the atlases need not fit beside stores that only a part of the model got
        if ((c->dyr || c->roi) && !c->scratch_captured) {
            col_release(c->vol_col);
            col_release(c->col1);
            col_release(c->tau_col);
            c->tau_col_set = false;
        }
        return CTREX_OK;
    }
    if (e == cudaSuccess) e = col_upload(c->vol_col, vol, vdt, c->stream, c->dyr);
    if (e == cudaSuccess && (c->dyr || c->roi))
        e = col_upload(c->col1, static_cast<const char *>(vol) + grid_voxels(c->grid) * dtype_size(vdt), vdt,
                       c->stream, c->dyr);
    if (e != cudaSuccess) return cuda_fail(c, e, "volume column layout");
    a.column = &c->vol_col;
    a.column1 = &c->col1;
    a.column_tau = &c->tau_col;
    return CTREX_OK;
}

// Uploads vol into the context's texture atlas and points a.atlas at it; if
// the volume does not fit the 2D texture limits the row-major path is used.
int prepare_atlas(ctrex_ctx *c, FwdArgs &a, const void *vol, int vdt)
{
    if (!c->has_motion && column_forward(c, vdt)) {
        const int e = prepare_columns(c, a, vol, vdt);
        if (e != CTREX_OK || a.column) return e;
    }
    if (c->projector == CTREX_PROJ_JOSEPH) {
        // x-, y- and z-slice stacks in one atlas; no row-major fallback
        const int nx = c->grid.nx, ny = c->grid.ny, nz = c->grid.nz;
        cudaError_t e = alloc_or_release(c, [&] {
            return atlas_ensure(c->jos_atlas, nx > ny ? nx : ny, ny > nz ? ny : nz, nx + ny + nz,
                                vdt == CTREX_BF16, c->device, false);
        });
        if (e == cudaErrorInvalidValue) {
            cudaGetLastError();
            return fail(c, CTREX_E_SHAPE, "Joseph projector: volume exceeds the 2D texture limits of the device");
        }
        if (e != cudaSuccess) return cuda_fail(c, e, "Joseph atlas allocation");
        e = atlas_upload_joseph(c->jos_atlas, vol, nx, ny, nz, c->stream);
        if (e != cudaSuccess) return cuda_fail(c, e, "Joseph atlas upload");
        c->jos_atlas_view = atlas_view(c->jos_atlas);
        a.atlas = &c->jos_atlas_view;
        return CTREX_OK;
    }
    if (c->dyr) {
        // initial values into the volume atlas, final values into their own;
        // the transition times were uploaded by set_dyrect; no row-major fallback
        const size_t off = grid_voxels(c->grid) * dtype_size(vdt);
        AtlasStore *st[2] = {&c->vol_atlas, &c->dyr_atlas1};
        Atlas *vw[2] = {&c->vol_atlas_view, &c->dyr_atlas1_view};
        for (int i = 0; i < 2; ++i) {
            cudaError_t e = alloc_or_release(c, [&] {
                return atlas_ensure(*st[i], c->grid.nx, c->grid.ny, c->grid.nz, vdt == CTREX_BF16, c->device, false);
            });
            if (e == cudaErrorInvalidValue) {
                cudaGetLastError();
                return fail(c, CTREX_E_SHAPE, "event model: the volume exceeds the 2D texture limits of the device");
            }
            if (e != cudaSuccess) return cuda_fail(c, e, "event-model atlas allocation");
            e = atlas_upload(*st[i], static_cast<const char *>(vol) + (i ? off : 0), c->stream);
            if (e != cudaSuccess) return cuda_fail(c, e, "event-model atlas upload");
            *vw[i] = atlas_view(*st[i]);
        }
        c->dyra.mu1 = &c->dyr_atlas1_view;
        c->dyra.tau_atlas = &c->tau_atlas_view;
        a.atlas = &c->vol_atlas_view;
        return CTREX_OK;
    }
    if (c->roi) {
        // context and ROI grids in atlases of their own; no row-major fallback
        const size_t off = grid_voxels(c->grid) * dtype_size(vdt);
        const Grid *gs[2] = {&c->grid, &c->roi_grid};
        AtlasStore *st[2] = {&c->vol_atlas, &c->roi_atlas};
        Atlas *vw[2] = {&c->vol_atlas_view, &c->roi_atlas_view};
        for (int i = 0; i < 2; ++i) {
            cudaError_t e = alloc_or_release(c, [&] {
                return atlas_ensure(*st[i], gs[i]->nx, gs[i]->ny, gs[i]->nz, vdt == CTREX_BF16, c->device, false);
            });
            if (e == cudaErrorInvalidValue) {
                cudaGetLastError();
                return fail(c, CTREX_E_SHAPE, "ROI projection: a grid exceeds the 2D texture limits of the device");
            }
            if (e != cudaSuccess) return cuda_fail(c, e, "ROI atlas allocation");
            e = atlas_upload(*st[i], static_cast<const char *>(vol) + (i ? off : 0), c->stream);
            if (e != cudaSuccess) return cuda_fail(c, e, "ROI atlas upload");
            *vw[i] = atlas_view(*st[i]);
        }
        a.atlas = &c->vol_atlas_view;
        a.roi_atlas = &c->roi_atlas_view;
        return CTREX_OK;
    }
    if (c->cyl) {
        // cylindrical domain: z-slice tiles of N_r x (N_phi + 1), the last row
        // repeating sector 0; no row-major fallback
        cudaError_t e = alloc_or_release(c, [&] {
            return atlas_ensure(c->vol_atlas, c->grid.nx, c->grid.ny, c->grid.nz, vdt == CTREX_BF16, c->device,
                                false, true);
        });
        if (e == cudaErrorInvalidValue) {
            cudaGetLastError();
            return fail(c, CTREX_E_SHAPE, "cylindrical volume exceeds the 2D texture limits of the device");
        }
        if (e != cudaSuccess) return cuda_fail(c, e, "volume atlas allocation");
        e = atlas_upload(c->vol_atlas, vol, c->stream);
        if (e != cudaSuccess) return cuda_fail(c, e, "volume atlas upload");
        c->vol_atlas_view = atlas_view(c->vol_atlas);
        a.atlas = &c->vol_atlas_view;
        return CTREX_OK;
    }
    if (c->atlas_unfit) return CTREX_OK;
    // BF16 volumes: slice pairs packed in 32-bit texels, one gather per sample
    cudaError_t e = alloc_or_release(c, [&] {
        return atlas_ensure(c->vol_atlas, c->grid.nx, c->grid.ny, c->grid.nz, vdt == CTREX_BF16, c->device,
                            vdt == CTREX_BF16);
    });
    if (e == cudaErrorInvalidValue) {
        cudaGetLastError();
        c->atlas_unfit = true;
        return CTREX_OK;
    }
    if (e != cudaSuccess) return cuda_fail(c, e, "volume atlas allocation");
    e = atlas_upload(c->vol_atlas, vol, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "volume atlas upload");
    c->vol_atlas_view = atlas_view(c->vol_atlas);
    a.atlas = &c->vol_atlas_view;
    return CTREX_OK;
}

// 3x3 helpers (FP64, host)
double det3(const double *m)
{
    return m[0] * (m[4] * m[8] - m[5] * m[7]) - m[1] * (m[3] * m[8] - m[5] * m[6]) + m[2] * (m[3] * m[7] - m[4] * m[6]);
}

void inv3(const double *m, double *r)
{
    const double d = det3(m);
    r[0] = (m[4] * m[8] - m[5] * m[7]) / d;
    r[1] = (m[2] * m[7] - m[1] * m[8]) / d;
    r[2] = (m[1] * m[5] - m[2] * m[4]) / d;
    r[3] = (m[5] * m[6] - m[3] * m[8]) / d;
    r[4] = (m[0] * m[8] - m[2] * m[6]) / d;
    r[5] = (m[2] * m[3] - m[0] * m[5]) / d;
    r[6] = (m[3] * m[7] - m[4] * m[6]) / d;
    r[7] = (m[1] * m[6] - m[0] * m[7]) / d;
    r[8] = (m[0] * m[4] - m[1] * m[3]) / d;
}

void set_clip_box(ctrex_ctx *c)
{
    const int n[3] = {c->grid.nx, c->grid.ny, c->grid.nz};
    const double m = c->has_motion ? c->margin : 0.0;
    for (int a = 0; a < 3; ++a) {
        c->grid.lo[a] = (float)(-0.5 - m / c->vox[a]);
        c->grid.hi[a] = (float)(n[a] - 0.5 + m / c->vox[a]);
    }
}

}  // namespace

extern "C" {

const char *ctrex_version(void) { return "ctrex-gb300 0.1 (sm_103a)"; }

const char *ctrex_last_error(const ctrex_ctx *c) { return c ? c->err.c_str() : g_static_err; }

int ctrex_create(ctrex_ctx **out, int device, void *stream)
{
    if (!out) return CTREX_E_ARG;
    *out = nullptr;
    int ndev = 0;
    cudaError_t e = cudaGetDeviceCount(&ndev);
    if (e != cudaSuccess || device < 0 || device >= ndev) {
        cudaGetLastError();
        return CTREX_E_CUDA;
    }
    ctrex_ctx *c = new (std::nothrow) ctrex_ctx();
    if (!c) return CTREX_E_NOMEM;
    c->device = device;
    c->stream = (cudaStream_t)stream;
    DeviceGuard g(device);
    if (cudaMalloc((void **)&c->d_sums, 2 * sizeof(double)) != cudaSuccess ||
        cudaMalloc((void **)&c->d_devcheck, sizeof(unsigned)) != cudaSuccess ||
        cudaMalloc((void **)&c->d_count, sizeof(unsigned long long)) != cudaSuccess ||
        cudaEventCreateWithFlags(&c->scratch_done, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        ctrex_destroy(c);
        return CTREX_E_NOMEM;
    }
    cudaMemset(c->d_devcheck, 0, sizeof(unsigned));
    *out = c;
    return CTREX_OK;
}

int ctrex_destroy(ctrex_ctx *c)
{
    if (!c) return CTREX_E_ARG;
    {
        DeviceGuard g(c->device);
        cudaStreamSynchronize(c->stream);
        dfree(c->d_views);
        dfree(c->d_motion);
        dfree(c->d_theta);
        dfree(c->d_coef);
        dfree(c->d_spline);
        dfree(c->d_dRdw);
        dfree(c->d_gM);
        dfree(c->d_gb);
        dfree(c->d_gcoef);
        dfree(c->d_partials);
        dfree(c->d_sums);
        dfree(c->d_devcheck);
        dfree(c->d_count);
        dfree(c->d_r);
        dfree(c->d_hvol);
        dfree(c->d_hp);
        dfree(c->d_hw);
        dfree(c->d_hq);
        dfree(c->d_hrs);
        dfree(c->d_hcs);
        if (c->copy_stream) cudaStreamDestroy(c->copy_stream);
        if (c->ev_vol) cudaEventDestroy(c->ev_vol);
        if (c->ev_p) cudaEventDestroy(c->ev_p);
        if (c->scratch_done) cudaEventDestroy(c->scratch_done);
        if (c->sums_done) cudaEventDestroy(c->sums_done);
        if (c->h_sums) cudaFreeHost(c->h_sums);
        dfree(c->d_subset_views);
        dfree(c->d_window);
        dfree(c->d_subset_sums);
        atlas_release(c->vol_atlas);
        col_release(c->vol_col);
        col_release(c->img_col);
        dfree(c->d_adj);
        atlas_release(c->img_atlas);
        atlas_release(c->jos_atlas);
        atlas_release(c->roi_atlas);
        dfree(c->d_views_roi);
        dyr_release(c);  // col1 with it
    }
    delete c;
    return CTREX_OK;
}

int ctrex_set_stream(ctrex_ctx *c, void *stream)
{
    if (!c) return CTREX_E_ARG;
    c->stream = (cudaStream_t)stream;
    return CTREX_OK;
}

int ctrex_device_status(ctrex_ctx *c)
{
    if (!c) return CTREX_E_ARG;
    DeviceGuard g(c->device);
    unsigned h = 0;
    CT_CUDA(c, cudaMemcpyAsync(&h, c->d_devcheck, sizeof h, cudaMemcpyDeviceToHost, c->stream));
    CT_CUDA(c, cudaStreamSynchronize(c->stream));
    if (h) {
        CT_CUDA(c, cudaMemsetAsync(c->d_devcheck, 0, sizeof(unsigned), c->stream));
        return fail(c, CTREX_E_DEVICE_CHECK, "a kernel bounds check fired (flags 0x%x): view index out of range", h);
    }
    return CTREX_OK;
}

// Shared by the Cartesian and the cylindrical set-up.  P maps the frame the
// grid is indexed in (mm) to pixels; voxel i of axis a sits at origin[a] +
// i vox[a] in that frame; ctr is the volume centre (sign normalisation of P);
// min_pitch the smallest physical pitch (step and row-sum threshold).
// Per-(view, sub) FP32 parameters of P on a grid (vox, origin); ctr fixes
// the sign normalisation.
static int compute_views(ctrex_ctx *c, const double *P, int nvs, int n_sub, const double vox[3],
                         const double origin[3], const double ctr[3], double uc, double vc, std::vector<ViewGPU> &hv)
{
    hv.assign((size_t)nvs, ViewGPU{});
    for (int q = 0; q < nvs; ++q) {
        const double *Pi = P + 12 * (size_t)q;
        double M[9], fro = 0.0;
        for (int k = 0; k < 12; ++k)
            if (!isfinite(Pi[k])) return fail(c, CTREX_E_GEOMETRY, "view %d sub %d: non-finite matrix", q / n_sub, q % n_sub);
        for (int r = 0; r < 3; ++r)
            for (int cc = 0; cc < 3; ++cc) {
                M[3 * r + cc] = Pi[4 * r + cc];
                fro += M[3 * r + cc] * M[3 * r + cc];
            }
        fro = sqrt(fro);
        if (!(fabs(det3(M)) > 1e-12 * fro * fro * fro))
            return fail(c, CTREX_E_GEOMETRY, "view %d sub %d: singular projection matrix", q / n_sub, q % n_sub);
        const double depth = Pi[8] * ctr[0] + Pi[9] * ctr[1] + Pi[10] * ctr[2] + Pi[11];
        if (!(depth != 0.0))
            return fail(c, CTREX_E_GEOMETRY, "view %d sub %d: volume centre on the source plane", q / n_sub, q % n_sub);
        const double sgn = depth > 0 ? 1.0 : -1.0;
        double Pn[12];
        for (int k = 0; k < 12; ++k) Pn[k] = sgn * Pi[k];
        for (int r = 0; r < 3; ++r)
            for (int cc = 0; cc < 3; ++cc) M[3 * r + cc] = Pn[4 * r + cc];
        double Mi[9];
        inv3(M, Mi);
        double src[3];
        for (int r = 0; r < 3; ++r) src[r] = -(Mi[3 * r] * Pn[3] + Mi[3 * r + 1] * Pn[7] + Mi[3 * r + 2] * Pn[11]);
        const double lam = sgn * depth;  // depth of the volume centre, > 0
        ViewGPU &V = hv[(size_t)q];
        for (int a = 0; a < 3; ++a) {
            const double mc = Mi[3 * a] * uc + Mi[3 * a + 1] * vc + Mi[3 * a + 2];
            const double dref = lam * mc;  // X(uc,vc) - source, mm
            V.dref[a] = (float)(dref / vox[a]);
            V.ref[a] = (float)((src[a] + dref - origin[a]) / vox[a]);
            V.qu[a] = (float)(lam * Mi[3 * a] / vox[a]);
            V.qv[a] = (float)(lam * Mi[3 * a + 1] / vox[a]);
        }
        // h = Pn [origin + vox * i; 1]
        for (int r = 0; r < 3; ++r) {
            double acc = Pn[4 * r + 3];
            for (int a = 0; a < 3; ++a) {
                V.P[4 * r + a] = (float)(Pn[4 * r + a] * vox[a]);
                acc += Pn[4 * r + a] * origin[a];
            }
            V.P[4 * r + 3] = (float)acc;
        }
    }
    return CTREX_OK;
}

// A pixel step along a detector column, in index coordinates at the volume's
// depth: its sideways part over its part along z, the latter, and its length
// (means over the views).
static void detector_column_step(const std::vector<ViewGPU> &hv, double &lean, double &step, double &pixel)
{
    lean = step = pixel = 0.0;
    for (const ViewGPU &V : hv) {
        const double xy = sqrt((double)V.qv[0] * V.qv[0] + (double)V.qv[1] * V.qv[1]), z = fabs((double)V.qv[2]);
        lean += xy <= 10.0 * z ? xy / z : 10.0;
        step += z;
        pixel += sqrt(xy * xy + z * z);
    }
    lean /= (double)hv.size();
    step /= (double)hv.size();
    pixel /= (double)hv.size();
}

// What share of the backprojection's blocks (columns side by side, 64 slices)
// project inside the detector or the window and take the short path, from a
// sample: eight views, nine places in x and y, the first, a middle and the last
// block of slices (0.05 ms).
static void set_bp_inside(ctrex_ctx *c)
{
    const Grid &G = c->grid;
    const int n = (int)c->hviews.size(), blocks = (G.nz + 63) / 64, nv = n < 8 ? n : 8;
    int inside = 0, all = 0;
    for (int i = 0; i < nv; ++i) {
        const int view = (int)((long long)i * n / nv);
        const int4 win = c->has_window ? c->hwindow[(size_t)(view / G.n_sub)] : make_int4(0, G.nu - 1, 0, G.nv - 1);
        for (int q = 0; q < 9; ++q)
            for (int z = 0; z < 3 && z < blocks; ++z) {
                const int zb = z == 0 ? 0 : (z == 1 ? (blocks - 1 + (blocks > 2)) / 2 : blocks - 1);
                const int z0 = zb * 64 + 64 > G.nz && G.nz > 64 ? G.nz - 64 : zb * 64;
                float lo[3], hi[3];
                if (c->cyl) {  // the axis and eight places around it
                    const double a = 0.25 * M_PI * q, r = q == 8 ? 0.0 : 0.7 * c->cylg.R;
                    const double p[2] = {r * cos(a), r * sin(a)};
                    for (int k = 0; k < 2; ++k) {
                        lo[k] = (float)(p[k] - 4.0 * c->cylg.dr);
                        hi[k] = (float)(p[k] + 4.0 * c->cylg.dr);
                    }
                    lo[2] = (z0 - c->cylg.zc) * c->cylg.dz;
                    hi[2] = (z0 + 63 - c->cylg.zc) * c->cylg.dz;
                } else {
                    const int wide = G.nx < 8 ? G.nx : 8;  // the first, middle and last columns
                    lo[0] = (float)((G.nx - wide) * (q % 3) / 2);
                    hi[0] = lo[0] + wide - 1;
                    lo[1] = hi[1] = (float)((G.ny - 1) * (q / 3) / 2);
                    lo[2] = (float)z0;
                    hi[2] = (float)(z0 + 63);
                }
                inside += backproject_box(c->hviews[(size_t)view], lo, hi, win);
                ++all;
            }
    }
    c->bp_inside = (double)inside / all;
}

// Gives back the stores of an earlier geometry that this one does not use.
static void drop_unused_columns(ctrex_ctx *c)
{
    DeviceGuard g(c->device);
    if (!column_forward(c, CTREX_F32) && !column_forward(c, CTREX_BF16)) col_release(c->vol_col);
    if (!column_backproject(c, CTREX_F32) && !column_backproject(c, CTREX_BF16)) col_release(c->img_col);
}

static int build_geometry(ctrex_ctx *c, const double *P, int n_views, int n_sub, const int n[3], const double vox[3],
                          const double origin[3], const double ctr[3], double min_pitch, const ctrex_det_grid *det,
                          double step_vox)
{
    DeviceGuard g(c->device);
    const int nvs = n_views * n_sub;
    std::vector<ViewGPU> hv;
    const double uc = 0.5 * (det->nu - 1), vc = 0.5 * (det->nv - 1);
    int e = compute_views(c, P, nvs, n_sub, vox, origin, ctr, uc, vc, hv);
    if (e) return e;
    // the world matrices and the centre, for a later ROI grid
    c->hostP.assign(P, P + 12 * (size_t)nvs);
    for (int a = 0; a < 3; ++a) c->ctr[a] = ctr[a];
    dfree(c->d_views);
    dfree(c->d_views_roi);
    c->roi = false;
    atlas_release(c->roi_atlas);
    dyr_release(c);
    dfree(c->d_window);
    c->has_window = false;
    // motion buffers are sized by n_views: drop them with the old geometry
    dfree(c->d_motion);
    dfree(c->d_dRdw);
    dfree(c->d_theta);
    dfree(c->d_coef);
    dfree(c->d_spline);
    dfree(c->d_gM);
    dfree(c->d_gb);
    dfree(c->d_gcoef);
    c->coef_valid = c->theta_valid = false;
    CT_CUDA(c, cudaMalloc((void **)&c->d_views, sizeof(ViewGPU) * (size_t)nvs));
    CT_CUDA(c, cudaMemcpy(c->d_views, hv.data(), sizeof(ViewGPU) * (size_t)nvs, cudaMemcpyHostToDevice));
    Grid &G = c->grid;
    G.nx = n[0];
    G.ny = n[1];
    G.nz = n[2];
    G.nu = det->nu;
    G.nv = det->nv;
    G.n_views = n_views;
    G.n_sub = n_sub;
    const double minv = min_pitch;
    for (int a = 0; a < 3; ++a) {
        c->vox[a] = vox[a];
        c->origin[a] = origin[a];
        G.vox[a] = (float)vox[a];
        G.spl_scale[a] = (float)(5.0 / n[a]);
    }
    c->step_vox = step_vox;
    G.step_mm = (float)(step_vox * minv);
    G.uc = (float)uc;
    G.vc = (float)vc;
    G.eps_R = (float)(1e-6 * minv);
    G.inv_sub = (float)(1.0 / n_sub);
    c->has_motion = false;
    c->cyl = false;
    c->has_geom = true;
    c->atlas_unfit = false;
    c->img_atlas_unfit = false;
    detector_column_step(hv, c->col_lean, c->col_step, c->col_pixel);
    c->bp_flat = backproject_flat(G, hv.data(), nvs);
    c->hviews.swap(hv);
    c->hwindow.clear();
    set_bp_inside(c);
    set_clip_box(c);
    return CTREX_OK;
}


int ctrex_set_geometry(ctrex_ctx *c, const double *P, int n_views, int n_sub, const ctrex_vol_grid *vol,
                       const ctrex_det_grid *det, double step_vox)
{
    if (!c) return CTREX_E_ARG;
    if (!P || !vol || !det) return fail(c, CTREX_E_ARG, "set_geometry: NULL argument");
    if (n_views < 1 || n_sub < 1 || (long long)n_views * n_sub > (1 << 24))
        return fail(c, CTREX_E_SHAPE, "set_geometry: bad n_views %d / n_sub %d", n_views, n_sub);
    if (vol->nx < 1 || vol->ny < 1 || vol->nz < 1 || (long long)vol->nx * vol->ny * vol->nz >= (1LL << 31))
        return fail(c, CTREX_E_SHAPE, "set_geometry: volume %d x %d x %d unsupported", vol->nx, vol->ny, vol->nz);
    if (det->nu < 1 || det->nv < 1 || det->nv > 4 * 65535 || (long long)det->nu * det->nv >= (1LL << 31))
        return fail(c, CTREX_E_SHAPE, "set_geometry: detector %d x %d unsupported", det->nu, det->nv);
    for (int a = 0; a < 3; ++a)
        if (!(vol->vox[a] > 0.0) || !isfinite(vol->origin[a]))
            return fail(c, CTREX_E_ARG, "set_geometry: voxel pitch must be > 0 and origin finite");
    // bounded step keeps every ray's sample count (and kernel run time) bounded
    if (!(step_vox >= 1e-2 && step_vox <= 100.0))
        return fail(c, CTREX_E_ARG, "set_geometry: step_vox must lie in [0.01, 100]");
    const int n[3] = {vol->nx, vol->ny, vol->nz};
    double ctr[3], minv = vol->vox[0];
    for (int a = 0; a < 3; ++a) {
        ctr[a] = vol->origin[a] + 0.5 * (n[a] - 1) * vol->vox[a];
        minv = fmin(minv, vol->vox[a]);
    }
    const int e = build_geometry(c, P, n_views, n_sub, n, vol->vox, vol->origin, ctr, minv, det, step_vox);
    if (e == CTREX_OK) drop_unused_columns(c);
    return e;
}

int ctrex_set_geometry_cylinder(ctrex_ctx *c, const double *P, int n_views, int n_sub, const ctrex_cyl_grid *cyl,
                                const ctrex_det_grid *det, double step_vox)
{
    if (!c) return CTREX_E_ARG;
    if (!P || !cyl || !det) return fail(c, CTREX_E_ARG, "set_geometry_cylinder: NULL argument");
    if (n_views < 1 || n_sub < 1 || (long long)n_views * n_sub > (1 << 24))
        return fail(c, CTREX_E_SHAPE, "set_geometry_cylinder: bad n_views %d / n_sub %d", n_views, n_sub);
    if (cyl->n_r < 1 || cyl->n_phi < 3 || cyl->n_z < 1 ||
        (long long)cyl->n_r * (cyl->n_phi + 1) * cyl->n_z >= (1LL << 31))
        return fail(c, CTREX_E_SHAPE, "set_geometry_cylinder: grid %d x %d x %d unsupported", cyl->n_r, cyl->n_phi,
                    cyl->n_z);
    if (det->nu < 1 || det->nv < 1 || det->nv > 4 * 65535 || (long long)det->nu * det->nv >= (1LL << 31))
        return fail(c, CTREX_E_SHAPE, "set_geometry_cylinder: detector %d x %d unsupported", det->nu, det->nv);
    if (!(cyl->dr > 0.0 && isfinite(cyl->dr) && cyl->dz > 0.0 && isfinite(cyl->dz)))
        return fail(c, CTREX_E_ARG, "set_geometry_cylinder: dr and dz must be finite and > 0");
    if (!(step_vox >= 1e-2 && step_vox <= 100.0))
        return fail(c, CTREX_E_ARG, "set_geometry_cylinder: step_vox must lie in [0.01, 100]");
    // the pose must be a rigid motion: Rc orthonormal with det +1
    const double *T = cyl->pose;
    for (int k = 0; k < 12; ++k)
        if (!isfinite(T[k])) return fail(c, CTREX_E_ARG, "set_geometry_cylinder: non-finite pose");
    double Rc[9];
    for (int r = 0; r < 3; ++r)
        for (int k = 0; k < 3; ++k) Rc[3 * r + k] = T[4 * r + k];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            const double d = Rc[i] * Rc[j] + Rc[3 + i] * Rc[3 + j] + Rc[6 + i] * Rc[6 + j];
            if (fabs(d - (i == j ? 1.0 : 0.0)) > 1e-9)
                return fail(c, CTREX_E_ARG, "set_geometry_cylinder: pose rotation is not orthonormal");
        }
    if (!(det3(Rc) > 0.0)) return fail(c, CTREX_E_ARG, "set_geometry_cylinder: pose rotation is a reflection");
    // P_q = P [Rc^T | -Rc^T tc]: the matrices act on cylinder-frame mm
    const size_t nvs = (size_t)n_views * n_sub;
    std::vector<double> Pq(12 * nvs);
    const double tc[3] = {T[3], T[7], T[11]};
    double inv[12];
    for (int r = 0; r < 3; ++r) {
        for (int k = 0; k < 3; ++k) inv[4 * r + k] = Rc[3 * k + r];
        inv[4 * r + 3] = -(Rc[r] * tc[0] + Rc[3 + r] * tc[1] + Rc[6 + r] * tc[2]);
    }
    for (size_t q = 0; q < nvs; ++q) {
        const double *Pi = P + 12 * q;
        double *Po = Pq.data() + 12 * q;
        for (int r = 0; r < 3; ++r)
            for (int k = 0; k < 4; ++k) {
                double acc = k == 3 ? Pi[4 * r + 3] : 0.0;
                for (int m = 0; m < 3; ++m) acc += Pi[4 * r + m] * inv[4 * m + k];
                Po[4 * r + k] = acc;
            }
    }
    const int n[3] = {cyl->n_r, cyl->n_phi, cyl->n_z};
    const double one[3] = {1.0, 1.0, 1.0}, zero[3] = {0.0, 0.0, 0.0};
    const int e = build_geometry(c, Pq.data(), n_views, n_sub, n, one, zero, zero, fmin(cyl->dr, cyl->dz), det,
                                 step_vox);
    if (e) return e;
    CylGPU &C = c->cylg;
    const double two_pi = 6.283185307179586476925286766559;
    C.n_r = cyl->n_r;
    C.n_phi = cyl->n_phi;
    C.n_z = cyl->n_z;
    C.dr = (float)cyl->dr;
    C.dphi = (float)(two_pi / cyl->n_phi);
    C.dz = (float)cyl->dz;
    C.inv_dr = (float)(1.0 / cyl->dr);
    C.inv_dphi = (float)(cyl->n_phi / two_pi);
    C.inv_dz = (float)(1.0 / cyl->dz);
    C.zc = (float)(0.5 * (cyl->n_z - 1));
    C.R = (float)(cyl->n_r * cyl->dr);
    C.Z = (float)(0.5 * cyl->n_z * cyl->dz);
    // bounding box of the cylinder (frame mm), for anything that reads the clip box
    for (int a = 0; a < 2; ++a) {
        c->grid.lo[a] = -C.R;
        c->grid.hi[a] = C.R;
    }
    c->grid.lo[2] = -C.Z;
    c->grid.hi[2] = C.Z;
    c->cyl = true;
    c->col_step /= cyl->dz;  // frame mm to slices
    c->col_pixel /= cyl->dz;
    set_bp_inside(c);
    c->projector = CTREX_PROJ_TRILINEAR;
    drop_unused_columns(c);
    return CTREX_OK;
}

int ctrex_set_motion(ctrex_ctx *c, const float *theta, const float *coef, const float *s_view, double margin_mm)
{
    if (!c) return CTREX_E_ARG;
    if (!c->has_geom) return fail(c, CTREX_E_STATE, "set_motion before set_geometry");
    if ((c->cyl || c->roi || c->dyr || c->projector == CTREX_PROJ_JOSEPH) && (theta || coef || s_view))
        return fail(c, CTREX_E_STATE, "set_motion: the motion model is defined for the trilinear projector on the "
                                      "Cartesian grid only, without the event model");
    double box = 0.0;
    const int nn[3] = {c->grid.nx, c->grid.ny, c->grid.nz};
    for (int a = 0; a < 3; ++a) box = fmax(box, nn[a] * c->vox[a]);
    if (!(margin_mm >= 0.0 && margin_mm <= box))
        return fail(c, CTREX_E_ARG, "set_motion: margin must lie in [0, largest box edge]");
    DeviceGuard g(c->device);
    if (!theta && !coef && !s_view) {
        c->has_motion = false;
        set_clip_box(c);
        return CTREX_OK;
    }
    const int V = c->grid.n_views;
    if (!c->d_motion) {
        CT_CUDA(c, cudaMalloc((void **)&c->d_motion, sizeof(MotionGPU) * (size_t)V));
        CT_CUDA(c, cudaMalloc((void **)&c->d_dRdw, sizeof(float) * 27 * (size_t)V));
        CT_CUDA(c, cudaMalloc((void **)&c->d_theta, sizeof(float) * 15 * (size_t)V));
        CT_CUDA(c, cudaMalloc((void **)&c->d_coef, sizeof(float) * 1536));
        CT_CUDA(c, cudaMalloc((void **)&c->d_spline, sizeof(float4) * SPLINE_TABLE));
        CT_CUDA(c, cudaMalloc((void **)&c->d_gM, sizeof(double) * 9 * (size_t)V));
        CT_CUDA(c, cudaMalloc((void **)&c->d_gb, sizeof(double) * 3 * (size_t)V));
        CT_CUDA(c, cudaMalloc((void **)&c->d_gcoef, sizeof(double) * 1536));
    }
    const float *th = nullptr;
    if (theta) {
        CT_CUDA(c, cudaMemcpyAsync(c->d_theta, theta, sizeof(float) * 15 * (size_t)V, cudaMemcpyDeviceToDevice, c->stream));
        th = c->d_theta;
    }
    const float *co = nullptr;
    if (coef) {
        CT_CUDA(c, cudaMemcpyAsync(c->d_coef, coef, sizeof(float) * 1536, cudaMemcpyDeviceToDevice, c->stream));
        co = c->d_coef;
    }
    const float *sv = nullptr;
    // s_view is consumed by the set-up kernel straight from the caller's buffer
    if (s_view) sv = s_view;
    c->margin = margin_mm;
    c->has_motion = true;
    cudaError_t e = launch_motion_setup(th, co, sv, V, c->grid, c->vox, c->origin, c->d_motion, c->d_spline,
                                        c->d_dRdw, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "motion set-up");
    c->coef_valid = co != nullptr;
    c->theta_valid = th != nullptr;
    set_clip_box(c);
    return CTREX_OK;
}

int ctrex_set_bp_window(ctrex_ctx *c, const int *window)
{
    if (!c) return CTREX_E_ARG;
    if (!c->has_geom) return fail(c, CTREX_E_STATE, "set_bp_window before set_geometry");
    if (!window) {
        c->has_window = false;
        set_bp_inside(c);
        return CTREX_OK;
    }
    const int V = c->grid.n_views;
    std::vector<int4> hw((size_t)V);
    for (int v = 0; v < V; ++v) {
        const int *q = window + 4 * (size_t)v;
        hw[(size_t)v] = make_int4(q[0] > 0 ? q[0] : 0, q[1] < c->grid.nu - 1 ? q[1] : c->grid.nu - 1,
                                  q[2] > 0 ? q[2] : 0, q[3] < c->grid.nv - 1 ? q[3] : c->grid.nv - 1);
    }
    DeviceGuard g(c->device);
    if (!c->d_window) CT_CUDA(c, cudaMalloc((void **)&c->d_window, sizeof(int4) * (size_t)V));
    CT_CUDA(c, cudaMemcpyAsync(c->d_window, hw.data(), sizeof(int4) * (size_t)V, cudaMemcpyHostToDevice, c->stream));
    CT_CUDA(c, cudaStreamSynchronize(c->stream));  // hw is a local buffer
    c->has_window = true;
    c->hwindow.swap(hw);
    set_bp_inside(c);
    return CTREX_OK;
}

int ctrex_set_roi(ctrex_ctx *c, const ctrex_vol_grid *roi)
{
    if (!c) return CTREX_E_ARG;
    if (!c->has_geom) return fail(c, CTREX_E_STATE, "set_roi before set_geometry");
    DeviceGuard g(c->device);
    if (!roi) {
        c->roi = false;
        dfree(c->d_views_roi);
        atlas_release(c->roi_atlas);
        col_release(c->col1);
        return CTREX_OK;
    }
    if (c->cyl || c->has_motion || c->dyr || c->projector != CTREX_PROJ_TRILINEAR)
        return fail(c, CTREX_E_STATE, "set_roi: the ROI projector is the trilinear one on a Cartesian grid without "
                                      "motion or the event model");
    if (roi->nx < 1 || roi->ny < 1 || roi->nz < 1 ||
        (long long)roi->nx * roi->ny * roi->nz + (long long)grid_voxels(c->grid) >= (1LL << 31))
        return fail(c, CTREX_E_SHAPE, "set_roi: grid %d x %d x %d unsupported", roi->nx, roi->ny, roi->nz);
    const int n[3] = {roi->nx, roi->ny, roi->nz}, nc[3] = {c->grid.nx, c->grid.ny, c->grid.nz};
    double lo[3], hi[3];
    for (int a = 0; a < 3; ++a) {
        if (!(roi->vox[a] > 0.0) || !isfinite(roi->vox[a]) || !isfinite(roi->origin[a]))
            return fail(c, CTREX_E_ARG, "set_roi: voxel pitch must be > 0 and origin finite");
        // the ROI box must lie inside the context grid's box
        lo[a] = roi->origin[a] - 0.5 * roi->vox[a];
        hi[a] = roi->origin[a] + (n[a] - 0.5) * roi->vox[a];
        const double clo = c->origin[a] - 0.5 * c->vox[a], chi = c->origin[a] + (nc[a] - 0.5) * c->vox[a];
        const double tol = 1e-9 * (chi - clo);
        if (lo[a] < clo - tol || hi[a] > chi + tol)
            return fail(c, CTREX_E_ARG, "set_roi: the ROI box leaves the context grid's box on axis %d", a);
    }
    const int nvs = c->grid.n_views * c->grid.n_sub;
    std::vector<ViewGPU> hv;
    int e = compute_views(c, c->hostP.data(), nvs, c->grid.n_sub, roi->vox, roi->origin, c->ctr, c->grid.uc,
                          c->grid.vc, hv);
    if (e) return e;
    dfree(c->d_views_roi);
    CT_CUDA(c, cudaMalloc((void **)&c->d_views_roi, sizeof(ViewGPU) * (size_t)nvs));
    CT_CUDA(c, cudaMemcpy(c->d_views_roi, hv.data(), sizeof(ViewGPU) * (size_t)nvs, cudaMemcpyHostToDevice));
    Grid &F = c->roi_grid;
    F = c->grid;
    F.nx = n[0];
    F.ny = n[1];
    F.nz = n[2];
    double minf = roi->vox[0];
    for (int a = 0; a < 3; ++a) {
        F.vox[a] = (float)roi->vox[a];
        minf = fmin(minf, roi->vox[a]);
        F.lo[a] = -0.5f;
        F.hi[a] = (float)(n[a] - 0.5);
    }
    c->bp_flat_roi = backproject_flat(F, hv.data(), nvs);
    F.step_mm = (float)(c->step_vox * minf);
    RoiGPU &R = c->roig;
    for (int a = 0; a < 3; ++a) {
        R.sc[a] = (float)(c->vox[a] / roi->vox[a]);
        R.oc[a] = (float)((c->origin[a] - roi->origin[a]) / roi->vox[a]);
        R.lo[a] = (float)((lo[a] - c->origin[a]) / c->vox[a]);
        R.hi[a] = (float)((hi[a] - c->origin[a]) / c->vox[a]);
    }
    R.step_mm = F.step_mm;
    for (int a = 0; a < 3; ++a) R.n[a] = n[a];
    c->roi = true;
    return CTREX_OK;
}

int ctrex_set_projector(ctrex_ctx *c, int kind)
{
    if (!c) return CTREX_E_ARG;
    if (kind != CTREX_PROJ_TRILINEAR && kind != CTREX_PROJ_JOSEPH)
        return fail(c, CTREX_E_ARG, "set_projector: unknown projector %d", kind);
    if (kind == CTREX_PROJ_JOSEPH && (c->cyl || c->has_motion || c->roi || c->dyr))
        return fail(c, CTREX_E_STATE, "set_projector: the Joseph projector is defined on the Cartesian grid "
                                      "without motion or the event model");
    c->projector = kind;
    if (kind != CTREX_PROJ_JOSEPH) atlas_release(c->jos_atlas);
    return CTREX_OK;
}

int ctrex_set_bp_subvoxel(ctrex_ctx *c, int s)
{
    if (!c) return CTREX_E_ARG;
    if (s < 1 || s > CTREX_MAX_SUBVOXEL) return fail(c, CTREX_E_ARG, "set_bp_subvoxel: s must be in [1, 8]");
    if (s > 1 && c->dyr) return fail(c, CTREX_E_STATE, "set_bp_subvoxel: not defined with the event model");
    c->bp_subvoxel = s;
    return CTREX_OK;
}

int ctrex_set_dyrect(ctrex_ctx *c, const float *tau, const float *t_view)
{
    if (!c) return CTREX_E_ARG;
    if (!c->has_geom) return fail(c, CTREX_E_STATE, "set_dyrect before set_geometry");
    DeviceGuard g(c->device);
    if (!tau) {
        dyr_release(c);
        return CTREX_OK;
    }
    if (!t_view) return fail(c, CTREX_E_ARG, "set_dyrect: t_view is NULL");
    if (c->cyl || c->roi || c->has_motion || c->projector != CTREX_PROJ_TRILINEAR || c->bp_subvoxel > 1)
        return fail(c, CTREX_E_STATE, "set_dyrect: the event model is defined for the trilinear projector on one "
                                      "Cartesian grid, without motion, ROI or sub-voxel backprojection");
    if (2 * (long long)grid_voxels(c->grid) >= (1LL << 31))
        return fail(c, CTREX_E_SHAPE, "set_dyrect: the two value fields exceed 2^31 elements");
    const size_t nvox = grid_voxels(c->grid), V = (size_t)c->grid.n_views;
    if (!c->d_tau) CT_CUDA(c, cudaMalloc((void **)&c->d_tau, sizeof(float) * nvox));
    if (!c->d_tview) CT_CUDA(c, cudaMalloc((void **)&c->d_tview, sizeof(float) * V));
    CT_CUDA(c, cudaMemcpyAsync(c->d_tau, tau, sizeof(float) * nvox, cudaMemcpyDeviceToDevice, c->stream));
    CT_CUDA(c, cudaMemcpyAsync(c->d_tview, t_view, sizeof(float) * V, cudaMemcpyDeviceToDevice, c->stream));
    cudaError_t e = alloc_or_release(c, [&] {
        return atlas_ensure(c->tau_atlas, c->grid.nx, c->grid.ny, c->grid.nz, false, c->device, false);
    });
    if (e == cudaErrorInvalidValue) {
        cudaGetLastError();
        dyr_release(c);
        return fail(c, CTREX_E_SHAPE, "set_dyrect: the volume exceeds the 2D texture limits of the device");
    }
    if (e != cudaSuccess) return cuda_fail(c, e, "transition-time atlas allocation");
    e = atlas_upload(c->tau_atlas, c->d_tau, c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "transition-time atlas upload");
    c->tau_atlas_view = atlas_view(c->tau_atlas);
    const int bnx = (c->grid.nx + 7) / 8, bny = (c->grid.ny + 7) / 8, bnz = (c->grid.nz + 7) / 8;
    if (!c->d_tau_brick)
        CT_CUDA(c, cudaMalloc((void **)&c->d_tau_brick, sizeof(float2) * (size_t)bnx * bny * bnz));
    if (!c->d_tau_block)
        CT_CUDA(c, cudaMalloc((void **)&c->d_tau_block, sizeof(float2) * (size_t)bnx * bny * bnz));
    const int cnx = (c->grid.nx + 3) / 4, cny = (c->grid.ny + 3) / 4, cnz = (c->grid.nz + 3) / 4;
    if (!c->d_tau_cell)
        CT_CUDA(c, cudaMalloc((void **)&c->d_tau_cell, sizeof(float2) * (size_t)cnx * cny * cnz));
    e = launch_tau_bricks(c->d_tau, c->grid.nx, c->grid.ny, c->grid.nz, c->d_tau_cell, c->d_tau_brick, c->d_tau_block,
                          c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "transition-time bricks");
    c->tau_col_set = false;
    c->dyra.tau_brick = c->d_tau_brick;
    c->dyra.tau_block = c->d_tau_block;
    c->dyra.bnx = bnx;
    c->dyra.bny = bny;
    c->dyra.tau = c->d_tau;
    c->dyra.t_view = c->d_tview;
    c->dyra.tau_atlas = &c->tau_atlas_view;
    c->dyra.mu1 = &c->dyr_atlas1_view;
    c->dyr = true;
    return CTREX_OK;
}

int ctrex_fwd_project(ctrex_ctx *c, const void *vol, int vdt, void *proj, int pdt, float *rowsum,
                      const int *view_idx, int n_idx)
{
    if (!c) return CTREX_E_ARG;
    int e = check_views(c, view_idx, n_idx);
    if (e) return e;
    if (n_idx == 0) return CTREX_OK;  // nothing to project
    if (!vol || !proj) return fail(c, CTREX_E_ARG, "fwd_project: NULL buffer");
    if (!dtype_ok(vdt) || !dtype_ok(pdt)) return fail(c, CTREX_E_DTYPE, "fwd_project: bad dtype");
    DeviceGuard g(c->device);
    ScratchUse use(c);
    FwdArgs a = fwd_args(c, vol, vdt, view_idx, n_idx);
    e = prepare_atlas(c, a, vol, vdt);
    if (e) return e;
    cudaError_t ce = launch_forward(a, proj, pdt, rowsum);
    if (ce != cudaSuccess) return cuda_fail(c, ce, "fwd_project launch");
    return CTREX_OK;
}

static int ensure_partials(ctrex_ctx *c, int n_idx)
{
    const int need = forward_partials_needed(c->grid, n_idx);
    if (need <= c->partials_cap) return CTREX_OK;
    size_t have = (size_t)c->partials_cap * 2 * sizeof(float);
    int e = ensure(c, (void **)&c->d_partials, &have, (size_t)need * 2 * sizeof(float), "residual partials");
    if (e) return e;
    c->partials_cap = need;
    return CTREX_OK;
}

int ctrex_fwd_correct(ctrex_ctx *c, const void *vol, int vdt, const void *p, int pdt, void *r, int rdt,
                      double *sums, const int *view_idx, int n_idx)
{
    if (!c) return CTREX_E_ARG;
    int e = check_views(c, view_idx, n_idx);
    if (e) return e;
    if (n_idx == 0) {  // empty view list: zero norms, no images
        if (sums) CT_CUDA(c, cudaMemsetAsync(sums, 0, 2 * sizeof(double), c->stream));
        return CTREX_OK;
    }
    if (!vol || !p || !r) return fail(c, CTREX_E_ARG, "fwd_correct: NULL buffer");
    if (!dtype_ok(vdt) || !dtype_ok(pdt) || !dtype_ok(rdt)) return fail(c, CTREX_E_DTYPE, "fwd_correct: bad dtype");
    if (pdt != rdt) return fail(c, CTREX_E_DTYPE, "fwd_correct: p and r must share one dtype");
    DeviceGuard g(c->device);
    ScratchUse use(c);
    e = ensure_partials(c, n_idx);
    if (e) return e;
    FwdArgs a = fwd_args(c, vol, vdt, view_idx, n_idx);
    a.norm_tiles = true;
    e = prepare_atlas(c, a, vol, vdt);
    if (e) return e;
    cudaError_t ce = launch_forward_correct(a, p, pdt, r, rdt, c->d_partials, c->partials_cap, sums);
    if (ce != cudaSuccess) return cuda_fail(c, ce, "fwd_correct launch");
    return CTREX_OK;
}

// The images of a backprojection into the layout that it reads.
static int bp_images(ctrex_ctx *c, BpArgs &a, const void *r, int rdt, int n_idx)
{
    if (n_idx > 0 && column_backproject(c, rdt)) {
        CT_CUDA(c, scratch_begin(c));
        cudaError_t ae = col_ensure_images(c->img_col, c->grid.nu, c->grid.nv, n_idx, c->stream);
        if (ae == cudaSuccess) {
            ae = col_upload_images(c->img_col, r, rdt, n_idx, c->stream);
            if (ae != cudaSuccess) return cuda_fail(c, ae, "image column upload");
            a.column = &c->img_col;
        } else if (ae != cudaErrorInvalidValue) {
            return cuda_fail(c, ae, "image column layout");
        }
    }
    if (n_idx > 0 && !a.column && !c->img_atlas_unfit) {
        cudaError_t ae = alloc_or_release(c, [&] {
            return atlas_ensure(c->img_atlas, c->grid.nu, c->grid.nv, n_idx, rdt == CTREX_BF16, c->device);
        });
        if (ae == cudaErrorInvalidValue) {
            cudaGetLastError();
            c->img_atlas_unfit = true;
        } else if (ae != cudaSuccess) {
            return cuda_fail(c, ae, "image atlas allocation");
        } else {
            ae = atlas_upload(c->img_atlas, r, c->stream);
            if (ae != cudaSuccess) return cuda_fail(c, ae, "image atlas upload");
            c->img_atlas_view = atlas_view(c->img_atlas);
            a.atlas = &c->img_atlas_view;
        }
    }
    return CTREX_OK;
}

// The backprojection of images that bp_images() has laid out in `a`.
static int bp_run(ctrex_ctx *c, BpArgs &a, const void *r, int rdt, void *vol, int vdt, const float *w, float alpha,
                  int normalize, int accumulate, const int *view_idx, int n_idx)
{
    a.grid = &c->grid;
    a.views = c->d_views;
    a.view_idx = view_idx;
    a.n_idx = n_idx;
    a.r = r;
    a.r_dtype = rdt;
    a.vol = vol;
    a.vol_dtype = vdt;
    a.w = w;
    a.alpha = alpha;
    a.normalize = normalize ? 1 : 0;
    a.accumulate = accumulate ? 1 : 0;
    a.stream = c->stream;
    a.window = c->has_window ? c->d_window : nullptr;
    a.subvox = c->bp_subvoxel;
    a.cyl = c->cyl ? &c->cylg : nullptr;
    a.dyr = c->dyr ? &c->dyra : nullptr;
    a.flat = c->bp_flat && !c->cyl;
    cudaError_t ce = launch_backproject(a);
    if (ce != cudaSuccess) return cuda_fail(c, ce, "back_project launch");
    if (c->roi) {  // the ROI grid's voxels follow the context grid's
        const size_t nc = grid_voxels(c->grid);
        a.grid = &c->roi_grid;
        a.views = c->d_views_roi;
        a.flat = c->bp_flat_roi;
        a.vol = static_cast<char *>(vol) + nc * dtype_size(vdt);
        a.w = w ? w + nc : nullptr;
        ce = launch_backproject(a);
        if (ce != cudaSuccess) return cuda_fail(c, ce, "back_project launch (ROI grid)");
    }
    return CTREX_OK;
}

int ctrex_back_project(ctrex_ctx *c, const void *r, int rdt, void *vol, int vdt, const float *w, float alpha,
                       int normalize, int accumulate, const int *view_idx, int n_idx)
{
    if (!c) return CTREX_E_ARG;
    int e = check_views(c, view_idx, n_idx);
    if (e) return e;
    if (!vol || (!r && n_idx > 0)) return fail(c, CTREX_E_ARG, "back_project: NULL buffer");
    if (!dtype_ok(vdt) || !dtype_ok(rdt)) return fail(c, CTREX_E_DTYPE, "back_project: bad dtype");
    if (!isfinite(alpha)) return fail(c, CTREX_E_ARG, "back_project: alpha not finite");
    DeviceGuard g(c->device);
    ScratchUse use(c);
    BpArgs a;
    e = bp_images(c, a, r, rdt, n_idx);
    return e ? e : bp_run(c, a, r, rdt, vol, vdt, w, alpha, normalize, accumulate, view_idx, n_idx);
}

int ctrex_adjoint_project(ctrex_ctx *c, const float *proj, float *vol, const int *view_idx, int n_idx)
{
    if (!c) return CTREX_E_ARG;
    int e = check_views(c, view_idx, n_idx);
    if (e) return e;
    if (c->cyl || c->roi || c->projector == CTREX_PROJ_JOSEPH)
        return fail(c, CTREX_E_STATE, "adjoint_project: the transpose of the trilinear projector on one Cartesian "
                                      "grid only");
    if (n_idx == 0) return CTREX_OK;
    if (!proj || !vol) return fail(c, CTREX_E_ARG, "adjoint_project: NULL buffer");
    DeviceGuard g(c->device);
    ScratchUse use(c);
    const FwdArgs a = fwd_args(c, nullptr, CTREX_F32, view_idx, n_idx);
    cudaError_t ce;
    if (column_adjoint(c, n_idx)) {
        CT_CUDA(c, scratch_begin(c));
        ce = launch_adjoint_column(a, adjoint_along_z(c), proj, vol, c->d_adj);
    } else {
        ce = launch_adjoint(a, proj, vol);
    }
    if (ce != cudaSuccess) return cuda_fail(c, ce, "adjoint_project launch");
    return CTREX_OK;
}

int ctrex_motion_grad(ctrex_ctx *c, const void *vol, int vdt, const float *gproj, float *grad_theta,
                      float *grad_coef, const int *view_idx, int n_idx)
{
    if (!c) return CTREX_E_ARG;
    int e = check_views(c, view_idx, n_idx);
    if (e) return e;
    if (!c->has_motion || c->dyr) return fail(c, CTREX_E_STATE, "motion_grad: set_motion has not been called");
    if (n_idx == 0) return CTREX_OK;
    if (!vol || !gproj) return fail(c, CTREX_E_ARG, "motion_grad: NULL buffer");
    if (!dtype_ok(vdt)) return fail(c, CTREX_E_DTYPE, "motion_grad: bad dtype");
    if (grad_theta && !c->theta_valid)
        return fail(c, CTREX_E_STATE, "motion_grad: grad_theta requested but no theta was set");
    if (grad_coef && !c->coef_valid)
        return fail(c, CTREX_E_STATE, "motion_grad: grad_coef requested but no coefficients were set");
    DeviceGuard g(c->device);
    ScratchUse use(c);
    const int V = c->grid.n_views;
    CT_CUDA(c, scratch_begin(c));
    CT_CUDA(c, cudaMemsetAsync(c->d_gM, 0, sizeof(double) * 9 * (size_t)V, c->stream));
    CT_CUDA(c, cudaMemsetAsync(c->d_gb, 0, sizeof(double) * 3 * (size_t)V, c->stream));
    CT_CUDA(c, cudaMemsetAsync(c->d_gcoef, 0, sizeof(double) * 1536, c->stream));
    FwdArgs a = fwd_args(c, vol, vdt, view_idx, n_idx);
    // the volume from its column store if that can be had and the rays outweigh
    // its layout (256^3, 128^2 pixels, pose alone: 1 view 0.50 ms, 0.30
    // row-major; 12 views 0.65, 1.27), row-major otherwise
    if (!capturing(c) && ray_voxels(c, n_idx) >= 0.8 * (double)grid_voxels(c->grid) &&
        col_ensure(c->vol_col, c->grid.nx, c->grid.ny, c->grid.nz, c->stream) == cudaSuccess) {
        CT_CUDA(c, col_upload(c->vol_col, vol, vdt, c->stream));
        a.column = &c->vol_col;
    }
    cudaError_t ce = launch_motion_grad(a, gproj, c->d_gM, c->d_gb, grad_coef ? c->d_gcoef : nullptr);
    if (ce != cudaSuccess) return cuda_fail(c, ce, "motion_grad launch");
    ce = launch_motion_grad_finish(c->theta_valid ? c->d_theta : nullptr, c->d_dRdw, c->d_gM, c->d_gb, c->d_gcoef, V,
                                   c->grid, c->vox, c->origin, grad_theta, grad_coef, c->stream);
    if (ce != cudaSuccess) return cuda_fail(c, ce, "motion_grad finish");
    return CTREX_OK;
}

int ctrex_sirt_iterate(ctrex_ctx *c, void *vol, int vdt, const void *p, int pdt, int max_iter, float alpha,
                       const float *w, float tol, float *hist, int *iters_done)
{
    if (!c) return CTREX_E_ARG;
    if (iters_done) *iters_done = 0;
    int e = check_views(c, nullptr, c->has_geom ? c->grid.n_views : 0);
    if (e) return e;
    if (!vol || !p) return fail(c, CTREX_E_ARG, "sirt_iterate: NULL buffer");
    if (!dtype_ok(vdt) || !dtype_ok(pdt)) return fail(c, CTREX_E_DTYPE, "sirt_iterate: bad dtype");
    if (max_iter < 0) return fail(c, CTREX_E_ARG, "sirt_iterate: max_iter < 0");
    DeviceGuard g(c->device);
    ScratchUse use(c);
    const int V = c->grid.n_views;
    const size_t rb = (size_t)V * c->grid.nu * c->grid.nv * dtype_size(pdt);
    e = ensure(c, &c->d_r, &c->r_bytes, rb, "SIRT correction images");
    if (e) return e;
    e = ensure_partials(c, V);
    if (e) return e;
    if (!c->sums_done) CT_CUDA(c, cudaEventCreateWithFlags(&c->sums_done, cudaEventDisableTiming));
    if (!c->h_sums) CT_CUDA(c, cudaMallocHost((void **)&c->h_sums, 2 * sizeof(double)));
    for (int k = 0; k < max_iter; ++k) {
        FwdArgs a = fwd_args(c, vol, vdt, nullptr, V);
        e = prepare_atlas(c, a, vol, vdt);
        if (e) return e;
        cudaError_t ce = launch_forward_correct(a, p, pdt, c->d_r, pdt, c->d_partials, c->partials_cap, c->d_sums);
        if (ce != cudaSuccess) return cuda_fail(c, ce, "sirt: fwd_correct");
        // the images' layout for the backprojection is under way while the host
        // waits for the residual
        CT_CUDA(c, cudaMemcpyAsync(c->h_sums, c->d_sums, 2 * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
        CT_CUDA(c, cudaEventRecord(c->sums_done, c->stream));
        BpArgs b;
        const int be = bp_images(c, b, c->d_r, pdt, V);
        CT_CUDA(c, cudaEventSynchronize(c->sums_done));
        const double s[2] = {c->h_sums[0], c->h_sums[1]};
        const double rho = s[1] > 0.0 ? sqrt(s[0] / s[1]) : sqrt(s[0]);
        if (hist) hist[k] = (float)rho;
        if (!isfinite(rho)) return fail(c, CTREX_E_DIVERGED, "sirt: residual not finite at iteration %d", k);
        if (rho <= (double)tol) break;
        if (be) return be;
        if (!isfinite(alpha)) return fail(c, CTREX_E_ARG, "back_project: alpha not finite");
        e = bp_run(c, b, c->d_r, pdt, vol, vdt, w, alpha, 1, 1, nullptr, V);
        if (e) return e;
        if (iters_done) *iters_done = k + 1;
    }
    return ctrex_device_status(c);
}

int ctrex_os_sirt_iterate(ctrex_ctx *c, void *vol, int vdt, const void *p, int pdt, const int *subset_views,
                          const int *subset_offsets, int n_sets, int max_cycles, float alpha, const float *w,
                          float tol, float *hist, int *cycles_done)
{
    if (!c) return CTREX_E_ARG;
    if (cycles_done) *cycles_done = 0;
    if (!c->has_geom) return fail(c, CTREX_E_STATE, "set_geometry has not been called");
    if (!vol || !p || !subset_views || !subset_offsets) return fail(c, CTREX_E_ARG, "os_sirt: NULL argument");
    if (!dtype_ok(vdt) || !dtype_ok(pdt)) return fail(c, CTREX_E_DTYPE, "os_sirt: bad dtype");
    if (n_sets < 1 || max_cycles < 0) return fail(c, CTREX_E_ARG, "os_sirt: need n_sets >= 1, max_cycles >= 0");
    const int V = c->grid.n_views;
    if (subset_offsets[0] != 0) return fail(c, CTREX_E_ARG, "os_sirt: subset_offsets[0] must be 0");
    int maxlen = 0;
    for (int s = 0; s < n_sets; ++s) {
        const int n = subset_offsets[s + 1] - subset_offsets[s];
        if (n < 0 || n > 65535) return fail(c, CTREX_E_SHAPE, "os_sirt: subset %d has size %d", s, n);
        if (n > maxlen) maxlen = n;
    }
    const int total = subset_offsets[n_sets];
    for (int i = 0; i < total; ++i)
        if (subset_views[i] < 0 || subset_views[i] >= V)
            return fail(c, CTREX_E_SHAPE, "os_sirt: view %d out of range", subset_views[i]);
    DeviceGuard g(c->device);
    ScratchUse use(c);
    int e = ensure(c, (void **)&c->d_subset_views, &c->subset_views_bytes, sizeof(int) * (size_t)(total > 0 ? total : 1),
                   "subset view lists");
    if (e) return e;
    e = ensure(c, (void **)&c->d_subset_sums, &c->subset_sums_bytes, sizeof(double) * 2 * (size_t)n_sets,
               "subset residual norms");
    if (e) return e;
    const size_t rb = (size_t)(maxlen > 0 ? maxlen : 1) * c->grid.nu * c->grid.nv * dtype_size(pdt);
    e = ensure(c, &c->d_r, &c->r_bytes, rb, "correction images");
    if (e) return e;
    e = ensure_partials(c, maxlen > 0 ? maxlen : 1);
    if (e) return e;
    if (total > 0)
        CT_CUDA(c, cudaMemcpyAsync(c->d_subset_views, subset_views, sizeof(int) * (size_t)total, cudaMemcpyHostToDevice,
                                   c->stream));
    CT_CUDA(c, cudaMemsetAsync(c->d_subset_sums, 0, sizeof(double) * 2 * (size_t)n_sets, c->stream));
    std::vector<double> sums(2 * (size_t)n_sets);
    for (int k = 0; k < max_cycles; ++k) {
        for (int s = 0; s < n_sets; ++s) {
            const int n = subset_offsets[s + 1] - subset_offsets[s];
            if (n == 0) continue;
            const int *vs = c->d_subset_views + subset_offsets[s];
            FwdArgs a = fwd_args(c, vol, vdt, vs, n);
            a.p_by_view = 1;
            e = prepare_atlas(c, a, vol, vdt);
            if (e) return e;
            cudaError_t ce = launch_forward_correct(a, p, pdt, c->d_r, pdt, c->d_partials, c->partials_cap,
                                                    c->d_subset_sums + 2 * (size_t)s);
            if (ce != cudaSuccess) return cuda_fail(c, ce, "os_sirt: fwd_correct");
            int be = ctrex_back_project(c, c->d_r, pdt, vol, vdt, w, alpha, 1, 1, vs, n);
            if (be) return be;
        }
        CT_CUDA(c, cudaMemcpyAsync(sums.data(), c->d_subset_sums, sizeof(double) * 2 * (size_t)n_sets,
                                   cudaMemcpyDeviceToHost, c->stream));
        CT_CUDA(c, cudaStreamSynchronize(c->stream));
        double acc = 0.0, p2 = 0.0;
        for (int s = 0; s < n_sets; ++s) {
            if (subset_offsets[s + 1] == subset_offsets[s]) continue;
            acc += sums[2 * (size_t)s];
            p2 += sums[2 * (size_t)s + 1];
        }
        const double rho = p2 > 0.0 ? sqrt(acc / p2) : sqrt(acc);
        if (hist) hist[k] = (float)rho;
        if (cycles_done) *cycles_done = k + 1;
        if (!isfinite(rho)) return fail(c, CTREX_E_DIVERGED, "os_sirt: residual not finite in cycle %d", k);
        if (rho <= (double)tol) break;
    }
    return ctrex_device_status(c);
}

int ctrex_sirt_host(ctrex_ctx *c, void *vol_h, int vdt, const void *p_h, int pdt, int max_iter, float alpha,
                    const float *w_h, float tol, float *hist, int *iters_done)
{
    if (!c) return CTREX_E_ARG;
    if (!c->has_geom) return fail(c, CTREX_E_STATE, "set_geometry has not been called");
    if (!vol_h || !p_h) return fail(c, CTREX_E_ARG, "sirt_host: NULL buffer");
    if (!dtype_ok(vdt) || !dtype_ok(pdt)) return fail(c, CTREX_E_DTYPE, "sirt_host: bad dtype");
    DeviceGuard g(c->device);
    ScratchUse use(c);
    const Grid &G = c->grid;
    const size_t nvox = volume_elems(c);
    const size_t vb = nvox * dtype_size(vdt);
    const size_t pb = (size_t)G.n_views * G.nu * G.nv * dtype_size(pdt);
    int e = ensure(c, &c->d_hvol, &c->hvol_bytes, vb, "host-SIRT volume");
    if (e) return e;
    e = ensure(c, &c->d_hp, &c->hp_bytes, pb, "host-SIRT projections");
    if (e) return e;
    const float *dw = nullptr;
    if (w_h) {
        e = ensure(c, (void **)&c->d_hw, &c->hw_bytes, nvox * sizeof(float), "host-SIRT weights");
        if (e) return e;
        CT_CUDA(c, cudaMemcpyAsync(c->d_hw, w_h, nvox * sizeof(float), cudaMemcpyHostToDevice, c->stream));
        dw = c->d_hw;
    }
    CT_CUDA(c, cudaMemcpyAsync(c->d_hvol, vol_h, vb, cudaMemcpyHostToDevice, c->stream));
    if (iters_done) *iters_done = 0;
    int first = 0;  // iterations done here, before ctrex_sirt_iterate takes over
    if (pdt == CTREX_F32 && max_iter >= 1) {
        // First iteration: the projections (the larger upload) travel on a
        // copy stream while the forward projection runs; the correction
        // r = R (p - A x) waits for them (the kernels of
        // ctrex_correct_static with this context's own scratch).  Same
        // arithmetic as the fused correction (A x and the row sums are FP32
        // either way); only the residual norms are summed in another order.
        const size_t npix = (size_t)G.n_views * G.nu * G.nv;
        e = ensure(c, &c->d_hq, &c->hq_bytes, npix * sizeof(float), "host-SIRT forward projection");
        if (e) return e;
        e = ensure(c, (void **)&c->d_hrs, &c->hrs_bytes, npix * sizeof(float), "host-SIRT row sums");
        if (e) return e;
        e = ensure(c, &c->d_r, &c->r_bytes, npix * sizeof(float), "SIRT correction images");
        if (e) return e;
        const size_t pairs = (size_t)correct_scratch_pairs((long long)npix);
        e = ensure(c, (void **)&c->d_hcs, &c->hcs_bytes, 2 * sizeof(double) * pairs, "host-SIRT correction partials");
        if (e) return e;
        if (!c->copy_stream) CT_CUDA(c, cudaStreamCreateWithFlags(&c->copy_stream, cudaStreamNonBlocking));
        if (!c->ev_vol) CT_CUDA(c, cudaEventCreateWithFlags(&c->ev_vol, cudaEventDisableTiming));
        if (!c->ev_p) CT_CUDA(c, cudaEventCreateWithFlags(&c->ev_p, cudaEventDisableTiming));
        CT_CUDA(c, cudaEventRecord(c->ev_vol, c->stream));  // the volume's upload (and earlier work) first
        CT_CUDA(c, cudaStreamWaitEvent(c->copy_stream, c->ev_vol, 0));
        CT_CUDA(c, cudaMemcpyAsync(c->d_hp, p_h, pb, cudaMemcpyHostToDevice, c->copy_stream));
        CT_CUDA(c, cudaEventRecord(c->ev_p, c->copy_stream));
        FwdArgs a = fwd_args(c, c->d_hvol, vdt, nullptr, G.n_views);
        e = prepare_atlas(c, a, c->d_hvol, vdt);
        if (e) return e;
        cudaError_t ce = launch_forward(a, c->d_hq, CTREX_F32, c->d_hrs);
        if (ce != cudaSuccess) return cuda_fail(c, ce, "sirt_host: forward projection");
        CT_CUDA(c, cudaStreamWaitEvent(c->stream, c->ev_p, 0));
        ce = launch_correct(c->d_hp, c->d_hq, c->d_hrs, c->d_r, CTREX_F32, (long long)npix, G.eps_R, c->d_sums,
                            c->d_hcs, c->stream);
        if (ce != cudaSuccess) return cuda_fail(c, ce, "sirt_host: correction of the first iteration");
        double s[2];
        CT_CUDA(c, cudaMemcpyAsync(s, c->d_sums, sizeof s, cudaMemcpyDeviceToHost, c->stream));
        CT_CUDA(c, cudaStreamSynchronize(c->stream));
        const double rho = s[1] > 0.0 ? sqrt(s[0] / s[1]) : sqrt(s[0]);
        if (hist) hist[0] = (float)rho;
        if (!isfinite(rho)) return fail(c, CTREX_E_DIVERGED, "sirt: residual not finite at iteration 0");
        first = 1;
        if (rho <= (double)tol) {
            max_iter = first;  // converged before the first update
        } else {
            e = ctrex_back_project(c, c->d_r, CTREX_F32, c->d_hvol, vdt, dw, alpha, 1, 1, nullptr, G.n_views);
            if (e) return e;
            if (iters_done) *iters_done = 1;
        }
    } else {
        CT_CUDA(c, cudaMemcpyAsync(c->d_hp, p_h, pb, cudaMemcpyHostToDevice, c->stream));
    }
    int rest = 0;
    e = ctrex_sirt_iterate(c, c->d_hvol, vdt, c->d_hp, pdt, max_iter - first, alpha, dw, tol,
                           hist ? hist + first : nullptr, &rest);
    if (iters_done && max_iter - first > 0) *iters_done = first + rest;
    if (e) return e;
    CT_CUDA(c, cudaMemcpyAsync(vol_h, c->d_hvol, vb, cudaMemcpyDeviceToHost, c->stream));
    CT_CUDA(c, cudaStreamSynchronize(c->stream));
    return CTREX_OK;
}

int ctrex_count_samples(ctrex_ctx *c, const int *view_idx, int n_idx, long long *out)
{
    if (!c) return CTREX_E_ARG;
    int e = check_views(c, view_idx, n_idx);
    if (e) return e;
    if (!out) return fail(c, CTREX_E_ARG, "count_samples: NULL output");
    DeviceGuard g(c->device);
    cudaError_t ce = launch_count_samples(fwd_args(c, nullptr, CTREX_F32, view_idx, n_idx), c->d_count);
    if (ce != cudaSuccess) return cuda_fail(c, ce, "count_samples launch");
    unsigned long long h = 0;
    CT_CUDA(c, cudaMemcpyAsync(&h, c->d_count, sizeof h, cudaMemcpyDeviceToHost, c->stream));
    CT_CUDA(c, cudaStreamSynchronize(c->stream));
    *out = (long long)h;
    return CTREX_OK;
}

}  // extern "C"
