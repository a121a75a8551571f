// adjoint_column.cu -- the matched adjoint of adjoint.cu for scans whose
// detector columns run along z (column.cuh): the rays of a warp that share a
// detector column scatter into neighbouring voxels of one z column, so the
// scatter goes to a zeroed volume with z contiguous, where one reduction
// instruction of a warp covers a few sectors instead of 32 scattered ones;
// a last pass adds it to the caller's volume.
//
// 45 views of the 256^3 motion geometry, scattered in place / here: 16.6 /
// 5.7 ms without motion (bound there by the reductions' path through L1), 39.0
// / 23.5 ms with motion (bound by the spline: issue 65 %, L1 75 %), 15.2 ms
// with the deformation run by run (ray.cuh).
#include "fwd_column.cuh"

namespace ctrex {

// Lanes of a warp along v.  Without motion all 32 (45 views of the 256^3
// motion geometry: 5.7 ms; 16: 6.2, 8: 7.7); with motion 8, so that a warp's
// samples share spline cells more often (23.5 ms; 16: 23.9, 4: 27.5).
constexpr int ADJ_LV = 32, ADJ_LV_PATCH = 8;
// CTAs per SM: the spline needs 168 registers to keep out of local memory (4
// CTAs at 128: 30.3 ms, 2: 26.6).
constexpr int ADJ_MIN_BLOCKS = 8, ADJ_MIN_BLOCKS_MOTION = 3;
// Shared memory that a CTA of the pose's patches asks for and leaves alone: three
// CTAs per SM, as with the spline.  More warps at a time reduce into lines
// further apart (256 x 256 x 24, 4 views turned by 20 degrees, 0.7 voxels a
// pixel: 0.32 ms; with 64 registers and as many CTAs as fit 0.65).
constexpr int ADJ_POSE_SHARED = 72 * 1024;
// Samples per spline cell from which the deformation goes by runs.  60 views
// at 64^3 / 80^3 / 96^3 (26 / 32 / 38 samples), by pairs: 0.76 / 1.36 / 2.14
// ms, by runs: 0.82 / 1.30 / 1.90 ms.
constexpr float ADJ_RUN_MIN = 30.0f;

// The scatter volume: padded index (i, j, k) (one border element on every
// side, never added back) at ((k >> 5) chunks + j rows + i) * 32 + (k & 31).
struct AdjVolume {
    float *p;
    unsigned sy;  // elements from row to row
    unsigned sz;  // elements from chunk to chunk, less the 32 that k itself counts
    int nx, ny, nz;
    __device__ __forceinline__ unsigned index(unsigned i, unsigned j, unsigned k) const
    {
        return j * sy + ((k >> 5) * sz + ((i << 5) + k));
    }
};

// The footprint that a thread's last samples share, not yet scattered: its
// lower corner and the summed weight of its eight taps.
struct AdjFoot {
    unsigned i = 0, j = 0, k = 0;
    bool live = false;
    float w[2][2][2];  // [z][y][x]

    __device__ __forceinline__ void flush(const AdjVolume &V)
    {
#pragma unroll
        for (int dz = 0; dz < 2; ++dz) {
            float *q = V.p + V.index(i, j, k + dz), *r = q + V.sy;
            atomicAdd(q, w[dz][0][0]);
            atomicAdd(q + 32, w[dz][0][1]);
            atomicAdd(r, w[dz][1][0]);
            atomicAdd(r + 32, w[dz][1][1]);
        }
    }
    // val at the point of cell (ci, cj, ck) (padded) with fractions ax, ay, az
    __device__ __forceinline__ void add(const AdjVolume &V, unsigned ci, unsigned cj, unsigned ck, float ax, float ay,
                                        float az, float val)
    {
        if (live && (ci != i || cj != j || ck != k)) {
            flush(V);
            live = false;
        }
        if (!live) {
            i = ci;
            j = cj;
            k = ck;
            live = true;
#pragma unroll
            for (int t = 0; t < 8; ++t) w[t >> 2][(t >> 1) & 1][t & 1] = 0.0f;
        }
        const float v1 = val * az, v0 = val - v1;
#pragma unroll
        for (int dz = 0; dz < 2; ++dz) {
            const float v = dz ? v1 : v0, y1 = v * ay, y0 = v - y1;
            w[dz][0][0] = fmaf(y0, 1.0f - ax, w[dz][0][0]);
            w[dz][0][1] = fmaf(y0, ax, w[dz][0][1]);
            w[dz][1][0] = fmaf(y1, 1.0f - ax, w[dz][1][0]);
            w[dz][1][1] = fmaf(y1, ax, w[dz][1][1]);
        }
    }
};

// LV: lanes of a warp along v; the other 32 / LV and the four warps of the
// CTA run along u.
// KIND: how the samples' positions are formed.  The pose alone in a kernel
// without the spline's registers (60 views of 128^3, pixels of a voxel: 1.81 ->
// 1.47 ms; 64^3, pixels of half a voxel: 1.47 -> 0.93).
enum AdjKind { ADJ_STILL, ADJ_POSE, ADJ_PAIRS, ADJ_RUNS };

template <int KIND, int LV>
__global__ void __launch_bounds__(128, KIND == ADJ_PAIRS || KIND == ADJ_RUNS ? ADJ_MIN_BLOCKS_MOTION : ADJ_MIN_BLOCKS)
    adjoint_column_kernel(Grid G, const ViewGPU *__restrict__ views, const MotionGPU *__restrict__ motion,
                          const float4 *spline, const int *__restrict__ view_idx, const float *__restrict__ proj,
                          const AdjVolume V, unsigned *devcheck, int n_strips)
{
    constexpr int LU = 32 / LV;
    constexpr bool SPLINE = KIND == ADJ_PAIRS || KIND == ADJ_RUNS;
    const int k = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int view = view_idx ? view_idx[k] : k;
    if (view < 0 || view >= G.n_views) {
        if (tid == 0) atomicOr(devcheck, (unsigned)DEVCHECK_OOB);
        return;
    }
    __shared__ float4 s_spline[SPLINE ? SPLINE_TABLE : 1];
    MotionGPU mo;
    if (KIND != ADJ_STILL) mo = motion[view];
    if (SPLINE) {
        load_spline(s_spline, spline, tid, 128);
        spline = s_spline;
        __syncthreads();
    }
    const int strip = blockIdx.z % n_strips, band = blockIdx.z / n_strips;
    const int iu = ((strip * gridDim.x + blockIdx.x) * 4 + warp) * LU + lane / LV, iv = band * LV + lane % LV;
    if (iu >= G.nu || iv >= G.nv) return;
    const float y = proj[((size_t)k * G.nv + iv) * G.nu + iu] * G.inv_sub;
    if (y == 0.0f) return;
    float cen[3];
    grid_centre(G, cen);
    const float n[3] = {(float)G.nx, (float)G.ny, (float)G.nz};
    AdjFoot F;
    // val at index coordinates base (whole numbers) + q, if a tap lies inside the grid
    auto point = [&](const float *base, const float *q, float val) {
        const float fx = floorf(q[0]), fy = floorf(q[1]), fz = floorf(q[2]);
        const float x = fx + base[0], y = fy + base[1], z = fz + base[2];
        if (!(val != 0.0f && x >= -1.0f && x < n[0] && y >= -1.0f && y < n[1] && z >= -1.0f && z < n[2])) return;
        F.add(V, (int)x + 1, (int)y + 1, (int)z + 1, q[0] - fx, q[1] - fy, q[2] - fz, val);
    };
    for (int s = 0; s < G.n_sub; ++s) {
        Ray R;  // sample positions relative to the grid centre
        if (!setup_ray(G, views[view * G.n_sub + s], (float)iu, (float)iv, R, cen)) continue;
        if (KIND == ADJ_POSE || KIND == ADJ_RUNS) {
            float d0[3], ds[3];
            pose_line(mo, R, d0, ds);
            const float kl = last_kappa(G, R);
            // the pose alone (a view whose time scale is 0 sees no deformation,
            // whatever the coefficients are)
            if (KIND == ADJ_POSE || mo.s == 0.0f) {
#pragma unroll 1
                for (int k = 0; k < R.K; ++k) {
                    const bool last = k == R.K - 1;
                    const float kap = last ? kl : (float)k, w = last ? fmaxf(R.w_last, 0.0f) : G.step_mm;
                    float q[3];
#pragma unroll
                    for (int r = 0; r < 3; ++r) q[r] = fmaf(kap, R.sg[r], R.g0[r]) + fmaf(kap, ds[r], d0[r]);
                    point(cen, q, y * w);
                }
                continue;
            }
            SplineLine L;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                L.x0[r] = fmaf(R.g0[r] + d0[r] + cen[r] + 0.5f, G.spl_scale[r], 1.0f);
                L.xs[r] = (R.sg[r] + ds[r]) * G.spl_scale[r];
            }
            for (int k = 0; k < R.K;) {
                SplineRun run;
                const int end = run.find(L, k, R.K, kl);
                float2 axy[CHEB_N];
                float az[CHEB_N];
                run.fit(spline, L, axy, az);
                const float ih = 1.0f / run.half;
                // positions from the run's middle, less its whole number (which
                // keeps their rounding below that of the pairs' positions)
                float m[3], base[3];
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    const float whole = rintf(fmaf(run.mid, R.sg[r], R.g0[r]));
                    m[r] = fmaf(run.mid, R.sg[r], R.g0[r] - whole);
                    base[r] = whole + cen[r];
                }
#pragma unroll 1
                for (; k < end; ++k) {
                    const bool last = k == R.K - 1;
                    const float kap = last ? kl : (float)k, w = last ? fmaxf(R.w_last, 0.0f) : G.step_mm;
                    float T[CHEB_N], u[3], q[3];
                    cheb_values((kap - run.mid) * ih, T);
                    SplineRun::value(axy, az, T, u);
#pragma unroll
                    for (int r = 0; r < 3; ++r)
                        q[r] = fmaf(kap - run.mid, R.sg[r], m[r]) + fmaf(mo.s, u[r], fmaf(kap, ds[r], d0[r]));
                    point(base, q, y * w);
                }
            }
        } else if (KIND == ADJ_PAIRS) {
            for (int kk = 0; kk < R.K; kk += 2) {
                float g[2][3], w[2], gc[2][3];
                sample_pair(G, R, kk, g, w);
                warp_pair_c(G, mo, spline, g, gc);
#pragma unroll 1
                for (int m = 0; m < 2; ++m) {
                    const float q[3] = {m ? gc[1][0] : gc[0][0], m ? gc[1][1] : gc[0][1], m ? gc[1][2] : gc[0][2]};
                    point(cen, q, y * (m ? w[1] : w[0]));
                }
            }
        } else {
            const float ys = y * G.step_mm;
            for (int kk = 0; kk < R.K - 1; ++kk) {
                const float kf = (float)kk;
                const float q[3] = {fmaf(kf, R.sg[0], R.g0[0]), fmaf(kf, R.sg[1], R.g0[1]), fmaf(kf, R.sg[2], R.g0[2])};
                point(cen, q, ys);
            }
            if (R.w_last > 0.0f) point(cen, R.g_last, y * R.w_last);
        }
    }
    if (F.live) F.flush(V);
}

// vol += the scatter volume: 32 x 32 (x, z) tiles of row y, turned in shared
// memory.
__global__ void __launch_bounds__(256) adjoint_add_kernel(const AdjVolume V, float *__restrict__ vol)
{
    __shared__ float tile[32][33];  // [x][z]
    const int x0 = blockIdx.x * 32, z0 = blockIdx.z * 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int y = blockIdx.y; y < V.ny; y += gridDim.y) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int x = x0 + warp + 8 * i, z = z0 + lane;
            tile[warp + 8 * i][lane] = x < V.nx && z < V.nz ? V.p[V.index(x + 1, y + 1, z + 1)] : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int x = x0 + lane, z = z0 + warp + 8 * i;
            if (x < V.nx && z < V.nz) vol[((size_t)z * V.ny + y) * V.nx + x] += tile[lane][warp + 8 * i];
        }
        __syncthreads();
    }
}

static AdjVolume adj_layout(const Grid &G, float *p, size_t &n)
{
    const size_t sy = ((size_t)G.nx + 2) * 32, sz = sy * ((size_t)G.ny + 2);
    n = sz * (((size_t)G.nz + 1) / 32 + 1);
    return {p, (unsigned)sy, (unsigned)(sz - 32), G.nx, G.ny, G.nz};
}

size_t adjoint_column_elems(const Grid &G)
{
    size_t n;
    adj_layout(G, nullptr, n);
    return n < (1ull << 32) && (G.nz + 31) / 32 <= 65535 ? n : 0;
}

// Tiles of a strip, list entries, strips x bands, with lv lanes along v.
static dim3 adj_grid(const Grid &G, int n_idx, int lv, int &n_strips)
{
    const int tu = 4 * (32 / lv);  // columns per CTA
    const int tiles = (G.nu + tu - 1) / tu, strip = 128 / tu, per = tiles < strip ? tiles : strip;
    n_strips = (tiles + per - 1) / per;
    return dim3(per, n_idx, (unsigned)n_strips * (unsigned)((G.nv + lv - 1) / lv));
}

static int adj_lanes(bool spline, bool along_z) { return !spline && along_z ? ADJ_LV : ADJ_LV_PATCH; }

bool adjoint_column_fits(const Grid &G, bool spline, bool along_z)
{
    int n_strips;
    return adj_grid(G, 1, adj_lanes(spline, along_z), n_strips).z <= 65535;
}

template <int KIND, int LV>
static cudaError_t adj_launch(const FwdArgs &a, const float *proj, const AdjVolume &V)
{
    const Grid &G = *a.grid;
    int n_strips;
    const dim3 grid = adj_grid(G, a.n_idx, LV, n_strips);
    const int shared = KIND == ADJ_POSE && LV == ADJ_LV_PATCH ? ADJ_POSE_SHARED : 0;
    if (shared) {
        const cudaError_t e = cudaFuncSetAttribute(adjoint_column_kernel<KIND, LV>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, shared);
        if (e != cudaSuccess) return e;
    }
    adjoint_column_kernel<KIND, LV><<<grid, 128, shared, a.stream>>>(G, a.views, a.motion, a.spline, a.view_idx, proj,
                                                                     V, a.devcheck, n_strips);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_column(const FwdArgs &a, bool along_z, const float *proj, float *vol, float *scratch)
{
    const Grid &G = *a.grid;
    size_t n;
    const AdjVolume V = adj_layout(G, scratch, n);
    cudaError_t e = cudaMemsetAsync(scratch, 0, n * sizeof(float), a.stream);
    if (e != cudaSuccess) return e;
    if (a.spline)
        e = spline_runs(G, ADJ_RUN_MIN) ? adj_launch<ADJ_RUNS, ADJ_LV_PATCH>(a, proj, V)
                                        : adj_launch<ADJ_PAIRS, ADJ_LV_PATCH>(a, proj, V);
    else if (a.motion)
        e = along_z ? adj_launch<ADJ_POSE, ADJ_LV>(a, proj, V) : adj_launch<ADJ_POSE, ADJ_LV_PATCH>(a, proj, V);
    else
        e = along_z ? adj_launch<ADJ_STILL, ADJ_LV>(a, proj, V) : adj_launch<ADJ_STILL, ADJ_LV_PATCH>(a, proj, V);
    if (e != cudaSuccess) return e;
    const dim3 grid((G.nx + 31) / 32, G.ny < 65535 ? G.ny : 65535, (G.nz + 31) / 32);
    adjoint_add_kernel<<<grid, 256, 0, a.stream>>>(V, vol);
    return cudaGetLastError();
}

}  // namespace ctrex
