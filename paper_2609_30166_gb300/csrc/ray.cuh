// ray.cuh -- per-ray set-up, sampling and interpolation shared by the
// ray-driven kernels (forward, fused correction, adjoint, motion gradient).
#pragma once

#include "ctrex_internal.cuh"

namespace ctrex {

// Geometry of one ray in voxel-index coordinates.  Samples k = 0..K-2 sit at
// g0 + k * sg with weight step_mm; the last one at g_last with weight w_last
// (truncated-midpoint rule of the clipped segment, Sec. 4.1 "weighted by
// their path lengths").
struct Ray {
    float g0[3];
    float sg[3];
    float g_last[3];
    float w_last;
    int K;
};

// The line of view parameters V through detector point (u, v): X, a point
// near the volume, and dg, index units per mm along the ray; the source sits
// at t = -len (t in mm from X).
__device__ __forceinline__ void ray_line(const Grid &G, const ViewGPU &V, float u, float v, float X[3], float dg[3],
                                         float &len)
{
    const float du = u - G.uc, dv = v - G.vc;
    float D[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        X[a] = fmaf(dv, V.qv[a], fmaf(du, V.qu[a], V.ref[a]));
        D[a] = fmaf(dv, V.qv[a], fmaf(du, V.qu[a], V.dref[a]));
    }
    const float m0 = D[0] * G.vox[0], m1 = D[1] * G.vox[1], m2 = D[2] * G.vox[2];
    len = sqrtf(fmaf(m0, m0, fmaf(m1, m1, m2 * m2)));
    const float il = 1.0f / len;
    dg[0] = D[0] * il;
    dg[1] = D[1] * il;
    dg[2] = D[2] * il;
}

// Samples of the clipped segment [t0, t1] (truncated-midpoint rule).
__device__ __forceinline__ void finish_ray(const Grid &G, const float X[3], const float dg[3], float t0, float t1,
                                           Ray &R)
{
    const float step = G.step_mm;
    const float L = t1 - t0;
    int K = (int)ceilf(L / step);
    if (K < 1) K = 1;
    const float th = t0 + 0.5f * step;
    const float a_last = fmaf((float)(K - 1), step, t0);
    const float t_last = 0.5f * (a_last + t1);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        R.g0[a] = fmaf(th, dg[a], X[a]);
        R.sg[a] = step * dg[a];
        R.g_last[a] = fmaf(t_last, dg[a], X[a]);
    }
    R.w_last = t1 - a_last;
    R.K = K;
}

// Sets up the ray of view parameters V through detector point (u, v).
// Returns false if the half line from the source misses the clip box.  With
// an offset off, the sample positions come out as index coordinates minus
// off (the clip itself is unchanged): for off = the integer grid centre they
// are formed at magnitudes up to n / 2, which halves their rounding.
__device__ __forceinline__ bool setup_ray(const Grid &G, const ViewGPU &V, float u, float v, Ray &R,
                                          const float *off = nullptr)
{
    float X[3], dg[3], len;
    ray_line(G, V, u, v, X, dg, len);
    float t0 = -len, t1 = INFINITY;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (dg[a] != 0.0f) {
            const float inv = 1.0f / dg[a];
            const float ta = (G.lo[a] - X[a]) * inv, tb = (G.hi[a] - X[a]) * inv;
            t0 = fmaxf(t0, fminf(ta, tb));
            t1 = fminf(t1, fmaxf(ta, tb));
        } else if (X[a] < G.lo[a] || X[a] > G.hi[a]) {
            return false;
        }
    }
    if (!(t1 > t0)) return false;
    if (off) {
        const float Xo[3] = {X[0] - off[0], X[1] - off[1], X[2] - off[2]};
        finish_ray(G, Xo, dg, t0, t1, R);
    } else {
        finish_ray(G, X, dg, t0, t1, R);
    }
    return true;
}

// Samples k of the interior range [ka, kb) have every trilinear tap inside the
// grid: g0 + k sg in [eps, n - 1 - eps] on each axis, with a margin eps far
// above the rounding of the sample positions, so the short path is exact.
__device__ __forceinline__ void interior_range(const Grid &G, const Ray &R, int &ka, int &kb)
{
    const float eps = 1e-2f;
    const int n[3] = {G.nx, G.ny, G.nz};
    float lo = 0.0f, hi = (float)(R.K - 1);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float l = eps, h = (float)(n[a] - 1) - eps;
        if (!(h >= l)) {  // one voxel along this axis: nothing is interior
            hi = -1.0f;
        } else if (R.sg[a] != 0.0f) {
            const float inv = 1.0f / R.sg[a];
            const float t0 = (l - R.g0[a]) * inv, t1 = (h - R.g0[a]) * inv;
            lo = fmaxf(lo, fminf(t0, t1));
            hi = fminf(hi, fmaxf(t0, t1));
        } else if (!(R.g0[a] >= l && R.g0[a] <= h)) {
            hi = -1.0f;
        }
    }
    ka = (int)ceilf(lo);
    kb = (int)floorf(hi) + 1;
    // keep one sample of rounding slack on each side in the exact path
    ka = min(max(ka + 1, 0), R.K - 1);
    kb = max(min(kb - 1, R.K - 1), ka);
}

// Zero-padded trilinear interpolation at index coordinate g (reading: taps
// outside [0, n-1] contribute nothing).  wsum receives the summed weight of
// the in-range taps (the interpolant of an all-ones volume, for row sums).
template <typename TV>
__device__ __forceinline__ float trilinear(const TV *__restrict__ vol, int nx, int ny, int nz,
                                           float gx, float gy, float gz, float &wsum)
{
    const float fx = floorf(gx), fy = floorf(gy), fz = floorf(gz);
    const int ix = (int)fx, iy = (int)fy, iz = (int)fz;
    const float ax = gx - fx, ay = gy - fy, az = gz - fz;
    const float wx0 = ((unsigned)ix < (unsigned)nx) ? 1.0f - ax : 0.0f;
    const float wx1 = ((unsigned)(ix + 1) < (unsigned)nx) ? ax : 0.0f;
    const float wy0 = ((unsigned)iy < (unsigned)ny) ? 1.0f - ay : 0.0f;
    const float wy1 = ((unsigned)(iy + 1) < (unsigned)ny) ? ay : 0.0f;
    const float wz0 = ((unsigned)iz < (unsigned)nz) ? 1.0f - az : 0.0f;
    const float wz1 = ((unsigned)(iz + 1) < (unsigned)nz) ? az : 0.0f;
    const int x0 = min(max(ix, 0), nx - 1), x1 = min(max(ix + 1, 0), nx - 1);
    const int y0 = min(max(iy, 0), ny - 1), y1 = min(max(iy + 1, 0), ny - 1);
    const int z0 = min(max(iz, 0), nz - 1), z1 = min(max(iz + 1, 0), nz - 1);
    const TV *r00 = vol + (z0 * ny + y0) * nx;
    const TV *r01 = vol + (z0 * ny + y1) * nx;
    const TV *r10 = vol + (z1 * ny + y0) * nx;
    const TV *r11 = vol + (z1 * ny + y1) * nx;
    const float v000 = Storage<TV>::load(r00 + x0), v001 = Storage<TV>::load(r00 + x1);
    const float v010 = Storage<TV>::load(r01 + x0), v011 = Storage<TV>::load(r01 + x1);
    const float v100 = Storage<TV>::load(r10 + x0), v101 = Storage<TV>::load(r10 + x1);
    const float v110 = Storage<TV>::load(r11 + x0), v111 = Storage<TV>::load(r11 + x1);
    const float c00 = fmaf(wx0, v000, wx1 * v001), c01 = fmaf(wx0, v010, wx1 * v011);
    const float c10 = fmaf(wx0, v100, wx1 * v101), c11 = fmaf(wx0, v110, wx1 * v111);
    const float c0 = fmaf(wy0, c00, wy1 * c01), c1 = fmaf(wy0, c10, wy1 * c11);
    wsum = (wx0 + wx1) * (wy0 + wy1) * (wz0 + wz1);
    return fmaf(wz0, c0, wz1 * c1);
}

// The deformation.  Along x the uniform cubic B-spline is held as one cubic
// polynomial per cell (between two control planes), along y and z by its
// basis functions: x by Horner's scheme (3 multiply-adds a row and component
// instead of 4, and no x weights), then weighted sums over y and z.  One pass
// over a cell's 64 coefficients serves two samples of a ray (their loads are
// what bounds it: a vector load fills a register of every lane, shared
// address or not).  Table: [z 8][y 8][cell 5][power of f 4] float4 (x, y, z
// components in voxels), 21 KB, copied to shared memory by each CTA.
//
// 45 views of the 256^3 motion workload, basis functions on three axes and a
// pass per sample / this: projector 29.7 / 23.8 ms, gradient 118.7 / 104.3 ms
// (all 64 monomials per cell from a 125 KB table in global memory: 39.5 ms).
// Rows and planes are padded to 5 and 1 mod 8 elements, so that lanes in
// different cells read different banks (unpadded, cells above one another hit
// the same ones: adjoint with motion, 128 x 128 x 8, 60 views, 1.37 -> 0.64 ms).
constexpr int SPL_ROW = 5 * 4 + 1, SPL_PLANE = 8 * SPL_ROW + 1;
static_assert(SPLINE_TABLE == 8 * SPL_PLANE, "spline table size");

__device__ __forceinline__ void load_spline(float4 *s, const float4 *__restrict__ table, int tid, int nthreads)
{
#pragma unroll 5
    for (int i = tid; i < SPLINE_TABLE; i += nthreads) s[i] = __ldg(table + i);
}

// Uniform cubic B-spline weights of the cell's control points at fraction f,
// and their derivatives.
__device__ __forceinline__ void bspline_weights(float f, float w[4])
{
    const float f2 = f * f, f3 = f2 * f, g = 1.0f - f;
    w[0] = g * g * g * (1.0f / 6.0f);
    w[1] = fmaf(0.5f, f3, fmaf(-1.0f, f2, 2.0f / 3.0f));
    w[2] = fmaf(-0.5f, f3, fmaf(0.5f, f2, fmaf(0.5f, f, 1.0f / 6.0f)));
    w[3] = f3 * (1.0f / 6.0f);
}

__device__ __forceinline__ void bspline_dweights(float f, float d[4])
{
    const float f2 = f * f, g = 1.0f - f;
    d[0] = -0.5f * g * g;
    d[1] = fmaf(1.5f, f2, -2.0f * f);
    d[2] = fmaf(-1.5f, f2, fmaf(1.0f, f, 0.5f));
    d[3] = 0.5f * f2;
}

// Power-basis coefficients (f^0 .. f^3) of the uniform cubic B-spline piece m
// (m = 0..3: weight of control point i0 - 1 + m at fraction f).
__host__ __device__ __forceinline__ float4 bspline_piece(int m)
{
    return m == 0 ? make_float4(1.0f / 6.0f, -0.5f, 0.5f, -1.0f / 6.0f)
                  : (m == 1 ? make_float4(2.0f / 3.0f, 0.0f, -1.0f, 0.5f)
                            : (m == 2 ? make_float4(1.0f / 6.0f, 0.5f, 0.5f, -0.5f)
                                      : make_float4(0.0f, 0.0f, 0.0f, 1.0f / 6.0f)));
}

// Cell i in [0, 4] and fraction f in [0, 1] of a spline coordinate (clamped
// to [1, 6]); `active` is false where the clamp holds.
__device__ __forceinline__ void spline_cell_of(float xi, int &i, float &f, bool &active)
{
    active = (xi > 1.0f) && (xi < 6.0f);
    xi = fminf(fmaxf(xi, 1.0f), 6.0f);
    const float fl = fminf(floorf(xi), 5.0f);
    i = (int)fl - 1;
    f = xi - fl;
}

// The same of index coordinate gp along one axis.
__device__ __forceinline__ void spline_coord(float gp, float scale, int &i, float &f, bool &active)
{
    spline_cell_of(fmaf(gp + 0.5f, scale, 1.0f), i, f, active);
}

__device__ __forceinline__ const float4 *spline_cell(const float4 *table, const int i[3])
{
    return table + i[2] * SPL_PLANE + i[1] * SPL_ROW + i[0] * 4;
}

// Displacement u (voxels) of N samples in the cell at `c`, fractions f.
// ROLLED: the z loop stays a loop (its weights picked by selects), where the
// registers of the unrolled one's loads are not to be had.
template <int N, bool ROLLED = false>
__device__ __forceinline__ void spline_value(const float4 *c, const float (&f)[N][3], float (&u)[N][3])
{
    float wy[N][4], wz[N][4];
#pragma unroll
    for (int n = 0; n < N; ++n) {
        bspline_weights(f[n][1], wy[n]);
        bspline_weights(f[n][2], wz[n]);
    }
    float2 uxy[N];
    float uz[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
        uxy[n] = two(0.0f);
        uz[n] = 0.0f;
    }
#pragma unroll(ROLLED ? 1 : 4)
    for (int k = 0; k < 4; ++k) {
        float2 yxy[N];
        float yz[N];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 *row = c + k * SPL_PLANE + j * SPL_ROW;
            const float4 c3 = row[3], c2 = row[2], c1 = row[1], c0 = row[0];
#pragma unroll
            for (int n = 0; n < N; ++n) {
                const float2 fx = make_float2(f[n][0], f[n][0]), w = make_float2(wy[n][j], wy[n][j]);
                float2 r = __ffma2_rn(fx, make_float2(c3.x, c3.y), make_float2(c2.x, c2.y));
                r = __ffma2_rn(fx, r, make_float2(c1.x, c1.y));
                r = __ffma2_rn(fx, r, make_float2(c0.x, c0.y));
                const float z = fmaf(f[n][0], fmaf(f[n][0], fmaf(f[n][0], c3.z, c2.z), c1.z), c0.z);
                yxy[n] = j == 0 ? __fmul2_rn(w, r) : __ffma2_rn(w, r, yxy[n]);
                yz[n] = j == 0 ? w.x * z : fmaf(w.x, z, yz[n]);
            }
        }
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const float w = k == 0 ? wz[n][0] : (k == 1 ? wz[n][1] : (k == 2 ? wz[n][2] : wz[n][3]));
            uxy[n] = __ffma2_rn(two(w), yxy[n], uxy[n]);
            uz[n] = fmaf(w, yz[n], uz[n]);
        }
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
        u[n][0] = uxy[n].x;
        u[n][1] = uxy[n].y;
        u[n][2] = uz[n];
    }
}

// Runs of a ray inside one spline cell.  The position is linear in the sample
// index, so within a cell the displacement is a polynomial of degree 9 in it
// (three cubics' products), and its values at 10 Chebyshev nodes determine it
// exactly: u(t) = sum_j a_j T_j(t), t in [-1, 1] over the run, with
//   a_j = (2 - [j = 0]) / 10 sum_n u(tau_n) T_j(tau_n),  tau_n = cos((2 n + 1) pi / 20).
// A cell is 1/5 of the volume wide: at 128^3 a run has about 51 samples, so
// 10 passes over the cell's 64 coefficients replace 26 (of two samples each).
// (The Chebyshev form keeps the coefficients' rounding at that of u; powers of
// t would not.)
constexpr int CHEB_N = 10;
__host__ __device__ constexpr float cheb_cos20(int m)  // cos(m pi / 20)
{
    const float c[11] = {1.0f,          0.98768834059513773f, 0.95105651629515357f, 0.89100652418836786f,
                         0.80901699437494742f, 0.70710678118654752f, 0.58778525229247313f, 0.45399049973954675f,
                         0.30901699437494742f, 0.15643446504023086f, 0.0f};
    m %= 40;
    if (m > 20) m = 40 - m;
    return m <= 10 ? c[m] : -c[20 - m];
}
struct ChebTable {
    float t[CHEB_N / 2][CHEB_N];  // T_j(tau_n) of the nodes tau_n > 0; T_j(-tau) = (-1)^j T_j(tau)
    constexpr ChebTable() : t()
    {
        for (int n = 0; n < CHEB_N / 2; ++n)
            for (int j = 0; j < CHEB_N; ++j) t[n][j] = cheb_cos20(j * (2 * n + 1));
    }
};
static __constant__ ChebTable c_cheb = ChebTable();

// T_0 .. T_9 at t.
__device__ __forceinline__ void cheb_values(float t, float T[CHEB_N])
{
    const float t2 = t + t;
    T[0] = 1.0f;
    T[1] = t;
#pragma unroll
    for (int j = 2; j < CHEB_N; ++j) T[j] = fmaf(t2, T[j - 1], -T[j - 2]);
}

// Whether a cell holds at least `least` samples along its shortest axis, so
// that the runs pay (51 at 128^3, 38 at 96^3, 26 at 64^3).
inline bool spline_runs(const Grid &G, float least)
{
    float cell = 1.0f / 0.0f;
    for (int a = 0; a < 3; ++a) cell = fminf(cell, G.vox[a] / (G.spl_scale[a] * G.step_mm));
    return cell >= least;
}

// A ray's spline coordinates, linear in the sample index kappa.
struct SplineLine {
    float x0[3], xs[3];
};

// The run of samples k, k + 1, .. in the cell of sample k.
struct SplineRun {
    int cell[3];
    float base[3];  // fraction along axis a: kappa xs + base where it moves, base (0 or 1) where the clamp holds
    bool on[3];
    float mid, half;  // t = (kappa - mid) / half

    // kappa of the ray's samples: their index, except kl for the last one.
    // Returns the first sample after the run.
    __device__ __forceinline__ int find(const SplineLine &L, int k, int K, float kl)
    {
        const float kap = k == K - 1 ? kl : (float)k;
        int end = K;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float xi = fmaf(kap, L.xs[a], L.x0[a]);
            float face;  // the spline coordinate at which the ray leaves
            bool leaves = L.xs[a] != 0.0f;
            on[a] = xi > 1.0f && xi < 6.0f;
            if (on[a]) {
                const float fl = floorf(xi);
                cell[a] = (int)fl - 1;
                base[a] = L.x0[a] - fl;
                face = L.xs[a] > 0.0f ? fl + 1.0f : fl;
            } else {
                const bool above = xi >= 6.0f;
                cell[a] = above ? 4 : 0;
                base[a] = above ? 1.0f : 0.0f;
                face = above ? 6.0f : 1.0f;
                leaves = above ? L.xs[a] < 0.0f : L.xs[a] > 0.0f;
            }
            const float e = (face - L.x0[a]) / L.xs[a];
            if (leaves && e < (float)K) end = min(end, max((int)ceilf(e), k + 1));
        }
        const float last = end == K ? kl : (float)(end - 1);
        mid = 0.5f * (kap + last);
        half = fmaxf(0.5f * (last - kap), 0.5f);
        return end;
    }
    __device__ __forceinline__ void fraction(const SplineLine &L, float kap, float f[3]) const
    {
#pragma unroll
        for (int a = 0; a < 3; ++a) f[a] = on[a] ? fmaf(kap, L.xs[a], base[a]) : base[a];
    }
    // Chebyshev coefficients of the displacement (voxels): x and y packed, z.
    __device__ __forceinline__ void fit(const float4 *table, const SplineLine &L, float2 axy[CHEB_N],
                                        float az[CHEB_N]) const
    {
        const float4 *c = spline_cell(table, cell);
#pragma unroll
        for (int j = 0; j < CHEB_N; ++j) {
            axy[j] = two(0.0f);
            az[j] = 0.0f;
        }
#pragma unroll 1
        for (int n = 0; n < CHEB_N / 2; ++n) {
            const float tau = half * c_cheb.t[n][1];
            float f[2][3], u[2][3];
            fraction(L, mid + tau, f[0]);
            fraction(L, mid - tau, f[1]);
            spline_value<2, true>(c, f, u);
            // even j take the sum of the two nodes' values, odd j the difference
            const float2 e = make_float2(u[0][0] + u[1][0], u[0][1] + u[1][1]);
            const float2 o = make_float2(u[0][0] - u[1][0], u[0][1] - u[1][1]);
            const float ez = u[0][2] + u[1][2], oz = u[0][2] - u[1][2];
#pragma unroll
            for (int j = 0; j < CHEB_N; ++j) {
                const float w = c_cheb.t[n][j] * (j == 0 ? 0.1f : 0.2f);
                axy[j] = __ffma2_rn(two(w), j & 1 ? o : e, axy[j]);
                az[j] = fmaf(w, j & 1 ? oz : ez, az[j]);
            }
        }
    }
    static __device__ __forceinline__ void value(const float2 axy[CHEB_N], const float az[CHEB_N],
                                                 const float T[CHEB_N], float u[3])
    {
        float2 s = two(0.0f);  // the small terms first
        float z = 0.0f;
#pragma unroll
        for (int j = CHEB_N - 1; j >= 0; --j) {
            s = __ffma2_rn(two(T[j]), axy[j], s);
            z = fmaf(T[j], az[j], z);
        }
        u[0] = s.x;
        u[1] = s.y;
        u[2] = z;
    }
};

// Displacements of two samples at index coordinates g: one pass over the
// first one's cell serves both, and a second sample beyond its face (a step
// is a small part of a cell) takes a pass of its own.
__device__ __forceinline__ void spline_pair(const Grid &G, const float4 *table, const float g[2][3], float u[2][3])
{
    float f[2][3];
    int i[2][3];
    bool on;
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int a = 0; a < 3; ++a) spline_coord(g[n][a], G.spl_scale[a], i[n][a], f[n][a], on);
    float v[2][3];
    spline_value<2>(spline_cell(table, i[0]), f, v);
    if (i[0][0] != i[1][0] || i[0][1] != i[1][1] || i[0][2] != i[1][2]) {
        const float f1[1][3] = {{f[1][0], f[1][1], f[1][2]}};
        float w[1][3];
        spline_value<1>(spline_cell(table, i[1]), f1, w);
#pragma unroll
        for (int a = 0; a < 3; ++a) v[1][a] = w[0][a];
    }
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int a = 0; a < 3; ++a) u[n][a] = v[n][a];
}

// Pixel of this thread in a 32 x 4 pixel CTA tile.  Row layout: warp w is
// detector row w of the tile.  Patch layout (the motion kernels): warp w is
// the 8 x 4 pixel patch at columns 8w .. 8w + 7, so a warp's samples lie
// closer together and more often in one spline cell, whose coefficient
// loads are then shared by the warp.
template <bool PATCH>
__device__ __forceinline__ void tile_pixel(int tile_u0, int tile_v0, int &iu, int &iv)
{
    if (PATCH) {
        const int tid = threadIdx.y * 32 + threadIdx.x;
        const int w = tid >> 5, l = tid & 31;
        iu = tile_u0 + 8 * w + (l & 7);
        iv = tile_v0 + (l >> 3);
    } else {
        iu = tile_u0 + threadIdx.x;
        iv = tile_v0 + threadIdx.y;
    }
}

// Integer grid centre c = floor((n - 1) / 2) per axis (index coordinates).
__device__ __forceinline__ void grid_centre(const Grid &G, float c[3])
{
    c[0] = (float)((G.nx - 1) >> 1);
    c[1] = (float)((G.ny - 1) >> 1);
    c[2] = (float)((G.nz - 1) >> 1);
}

// Warp of two samples (Sec. 2.2.2 pose, then Sec. 3.1 displacement), in
// coordinates centred on the integer grid centre c: gc = g - c in (g index
// coordinates), yc = y - c out, with y = M g + b + s u(M g + b).  It runs as
// yc = gc + (D gc + bc + s u) with gc = g - c, D = M - I, bc = M c + b - c:
// the bracket is a displacement of a few voxels for a near-identity pose,
// so its roundings are small, and only the last addition rounds at the
// magnitude of the coordinate (up to n / 2).  Since c is an integer, floor
// and fraction of y follow exactly from yc.  table: the spline's table in shared
// memory, or nullptr.
__device__ __forceinline__ void warp_pair_c(const Grid &G, const MotionGPU &m, const float4 *table,
                                            const float gc[2][3], float yc[2][3])
{
    float c[3];
    grid_centre(G, c);
    float d[2][3], g[2][3], u[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};  // d: displacement D gc + bc
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            d[n][r] = fmaf(m.D[3 * r], gc[n][0],
                           fmaf(m.D[3 * r + 1], gc[n][1], fmaf(m.D[3 * r + 2], gc[n][2], m.bc[r])));
            g[n][r] = gc[n][r] + d[n][r] + c[r];
        }
    if (table != nullptr && m.s != 0.0f) spline_pair(G, table, g, u);
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int r = 0; r < 3; ++r) yc[n][r] = gc[n][r] + fmaf(m.s, u[n][r], d[n][r]);
}

// The same warp in plain index coordinates, as the forward projector uses it:
// y = M g + b + s u(M g + b) formed directly (fewer operations; the forward
// averages the position rounding out along the ray, so it needs no centring).
__device__ __forceinline__ void warp_pair(const Grid &G, const MotionGPU &m, const float4 *table, const float g[2][3],
                                          float y[2][3])
{
    float gp[2][3], u[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int r = 0; r < 3; ++r)
            gp[n][r] = fmaf(m.M[3 * r], g[n][0],
                            fmaf(m.M[3 * r + 1], g[n][1], fmaf(m.M[3 * r + 2], g[n][2], m.b[r])));
    if (table != nullptr && m.s != 0.0f) spline_pair(G, table, gp, u);
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int r = 0; r < 3; ++r) y[n][r] = fmaf(m.s, u[n][r], gp[n][r]);
}

// The last sample of a ray sits at the middle of the clipped segment's rest:
// its place in units of the sample index.
__device__ __forceinline__ float last_kappa(const Grid &G, const Ray &R)
{
    return (float)(R.K - 1) + 0.5f * (R.w_last / G.step_mm - 1.0f);
}

// Displacement of a ray's samples by the pose, D g + bc (g relative to the
// grid centre, as R's positions): d0 + kappa ds at sample index kappa.
__device__ __forceinline__ void pose_line(const MotionGPU &m, const Ray &R, float d0[3], float ds[3])
{
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const float *D = m.D + 3 * r;
        d0[r] = fmaf(D[0], R.g0[0], fmaf(D[1], R.g0[1], fmaf(D[2], R.g0[2], m.bc[r])));
        ds[r] = fmaf(D[0], R.sg[0], fmaf(D[1], R.sg[1], D[2] * R.sg[2]));
    }
}

// Samples kk and kk + 1 of a ray and their weights (mm): the last one is the
// clipped segment's remainder, one past it weighs nothing (and repeats it).
__device__ __forceinline__ void sample_pair(const Grid &G, const Ray &R, int kk, float g[2][3], float w[2])
{
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        const bool last = kk + n >= R.K - 1;
        const float kf = (float)(kk + n);
#pragma unroll
        for (int a = 0; a < 3; ++a) g[n][a] = last ? R.g_last[a] : fmaf(kf, R.sg[a], R.g0[a]);
        w[n] = last ? (kk + n == R.K - 1 ? fmaxf(R.w_last, 0.0f) : 0.0f) : G.step_mm;
    }
}

}  // namespace ctrex
