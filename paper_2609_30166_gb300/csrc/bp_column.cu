// bp_column.cu -- the weighted backprojection of backproject.cu for scans
// whose detector columns run along z: a warp takes 32 voxels of a z column,
// whose projections run along one detector column, and the correction images
// are in column layout (column.cuh).
#include "column.cuh"
#include "cylinder.cuh"

#include <type_traits>

namespace ctrex {

constexpr int BPC_WX = 8, BPC_WY = 1;  // z columns of a CTA (one per warp)
constexpr int BPC_COLS = BPC_WX * BPC_WY;
constexpr int BPC_THREADS = 32 * BPC_COLS;
constexpr int BPC_CHUNK = 128;  // views staged at a time
constexpr int BPC_MIN_BLOCKS = 5;  // 48 registers (4 and 6: 21.1 and 21.8 ms where 5 takes 18.8)
constexpr int BPC_SUBV_MIN_BLOCKS = 4;
constexpr size_t BPC_DEEP_MAX = 4 * 152;  // 4 CTAs on each of 152 SMs

// The correction images [n][nu][nv] in column layout: pair (u, v) of image k,
// padded indices (u + 1, v + 1), at k view + (v >> 4) sv + (u << 4) + v.
struct ColImages {
    const float2 *p;
    size_t view;    // pairs per image
    unsigned sv;    // pairs from chunk to chunk, less the 16 that v itself counts
    unsigned bias;  // -index(bits of 2^23, bits of 2^23): see bp_load
};

// One view of the staged chunk.
struct ColView {
    float4 p0, p1, p2;                   // rows of P; p2 = 0: skipped
    const float2 *img;
    // -1: every voxel of the CTA projects outside the window; 1: every one
    // inside it; 2: and at one depth along z, to FP32 rounding; 0: neither
    int inside;
    int pad;
};

__device__ __forceinline__ float col_recip(float x)
{
    float r0;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(x));
    return r0 * fmaf(-x, r0, 2.0f);
}

// The loads of a bilinear sample at (u, v), each in [-1, n), and its
// fractions: floor + 1 comes out of adding 2^23 + 1 rounded down (the low
// mantissa bits), without a conversion.
struct BpTaps {
    float2 q0, q1;
    float au, av;
};
__device__ __forceinline__ BpTaps bp_load(const ColImages &I, const float2 *img, float u, float v)
{
    constexpr float M = 8388609.0f;
    BpTaps t;
    const float mu = __fadd_rd(u, M), mv = __fadd_rd(v, M);
    t.au = u - (mu - M);
    t.av = v - (mv - M);
    const unsigned bu = __float_as_uint(mu), bv = __float_as_uint(mv);
    const unsigned i = (bv >> COL_LOG) * I.sv + ((bu << COL_LOG) + (bv + I.bias));
    const float2 *q = img + i;
    t.q0 = __ldg(q);
    t.q1 = __ldg(q + (1 << COL_LOG));
    return t;
}
__device__ __forceinline__ float bp_interp(const BpTaps &t)
{
    return lerp(col_value(t.q0, t.av), col_value(t.q1, t.av), t.au);
}

// One voxel-view term in general position, as bp_term in backproject.cu.
__device__ __forceinline__ void bp_edge(const ColImages &I, const float2 *img, float h1, float h2,
                                        float h3, float4 win, float &b, float &c)
{
    if (!(h3 > 0.0f)) return;
    const float inv = col_recip(h3);
    const float u = h1 * inv, v = h2 * inv;
    if (!(u > win.x - 1.0f && u < win.y + 1.0f && v > win.z - 1.0f && v < win.w + 1.0f)) return;
    const float fu = floorf(u), fv = floorf(v), au = u - fu, av = v - fv;
    // each value by itself: a difference would bring in one beyond the window
    const unsigned bu = (unsigned)((int)fu + 1) << COL_LOG, bv = (unsigned)((int)fv + 1);
    const float2 *r0 = img + ((bv >> COL_LOG) * I.sv + (bu + bv)),
                 *r1 = img + (((bv + 1) >> COL_LOG) * I.sv + (bu + bv + 1));
    const float2 q0 = make_float2(__ldg(&r0->x), __ldg(&r1->x)),
                 q1 = make_float2(__ldg(&r0[1 << COL_LOG].x), __ldg(&r1[1 << COL_LOG].x));
    const float wu0 = fu >= win.x ? 1.0f - au : 0.0f, wu1 = fu + 1.0f <= win.y ? au : 0.0f;
    const float wv0 = fv >= win.z ? 1.0f - av : 0.0f, wv1 = fv + 1.0f <= win.w ? av : 0.0f;
    b += fmaf(wv0, fmaf(wu0, q0.x, wu1 * q1.x), wv1 * fmaf(wu0, q0.y, wu1 * q1.y));
    c += (wu0 + wu1) * (wv0 + wv1);
}

// A voxel's sums over the views (field 0: b, c; field 1: b, c), each term in
// general position.  bp_interp's differences turn a mean with infinite values,
// or with values too far apart for FP32, into NaN or an infinity, so a voxel
// whose sum is not finite takes its terms again here.  Not inlined: within
// the kernels it cost their loops 2 to 4 %.
template <bool WINDOW, bool SUBV, bool CYL, bool DYR>
__device__ __noinline__ float4 bp_voxel(const ViewGPU *__restrict__ views, const int *__restrict__ view_idx, int total,
                                        int n_sub, int n_views, ColImages I, const int4 *__restrict__ window, float4 det,
                                        int ix, int iy, int iz, int sv, CylGPU cyl, float tau,
                                        const float *__restrict__ t_view)
{
    const int points = SUBV ? sv * sv * sv : 1;
    const float d = 1.0f / (float)sv, o = SUBV ? 0.5f * d - 0.5f : 0.0f;
    float4 sum = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int m = 0; m < total; ++m) {
        const int k = m / n_sub, view = view_idx ? view_idx[k] : k;
        if (view < 0 || view >= n_views) continue;
        const float *P = views[view * n_sub + (m - k * n_sub)].P;
        float4 win = det;
        if (WINDOW) {
            const int4 w = window[view];
            win = make_float4((float)w.x, (float)w.y, (float)w.z, (float)w.w);
        }
        float b = 0.0f, c = 0.0f;
        for (int i = 0; i < points; ++i) {
            float x = (float)ix, y = (float)iy, z = (float)iz;
            if (SUBV) {
                x += fmaf((float)(i % sv), d, o);
                y += fmaf((float)(i / sv % sv), d, o);
                z += fmaf((float)(i / (sv * sv)), d, o);
            }
            if (CYL) cyl_point(cyl, x, y, z, x, y, z);
            auto row = [&](const float *p) { return fmaf(p[0], x, fmaf(p[1], y, fmaf(p[2], z, p[3]))); };
            bp_edge(I, I.p + (size_t)k * I.view, row(P), row(P + 4), row(P + 8), win, b, c);
        }
        if (DYR && !(t_view[view] < tau)) {
            sum.z += b;
            sum.w += c;
        } else {
            sum.x += b;
            sum.y += c;
        }
        if (!DYR && isnan(sum.x)) break;  // and stays it, whatever the weights
    }
    return sum;
}

// ColView::inside of the points of a box: its corners decide (the image of a
// box in front of the source is the hull of its corners' images), by a margin
// that covers the rounding of u and v, bounded from the size of the terms
// they are summed from.
__host__ __device__ __forceinline__ int box_inside(float4 p0, float4 p1, float4 p2, const float lo[3], const float hi[3],
                                          float4 win)
{
    const float e = 0.02f;
    float m[3], h3min = INFINITY, u0 = INFINITY, u1 = -INFINITY, v0 = INFINITY, v1 = -INFINITY;
#pragma unroll
    for (int a = 0; a < 3; ++a) m[a] = fmaxf(fabsf(lo[a]), fabsf(hi[a]));
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float x = i & 1 ? hi[0] : lo[0], y = i & 2 ? hi[1] : lo[1], z = i & 4 ? hi[2] : lo[2];
        const float h3 = fmaf(p2.x, x, fmaf(p2.y, y, fmaf(p2.z, z, p2.w)));
        const float u = fmaf(p0.x, x, fmaf(p0.y, y, fmaf(p0.z, z, p0.w))) / h3;
        const float v = fmaf(p1.x, x, fmaf(p1.y, y, fmaf(p1.z, z, p1.w))) / h3;
        h3min = fminf(h3min, h3);
        u0 = fminf(u0, u);
        u1 = fmaxf(u1, u);
        v0 = fminf(v0, v);
        v1 = fmaxf(v1, v);
    }
    const float s1 = fabsf(p0.x) * m[0] + fabsf(p0.y) * m[1] + fabsf(p0.z) * m[2] + fabsf(p0.w);
    const float s2 = fabsf(p1.x) * m[0] + fabsf(p1.y) * m[1] + fabsf(p1.z) * m[2] + fabsf(p1.w);
    const float s3 = fabsf(p2.x) * m[0] + fabsf(p2.y) * m[1] + fabsf(p2.z) * m[2] + fabsf(p2.w);
    const float umax = fmaxf(fabsf(u0), fabsf(u1)), vmax = fmaxf(fabsf(v0), fabsf(v1));
    if (!(h3min > 0.0f && fmaxf(s1 + umax * s3, s2 + vmax * s3) * 1e-6f < e * h3min)) return 0;
    if (u1 < win.x - 1.0f - e || u0 > win.y + 1.0f + e || v1 < win.z - 1.0f - e || v0 > win.w + 1.0f + e) return -1;
    if (!(u0 >= win.x + e && u1 <= win.y - e && v0 >= win.z + e && v1 <= win.w - e)) return 0;
    // depth changes by less than half a unit in the last place along z
    return fabsf(p2.z) * (hi[2] - lo[2]) < h3min * 0x1p-25f ? 2 : 1;
}

// The sums of a CTA (b / c of field f, c already times `mean`) into the volume,
// by way of shared memory, so that the threads run along x: a z column's own
// order would touch a line per voxel.
template <typename TV, int VZ>
__device__ __forceinline__ void bp_store(const Grid &G, float2 (*out)[BPC_COLS + 1], TV *__restrict__ vol,
                                         const float *__restrict__ w, const float b[VZ], const float c[VZ], float mean,
                                         float alpha, int normalize, int accumulate, int z0, int zfirst, int f)
{
    const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
    const size_t nvox = (size_t)G.nx * G.ny * G.nz;
    const int oc = tid % BPC_COLS, ox = blockIdx.x * BPC_WX + oc % BPC_WX, oy = blockIdx.y * BPC_WY + oc / BPC_WX;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < VZ; ++q)
        out[lane + 32 * q][warp] =
            make_float2(b[q] * mean, normalize ? alpha * (c[q] > 1e-6f ? 1.0f / c[q] : 0.0f) : alpha);
    __syncthreads();
    if (ox >= G.nx || oy >= G.ny) return;
    for (int r = tid / BPC_COLS; r < 32 * VZ; r += BPC_THREADS / BPC_COLS) {
        const int oz = z0 + r;
        if (oz < zfirst || oz >= G.nz) continue;
        const size_t j = ((size_t)oz * G.ny + oy) * G.nx + ox + (size_t)f * nvox;
        const float2 o = out[r][oc];
        const float upd = (w ? o.y * __ldg(w + j) : o.y) * o.x;
        Storage<TV>::store(vol + j, accumulate ? Storage<TV>::load(vol + j) + upd : upd);
    }
}

// VZ: voxels per thread, 32 slices apart.  SUBV, CYL: as bp_kernel in backproject.cu; DYR: as bp_dyrect_kernel.
template <typename TV, int VZ, bool WINDOW, bool SUBV, bool CYL, bool DYR>
__global__ void __launch_bounds__(BPC_THREADS, SUBV ? BPC_SUBV_MIN_BLOCKS : (DYR ? 4 : BPC_MIN_BLOCKS))
    bp_column_kernel(Grid G, const ViewGPU *__restrict__ views, const int *__restrict__ view_idx, int n_idx,
                     const ColImages I, const int4 *__restrict__ window, TV *__restrict__ vol,
                     const float *__restrict__ w, float alpha, int normalize, int accumulate, int sv, const CylGPU cyl,
                     const float *__restrict__ tau, const float *__restrict__ t_view)
{
    constexpr int NP = DYR ? 2 : 1;  // value fields
    __shared__ ColView sV[BPC_CHUNK];
    __shared__ float4 sWin[WINDOW ? BPC_CHUNK : 1];
    __shared__ float sT[DYR ? BPC_CHUNK : 1];
    __shared__ int sAll;  // the least `inside` of the chunk's views
    __shared__ float2 sOut[32 * VZ][BPC_COLS + 1];
    __shared__ float sXY[2][BPC_COLS];
    const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
    // (warps past the volume's edge repeat its last column and write nothing)
    const int ix = min(blockIdx.x * BPC_WX + warp % BPC_WX, G.nx - 1);
    const int iy = min(blockIdx.y * BPC_WY + warp / BPC_WX, G.ny - 1);
    // the last block of a column starts early enough to be full and writes
    // only the slices that the block before it did not take
    const int zfirst = blockIdx.z * (32 * VZ), z0 = max(min(zfirst, G.nz - 32 * VZ), 0), iz = z0 + lane;
    const float4 det = make_float4(0.0f, (float)(G.nu - 1), 0.0f, (float)(G.nv - 1));
    // the frame point of the first voxel, and the step to the next one
    float x = (float)ix, y = (float)iy, z = (float)iz, dz = 32.0f;
    float zlo = (float)z0, zhi = zlo + 32.0f * VZ - 1.0f;
    if (CYL && !SUBV) {
        cyl_point(cyl, x, y, (float)iz, x, y, z);
        dz = 32.0f * cyl.dz;
        zlo = (zlo - cyl.zc) * cyl.dz;
        zhi = (zhi - cyl.zc) * cyl.dz;
    }
    if (lane == 0) {
        sXY[0][warp] = x;
        sXY[1][warp] = y;
    }
    __syncthreads();
    // box of the CTA's points
    float lo[3] = {sXY[0][0], sXY[1][0], zlo}, hi[3] = {sXY[0][0], sXY[1][0], zhi};
#pragma unroll
    for (int i = 1; i < BPC_COLS; ++i)
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            lo[a] = fminf(lo[a], sXY[a][i]);
            hi[a] = fmaxf(hi[a], sXY[a][i]);
        }
    if (SUBV)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] -= 0.5f;
            hi[a] += 0.5f;
        }
    float ta[VZ] = {};
    if (DYR)
#pragma unroll
        for (int q = 0; q < VZ; ++q)
            ta[q] = iz + 32 * q < G.nz ? __ldg(tau + ((size_t)(iz + 32 * q) * G.ny + iy) * G.nx + ix) : 0.0f;
    float b[NP][VZ], c[NP][VZ];
#pragma unroll
    for (int f = 0; f < NP; ++f)
#pragma unroll
        for (int q = 0; q < VZ; ++q) b[f][q] = c[f][q] = 0.0f;
    const int total = n_idx * G.n_sub;
    for (int base = 0; base < total; base += BPC_CHUNK) {
        const int cnt = min(BPC_CHUNK, total - base);
        __syncthreads();
        if (tid == 0) sAll = SUBV ? 0 : 2;
        __syncthreads();
        for (int t = tid; t < cnt; t += BPC_THREADS) {
            const int k = (base + t) / G.n_sub, s = base + t - k * G.n_sub;
            int view = view_idx ? view_idx[k] : k;
            const bool ok = view >= 0 && view < G.n_views;
            if (!ok) view = 0;
            const float *P = views[view * G.n_sub + s].P;
            ColView V;
            V.p0 = make_float4(P[0], P[1], P[2], P[3]);
            V.p1 = make_float4(P[4], P[5], P[6], P[7]);
            // an invalid view index gets a zero depth row: it is skipped
            V.p2 = ok ? make_float4(P[8], P[9], P[10], P[11]) : make_float4(0.f, 0.f, 0.f, 0.f);
            V.img = I.p + (size_t)k * I.view;
            float4 win = det;
            if (WINDOW) {
                const int4 wd = window[view];
                win = make_float4((float)wd.x, (float)wd.y, (float)wd.z, (float)wd.w);
                sWin[t] = win;
            }
            V.inside = SUBV && CYL ? 0 : box_inside(V.p0, V.p1, V.p2, lo, hi, win);
            sV[t] = V;
            if (V.inside < 2) atomicMin(&sAll, V.inside);
            if (DYR) sT[t] = __ldg(t_view + view);
        }
        __syncthreads();
        // ALL: what is known of every view of the chunk
        auto term = [&](int m, auto all) {
            constexpr int ALL = decltype(all)::value;
            const float4 p0 = sV[m].p0, p1 = sV[m].p1, p2 = sV[m].p2;
            const float2 *img = sV[m].img;
            const bool inside = sV[m].inside > 0;
            if (ALL == 0 && sV[m].inside < 0) return;
            const float4 win = WINDOW ? sWin[m] : det;
            const float tv = DYR ? sT[m] : 0.0f;
            auto add = [&](int q, float tb, float tc) {
                if (DYR) {
                    const bool early = tv < ta[q];
                    b[0][q] += early ? tb : 0.0f;
                    c[0][q] += early ? tc : 0.0f;
                    b[NP - 1][q] += early ? 0.0f : tb;
                    c[NP - 1][q] += early ? 0.0f : tc;
                } else {
                    b[0][q] += tb;
                    c[0][q] += tc;
                }
            };
            // the VZ points h + q (d0, d1, d2); inside: all their loads first
            auto points = [&](float h1, float h2, float h3, float d0, float d1, float d2) {
                if (ALL || inside) {
                    BpTaps t[VZ];
                    const float inv0 = ALL == 2 ? col_recip(h3) : 0.0f;
#pragma unroll
                    for (int q = 0; q < VZ; ++q) {
                        const float inv = ALL == 2 ? inv0 : col_recip(fmaf((float)q, d2, h3));
                        t[q] = bp_load(I, img, fmaf((float)q, d0, h1) * inv, fmaf((float)q, d1, h2) * inv);
                    }
#pragma unroll
                    for (int q = 0; q < VZ; ++q) add(q, bp_interp(t[q]), ALL > 0 && !DYR ? 0.0f : 1.0f);
                } else {
#pragma unroll
                    for (int q = 0; q < VZ; ++q) {
                        float tb = 0.0f, tc = 0.0f;
                        bp_edge(I, img, fmaf((float)q, d0, h1), fmaf((float)q, d1, h2), fmaf((float)q, d2, h3), win, tb,
                                tc);
                        add(q, tb, tc);
                    }
                }
            };
            if (SUBV) {
                const float d = 1.0f / (float)sv, o = 0.5f * d - 0.5f;
                for (int az = 0; az < sv; ++az)
                    for (int ay = 0; ay < sv; ++ay) {
                        const float gy = (float)iy + fmaf((float)ay, d, o);
                        float sn = 0.0f, cs = 0.0f;
                        if (CYL) sincosf((gy + 0.5f) * cyl.dphi, &sn, &cs);
                        for (int ax = 0; ax < sv; ++ax) {
                            const float gx = (float)ix + fmaf((float)ax, d, o);
                            float X = gx, Y = gy, Z = (float)iz + fmaf((float)az, d, o), D = 32.0f;
                            if (CYL) {
                                const float r = (gx + 0.5f) * cyl.dr;
                                X = r * cs;
                                Y = r * sn;
                                Z = (Z - cyl.zc) * cyl.dz;
                                D = 32.0f * cyl.dz;
                            }
                            const float h1 = fmaf(p0.x, X, fmaf(p0.y, Y, fmaf(p0.z, Z, p0.w)));
                            const float h2 = fmaf(p1.x, X, fmaf(p1.y, Y, fmaf(p1.z, Z, p1.w)));
                            const float h3 = fmaf(p2.x, X, fmaf(p2.y, Y, fmaf(p2.z, Z, p2.w)));
                            points(h1, h2, h3, D * p0.z, D * p1.z, D * p2.z);
                        }
                    }
                return;
            }
            const float h1 = fmaf(p0.x, x, fmaf(p0.y, y, fmaf(p0.z, z, p0.w)));
            const float h2 = fmaf(p1.x, x, fmaf(p1.y, y, fmaf(p1.z, z, p1.w)));
            const float h3 = fmaf(p2.x, x, fmaf(p2.y, y, fmaf(p2.z, z, p2.w)));
            points(h1, h2, h3, dz * p0.z, dz * p1.z, dz * p2.z);
        };
        const int all = sAll;
        if (all == 2)
            for (int m = 0; m < cnt; ++m) term(m, std::integral_constant<int, 2>());
        else if (all == 1)
            for (int m = 0; m < cnt; ++m) term(m, std::integral_constant<int, 1>());
        else
            for (int m = 0; m < cnt; ++m) term(m, std::integral_constant<int, 0>());
        if (!DYR && all > 0)  // each view weighed 1
#pragma unroll
            for (int q = 0; q < VZ; ++q) c[0][q] += (float)cnt;
    }
#pragma unroll
    for (int q = 0; q < VZ; ++q)
        if (!isfinite(b[0][q]) || !isfinite(b[NP - 1][q])) {
            const float4 s = bp_voxel<WINDOW, SUBV, CYL, DYR>(views, view_idx, total, G.n_sub, G.n_views, I, window, det,
                                                              ix, iy, iz + 32 * q, sv, CYL ? cyl : CylGPU{}, ta[q], t_view);
            b[0][q] = s.x;
            c[0][q] = s.y;
            if (DYR) {
                b[NP - 1][q] = s.z;
                c[NP - 1][q] = s.w;
            }
        }
    const float mean = SUBV ? G.inv_sub / (float)(sv * sv * sv) : G.inv_sub;
#pragma unroll
    for (int f = 0; f < NP; ++f) {
#pragma unroll
        for (int q = 0; q < VZ; ++q) c[f][q] *= mean;
        bp_store<TV, VZ>(G, sOut, vol, w, b[f], c[f], mean, alpha, normalize, accumulate, z0, zfirst, f);
    }
}

// The same where every view has every voxel inside the detector and at one
// depth along z (backproject_flat): u and v are linear in z.  A warp takes 32
// views at a time: a lane forms one view's (u, v) at the column's first voxel
// and their steps, and a term is a broadcast of these and two multiply-adds a
// voxel.  In bp_column_kernel the view's rows took 3/10 of L1's data path (16
// wavefronts of broadcasts beside the taps' 37) and a quarter of the
// instructions.  144 views of the 512^3 scan 18.8 -> 17.5 ms, sparse 128^3
// 0.142 -> 0.129, 64^3 0.048 -> 0.044; with the event model's sums it was
// slower (256^3, 90 views: 2.57 ms for 2.31), which stays there.  u and v
// count from a whole column and a chunk of rows below them (the image pointer
// takes the rest), so that they round less.
// Two voxels a thread: six CTAs per SM (40 registers), four: five.
// DEEP: a grid of few CTAs (bpc_launch), which waits for its loads: four terms
// in flight, 64 registers.
template <typename TV, int VZ, bool DEEP>
__global__ void __launch_bounds__(BPC_THREADS, DEEP ? 4 : (VZ == 2 ? 6 : BPC_MIN_BLOCKS))
    bp_flat_kernel(Grid G, const ViewGPU *__restrict__ views, const int *__restrict__ view_idx, int n_idx,
                   const ColImages I, TV *__restrict__ vol, const float *__restrict__ w, float alpha, int normalize,
                   int accumulate)
{
    __shared__ union {
        struct {
            float4 f[BPC_COLS][32];  // u, u's step along z, v, v's step
            const float2 *img[BPC_COLS][32];
        } term;
        float2 out[32 * VZ][BPC_COLS + 1];
    } sh;
    const int lane = threadIdx.x, warp = threadIdx.y;
    const int ix = min(blockIdx.x * BPC_WX + warp % BPC_WX, G.nx - 1);
    const int iy = min(blockIdx.y * BPC_WY + warp / BPC_WX, G.ny - 1);
    const int zfirst = blockIdx.z * (32 * VZ), z0 = max(min(zfirst, G.nz - 32 * VZ), 0);
    float b[VZ], c[VZ];
#pragma unroll
    for (int q = 0; q < VZ; ++q) b[q] = 0.0f;
    int count = 0;
    const int total = n_idx * G.n_sub;
    for (int base = 0; base < total; base += 32) {
        const int m = base + lane, k = m / G.n_sub;
        const int view = m < total ? (view_idx ? view_idx[k] : k) : -1;
        const bool ok = view >= 0 && view < G.n_views;  // an invalid view index is skipped
        const unsigned mask = __ballot_sync(0xffffffffu, ok);
        const int n = __popc(mask), at = __popc(mask & ((1u << lane) - 1u));
        __syncwarp();
        if (ok) {
            const float x = (float)ix, y = (float)iy, z = (float)z0;
            const float *P = views[view * G.n_sub + (m - k * G.n_sub)].P;
            auto row = [&](const float *p) { return fmaf(p[0], x, fmaf(p[1], y, fmaf(p[2], z, p[3]))); };
            const float h1 = row(P), h2 = row(P + 4), h3 = row(P + 8), span = 32.0f * VZ;
            const float du = __fdiv_rn(P[2], h3), dv = __fdiv_rn(P[6], h3), u = __fdiv_rn(h1, h3), v = __fdiv_rn(h2, h3);
            const float bu = fmaxf(floorf(fminf(u, fmaf(span, du, u))), 0.0f),
                        bv = 16.0f * fmaxf(floorf(fminf(v, fmaf(span, dv, v)) * 0.0625f), 0.0f);
            sh.term.f[warp][at] = make_float4(__fdiv_rn(fmaf(-bu, h3, h1), h3), du, __fdiv_rn(fmaf(-bv, h3, h2), h3), dv);
            const unsigned iv = (unsigned)bv;
            sh.term.img[warp][at] =
                I.p + (size_t)k * I.view + ((size_t)(iv >> COL_LOG) * I.sv + ((unsigned)bu << COL_LOG) + iv);
        }
        __syncwarp();
        count += n;
#pragma unroll DEEP ? 4 : 1  // (2 at 48 registers: 18.8 ms)
        for (int i = 0; i < n; ++i) {
            const float4 f = sh.term.f[warp][i];
            const float2 *img = sh.term.img[warp][i];
            const float u = fmaf((float)lane, f.y, f.x), v = fmaf((float)lane, f.w, f.z);
            BpTaps t[VZ];
#pragma unroll
            for (int q = 0; q < VZ; ++q) t[q] = bp_load(I, img, fmaf(32.0f * q, f.y, u), fmaf(32.0f * q, f.w, v));
#pragma unroll
            for (int q = 0; q < VZ; ++q) b[q] += bp_interp(t[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < VZ; ++q)
        if (!isfinite(b[q]))
            b[q] = bp_voxel<false, false, false, false>(
                       views, view_idx, total, G.n_sub, G.n_views, I, nullptr,
                       make_float4(0.0f, (float)(G.nu - 1), 0.0f, (float)(G.nv - 1)), ix, iy, z0 + lane + 32 * q, 1,
                       CylGPU{}, 0.0f, nullptr)
                       .x;
    const float mean = G.inv_sub;
#pragma unroll
    for (int q = 0; q < VZ; ++q) c[q] = (float)count * mean;
    bp_store<TV, VZ>(G, sh.out, vol, w, b, c, mean, alpha, normalize, accumulate, z0, zfirst, 0);
}

template <typename TV, int VZ, bool SUBV, bool CYL, bool DYR>
static cudaError_t bpc_launch(const BpArgs &a)
{
    const Grid &G = *a.grid;
    const ColStore &s = *a.column;
    ColImages I;
    I.p = s.buf;
    I.view = s.view;
    I.sv = s.sy;
    const unsigned m = 0x4B000000u;  // the bits of 2^23
    I.bias = 0u - ((m >> COL_LOG) * I.sv + (m << COL_LOG) + m);
    const dim3 grid((G.nx + BPC_WX - 1) / BPC_WX, (G.ny + BPC_WY - 1) / BPC_WY, (G.nz + 32 * VZ - 1) / (32 * VZ));
    const CylGPU cyl = a.cyl ? *a.cyl : CylGPU{};
    const float *tau = a.dyr ? a.dyr->tau : nullptr, *tv = a.dyr ? a.dyr->t_view : nullptr;
    if constexpr (!SUBV && !CYL && !DYR)
        if (a.flat && !a.window) {
            // up to one wave of the deep form's CTAs (64^3 x 90 views: 0.044 ->
            // 0.042 ms; 512^3: 17.5 -> 19.6)
            const bool deep = (size_t)grid.x * grid.y * grid.z <= BPC_DEEP_MAX;
            auto *kernel = deep ? bp_flat_kernel<TV, VZ, true> : bp_flat_kernel<TV, VZ, false>;
            kernel<<<grid, dim3(32, BPC_COLS), 0, a.stream>>>(
                G, a.views, a.view_idx, a.n_idx, I, static_cast<TV *>(a.vol), a.w, a.alpha, a.normalize, a.accumulate);
            return cudaGetLastError();
        }
    if (a.window)
        bp_column_kernel<TV, VZ, true, SUBV, CYL, DYR><<<grid, dim3(32, BPC_COLS), 0, a.stream>>>(
            G, a.views, a.view_idx, a.n_idx, I, a.window, static_cast<TV *>(a.vol), a.w, a.alpha, a.normalize,
            a.accumulate, a.subvox, cyl, tau, tv);
    else
        bp_column_kernel<TV, VZ, false, SUBV, CYL, DYR><<<grid, dim3(32, BPC_COLS), 0, a.stream>>>(
            G, a.views, a.view_idx, a.n_idx, I, nullptr, static_cast<TV *>(a.vol), a.w, a.alpha, a.normalize,
            a.accumulate, a.subvox, cyl, tau, tv);
    return cudaGetLastError();
}

// Voxels per thread: 4 where 128-slice blocks fit the volume to within 14 %
// of 64-slice ones (144 views at 512^3: 21.7 ms with 4, 24.7 with 2, 27 with 8;
// 180 x 180 x 130, 100 views: 0.69 ms with 2, 0.83 with 1).  Four only from 128
// slices on: a block that reaches beyond the volume reaches beyond the
// detector (85 x 98 x 82, 34 helical views of 3 sub-angles: 0.32 ms with 4,
// 0.16 with 2).
static bool four_voxels(int nz)
{
    const int n4 = (nz + 127) / 128 * 128, n2 = (nz + 63) / 64 * 64;
    return nz >= 128 && 100 * n4 < 114 * n2;
}

// Slices that the kernel works through, the last block's repeats among them
// (two: the event model and sub-voxels always take two voxels per thread).
int backproject_column_slices(const Grid &G, bool two)
{
    const int b = !two && four_voxels(G.nz) ? 128 : 64;
    return (G.nz + b - 1) / b * b;
}

template <typename TV, bool CYL> static cudaError_t bpc_plain(const BpArgs &a)
{
    return four_voxels(a.grid->nz) ? bpc_launch<TV, 4, false, CYL, false>(a)
                                   : bpc_launch<TV, 2, false, CYL, false>(a);
}

template <typename TV> static cudaError_t bpc_dispatch(const BpArgs &a)
{
    if (a.dyr) {
        if (a.cyl || a.subvox > 1) return cudaErrorInvalidValue;
        return bpc_launch<TV, 2, false, false, true>(a);
    }
    if (a.subvox > 1)
        return a.cyl ? bpc_launch<TV, 2, true, true, false>(a) : bpc_launch<TV, 2, true, false, false>(a);
    return a.cyl ? bpc_plain<TV, true>(a) : bpc_plain<TV, false>(a);
}

cudaError_t launch_backproject_column(const BpArgs &a)
{
    return a.vol_dtype == CTREX_F32 ? bpc_dispatch<float>(a) : bpc_dispatch<__nv_bfloat16>(a);
}

bool backproject_column_fits(const Grid &G)
{
    return (G.ny + BPC_WY - 1) / BPC_WY <= 65535 && (G.nz + 63) / 64 <= 65535;
}

bool backproject_box(const ViewGPU &view, const float lo[3], const float hi[3], int4 w)
{
    const float *P = view.P;
    return box_inside(make_float4(P[0], P[1], P[2], P[3]), make_float4(P[4], P[5], P[6], P[7]),
                      make_float4(P[8], P[9], P[10], P[11]), lo, hi,
                      make_float4((float)w.x, (float)w.y, (float)w.z, (float)w.w)) > 0;
}

bool backproject_flat(const Grid &G, const ViewGPU *views, int n)
{
    // (a block of slices may reach beyond a thin volume)
    const int block = four_voxels(G.nz) ? 128 : 64;
    const float lo[3] = {0.0f, 0.0f, 0.0f},
                hi[3] = {G.nx - 1.0f, G.ny - 1.0f, (G.nz > block ? G.nz : block) - 1.0f};
    const float4 det = make_float4(0.0f, (float)(G.nu - 1), 0.0f, (float)(G.nv - 1));
    for (int i = 0; i < n; ++i) {
        const float *P = views[i].P;
        if (box_inside(make_float4(P[0], P[1], P[2], P[3]), make_float4(P[4], P[5], P[6], P[7]),
                       make_float4(P[8], P[9], P[10], P[11]), lo, hi, det) != 2)
            return false;
    }
    return true;
}

}  // namespace ctrex
