// fwd_column_models.cu -- the other forward models by z columns (see
// fwd_column.cu): event-based 4D values (dyrect.cuh), the multi-resolution ROI
// (roi.cuh), the cylindrical domain (cylinder.cuh) and the classical Joseph
// projector (joseph.cuh).  Each restates its model's integral on column
// stores; the geometry helpers are the texture versions' own.
//
// Forward + correction of 90 views of 768^2 (event: 384^2), texture gathers /
// columns: event model 256^3 with the 8-region scene 18.0 / 6.8 ms; ROI 256^3
// in 256^3 48.9 / 19.4 ms; cylinder 256 x 1024 x 512 73.5 / 51.3 ms (bound by
// issue: the square root and arctangent of each sample); Joseph 512^3 22.3 /
// 11.7 ms.
#include "cylinder.cuh"
#include "fwd_column.cuh"
#include "joseph.cuh"
#include "roi.cuh"

namespace ctrex {

// ---- event model -------------------------------------------------------------
//
// mu0, mu1 and tau in column stores of one shape, of pairs (a footprint may
// take its two z neighbours from different fields).  A run of DYR_BLOCK samples
// first looks up the (min, max) transition time of the voxels within 4 of its
// first sample's 8^3 brick: where the view's time lies outside it, the whole
// run reads one field like the static model.  Elsewhere each sample looks at
// its own brick, and only footprints that straddle the view's time read both
// fields and the transition times.
struct ColEvent {
    ColVolume v0;               // mu0; the other two differ in the pointer only
    const float2 *p1, *pt;      // mu1, tau
    const float *t_view;
    const float2 *brick, *block;
    int bnx, bny;
};
constexpr int DYR_BLOCK = 8;  // samples at most half a voxel apart: within 3.5 voxels of the first

struct PixelEvent {
    const ColEvent &E;
    const ViewGPU *views;
    const Grid &G;

    __device__ __forceinline__ ColPairs pick(unsigned i, float t) const
    {
        ColVolume v1 = E.v0, vt = E.v0;
        v1.p = E.p1;
        vt.p = E.pt;
        const ColTaps a = col_load(E.v0, i), b = col_load(v1, i), tt = col_load(vt, i);
        auto sel = [&](float2 x, float2 y, float2 z) {
            return make_float2(t < z.x ? x.x : y.x, t < z.y ? x.y : y.y);
        };
        return {sel(a.q00, b.q00, tt.q00), sel(a.q10, b.q10, tt.q10), sel(a.q01, b.q01, tt.q01),
                sel(a.q11, b.q11, tt.q11)};
    }
    __device__ __forceinline__ float2 look(const float2 *table, const ColRun &r) const
    {
        const int bx = ((int)(r.px >> 32) - 1) >> 3, by = ((int)(r.py >> 32) - 1) >> 3,
                  bz = ((int)(r.pz >> 32) - 1) >> 3;
        return __ldg(table + (bz * E.bny + by) * E.bnx + bx);
    }
    __device__ __forceinline__ void operator()(int view, float u, float v, float &val, float &rs) const
    {
        const float t = __ldg(E.t_view + view);
        auto taps = [&](unsigned i, unsigned j, unsigned k) { return pick(E.v0.index(i, j, k), t); };
        float acc = 0.0f, acc_rs = 0.0f;
        for (int s = 0; s < G.n_sub; ++s) {
            Ray R;
            if (!setup_ray(G, views[view * G.n_sub + s], u, v, R)) continue;
            const int Km1 = R.K - 1;
            int ka, kb;
            interior_range(G, R, ka, kb);
            ColRun run;
            if (!run.start(E.v0, R.g0, R.sg, ka, kb - ka)) kb = ka;
            float a = 0.0f, ars = 0.0f, ws;
            for (int k = ka > 0 ? 0 : kb; k < Km1; k = k + 1 == ka ? kb : k + 1) {
                const float kf = (float)k;
                a += col_edge(E.v0, fmaf(kf, R.sg[0], R.g0[0]), fmaf(kf, R.sg[1], R.g0[1]),
                              fmaf(kf, R.sg[2], R.g0[2]), ws, taps);
                ars += ws;
            }
            ars = (ars + (float)(kb - ka)) * G.step_mm;
            if (R.w_last > 0.0f) {
                acc = fmaf(R.w_last, col_edge(E.v0, R.g_last[0], R.g_last[1], R.g_last[2], ws, taps), acc);
                ars = fmaf(R.w_last, ws, ars);
            }
            acc_rs += ars;
            // longer steps (a coarse step_vox): shorter runs
            const float smax = fmaxf(fabsf(R.sg[0]), fmaxf(fabsf(R.sg[1]), fabsf(R.sg[2])));
            const int len = smax <= 0.5f ? DYR_BLOCK : (smax <= 3.5f ? 1 + (int)(3.5f / smax) : 1);
            for (int left = kb - ka; left > 0; left -= len) {
                const int n = min(len, left);
                const float2 lh = look(E.block, run);
                if (t < lh.x || t >= lh.y) {
                    ColVolume V = E.v0;
                    V.p = t < lh.x ? E.v0.p : E.p1;
                    a = run.sum<true>(V, n, a);
                } else {
                    for (int i = 0; i < n; ++i) {
                        const float2 b = look(E.brick, run);
                        const unsigned j = run.index(E.v0);
                        ColPairs q;
                        if (t < b.x || t >= b.y) {
                            ColVolume V = E.v0;
                            V.p = t < b.x ? E.v0.p : E.p1;
                            q = col_load_pairs(V, j);
                        } else {
                            q = pick(j, t);
                        }
                        a += run.interp(q);
                        run.next();
                    }
                }
            }
            acc = fmaf(a, G.step_mm, acc);
        }
        val = acc * G.inv_sub;
        rs = acc_rs * G.inv_sub;
    }
};

// ---- multi-resolution ROI ----------------------------------------------------

struct ColRoi {
    ColVolume ctx, roi;
    RoiGPU R;
};

// roi_piece of roi.cuh on a column store.
__device__ __forceinline__ void col_piece(const ColVolume &V, const int n[3], const float X[3], const float dg[3],
                                          float a, float b, float h, float &val, float &rs)
{
    if (!(b > a)) return;
    int K = (int)ceilf((b - a) / h);
    if (K < 1) K = 1;
    int ka, kb;
    piece_interior(X, dg, a, h, K, n, ka, kb);
    auto taps = [&](unsigned i, unsigned j, unsigned k) { return col_load(V, V.index(i, j, k)); };
    float g0[3], sg[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        g0[c] = fmaf(a + 0.5f * h, dg[c], X[c]);
        sg[c] = h * dg[c];
    }
    ColRun run;
    if (!run.start(V, g0, sg, ka, kb - ka)) kb = ka;
    float acc = 0.0f, wacc = 0.0f, ws;
    for (int k = ka > 0 ? 0 : kb; k < K - 1; k = k + 1 == ka ? kb : k + 1) {
        const float t = fmaf((float)k + 0.5f, h, a);
        acc += col_edge(V, fmaf(t, dg[0], X[0]), fmaf(t, dg[1], X[1]), fmaf(t, dg[2], X[2]), ws, taps);
        wacc += ws;
    }
    wacc += (float)(kb - ka);
    const float a_last = fmaf((float)(K - 1), h, a);
    const float t_last = 0.5f * (a_last + b), w_last = b - a_last;
    const float last =
        col_edge(V, fmaf(t_last, dg[0], X[0]), fmaf(t_last, dg[1], X[1]), fmaf(t_last, dg[2], X[2]), ws, taps);
    rs += fmaf(wacc, h, w_last * ws);
    val = fmaf(w_last, last, val);
    val = fmaf(run.sum(V, kb - ka, acc), h, val);
}

struct PixelRoi {
    const ColRoi &Q;
    const ViewGPU *views;
    const Grid &G;

    __device__ __forceinline__ void ray(const ViewGPU &V, float u, float v, float &val, float &rs) const
    {
        float X[3], dg[3], len;
        ray_line(G, V, u, v, X, dg, len);
        float t0, t1;
        if (!clip_box(X, dg, G.lo, G.hi, -len, t0, t1)) return;
        const RoiGPU &R = Q.R;
        float r0, r1;
        const bool hit = clip_box(X, dg, R.lo, R.hi, t0, r0, r1) && r0 < t1;
        const int nc[3] = {G.nx, G.ny, G.nz}, nr[3] = {R.n[0], R.n[1], R.n[2]};
        const float hc = G.step_mm;
        if (!hit) {
            col_piece(Q.ctx, nc, X, dg, t0, t1, hc, val, rs);
            return;
        }
        r1 = fminf(r1, t1);
        // the two context pieces by one call site, the ROI piece between them
#pragma unroll 1
        for (int i = 0; i < 2; ++i) col_piece(Q.ctx, nc, X, dg, i ? r1 : t0, i ? t1 : r0, hc, val, rs);
        // ROI index coordinates: g_roi = g_ctx * sc + oc per axis
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            X[a] = fmaf(X[a], R.sc[a], R.oc[a]);
            dg[a] *= R.sc[a];
        }
        col_piece(Q.roi, nr, X, dg, r0, r1, R.step_mm, val, rs);
    }
    __device__ __forceinline__ void operator()(int view, float u, float v, float &val, float &rs) const
    {
        for (int s = 0; s < G.n_sub; ++s) ray(views[view * G.n_sub + s], u, v, val, rs);
        val *= G.inv_sub;
        rs *= G.inv_sub;
    }
};

// ---- cylindrical domain ------------------------------------------------------
//
// Columns of (ring, sector); the store's row N_phi repeats sector 0.

struct ColCyl {
    ColVolume vol;
    CylGPU C;
};

struct PixelCyl {
    const ColCyl &Q;
    const ViewGPU *views;
    const Grid &G;

    // as CylSampler: r clamped at the first ring centre, phi periodic, zero
    // outside in r and z
    __device__ __forceinline__ float sample(float qx, float qy, float qz, float &ws) const
    {
        const CylGPU &C = Q.C;
        const float nphi = (float)C.n_phi;
        const float q2 = fmaf(qx, qx, qy * qy);
        const float r = q2 > 0.0f ? q2 * rsqrtf(q2) : 0.0f;
        float gp = fmaf(cyl_angle(qx, qy), C.inv_dphi, -0.5f);
        if (gp < 0.0f) gp += nphi;
        if (gp >= nphi) gp -= nphi;  // -tiny + N_phi rounded up to N_phi
        gp = fminf(fmaxf(gp, 0.0f), __uint_as_float(__float_as_uint(nphi) - 1u));  // below N_phi
        const float gr = fminf(fmaxf(fmaf(r, C.inv_dr, -0.5f), 0.0f), Q.vol.hx + 0.75f);
        const float gz = fminf(fmaxf(fmaf(qz, C.inv_dz, C.zc), -1.0f), Q.vol.hz + 0.75f);
        const float fr = floorf(gr), fp = floorf(gp), fz = floorf(gz);
        const float ar = gr - fr, ap = gp - fp, az = gz - fz;
        ws = col_inside(gr, ar, Q.vol.hx) * col_inside(gz, az, Q.vol.hz);
        return col_interp(col_load(Q.vol, Q.vol.index((int)fr + 1, (int)fp + 1, (int)fz + 1)), ar, ap, az);
    }
    __device__ __forceinline__ void operator()(int view, float u, float v, float &val, float &rs) const
    {
        float acc = 0.0f, acc_rs = 0.0f;
        for (int s = 0; s < G.n_sub; ++s) {
            Ray R;
            if (!setup_ray_cyl(G, Q.C, views[view * G.n_sub + s], u, v, R)) continue;
            float a = 0.0f, ars = 0.0f, ws, kf = 0.0f;
#pragma unroll 2
            for (int k = 0; k < R.K - 1; ++k, kf += 1.0f) {
                a += sample(fmaf(kf, R.sg[0], R.g0[0]), fmaf(kf, R.sg[1], R.g0[1]), fmaf(kf, R.sg[2], R.g0[2]), ws);
                ars += ws;
            }
            a *= G.step_mm;
            ars *= G.step_mm;
            if (R.w_last > 0.0f) {
                a = fmaf(R.w_last, sample(R.g_last[0], R.g_last[1], R.g_last[2], ws), a);
                ars = fmaf(R.w_last, ws, ars);
            }
            acc += a;
            acc_rs += ars;
        }
        val = acc * G.inv_sub;
        rs = acc_rs * G.inv_sub;
    }
};

// ---- classical Joseph --------------------------------------------------------
//
// One store serves all three principal axes: a slice across x or y is crossed
// between two columns (both z neighbours in each load), a slice across z
// between four.

struct PixelJoseph {
    const ColVolume &vol;
    const ViewGPU *views;
    const Grid &G;

    __device__ __forceinline__ void ray(const ViewGPU &V, float u, float v, float &val, float &rs) const
    {
        JRay J;
        if (!joseph_setup(G, V, u, v, J)) return;
        int a1, a2;
        joseph_axes(J.m, a1, a2);
        const int n1 = jsel(G.nx, G.ny, G.nz, a1), n2 = jsel(G.nx, G.ny, G.nz, a2);
        const int k0 = max(J.klo - 1, J.kmin), k1 = min(J.khi + 1, J.kmax);
        // crossings ka .. kb - 1 with all taps inside (one slice of slack)
        float lo = (float)k0, hi = (float)k1;
        const float c0[2] = {J.p0, J.q0}, r[2] = {J.r1, J.r2};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float h = (float)((i ? n2 : n1) - 1);
            if (r[i] != 0.0f) {
                const float ri = 1.0f / r[i], ta = -c0[i] * ri, tb = (h - c0[i]) * ri;
                lo = fmaxf(lo, fminf(ta, tb));
                hi = fminf(hi, fmaxf(ta, tb));
            } else if (!(c0[i] >= 0.0f && c0[i] <= h)) {
                hi = -2.0f;
            }
        }
        int ka = min(max((int)ceilf(lo) + 1, k0), k1 + 1), kb = max(min((int)floorf(hi), k1 + 1), ka);
        const float F = 4294967296.0f;
        const long long dp = __float2ll_rn(J.r1 * F), dq = __float2ll_rn(J.r2 * F);
        long long p = __float2ll_rn(J.p0 * F) + (1ll << 32) + ka * dp, q = __float2ll_rn(J.q0 * F) + (1ll << 32) + ka * dq;
        if (!(axis_inside(p, dp, J.r1, kb - ka, (float)(n1 - 1)) && axis_inside(q, dq, J.r2, kb - ka, (float)(n2 - 1))))
            kb = ka;
        const bool zslices = J.m == 2;
        // pairs from one value to the next along the slice's first axis and along the principal one
        const unsigned s1 = a1 == 0 ? 1u << COL_LOG : vol.sy, sm = J.m == 0 ? 1u << COL_LOG : vol.sy;
        auto at = [&](unsigned ip, unsigned iq, int k) {  // padded in-slice indices
            if (zslices) return vol.index(ip, iq, (unsigned)(k + 1));
            return ip * s1 + (unsigned)(k + 1) * sm + ((iq >> COL_LOG) * vol.sz + iq);
        };
        auto bilinear = [&](unsigned i, float ap, float aq) {
            if (zslices) {  // values at (x, y) .. (x + 1, y + 1): the first of each pair
                const float *f = reinterpret_cast<const float *>(vol.p + i);
                const float c00 = __ldg(f), c10 = __ldg(f + (2 << COL_LOG)), c01 = __ldg(f + 2 * (size_t)vol.sy),
                            c11 = __ldg(f + 2 * (size_t)vol.sy + (2 << COL_LOG));
                const float e0 = fmaf(ap, c10 - c00, c00), e1 = fmaf(ap, c11 - c01, c01);
                return fmaf(aq, e1 - e0, e0);
            }
            return lerp(col_value(__ldg(vol.p + i), aq), col_value(__ldg(vol.p + s1 + i), aq), ap);
        };
        float acc = 0.0f, wacc = 0.0f;
        for (int k = ka > k0 ? k0 : kb; k <= k1; k = k + 1 == ka ? kb : k + 1) {
            const float gp = fmaf((float)k, J.r1, J.p0), gq = fmaf((float)k, J.r2, J.q0);
            if (!(gp > -1.0f && gp < (float)n1 && gq > -1.0f && gq < (float)n2)) continue;  // no tap inside
            const float fp = floorf(gp), fq = floorf(gq);
            acc += bilinear(at((int)fp + 1, (int)fq + 1, k), gp - fp, gq - fq);
            wacc += col_inside(gp, gp - fp, (float)(n1 - 1)) * col_inside(gq, gq - fq, (float)(n2 - 1));
        }
        wacc += (float)(kb - ka);
        if (zslices) {
            for (int k = ka; k < kb; ++k) {
                acc += bilinear(at((unsigned)(p >> 32), (unsigned)(q >> 32), k), fixed_fraction((unsigned)p),
                                fixed_fraction((unsigned)q));
                p += dp;
                q += dq;
            }
        } else {
            unsigned base = (unsigned)(ka + 1) * sm;
#pragma unroll 4
            for (int left = kb - ka; left > 0; --left) {
                const unsigned iq = (unsigned)(q >> 32);
                const unsigned i = (unsigned)(p >> 32) * s1 + (base + ((iq >> COL_LOG) * vol.sz + iq));
                const float aq = fixed_fraction((unsigned)q);
                acc += lerp(col_value(__ldg(vol.p + i), aq), col_value(__ldg(vol.p + s1 + i), aq),
                            fixed_fraction((unsigned)p));
                p += dp;
                q += dq;
                base += sm;
            }
        }
        val = fmaf(acc, J.dl, val);
        rs = fmaf(wacc, J.dl, rs);
    }
    __device__ __forceinline__ void operator()(int view, float u, float v, float &val, float &rs) const
    {
        for (int s = 0; s < G.n_sub; ++s) ray(views[view * G.n_sub + s], u, v, val, rs);
        val *= G.inv_sub;
        rs *= G.inv_sub;
    }
};

// ---- launches ----------------------------------------------------------------

template <typename Pixel, typename Model, typename TP, int MODE>
__global__ void __launch_bounds__(32 * COL_TU, COL_MIN_BLOCKS)
    fwd_column_model_kernel(Grid G, const ViewGPU *__restrict__ views, const Model model,
                            const int *__restrict__ view_idx, TP *__restrict__ out, float *__restrict__ rowsum_out,
                            const TP *__restrict__ p, float *__restrict__ partials, unsigned *devcheck, int p_by_view,
                            int n_strips)
{
    col_body<TP, MODE>(G, view_idx, out, rowsum_out, p, partials, devcheck, p_by_view, n_strips,
                       Pixel{model, views, G});
}

template <typename Pixel, typename Model, typename TP, int MODE>
static cudaError_t launch(const FwdArgs &a, const Model &m, void *out, float *rowsum, const void *p, float *partials)
{
    int n_strips;
    const dim3 grid = col_grid(*a.grid, a.n_idx, n_strips);
    fwd_column_model_kernel<Pixel, Model, TP, MODE><<<grid, dim3(32, COL_TU), 0, a.stream>>>(
        *a.grid, a.views, m, a.view_idx, static_cast<TP *>(out), rowsum, static_cast<const TP *>(p), partials,
        a.devcheck, a.p_by_view, n_strips);
    return cudaGetLastError();
}

template <typename Pixel, typename Model>
static cudaError_t launch(const FwdArgs &a, const Model &m, bool correct, int pdt, void *out, float *rowsum,
                          const void *p, float *partials)
{
    if (pdt == CTREX_F32)
        return correct ? launch<Pixel, Model, float, MODE_CORRECT>(a, m, out, rowsum, p, partials)
                       : launch<Pixel, Model, float, MODE_PROJECT>(a, m, out, rowsum, p, partials);
    return correct ? launch<Pixel, Model, __nv_bfloat16, MODE_CORRECT>(a, m, out, rowsum, p, partials)
                   : launch<Pixel, Model, __nv_bfloat16, MODE_PROJECT>(a, m, out, rowsum, p, partials);
}

cudaError_t launch_forward_column_models(const FwdArgs &a, bool correct, int pdt, void *out, float *rowsum,
                                         const void *p, float *partials)
{
    const ColVolume v = col_view(*a.column);
    if (a.roi) {
        if (!a.column1) return cudaErrorInvalidValue;
        return launch<PixelRoi>(a, ColRoi{v, col_view(*a.column1), *a.roi}, correct, pdt, out, rowsum, p, partials);
    }
    if (a.dyr) {
        if (!a.column1 || !a.column_tau) return cudaErrorInvalidValue;
        const ColEvent e{v, a.column1->buf, a.column_tau->buf, a.dyr->t_view, a.dyr->tau_brick, a.dyr->tau_block,
                         a.dyr->bnx, a.dyr->bny};
        return launch<PixelEvent>(a, e, correct, pdt, out, rowsum, p, partials);
    }
    if (a.cyl) return launch<PixelCyl>(a, ColCyl{v, *a.cyl}, correct, pdt, out, rowsum, p, partials);
    return launch<PixelJoseph>(a, v, correct, pdt, out, rowsum, p, partials);
}

}  // namespace ctrex
