// unet_ops.cu -- the passes of the warm-start network around its
// convolutions (conv_tc.cu), and the network's forward pass as one call.
// All of them are bound by HBM; each reads its inputs and writes its outputs
// once, 16 bytes (8 BF16 channels) a thread.
//
// At 128^3 (batch 1 for the network, 2 for the gradient), as separate tensor
// operations / here: the ReLU mask and the bias gradient of a 16-channel
// layer 485 / 66 us; upsampling and skip concatenation of the top level 450 /
// 51 us; head 350 / 17 us; pooling of the top level 48 / 15 us; the network as
// a whole, launches included, 1888 / 873 us.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ctrex.h"

namespace {

typedef __nv_bfloat16 bf16;

union Vec8 {
    uint4 v;
    __nv_bfloat162 h[4];
};

unsigned blocks_for(long long n, int per) { return (unsigned)((n + per - 1) / per); }

// ---- ReLU mask and bias gradient ---------------------------------------------

constexpr int BG_THREADS = 256;
constexpr int BG_MAX_BLOCKS = 152 * 8;

// g = dy * (y > 0) (y null: g is not written and dy counts as it is), and
// this CTA's sum of it per channel.  A thread keeps one group of 8 channels:
// the grid's thread count is a multiple of the groups.  FP32 sums within a CTA
// (1 / 1216 of the voxels, 103 a thread at 2 x 200^3 and 16 channels), FP64 over
// the CTAs (bias_sum_kernel): 4e-8 of sum |g| at 25 M voxels of mean 1, where
// torch's FP32 sum was off by 8e-8.
__global__ void __launch_bounds__(BG_THREADS) bias_grad_kernel(const uint4 *__restrict__ dy,
                                                               const uint4 *__restrict__ y, uint4 *__restrict__ g,
                                                               long long n, int groups, float *__restrict__ partial)
{
    __shared__ float s[BG_THREADS][9];
    const int tid = threadIdx.x;
    const long long stride = (long long)gridDim.x * BG_THREADS;
    float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
    for (long long i = (long long)blockIdx.x * BG_THREADS + tid; i < n; i += stride) {
        Vec8 d, o;
        d.v = __ldg(dy + i);
        if (y) {
            Vec8 r;
            r.v = __ldg(y + i);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = __bfloat1622float2(d.h[q]), t = __bfloat1622float2(r.h[q]);
                o.h[q] = __floats2bfloat162_rn(f.x * (t.x > 0.0f ? 1.0f : 0.0f), f.y * (t.y > 0.0f ? 1.0f : 0.0f));
            }
            g[i] = o.v;
        } else {
            o.v = d.v;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 f = __bfloat1622float2(o.h[q]);
            a[2 * q] += f.x;
            a[2 * q + 1] += f.y;
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) s[tid][q] = a[q];
    __syncthreads();
    for (int c = tid; c < 8 * groups; c += BG_THREADS) {
        float sum = 0.0f;
        for (int t = c / 8; t < BG_THREADS; t += groups) sum += s[t][c % 8];
        partial[(size_t)blockIdx.x * 8 * groups + c] = sum;
    }
}

// db[c] = sum of the CTAs' partials, one CTA per channel, fixed order.
__global__ void __launch_bounds__(128) bias_sum_kernel(const float *__restrict__ partial, int blocks, int channels,
                                                       float *__restrict__ db)
{
    __shared__ double s[128];
    double a = 0.0;
    for (int b = threadIdx.x; b < blocks; b += 128) a += (double)partial[(size_t)b * channels + blockIdx.x];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int off = 64; off > 0; off >>= 1) {
        if (threadIdx.x < off) s[threadIdx.x] += s[threadIdx.x + off];
        __syncthreads();
    }
    if (threadIdx.x == 0) db[blockIdx.x] = (float)s[0];
}

// ---- network passes ----------------------------------------------------------

constexpr int LAYERS = 14;

struct CastTable {
    const float *src[LAYERS];
    bf16 *dst[LAYERS];
    int n[LAYERS];
};

// FP32 master weights to BF16, all layers in one launch (grid y = layer, four
// values a thread: every layer's count is a multiple of 4).
__global__ void __launch_bounds__(256) cast_weights_kernel(const CastTable t)
{
    const int l = blockIdx.y;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < t.n[l] / 4; i += gridDim.x * 256) {
        const float *s = t.src[l] + 4 * i;
        __nv_bfloat162 *o = reinterpret_cast<__nv_bfloat162 *>(t.dst[l] + 4 * i);
        o[0] = __floats2bfloat162_rn(__ldg(s), __ldg(s + 1));
        o[1] = __floats2bfloat162_rn(__ldg(s + 2), __ldg(s + 3));
    }
}

// The input volume as the first of 16 BF16 channels, zeros beside it.
__global__ void __launch_bounds__(256) input_kernel(const float *__restrict__ x, uint4 *__restrict__ out, long long n)
{
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;  // 16-byte half voxel
    if (i >= 2 * n) return;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (!(i & 1)) v.x = __bfloat16_as_ushort(__float2bfloat16_rn(__ldg(x + (i >> 1))));
    out[i] = v;
}

// 2 x 2 x 2 maximum (NaN propagates), channels last, G groups of 8 channels;
// h, w: the output's edges, planes: its planes over the batch.  Grid y runs
// over output rows (no 64-bit divisions per thread).
__global__ void __launch_bounds__(256) pool_kernel(const uint4 *__restrict__ x, uint4 *__restrict__ out, int planes,
                                                   int h, int w, int G)
{
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= w * G) return;
    const int X = i / G, c = i - X * G;
    for (long long row = blockIdx.y; row < (long long)planes * h; row += gridDim.y) {
        const long long Z = row / h;
        const int Y = (int)(row - Z * h);
        Vec8 m, t;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            t.v = __ldg(x + (((2 * Z + (q >> 2)) * 2 * h + 2 * Y + ((q >> 1) & 1)) * 2 * w + 2 * X + (q & 1)) * G + c);
            if (q == 0)
                m.v = t.v;
            else
#pragma unroll
                for (int r = 0; r < 4; ++r) m.h[r] = __hmax2_nan(m.h[r], t.h[r]);
        }
        out[row * w * G + i] = m.v;
    }
}

// Channels [nearest-upsampled low (Gl groups) | skip (Gs groups)]; h, w: the
// output's edges, twice low's, planes: its planes over the batch.
__global__ void __launch_bounds__(256) upcat_kernel(const uint4 *__restrict__ low, const uint4 *__restrict__ skip,
                                                    uint4 *__restrict__ out, int planes, int h, int w, int Gl, int Gs)
{
    const int G = Gl + Gs, i = blockIdx.x * 256 + threadIdx.x;
    if (i >= w * G) return;
    const int X = i / G, c = i - X * G;
    const long long rows = (long long)planes * h;
    // four rows a step, their loads before their stores
    for (long long r0 = 4ll * blockIdx.y; r0 < rows; r0 += 4ll * gridDim.y) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long row = min(r0 + k, rows - 1), Z = row / h;  // (a batch item has an even number of planes)
            const int Y = (int)(row - Z * h);
            v[k] = c >= Gl ? __ldg(skip + (row * w + X) * Gs + c - Gl)
                           : __ldg(low + (((Z >> 1) * (h / 2) + (Y >> 1)) * (w / 2) + (X >> 1)) * Gl + c);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (r0 + k < rows) out[(r0 + k) * w * G + i] = v[k];
    }
}

// y = x + (sum_c u[c] w[c] + b), G groups of 8 channels per voxel.
__global__ void __launch_bounds__(256) head_kernel(const uint4 *__restrict__ u, const float *__restrict__ w,
                                                   const float *__restrict__ b, const float *__restrict__ x,
                                                   float *__restrict__ y, long long n, int G)
{
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    float s = 0.0f;
    for (int c = 0; c < G; ++c) {
        Vec8 t;
        t.v = __ldg(u + i * G + c);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 f = __bfloat1622float2(t.h[q]);
            s = fmaf(f.x, __ldg(w + 8 * c + 2 * q), s);
            s = fmaf(f.y, __ldg(w + 8 * c + 2 * q + 1), s);
        }
    }
    y[i] = __ldg(x + i) + (s + __ldg(b));
}

// ---- the network's layers and workspace --------------------------------------

struct Layer {
    int level, cin, cout;
};

void net_layers(int c1, Layer l[LAYERS])
{
    const int c2 = 2 * c1, c3 = 4 * c1, c4 = 8 * c1;
    const Layer t[LAYERS] = {{0, 16, c1},      {0, c1, c1}, {1, c1, c2},      {1, c2, c2}, {2, c2, c3},
                             {2, c3, c3},      {3, c3, c4}, {3, c4, c4},      {2, c4 + c3, c3}, {2, c3, c3},
                             {1, c3 + c2, c2}, {1, c2, c2}, {0, c2 + c1, c1}, {0, c1, c1}};
    for (int i = 0; i < LAYERS; ++i) l[i] = t[i];
}

// Workspace (bytes from its start): the BF16 weights; per level an activation
// buffer a, the skip s and the concatenation cat (at the top level cat also
// holds the 16-channel input, at the bottom only a and s exist).
struct Plan {
    size_t w[LAYERS], a[4], s[4], cat[4], total;
};

Plan net_plan(long long vox, int c1)
{
    Plan p{};
    Layer l[LAYERS];
    net_layers(c1, l);
    size_t at = 0;
    auto take = [&](size_t elems) {
        const size_t r = at;
        at += (elems * sizeof(bf16) + 255) / 256 * 256;
        return r;
    };
    for (int i = 0; i < LAYERS; ++i) p.w[i] = take((size_t)27 * l[i].cin * l[i].cout);
    for (int v = 0; v < 4; ++v) {
        const size_t n = (size_t)(vox >> (3 * v)), c = (size_t)c1 << v;
        p.a[v] = take(n * c);
        p.s[v] = take(n * c);
        p.cat[v] = v < 3 ? take(n * (v == 0 && 3 * c < 16 ? 16 : 3 * c)) : 0;
    }
    p.total = at;
    return p;
}

bool net_shape_ok(int nb, int d, int h, int w, int base)
{
    return nb >= 1 && d >= 8 && h >= 8 && w >= 8 && !(d & 7) && !(h & 7) && !(w & 7) && base >= 8 && !(base & 7) &&
           base <= 512 && (long long)nb * d * h * w <= (1LL << 31) / (3 * base > 16 ? 3 * base : 16) * 8;
}

}  // namespace

extern "C" {

int ctrex_conv3d_bias_grad(const void *dy, const void *y, void *g, float *db, float *scratch, long long voxels,
                           int channels, void *stream)
{
    if (!dy || !db || !scratch || (y && !g)) return CTREX_E_ARG;
    if ((reinterpret_cast<uintptr_t>(dy) | reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(g)) & 15)
        return CTREX_E_ARG;
    const int groups = channels / 8;
    if (voxels < 1 || channels < 8 || (channels & 7) || BG_THREADS % groups) return CTREX_E_SHAPE;
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long n = voxels * groups;
    const long long want = (n + BG_THREADS * 4 - 1) / (BG_THREADS * 4);
    const int blocks = (int)(want < BG_MAX_BLOCKS ? want : BG_MAX_BLOCKS);
    bias_grad_kernel<<<blocks, BG_THREADS, 0, st>>>(static_cast<const uint4 *>(dy), static_cast<const uint4 *>(y),
                                                    static_cast<uint4 *>(g), n, groups, scratch);
    bias_sum_kernel<<<channels, 128, 0, st>>>(scratch, blocks, channels, db);
    return cudaGetLastError() == cudaSuccess ? CTREX_OK : CTREX_E_CUDA;
}

long long ctrex_unet_workspace(int nb, int d, int h, int w, int base)
{
    if (!net_shape_ok(nb, d, h, w, base)) return CTREX_E_SHAPE;
    return (long long)net_plan((long long)nb * d * h * w, base).total;
}

int ctrex_unet_forward(const float *x, float *y, const float *const *weights, const float *const *bias,
                       const float *head_w, const float *head_b, int nb, int d, int h, int w, int base, void *workspace,
                       int *status, void *stream)
{
    if (!x || !y || !weights || !bias || !head_w || !head_b || !workspace || !status) return CTREX_E_ARG;
    if (reinterpret_cast<uintptr_t>(workspace) & 255) return CTREX_E_ARG;
    for (int i = 0; i < LAYERS; ++i)
        if (!weights[i] || !bias[i]) return CTREX_E_ARG;
    if (!net_shape_ok(nb, d, h, w, base)) return CTREX_E_SHAPE;
    const cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long vox = (long long)nb * d * h * w;
    Layer l[LAYERS];
    net_layers(base, l);
    const Plan P = net_plan(vox, base);
    char *ws = static_cast<char *>(workspace);
    CastTable t;
    for (int i = 0; i < LAYERS; ++i) {
        t.src[i] = weights[i];
        t.dst[i] = reinterpret_cast<bf16 *>(ws + P.w[i]);
        t.n[i] = 27 * l[i].cin * l[i].cout;
    }
    cast_weights_kernel<<<dim3(128, LAYERS), 256, 0, st>>>(t);
    void *a[4], *s[4], *cat[4];
    for (int v = 0; v < 4; ++v) {
        a[v] = ws + P.a[v];
        s[v] = ws + P.s[v];
        cat[v] = ws + P.cat[v];
    }
    int rc = CTREX_OK;
    auto conv = [&](int i, const void *in, void *out) {
        const int v = l[i].level;
        if (rc == CTREX_OK)
            rc = ctrex_conv3d_fwd(in, ws + P.w[i], bias[i], out, CTREX_BF16, nb, d >> v, h >> v, w >> v, l[i].cin,
                                  l[i].cout, 1, status, stream);
    };
    auto groups = [&](int v) { return (base << v) / 8; };
    auto row_grid = [&](int v, int G, int per) {
        const long long rows = ((long long)nb * (d >> v) * (h >> v) + per - 1) / per;
        return dim3(blocks_for((long long)(w >> v) * G, 256), (unsigned)(rows < 65535 ? rows : 65535));
    };
    auto pool = [&](int v, const void *in, void *out) {  // level v - 1 to v
        const int G = groups(v - 1);
        pool_kernel<<<row_grid(v, G, 1), 256, 0, st>>>(static_cast<const uint4 *>(in), static_cast<uint4 *>(out),
                                                    nb * (d >> v), h >> v, w >> v, G);
    };
    auto upcat = [&](int v, const void *low) {  // level v + 1 to v, into cat[v]
        const int Gl = groups(v + 1), Gs = groups(v);
        upcat_kernel<<<row_grid(v, Gl + Gs, 4), 256, 0, st>>>(static_cast<const uint4 *>(low),
                                                           static_cast<const uint4 *>(s[v]),
                                                           static_cast<uint4 *>(cat[v]), nb * (d >> v), h >> v, w >> v,
                                                           Gl, Gs);
    };
    input_kernel<<<blocks_for(2 * vox, 256), 256, 0, st>>>(x, static_cast<uint4 *>(cat[0]), vox);
    conv(0, cat[0], a[0]);
    conv(1, a[0], s[0]);
    for (int v = 1; v < 4; ++v) {  // the pooled input of a level sits where its second convolution writes
        pool(v, s[v - 1], s[v]);
        conv(2 * v, s[v], a[v]);
        conv(2 * v + 1, a[v], s[v]);
    }
    const void *low = s[3];
    for (int v = 2; v >= 0; --v) {  // after the concatenation the skip's buffer is free
        upcat(v, low);
        conv(8 + 2 * (2 - v), cat[v], a[v]);
        conv(9 + 2 * (2 - v), a[v], s[v]);
        low = s[v];
    }
    head_kernel<<<blocks_for(vox, 256), 256, 0, st>>>(static_cast<const uint4 *>(low), head_w, head_b, x, y, vox,
                                                      groups(0));
    if (rc != CTREX_OK) return rc;
    return cudaGetLastError() == cudaSuccess ? CTREX_OK : CTREX_E_CUDA;
}

}  // extern "C"
