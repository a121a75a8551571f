// column.cu -- allocation and upload of column stores (column.cuh).
#include "column.cuh"

namespace ctrex {

void col_release(ColStore &s)
{
    if (s.buf) cudaFree(s.buf);
    s = ColStore();
}

// At least n zeroed pairs; a buffer that holds them and is not twice as large
// is kept, another one is replaced, and a refusal leaves the store as it was.
// Not in a capture, where the zeros would be written by the replay while the
// store counts as laid out at once.
static cudaError_t col_alloc(ColStore &s, size_t n, cudaStream_t stream)
{
    if (stream_capturing(stream)) return cudaErrorInvalidValue;
    const size_t bytes = n * sizeof(float2);
    if (bytes > s.bytes || bytes < s.bytes / 2) {
        size_t free = 0, total = 0;
        cudaError_t e = cudaMemGetInfo(&free, &total);
        if (e == cudaSuccess && bytes > (free + s.bytes) / 2) return cudaErrorInvalidValue;
        col_release(s);
        if (e == cudaSuccess) e = cudaMalloc(&s.buf, bytes);
        if (e != cudaSuccess) {
            cudaGetLastError();
            s.buf = nullptr;
            return cudaErrorInvalidValue;
        }
        s.bytes = bytes;
    }
    s.nx = 0;
    return cudaMemsetAsync(s.buf, 0, bytes, stream);
}

cudaError_t col_ensure(ColStore &s, int nx, int ny, int nz, cudaStream_t stream, bool wrap)
{
    if (s.buf && s.nx == nx && s.ny == ny && s.nz == nz && s.wrap == (wrap ? 1 : 0)) return cudaSuccess;
    const size_t sy = ((size_t)nx + 2) << COL_LOG, sz = sy * ((size_t)ny + 2);
    const size_t n = sz * ((((size_t)nz + 1) >> COL_LOG) + 1);
    if (n >= (1ull << 32)) return cudaErrorInvalidValue;
    const cudaError_t e = col_alloc(s, n, stream);
    if (e != cudaSuccess) return e;
    s.nx = nx;
    s.ny = ny;
    s.nz = nz;
    s.wrap = wrap ? 1 : 0;
    s.sy = (unsigned)sy;
    s.sz = (unsigned)(sz - (1u << COL_LOG));
    return cudaSuccess;
}

// Slices of rows v (vs elements apart) of nu values become columns: slice k
// starts at src + k ss and goes to dst + k ds, chunk to chunk `chunk` pairs
// further than the 16 that the pair's index counts.  A CTA takes 32 values
// along u by 64 pairs along v: read along u, turned in shared memory, written
// along v two pairs to a thread (HBM-bound; with 32 x 32 tiles and single
// pairs 90 images of 768^2 took 0.45 ms).  Pair j (padded) holds values j - 1
// and j, zero outside the slice.
template <typename T, bool PAIRS>
__global__ void __launch_bounds__(256) col_upload_kernel(const T *__restrict__ src, float2 *__restrict__ dst, int nu,
                                                         int nv, size_t vs, size_t ss, size_t ds, unsigned chunk,
                                                         int tiles_u, int n)
{
    __shared__ float tile[65][33];  // [j - j0][u - u0]
    const int u0 = (blockIdx.x % tiles_u) * 32, j0 = (int)(blockIdx.x / tiles_u) * 64;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, u = u0 + lane;
    for (int k = blockIdx.y; k < n; k += gridDim.y) {
        const T *s = src + (size_t)k * ss;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int r = warp + 8 * i, v = j0 - 1 + r;
            if (r < 65) tile[r][lane] = u < nu && v >= 0 && v < nv ? Storage<T>::load(s + (size_t)v * vs + u) : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int c = warp + 8 * i, r = 2 * lane;
            const unsigned j = j0 + r;
            if (u0 + c < nu && (int)j <= nv) {
                const float a = tile[r][c], b = tile[r + 1][c], e = tile[r + 2][c];
                *reinterpret_cast<float4 *>(dst + (size_t)k * ds + (size_t)(j >> COL_LOG) * chunk +
                                            ((size_t)(u0 + c + 1) << COL_LOG) + j) =
                    PAIRS ? make_float4(a, b, b, e) : make_float4(a, b - a, b, e - b);
            }
        }
        __syncthreads();
    }
}

static cudaError_t upload(const void *src, int dtype, float2 *dst, int nu, int nv, size_t vs, size_t ss, size_t ds,
                          unsigned chunk, int n, cudaStream_t stream, bool pairs = false)
{
    const int tu = (nu + 31) / 32;
    const dim3 grid(tu * ((nv + 1 + 63) / 64), n < 65535 ? n : 65535);
    auto go = [&](auto *kernel, auto *s) {
        kernel<<<grid, 256, 0, stream>>>(s, dst, nu, nv, vs, ss, ds, chunk, tu, n);
    };
    if (dtype == CTREX_BF16) {
        typedef __nv_bfloat16 T;
        go(pairs ? col_upload_kernel<T, true> : col_upload_kernel<T, false>, static_cast<const T *>(src));
    } else {
        go(pairs ? col_upload_kernel<float, true> : col_upload_kernel<float, false>, static_cast<const float *>(src));
    }
    return cudaGetLastError();
}

cudaError_t col_upload(const ColStore &s, const void *src, int dtype, cudaStream_t stream, bool pairs)
{
    cudaError_t e =
        upload(src, dtype, s.buf + s.sy, s.nx, s.nz, (size_t)s.nx * s.ny, s.nx, s.sy, s.sz, s.ny, stream, pairs);
    if (e == cudaSuccess && s.wrap)
        e = upload(src, dtype, s.buf + (size_t)s.sy * (s.ny + 1), s.nx, s.nz, (size_t)s.nx * s.ny, s.nx, s.sy, s.sz, 1,
                   stream);
    return e;
}

cudaError_t col_ensure_images(ColStore &s, int nu, int nv, int n, cudaStream_t stream)
{
    if (s.buf && s.nx == nu && s.ny == nv && s.nz >= n) return cudaSuccess;
    const size_t sv = ((size_t)nu + 2) << COL_LOG, view = sv * ((((size_t)nv + 1) >> COL_LOG) + 1);
    if (view >= (1ull << 32)) return cudaErrorInvalidValue;
    const cudaError_t e = col_alloc(s, view * (size_t)n, stream);
    if (e != cudaSuccess) return e;
    s.nx = nu;
    s.ny = nv;
    s.nz = n;
    s.sy = (unsigned)(sv - (1u << COL_LOG));
    s.view = view;
    return cudaSuccess;
}

cudaError_t col_upload_images(const ColStore &s, const void *src, int dtype, int n, cudaStream_t stream)
{
    return upload(src, dtype, s.buf, s.nx, s.ny, s.nx, (size_t)s.nx * s.ny, s.view, s.sy, n, stream);
}

}  // namespace ctrex
