// column.cuh -- stacks of 2D slices laid out as columns: for every (x, y) of
// a volume, or every u of a detector image, the values along z (along v) are
// contiguous, and each element is the pair (value k, value k + 1 less value k):
// a linear interpolation along the column is one multiply-add.
//
// Why: the rays of a detector column run nearly side by side in x and y and
// one voxel apart in z (a cone-beam scan about z; likewise the voxels of a
// z column project onto one detector column).  A warp that takes 32 pixels
// of a detector column (32 voxels of a z column) therefore reads 32
// neighbouring pairs of one column whatever the view angle: one 256-byte
// load instead of 32 scattered ones, and both z (v) neighbours of a bilinear
// column come in it.  A texture gather returns its 16 bytes at a quarter of
// that rate (see fwd_column.cu and bp_column.cu for what that measured).
//
// The store carries a border of zeros (one element below and above in every
// direction), so a footprint that straddles the grid's edge needs no clamp:
// element (i, j, k) of the grid sits at padded index (i + 1, j + 1, k + 1).
#pragma once

#include "ctrex_internal.cuh"

namespace ctrex {

// A store holds FP32 pairs for BF16 data too: unpacking 16-bit pairs costs the
// projector 8 more instructions a sample, and it is bound by issue as much as
// by loads (144 views of 512^3: 65.8 ms with packed BF16 pairs, 59.6 ms).
constexpr int COL_LOG = 4;  // pairs per 128-byte chunk = 1 << COL_LOG

// Padded index (i, j, k) of a store is at pair
//   ((k >> 4) * (ny + 2) + j) * sy + (i << 4) + (k & 15):
// chunks of 128 bytes along z, then x, then y, then the chunks.  The x
// neighbour of a pair is then 128 bytes on, an immediate offset of a load,
// whatever the volume's size.
struct ColVolume {
    const float2 *p;
    unsigned sy;       // pairs from row j to j + 1
    unsigned sz;       // pairs from chunk to chunk, less the 16 that k itself counts
    float hx, hy, hz;  // nx - 1, ny - 1, nz - 1
    __device__ __forceinline__ unsigned index(unsigned i, unsigned j, unsigned k) const
    {
        return j * sy + ((k >> COL_LOG) * sz + ((i << COL_LOG) + k));
    }
};

struct ColStore {
    float2 *buf = nullptr;
    size_t bytes = 0;
    int nx = 0, ny = 0, nz = 0;  // what it was laid out for (0: nothing)
    unsigned sy = 0, sz = 0;
    int wrap = 0;     // the row past the last repeats row 0 (periodic axis)
    size_t view = 0;  // image stacks: pairs per image (nz: images; sy: chunk to chunk)
};
void col_release(ColStore &s);
// Lays the store out for a volume (zero border written once); an allocation
// that fits, and is not twice as large, is kept.  cudaErrorInvalidValue: the layout's 32-bit indices
// cannot hold it, it would take more than half of the free device memory, or
// the stream is capturing (the caller keeps its other path).
cudaError_t col_ensure(ColStore &s, int nx, int ny, int nz, cudaStream_t stream, bool wrap = false);
// Transposes a [nz][ny][nx] volume into the store; pairs: elements (value k,
// value k + 1).
cudaError_t col_upload(const ColStore &s, const void *src, int dtype, cudaStream_t stream, bool pairs = false);

// The same for a stack of (at least) n detector images nu x nv, columns
// along v.
cudaError_t col_ensure_images(ColStore &s, int nu, int nv, int n, cudaStream_t stream);
cudaError_t col_upload_images(const ColStore &s, const void *src, int dtype, int n, cudaStream_t stream);

inline ColVolume col_view(const ColStore &s)
{
    ColVolume v;
    v.p = s.buf;
    v.sy = s.sy;
    v.sz = s.sz;
    v.hx = (float)(s.nx - 1);
    v.hy = (float)(s.ny - 1);
    v.hz = (float)(s.nz - 1);
    return v;
}

#ifdef __CUDACC__
// The four columns of a footprint: (value k, value k + 1 less it) at (x, y),
// (x + 1, y), (x, y + 1), (x + 1, y + 1).
struct ColTaps {
    float2 q00, q10, q01, q11;
};
__device__ __forceinline__ ColTaps col_load(const ColVolume &V, unsigned i)
{
    const float2 *a = V.p + i, *b = V.p + V.sy + i;
    return {__ldg(a), __ldg(a + (1 << COL_LOG)), __ldg(b), __ldg(b + (1 << COL_LOG))};
}
// a column's value at fraction f of the way to the next one
__device__ __forceinline__ float col_value(float2 q, float f) { return fmaf(f, q.y, q.x); }
__device__ __forceinline__ float lerp(float a, float b, float f) { return fmaf(f, b - a, a); }
__device__ __forceinline__ float2 lerp2(float2 a, float2 b, float2 f)
{
    return __ffma2_rn(f, __ffma2_rn(a, two(-1.0f), b), a);
}
// z first (one multiply-add a column), then x for both rows at once, then y: a
// packed multiply-add takes the issue port twice as long as a single one, so
// only the x step is packed.  144 views of 512^3 52.5 ms, 60 views of 128^3
// 0.466 ms (all single: 53.7, 0.481; x and y packed on pairs of values, then
// z: 55.5, 0.490).
__device__ __forceinline__ float col_interp(const ColTaps &t, float ax, float ay, float az)
{
    const float2 l = make_float2(col_value(t.q00, az), col_value(t.q01, az)),
                 r = make_float2(col_value(t.q10, az), col_value(t.q11, az));
    const float2 x = lerp2(l, r, two(ax));
    return lerp(x.x, x.y, ay);
}
// The same of a store of pairs.
struct ColPairs {
    float2 q00, q10, q01, q11;
};
__device__ __forceinline__ ColPairs col_load_pairs(const ColVolume &V, unsigned i)
{
    const ColTaps t = col_load(V, i);
    return {t.q00, t.q10, t.q01, t.q11};
}
__device__ __forceinline__ float col_interp(const ColPairs &t, float ax, float ay, float az)
{
    const float2 y = lerp2(lerp2(t.q00, t.q10, two(ax)), lerp2(t.q01, t.q11, two(ax)), two(ay));
    return lerp(y.x, y.y, az);
}

// Fraction of a 32.32 fixed-point number from its low word: its top 23 bits
// placed behind the exponent of 1.
__device__ __forceinline__ float fixed_fraction(unsigned lo)
{
    return __uint_as_float(__funnelshift_r(lo, 0x7Fu, 9)) - 1.0f;
}

// Summed weight of the taps inside [0, h] at a coordinate g in [-1, h + 1)
// with fraction a.
__device__ __forceinline__ float col_inside(float g, float a, float h)
{
    return g < 0.0f ? a : (g > h ? 1.0f - a : 1.0f);
}
#endif

}  // namespace ctrex
