// vr_bricks.cu -- cube-level kernels: exact min/max, brick gather with ghost voxels, and the
// 16-bit brick encoding with a per-brick power-of-two scale.
//
// Bricking follows the object-space partition of Section 2.2 (each part rendered on its own);
// the ghost layer makes every trilinear stencil of a sample a brick owns local to that brick.
#include <algorithm>

#include "vr_internal.cuh"

namespace vr {
namespace {

// Monotone map of float bits to unsigned ints (so atomicMin/atomicMax order floats exactly).
__device__ __forceinline__ unsigned int f2ord(float x) {
    unsigned int b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__global__ void k_minmax(const float *__restrict__ v, long long n, unsigned int *enc) {
    unsigned int lo = 0xffffffffu, hi = 0u;
    long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        unsigned int e = f2ord(__ldg(v + i));
        lo = min(lo, e);
        hi = max(hi, e);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMin(enc, lo);
        atomicMax(enc + 1, hi);
    }
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// A brick's rows are spread over kRowCtas CTAs of 8 warps; a warp takes kRows rows at a time, its
// lanes along x, so that it has that many independent loads in flight (a row is only 130 or 258
// floats).  One row a CTA turn, as before, left half of 256 threads idle on 130-voxel rows.
constexpr int kRows = 4;

// max |v|, min and max over each brick's stored region (core + ghost, clamped to the cube):
// maxbits[b] (float bits), and range[2b], range[2b+1] (order-preserving encodings).
// Bound by HBM (each stored voxel read once).  741 MB in 130^3 bricks: 657 -> 175 us, 4.4 TB/s.
__global__ void __launch_bounds__(256)
k_brick_maxabs(const float *__restrict__ cube, int nx, int ny, int nz, const DrawBrick *__restrict__ bricks,
               unsigned int *maxbits, unsigned int *range) {
    const DrawBrick &b = bricks[blockIdx.y];
    const int x0 = max(b.org[0], 0), x1 = min(b.org[0] + b.dim[0], nx);
    const int y0 = max(b.org[1], 0), ny1 = min(b.org[1] + b.dim[1], ny) - y0;
    const int z0 = max(b.org[2], 0), nz1 = min(b.org[2] + b.dim[2], nz) - z0;
    const long long rows = (long long)ny1 * nz1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float m = 0.0f, lo = INFINITY, hi = -INFINITY;
    for (long long r = ((long long)blockIdx.x * 8 + warp) * kRows; r < rows; r += (long long)gridDim.x * 8 * kRows) {
        const float *row[kRows];
#pragma unroll
        for (int k = 0; k < kRows; ++k) {           // past the end: the last row again
            const long long q = min(r + k, rows - 1);
            const int z = (int)(q / ny1), y = (int)(q - (long long)z * ny1);
            row[k] = cube + ((long long)(z0 + z) * ny + (y0 + y)) * nx;
        }
#pragma unroll 2
        for (int x = x0 + lane; x < x1; x += 32) {
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                const float v = __ldg(row[k] + x);
                m = fmaxf(m, fabsf(v));
                lo = fminf(lo, v);
                hi = fmaxf(hi, v);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    __shared__ float s_m[8], s_lo[8], s_hi[8];
    if (lane == 0) { s_m[warp] = m; s_lo[warp] = lo; s_hi[warp] = hi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) { m = fmaxf(m, s_m[w]); lo = fminf(lo, s_lo[w]); hi = fmaxf(hi, s_hi[w]); }
        atomicMax(maxbits + blockIdx.y, __float_as_uint(m));
        atomicMin(range + 2 * blockIdx.y, f2ord(lo));
        atomicMax(range + 2 * blockIdx.y + 1, f2ord(hi));
    }
}

// ceil(log2 m) from the exact frexp decomposition; FP16 keeps 14 bits of headroom below 2^15.
__device__ __forceinline__ int scale_exponent(float m, int storage) {
    if (!(m > 0.0f)) return 0;
    int e;
    float f = frexpf(m, &e);
    int cl = (f == 0.5f) ? e - 1 : e;
    return storage == 1 ? cl - 14 : cl;
}

// v 2^-e rounded to the storage: one multiplication by a power of two in the usual range (ldexpf's
// result), ldexpf beyond it.
template <int S>
__device__ __forceinline__ auto encode(float v, int e, bool usual, float scale) {
    if constexpr (S == 0) {
        return v;
    } else {
        const float u = usual ? __fmul_rn(v, scale) : ldexpf(v, -e);
        if constexpr (S == 1) return __half_as_ushort(__float2half_rn(u));
        else return __bfloat16_as_ushort(__float2bfloat16_rn(u));
    }
}

// ATLAS 0: the pool alone.  1: also the brick's slice atlas with copies of the columns' heads (3: without, its
// own instantiation: a test of the cell in the rows' loop takes 553 us instead of 441), 2: also its pair atlas (16-bit codes
// of slices z and z + 1 in one texel), through its array's surface: one pass over the source
// instead of a pass for the pool and one per brick reading the pool back.  Bound by HBM (source
// read, pool and atlas written): 741 MB into FP16 bricks of 130^3 with atlases 770 us and 120
// packs of 8 us -> 441 us, 3.5 TB/s.  Coordinates are in range by construction; the zero boundary mode
// makes any write outside the array a no-op rather than a fault.
template <int S, int ATLAS>
__global__ void __launch_bounds__(256)
k_brick_build(const float *__restrict__ cube, int nx, int ny, int nz, const DrawBrick *__restrict__ bricks,
              const unsigned int *__restrict__ maxbits, void *pool, int *exps, const AtlasCell *__restrict__ cells) {
    const DrawBrick &b = bricks[blockIdx.y];
    int e = 0;
    if (S != 0) e = scale_exponent(__uint_as_float(maxbits[blockIdx.y]), S);
    if (S != 0 && blockIdx.x == 0 && threadIdx.x == 0) exps[blockIdx.y] = e;
    const bool usual = e >= -126 && e <= 126;
    const float scale = usual ? __int_as_float((127 - e) << 23) : 0.0f;
    const int dx = b.dim[0], dy = b.dim[1], dz = b.dim[2], ox = b.org[0];
    const long long rows = (long long)dy * dz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    using T = decltype(encode<S>(0.0f, 0, true, 0.0f));
    T *out = static_cast<T *>(pool);
    AtlasCell cell{0ull, 0, 0, 1, 0};
    if (ATLAS) cell = cells[blockIdx.y];
    for (long long r = ((long long)blockIdx.x * 8 + warp) * kRows; r < rows; r += (long long)gridDim.x * 8 * kRows) {
        const float *row[kRows], *up[kRows];
        long long dst[kRows];
        int ax[kRows], ay[kRows], twice[kRows];
#pragma unroll
        for (int k = 0; k < kRows; ++k) {           // past the end: the last row again
            const long long q = min(r + k, rows - 1);
            const int z = (int)(q / dy), y = (int)(q - (long long)z * dy);
            const int gy = clampi(b.org[1] + y, 0, ny - 1), gz = clampi(b.org[2] + z, 0, nz - 1);
            row[k] = cube + ((long long)gz * ny + gy) * nx;
            // the brick's layout decides the strides (x need not be the contiguous axis)
            dst[k] = b.data_off + (long long)y * b.str[1] + (long long)z * b.str[2];
            if (ATLAS) {
                const int c = z / cell.rows, zr = z - c * cell.rows;
                ax[k] = cell.x0 + c * dx;
                ay[k] = cell.y0 + zr * dy + y;
                twice[k] = ATLAS == 1 && zr == 0 && c > 0 ? cell.y0 + cell.rows * dy + y : -1;
            }
            if (ATLAS == 2) {                        // no tile for the last slice
                up[k] = cube + ((long long)clampi(b.org[2] + z + 1, 0, nz - 1) * ny + gy) * nx;
                if (z == dz - 1) ay[k] = -1;
            }
        }
        for (int x = lane; x < dx; x += 32) {
            const int gx = clampi(ox + x, 0, nx - 1);
            T v[kRows];
#pragma unroll
            for (int k = 0; k < kRows; ++k) v[k] = encode<S>(__ldg(row[k] + gx), e, usual, scale);
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                out[dst[k] + (long long)x * b.str[0]] = v[k];
                if constexpr (ATLAS == 1 || ATLAS == 3) {
                    surf2Dwrite<T>(v[k], (cudaSurfaceObject_t)cell.surf, (ax[k] + x) * (int)sizeof(T), ay[k], cudaBoundaryModeZero);
                    if (twice[k] >= 0)
                        surf2Dwrite<T>(v[k], (cudaSurfaceObject_t)cell.surf, (ax[k] - dx + x) * (int)sizeof(T), twice[k], cudaBoundaryModeZero);
                }
                if constexpr (ATLAS == 2) {
                    if (ay[k] >= 0)
                        surf2Dwrite<unsigned int>((unsigned int)v[k] | ((unsigned int)encode<S>(__ldg(up[k] + gx), e, usual, scale) << 16),
                                                  (cudaSurfaceObject_t)cell.surf, (ax[k] + x) * 4, ay[k], cudaBoundaryModeZero);
                }
            }
        }
    }
}

// 16-byte pieces where both ends are aligned, in strips of 4 a thread; bound by HBM.  741 MB: 218 us,
// 6.8 TB/s of reads and writes, where a 3D memory copy takes 806 us.
__global__ void __launch_bounds__(256) k_copy(const float *__restrict__ src, float *__restrict__ dst, long long n) {
    const long long t = (long long)blockIdx.x * 256 + threadIdx.x, nt = (long long)gridDim.x * 256;
    const bool al = ((reinterpret_cast<unsigned long long>(src) | reinterpret_cast<unsigned long long>(dst)) & 15) == 0;
    const long long n4 = al ? n / 4 : 0;
    const float4 *s4 = reinterpret_cast<const float4 *>(src);
    float4 *d4 = reinterpret_cast<float4 *>(dst);
    long long i = t;
    for (; i + 3 * nt < n4; i += 4 * nt) {
        const float4 a = __ldcs(s4 + i), b = __ldcs(s4 + i + nt), c = __ldcs(s4 + i + 2 * nt), d = __ldcs(s4 + i + 3 * nt);
        d4[i] = a; d4[i + nt] = b; d4[i + 2 * nt] = c; d4[i + 3 * nt] = d;
    }
    for (; i < n4; i += nt) d4[i] = s4[i];
    for (long long j = 4 * n4 + t; j < n; j += nt) dst[j] = src[j];
}

// CTAs a brick: enough of them over all bricks to fill the chip a few times, 16 to 2048 (those beyond a
// brick's rows find nothing to do).
int row_ctas(int nbricks) { return std::min(2048, std::max(16, (152 * 8 * 4 + nbricks - 1) / nbricks)); }

}  // namespace

cudaError_t launch_copy(const float *src, float *dst, long long n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_copy<<<(int)std::min<long long>((n + 4095) / 4096, 152 * 8), 256, 0, s>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_minmax(const float *v, long long n, unsigned int *enc, cudaStream_t s) {
    long long blocks = (n + 255) / 256;
    int grid = (int)(blocks < 152 * 16 ? (blocks > 0 ? blocks : 1) : 152 * 16);
    k_minmax<<<grid, 256, 0, s>>>(v, n, enc);
    return cudaGetLastError();
}

cudaError_t launch_brick_maxabs(const float *cube, int nx, int ny, int nz, const DrawBrick *bricks,
                                int nbricks, unsigned int *maxbits, unsigned int *range,
                                cudaStream_t s) {
    if (nbricks <= 0) return cudaSuccess;
    const dim3 grid(row_ctas(nbricks), nbricks);
    k_brick_maxabs<<<grid, 256, 0, s>>>(cube, nx, ny, nz, bricks, maxbits, range);
    return cudaGetLastError();
}

// Atlas placement: slice z of the x-contiguous brick is row z mod K (rows = K) of column z / K; a
// slice that heads a later column is also stored below the column before it, so the slices iz
// and iz + 1 of any sample stand one below the other.  One CTA per strip of brick rows; raw
// bits are moved (codes stay codes).  PAIR: 32-bit texels of the codes at z and z + 1, no copies.
template <typename T, bool PAIR>
struct PackSrc {
    const T *src;
    int dx, dy;
    __device__ __forceinline__ auto get(size_t row, int x) const {
        if constexpr (PAIR)
            return (unsigned int)src[row * dx + x] | ((unsigned int)src[(row + dy) * dx + x] << 16);
        else
            return src[row * dx + x];
    }
};
struct PackLinear {
    char *atlas;
    size_t pitch;
    template <typename V>
    __device__ __forceinline__ void put(V v, int col, int row) const {
        reinterpret_cast<V *>(atlas + (size_t)row * pitch)[col] = v;
    }
};
// Through a surface: coordinates are in range by construction; the zero boundary mode makes any
// write outside the array a no-op rather than a fault.
struct PackSurf {
    cudaSurfaceObject_t surf;
    template <typename V>
    __device__ __forceinline__ void put(V v, int col, int row) const {
        surf2Dwrite<V>(v, surf, col * (int)sizeof(V), row, cudaBoundaryModeZero);
    }
};
template <typename T, bool PAIR, typename Dst>
__global__ void __launch_bounds__(256) k_atlas_pack(PackSrc<T, PAIR> src, int dx, int dy, int nt, int rows, bool copies, Dst dst) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n = (long long)dy * nt;
    for (long long r = (long long)blockIdx.x * 8 + warp; r < n; r += (long long)gridDim.x * 8) {
        const int z = (int)(r / dy), y = (int)(r - (long long)z * dy);
        const int c = z / rows, zr = z - c * rows;
        const bool twice = copies && zr == 0 && c > 0;
        for (int x = lane; x < dx; x += 32) {
            const auto v = src.get((size_t)r, x);
            dst.put(v, c * dx + x, zr * dy + y);
            if (twice) dst.put(v, (c - 1) * dx + x, rows * dy + y);
        }
    }
}

template <typename T, bool PAIR, typename Dst>
static cudaError_t pack(const void *brick, int dx, int dy, int nt, int rows, bool copies, Dst dst, cudaStream_t s) {
    const long long n = (long long)dy * nt;
    if (n <= 0 || dx <= 0) return cudaSuccess;
    const int grid = (int)std::min<long long>((n + 7) / 8, 152 * 8);
    k_atlas_pack<T, PAIR, Dst><<<grid, 256, 0, s>>>(PackSrc<T, PAIR>{static_cast<const T *>(brick), dx, dy}, dx, dy, nt, rows, copies, dst);
    return cudaGetLastError();
}

cudaError_t launch_atlas_pack_surf(const void *brick, int esz, int dx, int dy, int dz, int rows, bool copies,
                                   unsigned long long surf, cudaStream_t s) {
    const PackSurf d{(cudaSurfaceObject_t)surf};
    return esz == 4 ? pack<unsigned int, false>(brick, dx, dy, dz, rows, copies, d, s)
                    : pack<unsigned short, false>(brick, dx, dy, dz, rows, copies, d, s);
}

cudaError_t launch_atlas_pack(const void *brick, int esz, int dx, int dy, int dz, int rows, bool copies, void *atlas,
                              size_t pitch, cudaStream_t s) {
    const PackLinear d{static_cast<char *>(atlas), pitch};
    return esz == 4 ? pack<unsigned int, false>(brick, dx, dy, dz, rows, copies, d, s)
                    : pack<unsigned short, false>(brick, dx, dy, dz, rows, copies, d, s);
}

cudaError_t launch_pair_pack(const void *brick, int dx, int dy, int dz, int rows, void *atlas, size_t pitch,
                             cudaStream_t s) {
    return pack<unsigned short, true>(brick, dx, dy, dz - 1, rows, false, PackLinear{static_cast<char *>(atlas), pitch}, s);
}

template <int S>
static cudaError_t build(const float *cube, int nx, int ny, int nz, const DrawBrick *bricks, int nbricks,
                         const unsigned int *maxbits, void *pool, int *exps, const AtlasCell *cells, bool pair, bool copies, cudaStream_t s) {
    const dim3 grid(row_ctas(nbricks), nbricks);
    if (!cells)
        k_brick_build<S, 0><<<grid, 256, 0, s>>>(cube, nx, ny, nz, bricks, maxbits, pool, exps, cells);
    else if (copies)
        k_brick_build<S, 1><<<grid, 256, 0, s>>>(cube, nx, ny, nz, bricks, maxbits, pool, exps, cells);
    else if (S == 0 || !pair)
        k_brick_build<S, 3><<<grid, 256, 0, s>>>(cube, nx, ny, nz, bricks, maxbits, pool, exps, cells);
    else if constexpr (S != 0)
        k_brick_build<S, 2><<<grid, 256, 0, s>>>(cube, nx, ny, nz, bricks, maxbits, pool, exps, cells);
    return cudaGetLastError();
}

cudaError_t launch_brick_build(const float *cube, int nx, int ny, int nz, const DrawBrick *bricks,
                               int nbricks, const unsigned int *maxbits, int storage, void *pool,
                               int *exps, const AtlasCell *cells, bool pair, bool copies, cudaStream_t s) {
    if (nbricks <= 0) return cudaSuccess;
    if (storage == 0) return build<0>(cube, nx, ny, nz, bricks, nbricks, maxbits, pool, exps, cells, pair, copies, s);
    if (storage == 1) return build<1>(cube, nx, ny, nz, bricks, nbricks, maxbits, pool, exps, cells, pair, copies, s);
    return build<2>(cube, nx, ny, nz, bricks, nbricks, maxbits, pool, exps, cells, pair, copies, s);
}

}  // namespace vr
