// vr_wavelet.cu -- lossy wavelet compression of a cube kept in GPU memory (Section 6: wavelet
// compression of the cube portions stored in GPU memory, with fast decompression and random
// access, to store and render larger cubes).
//
// The cube is cut into 8x8x8 blocks on a global grid (border blocks padded by repeating the
// edge voxels).  Each block is transformed by three levels of the 3D Haar average/difference
// transform, s = (a + b)/2, d = (a - b)/2 along x, then y, then z, each level on the
// previous level's averages; the 511 detail coefficients are quantised to int8 with one
// power-of-two step per subband and the average is kept in FP32.  A block is one fixed-size
// record, so any block decodes on its own (random access at block granularity).  Every
// operation is an explicit IEEE binary32 operation in a fixed order, so the codes and the
// decoded values are exact functions of the input.
//
// Record (kWaveletRecordBytes = 544 bytes):
//   [0, 512)   int8 q[x + 8 y + 64 z] in the block's pyramid layout (entry 0 unused, 0)
//   [512, 516) FP32 average of the block (the level-3 approximation)
//   [516, 537) int8 e[7 (L - 1) + (bx + 2 by + 4 bz) - 1], the step 2^e of subband (bx, by, bz)
//              of level L; -128: the subband is all zero
//   [537, 544) zero
// Coefficient (x, y, z) belongs to level L (n = 8 >> (L - 1), h = n / 2) when it lies in
// [0, n)^3 but not in [0, h)^3, to subband bx = (x >= h), by = (y >= h), bz = (z >= h).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "vr_internal.cuh"

namespace vr {
namespace {

constexpr int kWarpsPerCta = 8;

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// 2^k as a float for k in [-126, 127] (built from its bits: exact).
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }

// How a warp holds a block: lane l and gg = 0, 1 hold the 2x2x2 group (i, j, k) = (l & 3, l >> 2 & 3,
// (l >> 4) + 2 gg) of level 1, voxels (2i + a, 2j + b, 2k + c).  The eight level-1 groups of a level-2
// group differ in lane bits 0, 2 and 4, the eight level-2 groups in lane bits 1 and 3 and in gg,
// so levels 2 and 3 are butterflies between lanes and nothing but the codes passes through
// shared memory.  Each pair's operations and their order (x, then y, then z; inverse z, y, x) are
// those of passes over the whole level: the same bits.

// One butterfly of the forward transform over lane bit `bit`: the lane with the bit clear keeps the
// pair's average, the other its half difference (even minus odd).
__device__ __forceinline__ float fwd_pair(float v, int bit, int lane) {
    const float o = __shfl_xor_sync(0xffffffffu, v, bit);
    return __fmul_rn((lane & bit) ? __fsub_rn(o, v) : __fadd_rn(v, o), 0.5f);
}
// ... of the inverse: the lanes hold s and d, and get s + d and s - d.
__device__ __forceinline__ float inv_pair(float v, int bit, int lane) {
    const float o = __shfl_xor_sync(0xffffffffu, v, bit);
    return (lane & bit) ? __fsub_rn(o, v) : __fadd_rn(v, o);
}

// A group's forward transform: voxels v[a + 2b + 4c] -> average in v[0], details in v[sb].
__device__ __forceinline__ void fwd_group(float v[8]) {
#pragma unroll
    for (int ax = 1; ax < 8; ax <<= 1)
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (!(c & ax)) {
                const float x0 = v[c], x1 = v[c | ax];
                v[c] = __fmul_rn(__fadd_rn(x0, x1), 0.5f);
                v[c | ax] = __fmul_rn(__fsub_rn(x0, x1), 0.5f);
            }
}

// |x| as bits: their order is that of the values, a NaN above all (its subband gets no codes).
__device__ __forceinline__ unsigned abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }

// Exponent of a subband's step: the smallest e in [-126, 120] with m <= 127 2^e; -128 for m = 0.
__device__ __forceinline__ int step_exponent(float m) {
    if (!(m > 0.0f)) return -128;
    int k;
    frexpf(m, &k);                           // m = f 2^k, 1/2 <= f < 1
    int e = k - 7;
    if (e >= -126 && m > __fmul_rn(127.0f, pow2f(e))) e += 1;
    return clampi(e, -126, 120);
}
__device__ __forceinline__ signed char quantise(float a, float inv_step) {
    return (signed char)clampi((int)rintf(__fmul_rn(a, inv_step)), -127, 127);
}

// Encoder: one warp per block, the whole transform in registers.  Bound by HBM: 768x768x512 voxels
// (1.21 GB read, 0.32 GB written) 1.81 -> 0.37 ms; the passes through shared memory with a division
// for every coefficient's place were the time.
__global__ void __launch_bounds__(32 * kWarpsPerCta)
k_wavelet_encode(const float *__restrict__ cube, int nx, int ny, int nz, int bnx, int bny, long long nblocks,
                 unsigned char *__restrict__ store) {
    __shared__ __align__(16) signed char s_q[kWarpsPerCta][512];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long blk = (long long)blockIdx.x * kWarpsPerCta + w;
    if (blk >= nblocks) return;                      // warp-uniform; no block-wide barrier below
    const int bx = (int)(blk % bnx), by = (int)((blk / bnx) % bny), bz = (int)(blk / ((long long)bnx * bny));
    const int i = lane & 3, j = (lane >> 2) & 3, k0 = lane >> 4;
    float v[2][8];
    if (8 * bx + 8 <= nx && 8 * by + 8 <= ny && 8 * bz + 8 <= nz && !(nx & 1)) {
        const float *p = cube + ((long long)(8 * bz + 2 * k0) * ny + 8 * by + 2 * j) * nx + 8 * bx + 2 * i;
#pragma unroll
        for (int gg = 0; gg < 2; ++gg)
#pragma unroll
            for (int r = 0; r < 4; ++r) {            // rows (b, c); pairs lie on 8-byte boundaries (nx even)
                const float2 f = __ldg(reinterpret_cast<const float2 *>(p + ((long long)(4 * gg + (r >> 1)) * ny + (r & 1)) * nx));
                v[gg][2 * r] = f.x;
                v[gg][2 * r + 1] = f.y;
            }
    } else {                                         // past the cube: the edge voxels again
#pragma unroll
        for (int gg = 0; gg < 2; ++gg)
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int x = min(8 * bx + 2 * i + (c & 1), nx - 1), y = min(8 * by + 2 * j + ((c >> 1) & 1), ny - 1);
                const int z = min(8 * bz + 2 * (k0 + 2 * gg) + (c >> 2), nz - 1);
                v[gg][c] = cube[((long long)z * ny + y) * nx + x];
            }
    }
    float l2[2], l3[2];
#pragma unroll
    for (int gg = 0; gg < 2; ++gg) {
        fwd_group(v[gg]);
        l2[gg] = fwd_pair(fwd_pair(fwd_pair(v[gg][0], 1, lane), 4, lane), 16, lane);
        l3[gg] = fwd_pair(fwd_pair(l2[gg], 2, lane), 8, lane);      // means something in lanes with bits 0, 2, 4 clear
    }
    const float s3 = __fmul_rn(__fadd_rn(l3[0], l3[1]), 0.5f), d3 = __fmul_rn(__fsub_rn(l3[0], l3[1]), 0.5f);
    l3[0] = s3;                                      // subband (bit 1, bit 3, gg)
    l3[1] = d3;
    // max |c| of subband slot s (7 (L - 1) + sb - 1) in lane s
    float m = 0.0f;
#pragma unroll
    for (int sb = 1; sb < 8; ++sb) {
        const unsigned r = __reduce_max_sync(0xffffffffu, max(abs_bits(v[0][sb]), abs_bits(v[1][sb])));
        if (lane == sb - 1) m = __uint_as_float(r);
    }
    unsigned m2 = max(abs_bits(l2[0]), abs_bits(l2[1]));
    m2 = max(m2, __shfl_xor_sync(0xffffffffu, m2, 2));
    m2 = max(m2, __shfl_xor_sync(0xffffffffu, m2, 8));
    const int sb = lane < 7 ? 0 : (lane - 7) % 7 + 1;          // lanes 7..20: slots of levels 2 and 3
    const float a2 = __uint_as_float(__shfl_sync(0xffffffffu, m2, (sb & 1) + 4 * ((sb >> 1) & 1) + 16 * (sb >> 2)));
    const float a30 = __shfl_sync(0xffffffffu, l3[0], 2 * (sb & 1) + 8 * ((sb >> 1) & 1));
    const float a31 = __shfl_sync(0xffffffffu, l3[1], 2 * (sb & 1) + 8 * ((sb >> 1) & 1));
    if (lane >= 7) m = lane < 14 ? a2 : fabsf((sb >> 2) ? a31 : a30);
    const int e = step_exponent(m);
    const float inv = e == -128 ? 0.0f : pow2f(-e);
    unsigned char *rec = store + blk * kWaveletRecordBytes;
    // bytes 512..543: the average, the 21 exponents, zeros
    const float avg = __shfl_sync(0xffffffffu, l3[0], 0);
    if (lane < 28) rec[516 + lane] = lane < 21 ? (unsigned char)(signed char)e : 0;
    if (lane == 0) *reinterpret_cast<float *>(rec + 512) = avg;
    signed char *q = s_q[w];
#pragma unroll
    for (int c = 1; c < 8; ++c) {
        const float f = __shfl_sync(0xffffffffu, inv, c - 1);
#pragma unroll
        for (int gg = 0; gg < 2; ++gg)
            q[(i + 4 * (c & 1)) + 8 * (j + 4 * ((c >> 1) & 1)) + 64 * (k0 + 2 * gg + 4 * (c >> 2))] = quantise(v[gg][c], f);
    }
    const int b2 = (lane & 1) + 2 * ((lane >> 2) & 1) + 4 * (lane >> 4);     // this lane's level-2 subband
    const float f2 = __shfl_sync(0xffffffffu, inv, 6 + max(b2, 1));
    const int b3 = ((lane >> 1) & 1) + 2 * ((lane >> 3) & 1);                // and level-3 one (gg = 0; + 4: gg = 1)
    const float f30 = __shfl_sync(0xffffffffu, inv, 13 + max(b3, 1)), f31 = __shfl_sync(0xffffffffu, inv, 17 + b3);
    if (b2) {
#pragma unroll
        for (int gg = 0; gg < 2; ++gg)
            q[(i >> 1) + 2 * (b2 & 1) + 8 * ((j >> 1) + 2 * ((b2 >> 1) & 1)) + 64 * (gg + 2 * (b2 >> 2))] = quantise(l2[gg], f2);
    } else {
        q[(b3 & 1) + 8 * (b3 >> 1)] = b3 ? quantise(l3[0], f30) : 0;
        q[(b3 & 1) + 8 * (b3 >> 1) + 64] = quantise(l3[1], f31);
    }
    __syncwarp();
    reinterpret_cast<uint4 *>(rec)[lane] = reinterpret_cast<const uint4 *>(q)[lane];
}

// Inverse of one level for one 2x2x2 group: c[a + 2b + 4c] holds the coarser average (c[0]) and
// the 7 details of subbands (a, b, c); the separable inverse pairs along z, then y, then x
// touch only these 8 values, so out[x + 2y + 4z] here is bit-identical to the whole-level
// passes (same pairs, same binary32 operations, same order).
__device__ __forceinline__ void inv_group(const float c[8], float out[8]) {
    float t[8], u[8];
#pragma unroll
    for (int ab = 0; ab < 4; ++ab) {              // along z
        t[ab] = __fadd_rn(c[ab], c[ab + 4]);
        t[ab + 4] = __fsub_rn(c[ab], c[ab + 4]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {                 // along y: r = a + 4z -> index a + 4z (+ 2)
        const int i0 = (r & 1) + 4 * (r >> 1);
        u[i0] = __fadd_rn(t[i0], t[i0 + 2]);
        u[i0 + 2] = __fsub_rn(t[i0], t[i0 + 2]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {                 // along x: r = y + 2z -> index 2y + 4z (+ 1)
        const int i0 = 2 * r;
        out[i0] = __fadd_rn(u[i0], u[i0 + 1]);
        out[i0 + 1] = __fsub_rn(u[i0], u[i0 + 1]);
    }
}

// Decoder into one brick's stored region: element (x, y, z) holds global voxel clamp(org + (x, y, z)),
// either in a dx*dy*dz x-contiguous FP32 array or (SURF) in the brick's slice atlas, columns of `rows`
// slices through a surface.  One warp per cube block that the region's clamped coordinates
// touch: the inverse transform in registers, the block's 512 voxels through shared memory in
// patches of 8 x 4, written to every element that maps to them.  A brick for an atlas frame goes
// straight to its atlas (before: into the slot, then a pack read it back).  Issue-bound (the
// transform and the addressing).  768x768x512, 18 bricks of 258^3 with atlases: decode 0.61 and
// pack 0.96 ms -> 0.52 ms.
template <bool SURF>
__global__ void __launch_bounds__(32 * kWarpsPerCta)
k_wavelet_decode(const unsigned char *__restrict__ store, int nx, int ny, int nz, int bnx, int bny, const WaveletJobs jobs) {
    __shared__ __align__(16) signed char s_q[kWarpsPerCta][512];
    __shared__ __align__(16) float s_v[kWarpsPerCta][512];
    const WaveletJob &jb = jobs.job[blockIdx.y];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long t = (long long)blockIdx.x * kWarpsPerCta + w;
    const int nbx = jb.nb[0], nby = jb.nb[1];
    if (t >= (long long)nbx * nby * jb.nb[2]) return;            // warp-uniform
    const int tz = (int)(t / ((long long)nbx * nby)), tr = (int)(t - (long long)tz * nbx * nby), ty = tr / nbx;
    const int cb[3] = {jb.b0[0] + tr - ty * nbx, jb.b0[1] + ty, jb.b0[2] + tz};
    const unsigned char *rec = store + (((long long)cb[2] * bny + cb[1]) * bnx + cb[0]) * kWaveletRecordBytes;
    signed char *q = s_q[w];
    reinterpret_cast<uint4 *>(q)[lane] = __ldg(reinterpret_cast<const uint4 *>(rec) + lane);
    float step = 0.0f;                               // lane s: the step of subband slot s
    if (lane < 21) {
        const int e = (int)(signed char)rec[516 + lane];
        step = e == -128 ? 0.0f : pow2f(e);
    }
    const float avg = __ldg(reinterpret_cast<const float *>(rec + 512));
    __syncwarp();
    const int i = lane & 3, j = (lane >> 2) & 3, k0 = lane >> 4;
    const int b2 = (lane & 1) + 2 * ((lane >> 2) & 1) + 4 * (lane >> 4), b3 = ((lane >> 1) & 1) + 2 * ((lane >> 3) & 1);
    const float f2 = __shfl_sync(0xffffffffu, step, 6 + max(b2, 1));
    const float f30 = __shfl_sync(0xffffffffu, step, 13 + max(b3, 1)), f31 = __shfl_sync(0xffffffffu, step, 17 + b3);
    const float c30 = b3 ? __fmul_rn((float)q[(b3 & 1) + 8 * (b3 >> 1)], f30) : avg;
    const float c31 = __fmul_rn((float)q[(b3 & 1) + 8 * (b3 >> 1) + 64], f31);
    float a[2] = {__fadd_rn(c30, c31), __fsub_rn(c30, c31)};     // level 3: z, then y, then x
    float *sv = s_v[w];
    float f1[8];
#pragma unroll
    for (int c = 1; c < 8; ++c) f1[c] = __shfl_sync(0xffffffffu, step, c - 1);
#pragma unroll
    for (int gg = 0; gg < 2; ++gg) {
        a[gg] = inv_pair(inv_pair(a[gg], 8, lane), 2, lane);
        const float d2 = __fmul_rn((float)q[(i >> 1) + 2 * (b2 & 1) + 8 * ((j >> 1) + 2 * ((b2 >> 1) & 1)) + 64 * (gg + 2 * (b2 >> 2))], f2);
        float c[8], o[8];
        c[0] = inv_pair(inv_pair(inv_pair(b2 ? d2 : a[gg], 16, lane), 4, lane), 1, lane);
#pragma unroll
        for (int sb = 1; sb < 8; ++sb)
            c[sb] = __fmul_rn((float)q[(i + 4 * (sb & 1)) + 8 * (j + 4 * ((sb >> 1) & 1)) + 64 * (k0 + 2 * gg + 4 * (sb >> 2))], f1[sb]);
        inv_group(c, o);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            *reinterpret_cast<float2 *>(sv + 2 * i + 8 * (2 * j + (r & 1)) + 64 * (2 * (k0 + 2 * gg) + (r >> 1))) =
                make_float2(o[2 * r], o[2 * r + 1]);
    }
    __syncwarp();
    // elements whose clamped global coordinate lies in this block, per axis [lo, hi)
    int lo[3], hi[3];
    const int n[3] = {nx, ny, nz};
    bool whole = true;                               // every voxel of the block lands once, unclamped
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        // clamp(org + e, 0, n - 1) in [8 cb, 8 cb + 8)  <=>  e in [lo, hi)
        const int g0 = 8 * cb[ax], g1 = min(8 * cb[ax] + 8, n[ax]);   // voxels of the block
        int l = g0 - jb.org[ax], h = g1 - jb.org[ax];
        if (g0 == 0) l = 0;                           // elements below the cube map to voxel 0
        if (g1 == n[ax]) h = jb.dim[ax];              // elements above it map to voxel n - 1
        lo[ax] = max(l, 0);
        hi[ax] = min(h, jb.dim[ax]);
        whole = whole && hi[ax] - lo[ax] == 8 && lo[ax] == g0 - jb.org[ax] && g0 + 8 <= n[ax];
    }
    const int dx = jb.dim[0], dy = jb.dim[1];
    // slice z of the atlas: row zr of column c, and, at the head of a later column, again below the one before
    auto put_atlas = [&](int x, int y, int c, int zr, float v) {
        surf2Dwrite<float>(v, (cudaSurfaceObject_t)jb.surf, (jb.x0 + c * dx + x) * 4, jb.y0 + zr * dy + y, cudaBoundaryModeZero);
        if (jb.copies && zr == 0 && c > 0)
            surf2Dwrite<float>(v, (cudaSurfaceObject_t)jb.surf, (jb.x0 + (c - 1) * dx + x) * 4, jb.y0 + jb.rows * dy + y,
                               cudaBoundaryModeZero);
    };
    if (whole) {
        const int x = lo[0] + (lane & 7), y = lo[1] + (lane >> 3);
        if constexpr (SURF) {
            int c = lo[2] / jb.rows, zr = lo[2] - c * jb.rows;
#pragma unroll
            for (int z = 0; z < 8; ++z) {
                put_atlas(x, y, c, zr, sv[lane + 64 * z]);
                put_atlas(x, y + 4, c, zr, sv[lane + 64 * z + 32]);
                if (++zr == jb.rows) { zr = 0; ++c; }
            }
        } else {
            float *d0 = jb.dst + ((long long)lo[2] * dy + y) * dx + x;
#pragma unroll
            for (int z = 0; z < 8; ++z, d0 += (long long)dy * dx) {
                d0[0] = sv[lane + 64 * z];
                d0[4ll * dx] = sv[lane + 64 * z + 32];
            }
        }
        return;
    }
    const int ex = hi[0] - lo[0], ey = hi[1] - lo[1], ez = hi[2] - lo[2];
    if (ex <= 0 || ey <= 0 || ez <= 0) return;
    for (int e = lane; e < ex * ey * ez; e += 32) {
        const int x = lo[0] + e % ex, y = lo[1] + (e / ex) % ey, z = lo[2] + e / (ex * ey);
        const int gx = clampi(jb.org[0] + x, 0, nx - 1) - 8 * cb[0], gy = clampi(jb.org[1] + y, 0, ny - 1) - 8 * cb[1];
        const int gz = clampi(jb.org[2] + z, 0, nz - 1) - 8 * cb[2];
        const float v = sv[gx + 8 * gy + 64 * gz];
        if constexpr (SURF) {
            const int c = z / jb.rows;
            put_atlas(x, y, c, z - c * jb.rows, v);
        } else {
            jb.dst[((long long)z * dy + y) * dx + x] = v;
        }
    }
}

}  // namespace

cudaError_t launch_wavelet_encode(const float *cube, int nx, int ny, int nz, unsigned char *store,
                                  cudaStream_t s) {
    const int bnx = (nx + 7) / 8, bny = (ny + 7) / 8, bnz = (nz + 7) / 8;
    const long long nb = (long long)bnx * bny * bnz;
    if (nb <= 0) return cudaSuccess;
    const long long grid = (nb + kWarpsPerCta - 1) / kWarpsPerCta;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
    k_wavelet_encode<<<(unsigned)grid, 32 * kWarpsPerCta, 0, s>>>(cube, nx, ny, nz, bnx, bny, nb, store);
    return cudaGetLastError();
}

cudaError_t launch_wavelet_decode(const unsigned char *store, int nx, int ny, int nz, WaveletJobs &jobs, int njobs, bool surf,
                                  cudaStream_t s) {
    const int bnx = (nx + 7) / 8, bny = (ny + 7) / 8;
    const int n[3] = {nx, ny, nz};
    long long most = 0;
    for (int q = 0; q < njobs; ++q) {
        WaveletJob &jb = jobs.job[q];
        for (int a = 0; a < 3; ++a) {
            const int g0 = std::min(std::max(jb.org[a], 0), n[a] - 1);
            const int g1 = std::min(std::max(jb.org[a] + jb.dim[a] - 1, 0), n[a] - 1);
            jb.b0[a] = g0 / 8;
            jb.nb[a] = g1 / 8 - jb.b0[a] + 1;
        }
        most = std::max(most, (long long)jb.nb[0] * jb.nb[1] * jb.nb[2]);
    }
    if (most <= 0) return cudaSuccess;
    const dim3 grid((unsigned)((most + kWarpsPerCta - 1) / kWarpsPerCta), njobs);
    if (surf) k_wavelet_decode<true><<<grid, 32 * kWarpsPerCta, 0, s>>>(store, nx, ny, nz, bnx, bny, jobs);
    else k_wavelet_decode<false><<<grid, 32 * kWarpsPerCta, 0, s>>>(store, nx, ny, nz, bnx, bny, jobs);
    return cudaGetLastError();
}

}  // namespace vr
