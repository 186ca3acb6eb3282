// vr_raycast.cu -- brick ray casting (DVR and MIP) and sort-last compositing.
//
// Section 2.4: every ray inside a part's rendering rectangle is tested against the part's box;
// rays that hit are sampled between entry and exit, colours accumulated front to back, with
// early ray termination; MIP keeps the maximum sampled value.  Section 2.5: the parts'
// sub-images are blended with the associative "over" operator.
//
// Sample positions lie on the global lattice t = k*step of each ray, so which samples exist
// does not depend on the bricking.  A brick owns the lattice indices k with
// ceil(t_in/step) <= k < ceil(t_out/step), t_in/t_out from its core box's slab planes.  Those
// decisions use IEEE binary32 operations in one fixed order (the __f*_rn intrinsics are never
// contracted), identical for every brick, so neighbouring bricks split each ray's samples
// exactly, with no sample lost or counted twice.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "vr_internal.cuh"

// Tuning knobs of the ray-cast kernels (build-time): unroll factor of the linear sample loops, samples
// fetched ahead (slice atlases, pair atlases, linear rows), the CTAs of 128 threads per SM (half as many of
// 256) the register allocation must allow for DVR frames read through these and for MIP frames (0: no
// constraint), and the same for the one-pass (global termination, 256 threads) kernel and the adjoint.
#ifndef VR_SAMPLE_UNROLL
#define VR_SAMPLE_UNROLL 1
#endif
#ifndef VR_AHEAD
#define VR_AHEAD 3
#endif
#ifndef VR_AHEAD_PAIR
#define VR_AHEAD_PAIR 4
#endif
#ifndef VR_AHEAD_ROWS
#define VR_AHEAD_ROWS 2
#endif
#ifndef VR_ATLAS_MIN_BLOCKS
#define VR_ATLAS_MIN_BLOCKS 6
#endif
#ifndef VR_PAIR_MIN_BLOCKS
#define VR_PAIR_MIN_BLOCKS 5
#endif
#ifndef VR_ROWS_MIN_BLOCKS
#define VR_ROWS_MIN_BLOCKS 8
#endif
#ifndef VR_MIP_MIN_BLOCKS
#define VR_MIP_MIN_BLOCKS 0
#endif
#ifndef VR_RAYMARCH_MIN_BLOCKS
#define VR_RAYMARCH_MIN_BLOCKS 5
#endif
#ifndef VR_ADJ_MIN_BLOCKS
#define VR_ADJ_MIN_BLOCKS 5
#endif
constexpr int kSampleUnroll = VR_SAMPLE_UNROLL;

namespace vr {
namespace {

// ----------------------------------------------------------------------------------------------
// FP32 decision arithmetic: ray generation and slab clipping
// ----------------------------------------------------------------------------------------------
// Pixel (i, j)'s ray before the view rotation: the offset y = e - t of its origin from the
// view translation (y2 = 0 - t2 for both projections, so only y0, y1 vary per pixel) and its
// direction in world space.
__device__ __forceinline__ void ray_eye(const Cam &c, int i, int j, float &y0, float &y1, float d[3]) {
    float sx = __fsub_rn(__fmul_rn(__fdiv_rn(__fadd_rn((float)i, 0.5f), (float)c.W), 2.0f), 1.0f);
    float sy = __fsub_rn(1.0f, __fmul_rn(__fdiv_rn(__fadd_rn((float)j, 0.5f), (float)c.H), 2.0f));
    float e0, e1, de0, de1, de2;
    if (c.proj == 0) {
        e0 = __fmul_rn(sx, c.half_w);
        e1 = __fmul_rn(sy, c.half_h);
        de0 = 0.0f; de1 = 0.0f; de2 = -1.0f;
    } else {
        e0 = e1 = 0.0f;
        float x = __fmul_rn(sx, c.th_w), y = __fmul_rn(sy, c.th), z = -1.0f;
        float n2 = __fadd_rn(__fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y)), __fmul_rn(z, z));
        float len = __fsqrt_rn(n2);
        de0 = __fdiv_rn(x, len); de1 = __fdiv_rn(y, len); de2 = __fdiv_rn(z, len);
    }
    y0 = __fsub_rn(e0, c.t[0]);
    y1 = __fsub_rn(e1, c.t[1]);
#pragma unroll
    for (int k = 0; k < 3; ++k)     // world = R^T (eye - t)
        d[k] = __fadd_rn(__fadd_rn(__fmul_rn(c.R[k], de0), __fmul_rn(c.R[3 + k], de1)),
                         __fmul_rn(c.R[6 + k], de2));
}

// World coordinate k of the origin of a ray whose eye-space offset is (y0, y1, 0 - t2).
__device__ __forceinline__ float ray_origin(const Cam &c, int k, float y0, float y1) {
    const float y2 = __fsub_rn(0.0f, c.t[2]);
    return __fadd_rn(__fadd_rn(__fmul_rn(c.R[k], y0), __fmul_rn(c.R[3 + k], y1)), __fmul_rn(c.R[6 + k], y2));
}

__device__ __forceinline__ void ray_for_pixel(const Cam &c, int i, int j, float o[3], float d[3]) {
    float y0, y1;
    ray_eye(c, i, j, y0, y1, d);
#pragma unroll
    for (int k = 0; k < 3; ++k) o[k] = ray_origin(c, k, y0, y1);
}

// Lattice range [k0, k1) of the samples inside the half-open box [lo, hi), t >= 0.
__device__ __forceinline__ bool box_krange(const float o[3], const float d[3], const float lo[3],
                                           const float hi[3], float step, int &k0, int &k1) {
    float tin = 0.0f, tout = INFINITY;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (d[a] == 0.0f) {
            if (!(lo[a] <= o[a] && o[a] < hi[a])) return false;
        } else {
            float t0 = __fdiv_rn(__fsub_rn(lo[a], o[a]), d[a]);
            float t1 = __fdiv_rn(__fsub_rn(hi[a], o[a]), d[a]);
            float en = t0 < t1 ? t0 : t1, ex = t0 < t1 ? t1 : t0;
            if (en > tin) tin = en;
            if (ex < tout) tout = ex;
        }
    }
    if (!(tout > tin) || !(tout < INFINITY)) return false;   // no direction: no samples
    k0 = (int)ceilf(__fdiv_rn(tin, step));
    k1 = (int)ceilf(__fdiv_rn(tout, step));
    // samples are counted in floats: with a direction far shorter than 1 (a view matrix whose rows are
    // not orthonormal) more of them would never be counted to the end.  The host admits no others.
    if (k1 - k0 > (1 << 24) + 1) k1 = k0 + (1 << 24) + 1;
    return k1 > k0;
}

// Local stored coordinate of sample k along one axis, x = o + (k*step)*d - c, evaluated with
// error-free transformations (two-sum, fma residuals) and rounded once, so the anchor is
// accurate to half an ulp of a brick-local coordinate even when t is thousands of voxels.
__device__ __forceinline__ float anchor(float o, float d, float c, int k, float step) {
    float kf = (float)k;
    float th = __fmul_rn(kf, step);
    float tl = __fmaf_rn(kf, step, -th);          // k*step = th + tl exactly
    float ph = __fmul_rn(th, d);
    float pl = __fmaf_rn(th, d, -ph);             // th*d = ph + pl exactly
    float s = __fsub_rn(o, c);                    // two-sum of o and -c
    float bb = __fsub_rn(s, o);
    float sl = __fadd_rn(__fsub_rn(o, __fsub_rn(s, bb)), __fsub_rn(-c, bb));
    float r = __fadd_rn(s, ph);                   // two-sum of s and ph
    float rb = __fsub_rn(r, s);
    float rl = __fadd_rn(__fsub_rn(s, __fsub_rn(r, rb)), __fsub_rn(ph, rb));
    float lo = __fadd_rn(__fadd_rn(rl, sl), __fadd_rn(pl, __fmul_rn(tl, d)));
    return __fadd_rn(r, lo);
}

template <int S>
__device__ __forceinline__ float ldv(const void *p, int i);
template <>
__device__ __forceinline__ float ldv<0>(const void *p, int i) { return __ldg(static_cast<const float *>(p) + i); }
template <>
__device__ __forceinline__ float ldv<1>(const void *p, int i) {
    return __half2float(__ldg(static_cast<const __half *>(p) + i));
}
template <>
__device__ __forceinline__ float ldv<2>(const void *p, int i) {
    return __bfloat162float(__ldg(static_cast<const __nv_bfloat16 *>(p) + i));
}

__device__ __forceinline__ float lerp_rn(float a, float b, float f) {
    return __fadd_rn(a, __fmul_rn(f, __fsub_rn(b, a)));
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// One DVR sample: trilinear value at local stored coordinate (x, y, z), table lookup.  Every
// operation is an explicit intrinsic (no contraction), so the forward kernel and the adjoint's
// replay of a ray produce bit-identical values.
struct DvrSample {
    int ix, iy, iz;         // lower stencil corner (stored indices)
    float fx, fy, fz;       // trilinear fractions
    float u;                // unclamped table coordinate (v - vmin) / (vmax - vmin)
    int li;                 // table interval
    float lf;               // fraction inside the interval
    float4 L0, D;           // the interval's first entry and the difference to the next
    float r, g, b, a;       // interpolated colour and opacity
};

// Cell of a sample: lower stencil corner (local stored index, clamped so the 2x2x2 stencil stays
// inside the stored brick) and the trilinear fractions.
struct Cell {
    int ix, iy, iz;
    float fx, fy, fz;
};

// floor(x) as a float and as an int, for |x| < 2^22, on the FMA and integer pipes (floorf and
// float <-> int conversions issue on the narrower conversion pipe, which the per-sample work
// kept a third busy): x + 1.5 * 2^23 rounded toward -infinity lands on the float grid of
// spacing 1, exactly at floor(x) + 1.5 * 2^23, so the difference is exact and the integer sits in
// the low mantissa bits.  (For x = -0 the float floor is +0 where floorf gives -0; the fraction
// x - floor is then -0 instead of +0: the same value.)
constexpr float kFloorMagic = 12582912.0f;          // 1.5 * 2^23
constexpr int kFloorMagicBits = 0x4B400000;         // its bit pattern
__device__ __forceinline__ int floor_split(float x, float &fl) {
    const float t = __fadd_rd(x, kFloorMagic);
    fl = __fsub_rn(t, kFloorMagic);
    return __float_as_int(t) - kFloorMagicBits;
}

// Brick-local coordinates are below 2^17 in magnitude (stored bricks span at most 65536 + 2
// voxels per axis), well inside floor_split's range.
template <bool CLAMP = true>
__device__ __forceinline__ void cell_of(float x, float y, float z, int mx, int my, int mz, Cell &c) {
    float flx, fly, flz;
    const int jx = floor_split(x, flx), jy = floor_split(y, fly), jz = floor_split(z, flz);
    c.fx = __fsub_rn(x, flx); c.fy = __fsub_rn(y, fly); c.fz = __fsub_rn(z, flz);
    if (CLAMP) {
        c.ix = clampi(jx, 0, mx); c.iy = clampi(jy, 0, my); c.iz = clampi(jz, 0, mz);
    } else {                          // caller has shown every index of the segment is in range
        c.ix = jx; c.iy = jy; c.iz = jz;
    }
}

// Shared-memory slots (float4) of table entry i and of its difference to entry i + 1, n entries:
// all entries, then all differences.  16-byte strides put any 8 consecutive entries in 8
// different bank groups (interleaved pairs repeat every 4 entries: measurably more conflicts).
__device__ __forceinline__ int tab_entry(int i, int) { return i; }
__device__ __forceinline__ int tab_diff(int i, int n) { return n + i; }

// Two binary32 operations in one instruction (sm_100+: fma / add / sub on a pair of registers),
// each half rounded like the scalar one, so a value is the same whichever form computed it.
__device__ __forceinline__ float2 pair2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long x, y, r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    float2 o;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
    return o;
}

// The stencil's four xy corners (x + 2y) at the sample's z.  z is interpolated first, then x,
// then y: a gather returns the four corners of one slice, so the z step of two corners is one
// packed operation.
struct Corners {
    float c0, c1, c2, c3;
};
__device__ __forceinline__ Corners lerp_z(const float v[8], float fz) {
    return Corners{__fmaf_rn(fz, __fsub_rn(v[4], v[0]), v[0]), __fmaf_rn(fz, __fsub_rn(v[5], v[1]), v[1]),
                   __fmaf_rn(fz, __fsub_rn(v[6], v[2]), v[2]), __fmaf_rn(fz, __fsub_rn(v[7], v[3]), v[3])};
}
// The same from two gathers (texels ordered (x0,y1), (x1,y1), (x1,y0), (x0,y0)).
__device__ __forceinline__ Corners lerp_z(const float4 &g0, const float4 &g1, float fz) {
    const float2 zz = pair2(fz, fz), a = pair2(g0.x, g0.y), b = pair2(g0.z, g0.w);
    const float2 hi = __ffma2_rn(zz, sub2(pair2(g1.x, g1.y), a), a), lo = __ffma2_rn(zz, sub2(pair2(g1.z, g1.w), b), b);
    return Corners{lo.y, lo.x, hi.x, hi.y};
}

// Trilinear value from the corners at the sample's z, then the table lookup.
__device__ __forceinline__ void interp_tf(const Corners &q, const Cell &c, bool scaled, float scale,
                                          float vmin, float inv_range, float lutmax, int lmax,
                                          const float4 *s_lut, DvrSample &o) {
    o.fx = c.fx; o.fy = c.fy; o.fz = c.fz;
    const float b0 = __fmaf_rn(c.fx, __fsub_rn(q.c1, q.c0), q.c0);
    const float b1 = __fmaf_rn(c.fx, __fsub_rn(q.c3, q.c2), q.c2);
    const float val = __fmaf_rn(c.fy, __fsub_rn(b1, b0), b0);
    // (a brick's scale is a power of two: val scale is exact, and the difference rounded once)
    const float off = scaled ? __fmaf_rn(val, scale, -vmin) : __fsub_rn(val, vmin);
    o.u = __fmul_rn(off, inv_range);
    const float uc = __saturatef(o.u);          // clamp to [0, 1] (one instruction)
    // interval floor(uc lutmax) of the exact product, and the fraction with one rounding.  uc = 1
    // takes entry n - 1 with fraction 0: its stored difference is 0, so the colour is entry n - 1
    // itself and no clamp of the interval is needed
    const float t = __fmaf_rd(uc, lutmax, kFloorMagic);
    o.li = __float_as_int(t) - kFloorMagicBits;
    o.lf = __fmaf_rn(uc, lutmax, -__fsub_rn(t, kFloorMagic));
    o.L0 = s_lut[tab_entry(o.li, lmax + 2)];
    o.D = s_lut[tab_diff(o.li, lmax + 2)];
    const float2 ff = pair2(o.lf, o.lf);
    const float2 rg = __ffma2_rn(ff, pair2(o.D.x, o.D.y), pair2(o.L0.x, o.L0.y));
    const float2 ba = __ffma2_rn(ff, pair2(o.D.z, o.D.w), pair2(o.L0.z, o.L0.w));
    o.r = rg.x; o.g = rg.y; o.b = ba.x; o.a = ba.y;
}
__device__ __forceinline__ void interp_tf(const float v[8], const Cell &c, bool scaled, float scale,
                                          float vmin, float inv_range, float lutmax, int lmax,
                                          const float4 *s_lut, DvrSample &o) {
    interp_tf(lerp_z(v, c.fz), c, scaled, scale, vmin, inv_range, lutmax, lmax, s_lut, o);
}

// The table in shared memory with its differences entry i+1 - entry i: the same IEEE
// subtractions a lookup would do, made once per block instead of once per sample.
constexpr size_t table_bytes(int n) { return 2 * sizeof(float4) * (size_t)n; }
__device__ __forceinline__ void load_table(const float4 *__restrict__ lut, int n, float4 *s) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float4 a = lut[i];
        const float4 b = i + 1 < n ? lut[i + 1] : a;
        s[tab_entry(i, n)] = a;
        s[tab_diff(i, n)] = make_float4(__fsub_rn(b.x, a.x), __fsub_rn(b.y, a.y), __fsub_rn(b.z, a.z),
                                   __fsub_rn(b.w, a.w));
    }
}

// Strides of x, y, z in the stored brick (its layout: any axis may be the contiguous one).
struct Strides {
    int x, y, z;
};

// A brick's atlas (see DrawBrick::atlas): the texture, the brick's place in it plus one texel,
// its stored slice's size, and 1 / K (rounded up) and -K for its K slices a column.
struct Atlas {
    unsigned long long tex;
    float2 org, dim;
    float inv, neg;
};
__device__ __forceinline__ Atlas atlas_of(const DrawBrick &b) {
    return Atlas{b.atlas, pair2(b.at_org[0], b.at_org[1]), pair2(b.at_dim[0], b.at_dim[1]), b.at_inv, b.at_neg};
}

// Gather coordinates of the 2x2 footprint at (ix, iy) of slice iz (whole numbers as floats).  A
// gather at unnormalised (x, y) returns the texels at floor(x - 1/2) and the next one on each
// axis, ordered ((x0,y1), (x1,y1), (x1,y0), (x0,y0)); x = ix + 1 selects exactly ix.  The texels
// are returned unfiltered, so the corners are the stored values themselves.  Slice iz is row
// iz - K c of column c = floor(iz / K); the product with 1 / K rounded up is exact and rounded
// down once, so c is exact for every slice of a stored brick (at most 65538).  Every
// operation is on whole numbers below 2^24: exact, on the FMA pipe, two coordinates at a time.
__device__ __forceinline__ float2 atlas_xy(const Atlas &a, float2 ixy, float iz) {
    const float c = __fsub_rn(__fmaf_rd(iz, a.inv, kFloorMagic), kFloorMagic);
    return __ffma2_rn(pair2(c, __fmaf_rn(c, a.neg, iz)), a.dim, __fadd2_rn(ixy, a.org));
}

// A BF16 code widened to binary32 (exact: the code is the top half of the float).
__device__ __forceinline__ float bf16_value(unsigned int c) { return __uint_as_float(c << 16); }

// One slice's footprint widened to binary32: FP32 texels, FP16 ones the texture unit widens
// (exactly), or BF16 codes as 16-bit unsigned texels.
template <int S>
__device__ __forceinline__ float4 gather_slice(unsigned long long tex, float2 xy) {
    if constexpr (S != 2) return tex2Dgather<float4>(tex, xy.x, xy.y, 0);
    const uint4 g = tex2Dgather<uint4>(tex, xy.x, xy.y, 0);
    return make_float4(bf16_value(g.x), bf16_value(g.y), bf16_value(g.z), bf16_value(g.w));
}

// The footprints of slices iz and iz + 1, two gathers.  Slice iz + 1 always lies dy rows below:
// the slice that heads a column is stored again below the column before it.  (Slices side by side
// instead of below one another: FP32 frames 3.3 % slower, texture cache set conflicts.)
// WRAP: no slice is stored again, so the next one's place is its own (bricks near the gather size, which have
// no room for the copies).
template <bool WRAP>
__device__ __forceinline__ float2 next_slice_xy(const Atlas &a, float2 ixy, float iz, float2 xy) {
    return WRAP ? atlas_xy(a, ixy, __fadd_rn(iz, 1.0f)) : __fadd2_rn(xy, pair2(0.0f, a.dim.y));
}
template <int S, bool WRAP>
__device__ __forceinline__ void gather_slices(const Atlas &a, float2 ixy, float iz, float4 &g0, float4 &g1) {
    const float2 xy = atlas_xy(a, ixy, iz);
    g0 = gather_slice<S>(a.tex, xy);
    g1 = gather_slice<S>(a.tex, next_slice_xy<WRAP>(a, ixy, iz, xy));
}
// The same as the stencil v[x + 2y + 4z].
__device__ __forceinline__ void gathers_to_stencil(const float4 &g0, const float4 &g1, float v[8]) {
    v[0] = g0.w; v[1] = g0.z; v[2] = g0.x; v[3] = g0.y;
    v[4] = g1.w; v[5] = g1.z; v[6] = g1.x; v[7] = g1.y;
}

// A 16-bit code of a pair texel widened to binary32 (exact): FP16 through the half conversion,
// BF16 as the top half of the float.
template <int S>
__device__ __forceinline__ float code_value(unsigned int c) {
    if constexpr (S == 1) return __half2float(__ushort_as_half((unsigned short)c));
    else return bf16_value(c);
}

// Pair atlas (16-bit bricks): tile iz holds, in each 32-bit texel (x, y), the codes of voxel
// (x, y, iz) (low half) and (x, y, iz + 1) (high half), so one gather at slice iz's footprint
// returns all 8 stencil corners -- 16 bytes of texels per sample instead of 32, one gather
// instead of two.  Tiles are placed like the slice atlas's, one per slice but the last, none twice.
__device__ __forceinline__ uint4 gather_pair(const Atlas &a, float2 ixy, float iz) {
    const float2 xy = atlas_xy(a, ixy, iz);
    return tex2Dgather<uint4>(a.tex, xy.x, xy.y, 0);
}

// The two slices' footprints of a pair gather.
template <int S>
__device__ __forceinline__ void unpack_pair(const uint4 g, float4 &g0, float4 &g1) {
    g0 = make_float4(code_value<S>(g.x & 0xffffu), code_value<S>(g.y & 0xffffu), code_value<S>(g.z & 0xffffu),
                     code_value<S>(g.w & 0xffffu));
    g1 = make_float4(code_value<S>(g.x >> 16), code_value<S>(g.y >> 16), code_value<S>(g.z >> 16), code_value<S>(g.w >> 16));
}

// The two slices' footprints by fetch mode F.
template <int S, int F>
__device__ __forceinline__ void gather_stencil(const Atlas &a, float2 ixy, float iz, float4 &g0, float4 &g1) {
    if constexpr (F == 5) unpack_pair<S>(gather_pair(a, ixy, iz), g0, g1);
    else gather_slices<S, F == 3>(a, ixy, iz, g0, g1);
}

// Whether fetch mode F reads rows of a linear copy without clamps, and the copy's contiguous axis.
constexpr bool straight(int F) { return F >= 6; }
constexpr int row_axis(int F) { return F - 6; }

// Samples whose stencils a fragment kernel's segment loop fetches before it composites the first.
constexpr int ahead(int F) { return F == 2 || F == 3 ? VR_AHEAD : F == 5 ? VR_AHEAD_PAIR : F >= 6 ? VR_AHEAD_ROWS : 1; }

// Whether fetch mode F reads a texture (the slice atlas, 2 and 3, or the pair atlas, 5).
constexpr bool gathers(int F) { return F == 2 || F == 3 || F == 5; }

template <int S>
__device__ __forceinline__ void fetch8(const void *src, int i0, const Strides &t, float v[8]) {
    v[0] = ldv<S>(src, i0);             v[1] = ldv<S>(src, i0 + t.x);
    v[2] = ldv<S>(src, i0 + t.y);       v[3] = ldv<S>(src, i0 + t.y + t.x);
    v[4] = ldv<S>(src, i0 + t.z);       v[5] = ldv<S>(src, i0 + t.z + t.x);
    v[6] = ldv<S>(src, i0 + t.z + t.y); v[7] = ldv<S>(src, i0 + t.z + t.y + t.x);
}

// The stencil at element p of a linear copy whose axis AX is contiguous: four rows, two neighbours each
// (the second at a constant offset: 4 addresses instead of 8).
template <int S, int AX>
__device__ __forceinline__ void fetch8_rows(const void *src, int i0, const Strides &t, float v[8], unsigned planes = 3) {
    using T = std::conditional_t<S == 0, float, unsigned short>;
    const T *p = static_cast<const T *>(src) + i0;
    const int s1 = AX == 0 ? t.y : t.x, s2 = AX == 2 ? t.y : t.z;
    constexpr int a = 1 << AX, b1 = AX == 0 ? 2 : 1, b2 = AX == 2 ? 2 : 4;
    const T *q = p + s1, *r = p + s2, *w = r + s1;
    // (corners of a z-plane not in `planes` keep their values)
    auto ld = [&](const T *row, int k, int c) {
        if ((planes >> (c >> 2)) & 1) v[c] = ldv<S>(row, k);
    };
    ld(p, 0, 0);       ld(p, 1, a);
    ld(q, 0, b1);      ld(q, 1, b1 | a);
    ld(r, 0, b2);      ld(r, 1, b2 | a);
    ld(w, 0, b2 | b1); ld(w, 1, b2 | b1 | a);
}

// Disabled spectral channels hold vmin (the bottom of the table range) in place of their data:
// the stencil's two z-planes are global channels org_z + iz and + 1 (clamped at the cube
// border, like the ghost copies).  `vcode` is vmin in the brick's stored units.
__device__ __forceinline__ void mask_channels(float v[8], int iz, int org_z, int nz,
                                              const unsigned char *chmask, float vcode) {
    const int z0 = clampi(org_z + iz, 0, nz - 1), z1 = clampi(org_z + iz + 1, 0, nz - 1);
    if (!chmask[z0]) { v[0] = vcode; v[1] = vcode; v[2] = vcode; v[3] = vcode; }
    if (!chmask[z1]) { v[4] = vcode; v[5] = vcode; v[6] = vcode; v[7] = vcode; }
}

// The same from a brick's plane bits in shared memory: bit 0 of byte iz is the channel of stored plane
// iz, bit 1 that of iz + 1 (one load a sample instead of two from global memory and their clamps).
__device__ __forceinline__ void load_mask_planes(const DrawBrick &b, int nz, const unsigned char *chmask, unsigned char *s) {
    for (int i = threadIdx.x; i < b.dim[2] - 1; i += blockDim.x)
        s[i] = (chmask[clampi(b.org[2] + i, 0, nz - 1)] ? 1 : 0) | (chmask[clampi(b.org[2] + i + 1, 0, nz - 1)] ? 2 : 0);
}
__device__ __forceinline__ void mask_planes(float v[8], unsigned m, float vcode) {
    if (!(m & 1)) { v[0] = vcode; v[1] = vcode; v[2] = vcode; v[3] = vcode; }
    if (!(m & 2)) { v[4] = vcode; v[5] = vcode; v[6] = vcode; v[7] = vcode; }
}

// Which of a cell's two z-planes are on: bit 0 the lower, bit 1 the upper one.
__device__ __forceinline__ unsigned plane_bits(const FrameConsts &fc, const unsigned char *s_mask, int iz, int org_z) {
    if (s_mask) return s_mask[iz];
    return (fc.chmask[clampi(org_z + iz, 0, fc.nz - 1)] ? 1u : 0u) | (fc.chmask[clampi(org_z + iz + 1, 0, fc.nz - 1)] ? 2u : 0u);
}

// A point's cell in whole-number floats: lower corner (x, y packed) and fractions, no clamps --
// for samples whose cell is known to lie inside the stored brick.
struct CellF {
    float2 ixy;
    float iz;
    float2 fxy;
    float fz;
};
__device__ __forceinline__ CellF cell_f(float2 xy, float z) {
    CellF c;
    const float2 m = pair2(kFloorMagic, kFloorMagic);
    c.ixy = sub2(__fadd2_rd(xy, m), m);
    c.iz = __fsub_rn(__fadd_rd(z, kFloorMagic), kFloorMagic);
    c.fxy = sub2(xy, c.ixy);
    c.fz = __fsub_rn(z, c.iz);
    return c;
}
__device__ __forceinline__ int small_float_int(float f) { return __float_as_int(__fadd_rn(f, kFloorMagic)) - kFloorMagicBits; }

// Stencil cache of one ray: the 8 corner values of the previous sample's cell.  Moving to an
// adjacent cell (each index changes by at most 1) keeps the corners the two cells share and
// gathers only the others; any larger jump reloads all 8.  `need` bit c marks corner c as
// still to be gathered; shifting the values shifts their bits too.
template <int S>
__device__ __forceinline__ void fetch8_cached(const void *src, const Strides &t, const Cell &c,
                                              int &px, int &py, int &pz, float v[8]) {
    const int ddx = c.ix - px, ddy = c.iy - py, ddz = c.iz - pz;
    unsigned need = 0u;
    if (ddx < -1 || ddx > 1 || ddy < -1 || ddy > 1 || ddz < -1 || ddz > 1) {
        need = 0xffu;
    } else {
        if (ddx == 1) {
            v[0] = v[1]; v[2] = v[3]; v[4] = v[5]; v[6] = v[7];
            need = ((need >> 1) & 0x55u) | 0xaau;
        } else if (ddx == -1) {
            v[1] = v[0]; v[3] = v[2]; v[5] = v[4]; v[7] = v[6];
            need = ((need << 1) & 0xaau) | 0x55u;
        }
        if (ddy == 1) {
            v[0] = v[2]; v[1] = v[3]; v[4] = v[6]; v[5] = v[7];
            need = ((need >> 2) & 0x33u) | 0xccu;
        } else if (ddy == -1) {
            v[2] = v[0]; v[3] = v[1]; v[6] = v[4]; v[7] = v[5];
            need = ((need << 2) & 0xccu) | 0x33u;
        }
        if (ddz == 1) {
            v[0] = v[4]; v[1] = v[5]; v[2] = v[6]; v[3] = v[7];
            need = ((need >> 4) & 0x0fu) | 0xf0u;
        } else if (ddz == -1) {
            v[4] = v[0]; v[5] = v[1]; v[6] = v[2]; v[7] = v[3];
            need = ((need << 4) & 0xf0u) | 0x0fu;
        }
    }
    px = c.ix; py = c.iy; pz = c.iz;
    const int i0 = c.ix * t.x + c.iy * t.y + c.iz * t.z;
    if (need & 0x01u) v[0] = ldv<S>(src, i0);
    if (need & 0x02u) v[1] = ldv<S>(src, i0 + t.x);
    if (need & 0x04u) v[2] = ldv<S>(src, i0 + t.y);
    if (need & 0x08u) v[3] = ldv<S>(src, i0 + t.y + t.x);
    if (need & 0x10u) v[4] = ldv<S>(src, i0 + t.z);
    if (need & 0x20u) v[5] = ldv<S>(src, i0 + t.z + t.x);
    if (need & 0x40u) v[6] = ldv<S>(src, i0 + t.z + t.y);
    if (need & 0x80u) v[7] = ldv<S>(src, i0 + t.z + t.y + t.x);
}

// Front-to-back "over" of one sample into (c, T): c += T a rgb, T *= 1 - a.
__device__ __forceinline__ void over(const DvrSample &s, float &c0, float &c1, float &c2, float &T) {
    const float w = __fmul_rn(T, s.a);
    const float2 c = __ffma2_rn(pair2(w, w), pair2(s.r, s.g), pair2(c0, c1));
    c0 = c.x;
    c1 = c.y;
    c2 = __fmaf_rn(w, s.b, c2);
    T = __fmaf_rn(-T, s.a, T);                 // T (1 - a), one rounding
}

// ----------------------------------------------------------------------------------------------
// ray cast: a work item = 32x8 (or 8x32) pixels of one brick's rendering rectangle, one or two CTAs; warp = 32 pixels
// along the image axis that the brick layout follows
// ----------------------------------------------------------------------------------------------
// One brick segment of a ray: n >= 1 lattice samples from the anchor q, composited front to back
// until the segment's transmittance reaches the threshold.  Returns the samples composited.
// F: how the stencil is read (FrameConsts::fetch).  MASK: a spectral-channel mask is set (its own
// instantiation, so unmasked frames carry none of its registers or branches).
//
// Atlas bricks: two slice gathers a sample return their texels over a 32-byte-a-cycle path, which
// is busy 93 % of the time on coherent FP32 rays (81 % on sparse ones) and sets the pace; pair
// atlases and global termination are bound by issue and the gathers' latency.  The loop is
// therefore written for few instructions (65 per 32 samples; 93 with integer cells and clamps): the
// x and y halves of position, floor, fraction and atlas coordinates in packed pairs, cells as
// whole-number floats, the slices placed so that no sample tests for a column's end, z
// interpolated first (packed), the two exits one branch.  No index is clamped: the host takes this
// path only for cameras near enough that rounding cannot move a sample half a voxel (kAtlasReach).
// The stencils of AHEAD samples are fetched before the first of them is looked up, and all are looked
// up before the first is composited, so that a ray waits once for several samples (short
// launches are bound by that chain: 64-sample segments, 128^3 at 256^2, 73 -> 62 us): three with slice
// atlases at 6 CTAs of 128 threads (72 registers), four with pair atlases at 5 (72).
// 1024^2 frames at step 1, ms: integer cells -> one sample at a time -> two (pair atlas three) ahead,
// composited one by one, 4 CTAs of 256 threads -> now.  1720x1720x1024 FP32 3.54 -> 3.41 -> 3.26 ->
// 3.18, FP16 2.95 -> 2.82 -> 2.74 -> 2.73, FP16 pair atlas 2.94 -> 2.92 -> 2.56 -> 2.43;
// 768x768x512 FP32 1.36 -> 1.31 -> 1.29 -> 1.24; 256^3 at 512^2, step 0.5: 0.35 -> 0.34 -> 0.31 -> 0.30;
// 2048x2048x256 BF16 pair atlas, step 0.5: 1.07 -> 1.06 -> 0.89 -> 0.82.  FP32 1720x1720x1024 and
// 768x768x512 with two ahead at 8 CTAs 3.25 and 1.26, three at 7 3.40 and 1.31, four at 5 3.24 and
// 1.28; pair atlas (FP16 1720x1720x1024) three at 6 2.51, three at 8 2.47, four at 7 2.43 (BF16 0.83).
// Global termination (one sample at a time: two spill) 768x768x512 0.64 -> 0.59.
// With a channel mask a slice whose channel is off is not gathered at all: its texels hold vcode.
// (A band of 20 % of the channels on, FP32: 1720x1720x1024 3.37 -> 2.26 ms, 768x768x512 1.33 -> 0.97,
// with global termination and an opaque table 1.51 -> 1.13; every slice gathered before.)
template <int S, int F, bool MASK>
__device__ __forceinline__ unsigned gather_masked(const Atlas &atl, const CellF &c, const FrameConsts &fc, const unsigned char *s_mask,
                                                  int org_z, float vcode, float4 &g0, float4 &g1) {
    unsigned m = 3;
    if constexpr (MASK) {
        m = plane_bits(fc, s_mask, small_float_int(c.iz), org_z);
        g0 = g1 = make_float4(vcode, vcode, vcode, vcode);
    }
    if constexpr (MASK && F != 5) {
        const float2 xy = atlas_xy(atl, c.ixy, c.iz);
        if (m & 1) g0 = gather_slice<S>(atl.tex, xy);
        if (m & 2) g1 = gather_slice<S>(atl.tex, next_slice_xy<F == 3>(atl, c.ixy, c.iz, xy));
    } else if (m) {
        gather_stencil<S, F>(atl, c.ixy, c.iz, g0, g1);
    }
    return m;
}
template <int S, int F, bool MASK>
__device__ __forceinline__ void shade(float4 g0, float4 g1, unsigned m, const CellF &c, float scale, const FrameConsts &fc,
                                      const float4 *s_lut, float vcode, DvrSample &sm) {
    const Cell cl{0, 0, 0, c.fxy.x, c.fxy.y, c.fz};
    if (MASK && F == 5) {              // (one gather brings both slices)
        if (!(m & 1)) g0 = make_float4(vcode, vcode, vcode, vcode);
        if (!(m & 2)) g1 = make_float4(vcode, vcode, vcode, vcode);
    }
    interp_tf(lerp_z(g0, g1, c.fz), cl, S != 0, scale, fc.vmin, fc.inv_range, fc.lutmax, fc.nlut - 2, s_lut, sm);
}

template <int S, int F, bool MASK, int AHEAD>
__device__ __forceinline__ int dvr_segment_atlas(const Atlas &atl, float scale, float qx, float qy, float qz,
                                                 const float d[3], int n, const FrameConsts &fc, const float4 *s_lut,
                                                 const unsigned char *s_mask, int org_z, float vcode, float &c0, float &c1, float &c2, float &T) {
    const float nf = (float)n;            // exact: n <= 2^24 + 1, checked by the host
    const float2 q = pair2(qx, qy), dd = pair2(d[0], d[1]);
    float jf = 0.0f;
    if constexpr (AHEAD > 1) {
        // the gathers of AHEAD samples, then the samples in order (past the segment's end: its last
        // sample's again, unused)
        const float nl = __fsub_rn(nf, 1.0f);
        for (;;) {
            CellF cl[AHEAD];
            float4 g0[AHEAD], g1[AHEAD];
            unsigned m[AHEAD];
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) {
                const float tj = __fmul_rn(u ? fminf(__fadd_rn(jf, (float)u), nl) : jf, fc.step);
                cl[u] = cell_f(__ffma2_rn(pair2(tj, tj), dd, q), __fmaf_rn(tj, d[2], qz));
                m[u] = gather_masked<S, F, MASK>(atl, cl[u], fc, s_mask, org_z, vcode, g0[u], g1[u]);
            }
            DvrSample sm[AHEAD];
#pragma unroll
            for (int u = 0; u < AHEAD; ++u)
                shade<S, F, MASK>(g0[u], g1[u], m[u], cl[u], scale, fc, s_lut, vcode, sm[u]);
#pragma unroll
            for (int u = 0; u < AHEAD; ++u) {
                over(sm[u], c0, c1, c2, T);
                jf = __fadd_rn(jf, 1.0f);
                if (T <= fc.thr || !(jf < nf)) return (int)jf;
            }
        }
    } else {
        do {
            const float tj = __fmul_rn(jf, fc.step);
            const CellF cl = cell_f(__ffma2_rn(pair2(tj, tj), dd, q), __fmaf_rn(tj, d[2], qz));
            float4 g0, g1;
            const unsigned m = gather_masked<S, F, MASK>(atl, cl, fc, s_mask, org_z, vcode, g0, g1);
            DvrSample sm;
            shade<S, F, MASK>(g0, g1, m, cl, scale, fc, s_lut, vcode, sm);
            over(sm, c0, c1, c2, T);
            jf = __fadd_rn(jf, 1.0f);
        } while (!(T <= fc.thr) && jf < nf);
        return (int)jf;
    }
}

// The segment loop over rows of a linear copy, for cameras near enough that no index needs a clamp.
// Bound by the loads' latency and their L1 wavefronts.  Few instructions, as in the atlas loop; cell
// indices come straight from the bits of the rounded-down positions, and the rows' second
// neighbours are constant offsets.  768x768x512, 1024^2 orbit, aligned copies kept: 1.66 -> 1.48 ms; with
// every third channel masked (plane bits in shared memory) 333x257x190 frames of 641x479 from the
// default layout take 336 -> 299 us.  CTAs of 128 threads and lookups before compositing: 1.53 -> 1.50 ms.
// Disabled channels are not loaded: the masked 333x257x190 frames 300 -> 227 us, a band of 20 % of the channels
// of 768x768x512 from the default layout 2.34 -> 1.10 ms (the stencil cache, which loads them, before).
template <int S, int AX, bool MASK, int AHEAD>
__device__ __forceinline__ int dvr_segment_rows(const void *src, const Strides &st, float scale, float qx, float qy, float qz,
                                                const float d[3], int n, const FrameConsts &fc, const float4 *s_lut,
                                                const unsigned char *s_mask, int org_z, float vcode,
                                                float &c0, float &c1, float &c2, float &T) {
    const float nf = (float)n;            // exact: n <= 2^24 + 1, checked by the host
    const float2 q = pair2(qx, qy), dd = pair2(d[0], d[1]), mm = pair2(kFloorMagic, kFloorMagic);
    // element of a cell: its rounded-down coordinates' bits times the strides, minus the magic's share
    const unsigned bias = (unsigned)kFloorMagicBits * (unsigned)(st.x + st.y + st.z);
    const float nl = __fsub_rn(nf, 1.0f);
    float jf = 0.0f;
    for (;;) {
        float v[AHEAD][8], fx[AHEAD], fy[AHEAD], fz[AHEAD];
        int iz[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {        // (past the end: the last sample's loads again)
            const float tj = __fmul_rn(u ? fminf(__fadd_rn(jf, (float)u), nl) : jf, fc.step);
            const float2 xy = __ffma2_rn(pair2(tj, tj), dd, q);
            const float z = __fmaf_rn(tj, d[2], qz);
            const float2 t = __fadd2_rd(xy, mm);
            const float tz = __fadd_rd(z, kFloorMagic);
            const float2 f = sub2(xy, sub2(t, mm));
            fx[u] = f.x;
            fy[u] = f.y;
            fz[u] = __fsub_rn(z, __fsub_rn(tz, kFloorMagic));
            iz[u] = __float_as_int(tz) - kFloorMagicBits;
            const unsigned i0 = __float_as_uint(t.x) * (AX == 0 ? 1u : (unsigned)st.x) + __float_as_uint(t.y) * (AX == 1 ? 1u : (unsigned)st.y) +
                                __float_as_uint(tz) * (AX == 2 ? 1u : (unsigned)st.z) - bias;
            unsigned planes = 3;
            if (MASK) {                    // disabled channels are not loaded
                planes = plane_bits(fc, s_mask, iz[u], org_z);
#pragma unroll
                for (int c = 0; c < 8; ++c) v[u][c] = vcode;
            }
            fetch8_rows<S, AX>(src, (int)i0, st, v[u], planes);
        }
        DvrSample sm[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            const Cell cl{0, 0, 0, fx[u], fy[u], fz[u]};
            interp_tf(v[u], cl, S != 0, scale, fc.vmin, fc.inv_range, fc.lutmax, fc.nlut - 2, s_lut, sm[u]);
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            over(sm[u], c0, c1, c2, T);
            jf = __fadd_rn(jf, 1.0f);
            if (T <= fc.thr || !(jf < nf)) return (int)jf;
        }
    }
}

template <int S, int F, bool CLAMP, bool MASK, int AHEAD>
__device__ __forceinline__ int dvr_segment(const void *src, const Strides &st, const Atlas &atl,
                                           int mx, int my, int mz,
                                           float scale, float qx, float qy, float qz, const float d[3],
                                           int n, const FrameConsts &fc, const float4 *s_lut,
                                           const unsigned char *s_mask, int org_z, float vcode,
                                           float &c0, float &c1, float &c2, float &T) {
    if constexpr (gathers(F))
        return dvr_segment_atlas<S, F, MASK, AHEAD>(atl, scale, qx, qy, qz, d, n, fc, s_lut, s_mask, org_z, vcode, c0, c1, c2, T);
    if constexpr (straight(F))
        return dvr_segment_rows<S, row_axis(F), MASK, AHEAD>(src, st, scale, qx, qy, qz, d, n, fc, s_lut, s_mask, org_z, vcode, c0, c1, c2, T);
    const float vmin = fc.vmin, inv_range = fc.inv_range, lutmax = fc.lutmax, thr = fc.thr;
    const int lmax = fc.nlut - 2;
    int px = -4, py = -4, pz = -4;        // no cell cached yet
    float v[8];
    // the sample index as a float (exact: n <= 2^24 + 1, checked by the host)
    const float nf = (float)n;
    float jf = 0.0f;
#pragma unroll kSampleUnroll
    for (; jf < nf; jf = __fadd_rn(jf, 1.0f)) {
        const float tj = __fmul_rn(jf, fc.step);
        Cell cl;
        cell_of<CLAMP>(__fmaf_rn(tj, d[0], qx), __fmaf_rn(tj, d[1], qy), __fmaf_rn(tj, d[2], qz),
                       mx, my, mz, cl);
        if (F == 1)
            fetch8_cached<S>(src, st, cl, px, py, pz, v);
        else
            fetch8<S>(src, cl.ix * st.x + cl.iy * st.y + cl.iz * st.z, st, v);
        DvrSample sm;
        static_assert(F != 1 || !MASK);       // (a cached stencil keeps the stored values)
        if (MASK) {
            if (s_mask) mask_planes(v, s_mask[cl.iz], vcode);
            else mask_channels(v, cl.iz, org_z, fc.nz, fc.chmask, vcode);
        }
        interp_tf(v, cl, S != 0, scale, vmin, inv_range, lutmax, lmax, s_lut, sm);
        over(sm, c0, c1, c2, T);
        if (T <= thr) return (int)jf + 1;
    }
    return (int)jf;
}

// F = 1: a ray keeps the stencil corners its next cell shares with the last one (fewer loads,
// more instructions; pays off when a warp's loads scatter over many cache lines); F = 0: all
// eight corners are loaded for every sample; F = 2: two gathers from the slice atlas.
// MODE 0: DVR, one fragment (colour, transmittance) per (brick, pixel of its rectangle);
// MODE 1: MIP, one maximum per (brick, pixel).
// Pixel (rx, ry) of a work item's rectangle that lane `lane` of warp `w` (0..7) ray-casts:
// lanes 0: a warp is 32 pixels along image x (tile 32x8); 1: along image y (tile 8x32).  (Warps
// of 8x4 pixels in 2x2 quads, for texture-quad locality, measured 10 % slower.)
__device__ __forceinline__ void thread_pixel(int lanes, const TileItem &it, int w, int lane, int &rx, int &ry) {
    if (lanes == 1) {
        rx = it.tx * kRcShort + w;
        ry = it.ty * kRcLong + lane;
    } else {
        rx = it.tx * kRcLong + lane;
        ry = it.ty * kRcShort + w;
    }
}

// Threads of a ray-cast CTA.  A CTA's registers and table are held until its last ray ends, so half
// a work item (4 warps) leaves fewer of them idle than a whole one: MIP 2 - 3 % faster, atlases
// up to 11 %.  (The halves of an item on two SMs both read the lines between them: FP32 frames of sparse rays
// move 6 % more DRAM bytes, 1720x1720x256 3.46 instead of 3.26 GB, in 0.89 instead of 0.92 ms.)  The stencil cache wants the whole item: its rows share lines in L1 (2.24 ms, halves 2.35).
// (HALF below.)  DVR CTAs each hold a whole table, though, and above some hundred entries the tables of
// twice as many CTAs take the shared memory that L1 and the texture cache would have, then the warps.
// 768x768x512 at step 1, 1024^2, us with halves / whole items: slice atlas FP32 256 entries 1242 / 1303,
// 768 1305 / 1321, 1024 2014 / 1325, 4096 5815 / 3060; pair atlas BF16 768 922 / 982, 1024 1303 / 990; rows
// FP32 256 1492 / 1529, 384 1564 / 1562, 512 1687 / 1627, 1024 2940 / 1879, 4096 7519 / 4297.
constexpr int kHalfTable = 768, kHalfTableRows = 384;
template <int MODE, int F>
constexpr bool rc_halves() {
    return MODE == 1 || gathers(F) || straight(F);
}

// The 32 rays of one warp: strip `strip` (0..7) of work item `it`; writes their fragments and
// adds the warp's samples to the counters.
template <int S, int MODE, int F, bool MASK, bool HALF>
__device__ __forceinline__ void rc_strip(const FrameConsts &fc, const float4 *__restrict__ lut,
                                         DrawBrick *__restrict__ dbs, const TileItem it, int strip, int lane,
                                         const void *__restrict__ pool, void *__restrict__ frags,
                                         Counters *__restrict__ ctr, float4 *s_lut, const unsigned char *s_mask) {
    const DrawBrick &b = dbs[it.db];
    // a warp's 32 rays are adjacent pixels along the image axis the brick layout follows
    int rx, ry;
    thread_pixel(fc.lanes_y, it, strip, lane, rx, ry);
    const int rw = b.rect[2];
    const bool inrect = rx < rw && ry < b.rect[3];
    int nsamp = 0;
    float o[3], d[3];
    int k0 = 0, k1 = 0;
    bool hit = false;
    if (inrect) {
        ray_for_pixel(fc.cam, b.rect[0] + rx, b.rect[1] + ry, o, d);
        hit = box_krange(o, d, b.lo, b.hi, fc.step, k0, k1);
    }
    float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, T = 1.0f;
    if (inrect) {
        const void *src = static_cast<const char *>(pool) +
                          b.data_off * (S == 0 ? 4 : 2);
        const Strides st{b.str[0], b.str[1], b.str[2]};
        const int mx = b.dim[0] - 2, my = b.dim[1] - 2, mz = b.dim[2] - 2;
        const float scale = S == 0 ? 1.0f : ldexpf(1.0f, b.exp2);
        const Atlas atl = gathers(F) ? atlas_of(b) : Atlas{};
        if (MODE == 0) {
            if (hit) {
                const float qx = anchor(o[0], d[0], b.org_c[0], k0, fc.step);
                const float qy = anchor(o[1], d[1], b.org_c[1], k0, fc.step);
                const float qz = anchor(o[2], d[2], b.org_c[2], k0, fc.step);
                const int n = k1 - k0;
                const float vcode = S == 0 ? fc.vmin : ldexpf(fc.vmin, -b.exp2);
                // (no clamps but for far cameras: every cell is inside the stored brick, kAtlasReach)
                const int j = dvr_segment<S, F, F == 0, MASK, ahead(F)>(src, st, atl, mx, my, mz, scale, qx, qy, qz, d, n, fc,
                                                              s_lut, s_mask, b.org[2], vcode, c0, c1, c2, T);
                nsamp = j;
            }
            // the pixel's place is formed again here, so that the sample loop's registers hold only its own state
            unsigned tid;
            asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
            if constexpr (HALF) {
                unsigned cta;
                asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(cta));
                tid += cta * 128 & 255u;
            }
            int wx, wy;
            thread_pixel(fc.lanes_y, it, (int)(tid >> 5), (int)(tid & 31), wx, wy);
            static_cast<float4 *>(frags)[b.frag_off + (long long)wy * b.rect[2] + wx] = make_float4(c0, c1, c2, T);
        } else {
            float m = -INFINITY;
            if (hit) {
                for (int k = k0; k < k1; ++k) {
                    const float t = __fmul_rn((float)k, fc.step);
                    const float px = __fadd_rn(o[0], __fmul_rn(t, d[0]));
                    const float py = __fadd_rn(o[1], __fmul_rn(t, d[1]));
                    const float pz = __fadd_rn(o[2], __fmul_rn(t, d[2]));
                    const float x = __fsub_rn(px, 0.5f), y = __fsub_rn(py, 0.5f), z = __fsub_rn(pz, 0.5f);
                    // floors on the FMA and integer pipes (world coordinates are far below 2^22)
                    float flx, fly, flz;
                    const int jx = floor_split(x, flx), jy = floor_split(y, fly), jz = floor_split(z, flz);
                    const float fx = __fsub_rn(x, flx), fy = __fsub_rn(y, fly), fz = __fsub_rn(z, flz);
                    float v[8];
                    int iz;
                    if (gathers(F)) {         // cells inside the stored brick (make_consts)
                        float4 g0, g1;
                        gather_stencil<S, F>(atl, sub2(pair2(flx, fly), pair2((float)b.org[0], (float)b.org[1])),
                                             __fsub_rn(flz, (float)b.org[2]), g0, g1);
                        gathers_to_stencil(g0, g1, v);
                        iz = jz - b.org[2];
                    } else if constexpr (straight(F)) {
                        iz = jz - b.org[2];
                        fetch8_rows<S, row_axis(F)>(src, (jx - b.org[0]) * st.x + (jy - b.org[1]) * st.y + iz * st.z, st, v);
                    } else {
                        const int ix = clampi(jx - b.org[0], 0, mx);
                        const int iy = clampi(jy - b.org[1], 0, my);
                        iz = clampi(jz - b.org[2], 0, mz);
                        fetch8<S>(src, ix * st.x + iy * st.y + iz * st.z, st, v);
                    }
                    if (MASK) {
                        const float vcode = S == 0 ? fc.vmin : ldexpf(fc.vmin, -b.exp2);
                        if (s_mask) mask_planes(v, s_mask[iz], vcode);
                        else mask_channels(v, iz, b.org[2], fc.nz, fc.chmask, vcode);
                    }
                    const float c00 = lerp_rn(v[0], v[1], fx);
                    const float c10 = lerp_rn(v[2], v[3], fx);
                    const float c01 = lerp_rn(v[4], v[5], fx);
                    const float c11 = lerp_rn(v[6], v[7], fx);
                    float val = lerp_rn(lerp_rn(c00, c10, fy), lerp_rn(c01, c11, fy), fz);
                    if (S != 0) val = __fmul_rn(val, scale);
                    m = val > m ? val : m;
                }
                nsamp = k1 - k0;
            }
            static_cast<float *>(frags)[b.frag_off + (long long)ry * rw + rx] = m;
        }
    }
    const unsigned int tot = __reduce_add_sync(0xffffffffu, (unsigned int)nsamp);
    if (lane == 0 && tot > 0) {
        atomicAdd(&ctr->samples, (unsigned long long)tot);
        if (atomicExch(&dbs[it.db].sampled, 1) == 0) {
            atomicAdd(&ctr->bricks_sampled, 1ull);
            atomicAdd(&ctr->brick_bytes_sampled, (unsigned long long)b.bytes);
        }
    }
}

// CTAs per SM the registers of k_raycast<., MODE, F, ., HALF> must allow (1: no constraint beyond one):
// the fewest that the samples fetched ahead fit without spills.
template <int MODE, int F, bool HALF>
constexpr int rc_min_blocks() {
    if (MODE != 0) return VR_MIP_MIN_BLOCKS > 0 ? VR_MIP_MIN_BLOCKS : 1;
    const int halves = F == 2 || F == 3 ? VR_ATLAS_MIN_BLOCKS : F == 5 ? VR_PAIR_MIN_BLOCKS : straight(F) ? VR_ROWS_MIN_BLOCKS : 1;
    return HALF ? halves : (halves + 1) / 2;
}

template <int S, int MODE, int F, bool MASK, bool HALF>
__global__ void __launch_bounds__(HALF ? 128 : 256, rc_min_blocks<MODE, F, HALF>())
k_raycast(const FrameConsts fc, const float4 *__restrict__ lut, DrawBrick *__restrict__ dbs,
          const TileItem *__restrict__ items, const void *__restrict__ pool, void *__restrict__ frags,
          Counters *__restrict__ ctr) {
    extern __shared__ float4 s_lut[];
    constexpr int per = HALF ? 2 : 1;                     // CTAs of a work item
    const int warp = (blockIdx.x % per) * (8 / per) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const TileItem it = items[blockIdx.x / per];
    unsigned char *s_mask = nullptr;
    if (MASK && fc.mask_planes > 0) {
        s_mask = reinterpret_cast<unsigned char *>(s_lut) + (MODE == 0 ? table_bytes(fc.nlut) : 0);
        load_mask_planes(dbs[it.db], fc.nz, fc.chmask, s_mask);
    }
    if (MODE == 0) load_table(lut, fc.nlut, s_lut);
    if (MODE == 0 || MASK) __syncthreads();
    rc_strip<S, MODE, F, MASK, HALF>(fc, lut, dbs, it, warp, lane, pool, frags, ctr, s_lut, s_mask);
}

// ----------------------------------------------------------------------------------------------
// staged ray cast (fetch 4): the rays of a work item cross their brick along its march axis M (the
// view's dominant axis other than the contiguous axis L of the brick copy); the block walks that
// axis in chunks of kStageC lower-stencil indices, copies each chunk's slab of the brick -- the
// bounding box of the tile's four corner rays across the chunk, widened by the stencil and a
// margin -- into shared memory with one bulk copy per row of the padded copy, one chunk ahead
// (two stages, an mbarrier each), and samples the stencils from there.  Each ray processes its
// samples in order, stopping at a chunk's end; a stencil outside the staged slab (or a chunk
// whose slab does not fit a stage, or a ray crossing M the other way) is read from global
// memory instead, so every sample and every frame is exactly the linear path's.
// ----------------------------------------------------------------------------------------------
constexpr int kStageC = 8;              // lower-stencil indices per chunk along the march axis
constexpr int kStageFloats = 7168;      // floats per stage (28 KB)
constexpr int kStageSpin = 1 << 21;     // bound of a wait for a stage's copies (polls ~32 ns apart:
                                        // ~0.1 s, against microseconds for a slab)

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(unsigned long long *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
// Whether the phase of `bar` with parity `parity` has completed (no blocking).
__device__ __forceinline__ bool mbar_test_wait(unsigned long long *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// One row of the slab: `bytes` (a multiple of 16) from 16-byte-aligned global `src` to
// 16-byte-aligned shared `dst`, counted on `bar`.
__device__ __forceinline__ void bulk_row(float *dst, const float *src, unsigned bytes, unsigned long long *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// The slab a stage holds: stored-brick index ranges [lo, lo + n) per world axis, the floats per
// shared row (its contiguous-axis extent, a multiple of 4) and the stage's bytes (0: nothing
// staged; the chunk's stencils are read from global memory).
struct StageBox {
    int lo[3], n[3];
    int row, bytes;
};

// Element a of a three-element register array by selects (a dynamic index would put the
// array in local memory).
__device__ __forceinline__ float pick3(const float v[3], int a) { return a == 0 ? v[0] : (a == 1 ? v[1] : v[2]); }
__device__ __forceinline__ int pick3(const int v[3], int a) { return a == 0 ? v[0] : (a == 1 ? v[1] : v[2]); }

// Warp 0: the slab of chunk c (march-axis lower indices [c C, c C + C)) from the tile's four corner
// rays, and its bulk copies into stage s.  Every lane takes a corner (lane & 3); lane 0 arms the
// stage's barrier with the slab's bytes before any lane issues a row.
__device__ __forceinline__ void stage_slab(const FrameConsts &fc, const DrawBrick &b, const TileItem &it, int M,
                                           int L, int O, int c, int s, float *stage, const float *__restrict__ pool,
                                           StageBox *box, unsigned long long *bar, bool off) {
    const int lane = threadIdx.x & 31;
    // the tile's pixel range inside the rectangle
    const int tw = fc.lanes_y ? kRcShort : kRcLong, th = fc.lanes_y ? kRcLong : kRcShort;
    const int px0 = it.tx * tw, py0 = it.ty * th;
    const int px1 = min(px0 + tw, b.rect[2]) - 1, py1 = min(py0 + th, b.rect[3]) - 1;
    const int cx = (lane & 1) ? px1 : px0, cy = (lane & 2) ? py1 : py0;
    float o[3], d[3];
    ray_for_pixel(fc.cam, b.rect[0] + cx, b.rect[1] + cy, o, d);
    const int dimM = b.dim[M], dimL = b.dim[L], dimO = b.dim[O];
    const int m0 = c * kStageC;
    int lo_l = 0x7fffffff, hi_l = -0x7fffffff, lo_o = 0x7fffffff, hi_o = -0x7fffffff;
    const float oM = pick3(o, M), dM = pick3(d, M), oL = pick3(o, L), dL = pick3(d, L), oO = pick3(o, O),
                dO = pick3(d, O);
    bool ok = dM != 0.0f;
    for (int e = 0; e < 2 && ok; ++e) {
        // the plane x_M = m0 (or m0 + C) of stored coordinates: x = p - org_c
        const float v = (float)(m0 + e * kStageC) + b.org_c[M];
        const float t = (v - oM) / dM;
        ok = t >= 0.0f;
        const float xl = fmaf(t, dL, oL) - b.org_c[L], xo = fmaf(t, dO, oO) - b.org_c[O];
        const int fl = (int)floorf(xl), fo = (int)floorf(xo);
        lo_l = min(lo_l, fl); hi_l = max(hi_l, fl);
        lo_o = min(lo_o, fo); hi_o = max(hi_o, fo);
    }
#pragma unroll
    for (int sh = 1; sh < 4; sh <<= 1) {
        lo_l = min(lo_l, __shfl_xor_sync(0xffffffffu, lo_l, sh));
        hi_l = max(hi_l, __shfl_xor_sync(0xffffffffu, hi_l, sh));
        lo_o = min(lo_o, __shfl_xor_sync(0xffffffffu, lo_o, sh));
        hi_o = max(hi_o, __shfl_xor_sync(0xffffffffu, hi_o, sh));
    }
    ok = __all_sync(0xffffffffu, ok) && !off && b.pad_off >= 0 && (unsigned)m0 <= (unsigned)(dimM - 1);
    // the stencil's upper neighbour and a margin of one voxel for rounding, inside the brick;
    // the contiguous axis from a 16-byte boundary, whole 16-byte pieces, within the padded row
    const int prow = (dimL + 3) & ~3;
    int l0 = max(lo_l - 1, 0) & ~3;
    int l1 = min(hi_l + 2, dimL - 1);
    int o0 = max(lo_o - 1, 0), o1 = min(hi_o + 2, dimO - 1);
    const int nm = min(kStageC + 1, dimM - m0);
    int row = ((l1 - l0 + 1) + 3) & ~3;
    if (l0 + row > prow) row = prow - l0;
    const int no = o1 - o0 + 1;
    long long floats = (long long)nm * no * row;
    // a stencil needs two indices along every axis of the slab
    if (!ok || l1 < l0 + 1 || o1 < o0 + 1 || nm < 2 || row < 4 || floats > kStageFloats) floats = 0;
    if (lane == 0) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            box->lo[a] = a == L ? l0 : (a == O ? o0 : m0);
            box->n[a] = a == L ? row : (a == O ? no : nm);
        }
        box->row = row;
        box->bytes = (int)(floats * 4);
        if (floats > 0) mbar_expect_tx(bar, (unsigned)(floats * 4));
    }
    __syncwarp();
    if (floats == 0) return;
    const float *base = pool + b.pad_off + (long long)l0;
    const int sM = b.pad_str[M], sO = b.pad_str[O];
    for (int mi = 0; mi < nm; ++mi)
        for (int oi = lane; oi < no; oi += 32)
            bulk_row(stage + ((long long)mi * no + oi) * row,
                     base + (long long)(m0 + mi) * sM + (long long)(o0 + oi) * sO, (unsigned)(row * 4), bar);
}

template <bool MASK>
__global__ void __launch_bounds__(256, 3)
k_raycast_staged(const FrameConsts fc, const float4 *__restrict__ lut, DrawBrick *__restrict__ dbs,
                 const TileItem *__restrict__ items, const float *__restrict__ pool, float4 *__restrict__ frags,
                 Counters *__restrict__ ctr) {
    extern __shared__ float4 s_lut[];
    float *stages = reinterpret_cast<float *>(s_lut + 2 * fc.nlut);      // 2 x kStageFloats
    __shared__ __align__(8) unsigned long long s_bar[2];
    __shared__ StageBox s_box[2];
    __shared__ int s_rng[2][8];
    __shared__ int s_err;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    load_table(lut, fc.nlut, s_lut);
    if (tid == 0) {
        mbar_init(&s_bar[0]);
        mbar_init(&s_bar[1]);
        mbar_fence_init();
        s_err = 0;
    }
    const TileItem it = items[blockIdx.x];
    DrawBrick &b = dbs[it.db];
    const int L = b.pad_str[0] == 1 ? 0 : (b.pad_str[1] == 1 ? 1 : 2);
    const int M = fc.stage_m, O = 3 - L - M;
    int rx, ry;
    thread_pixel(fc.lanes_y, it, warp, lane, rx, ry);
    const int rw = b.rect[2];
    const bool inrect = rx < rw && ry < b.rect[3];
    float o[3], d[3];
    int k0 = 0, k1 = 0;
    bool hit = false;
    if (inrect) {
        ray_for_pixel(fc.cam, b.rect[0] + rx, b.rect[1] + ry, o, d);
        hit = box_krange(o, d, b.lo, b.hi, fc.step, k0, k1);
    }
    const int mx = b.dim[0] - 2, my = b.dim[1] - 2, mz = b.dim[2] - 2;
    const int mM = b.dim[M] - 2;
    float q[3] = {0.0f, 0.0f, 0.0f};
    int n = 0;
    if (hit) {
        q[0] = anchor(o[0], d[0], b.org_c[0], k0, fc.step);
        q[1] = anchor(o[1], d[1], b.org_c[1], k0, fc.step);
        q[2] = anchor(o[2], d[2], b.org_c[2], k0, fc.step);
        n = k1 - k0;
    }
    const float dM = M == 0 ? d[0] : (M == 1 ? d[1] : d[2]);
    const float qM = M == 0 ? q[0] : (M == 1 ? q[1] : q[2]);
    const bool staged = hit && (fc.stage_dir > 0 ? dM > 0.2f : dM < -0.2f) && b.pad_off >= 0;
    // chunks of the ray's first and last samples (the loop's own position arithmetic)
    int cmin = 0x7fffffff, cmax = -1;
    if (staged) {
        const float tl = __fmul_rn((float)(n - 1), fc.step);
        float fl;
        const int i0 = clampi(floor_split(qM, fl), 0, mM);
        const int i1 = clampi(floor_split(__fmaf_rn(tl, dM, qM), fl), 0, mM);
        cmin = min(i0, i1) / kStageC;
        cmax = max(i0, i1) / kStageC;
    }
    for (int sh = 16; sh > 0; sh >>= 1) {
        cmin = min(cmin, __shfl_xor_sync(0xffffffffu, cmin, sh));
        cmax = max(cmax, __shfl_xor_sync(0xffffffffu, cmax, sh));
    }
    if (lane == 0) { s_rng[0][warp] = cmin; s_rng[1][warp] = cmax; }
    __syncthreads();                    // table, barriers and the warps' chunk ranges
    cmin = s_rng[0][0]; cmax = s_rng[1][0];
#pragma unroll
    for (int w = 1; w < 8; ++w) { cmin = min(cmin, s_rng[0][w]); cmax = max(cmax, s_rng[1][w]); }

    const float *src = pool + (b.pad_off >= 0 ? b.pad_off : b.data_off);
    const Strides gst = b.pad_off >= 0 ? Strides{b.pad_str[0], b.pad_str[1], b.pad_str[2]}
                                       : Strides{b.str[0], b.str[1], b.str[2]};
    const float vmin = fc.vmin, inv_range = fc.inv_range, lutmax = fc.lutmax, thr = fc.thr;
    const int lmax = fc.nlut - 2;
    float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, T = 1.0f;
    int j = 0;
    bool done = !hit;
    if (hit && !staged) {               // every stencil of this ray from global memory
        j = dvr_segment<0, 0, true, MASK, 1>(src, gst, Atlas{0ull, 0, 0, 0}, mx, my, mz, 1.0f, q[0], q[1], q[2], d,
                                          n, fc, s_lut, nullptr, b.org[2], fc.vmin, c0, c1, c2, T);
        done = true;
    }
    if (cmax >= cmin) {
        const int nch = cmax - cmin + 1;
        const int cbeg = fc.stage_dir > 0 ? cmin : cmax;
        unsigned phases = 0u;           // bit s: the parity stage s waits for next
        if (warp == 0) stage_slab(fc, b, it, M, L, O, cbeg, 0, stages, pool, &s_box[0], &s_bar[0], false);
        __syncthreads();
        for (int i = 0; i < nch; ++i) {
            const int cs = i & 1, c = cbeg + i * fc.stage_dir;
            if (i + 1 < nch && warp == 0)
                stage_slab(fc, b, it, M, L, O, c + fc.stage_dir, cs ^ 1, stages + (cs ^ 1) * kStageFloats, pool,
                           &s_box[cs ^ 1], &s_bar[cs ^ 1], s_err != 0);
            StageBox bx = s_box[cs];
            if (bx.bytes > 0) {         // this chunk's slab has landed
                bool ok = false;
                const unsigned par = (phases >> cs) & 1u;
                for (int r = 0; r < kStageSpin && !ok; ++r) {
                    ok = mbar_test_wait(&s_bar[cs], par);
                    if (!ok) __nanosleep(32);
                }
                phases ^= 1u << cs;
                if (!ok) {
                    s_err = 1;
                    atomicOr(reinterpret_cast<unsigned int *>(&ctr->pad), 1u);
                    bx.bytes = 0;
                }
            }
            const float *stage = stages + cs * kStageFloats;
            int so[3];                  // shared-memory strides of the slab by world axis
#pragma unroll
            for (int a = 0; a < 3; ++a) so[a] = a == L ? 1 : (a == O ? bx.row : bx.row * pick3(bx.n, O));
            const int mlo = c * kStageC, mhi = mlo + kStageC;
            float jf = (float)j;
            while (staged && !done && j < n) {
                const float tj = __fmul_rn(jf, fc.step);
                Cell cl;
                cell_of<true>(__fmaf_rn(tj, d[0], q[0]), __fmaf_rn(tj, d[1], q[1]), __fmaf_rn(tj, d[2], q[2]),
                              mx, my, mz, cl);
                const int im = M == 0 ? cl.ix : (M == 1 ? cl.iy : cl.iz);
                if (fc.stage_dir > 0 ? im >= mhi : im < mlo) break;   // the next chunk's sample
                float v[8];
                const int ux = cl.ix - bx.lo[0], uy = cl.iy - bx.lo[1], uz = cl.iz - bx.lo[2];
                if (bx.bytes > 0 && ux >= 0 && ux < bx.n[0] - 1 && uy >= 0 && uy < bx.n[1] - 1 && uz >= 0 &&
                    uz < bx.n[2] - 1) {
                    const float *p = stage + ux * so[0] + uy * so[1] + uz * so[2];
                    v[0] = p[0];                  v[1] = p[so[0]];
                    v[2] = p[so[1]];              v[3] = p[so[1] + so[0]];
                    v[4] = p[so[2]];              v[5] = p[so[2] + so[0]];
                    v[6] = p[so[2] + so[1]];      v[7] = p[so[2] + so[1] + so[0]];
                } else {
                    fetch8<0>(src, cl.ix * gst.x + cl.iy * gst.y + cl.iz * gst.z, gst, v);
                }
                if (MASK) mask_channels(v, cl.iz, b.org[2], fc.nz, fc.chmask, fc.vmin);
                DvrSample sm;
                interp_tf(v, cl, false, 1.0f, vmin, inv_range, lutmax, lmax, s_lut, sm);
                over(sm, c0, c1, c2, T);
                ++j;
                jf = __fadd_rn(jf, 1.0f);
                if (T <= thr) done = true;
            }
            if (j >= n) done = true;
            __syncthreads();            // the stage is read before it is refilled
        }
    }
    if (hit && !done && j < n) {        // samples no chunk took (not expected): from global memory
        for (float jf = (float)j; j < n; ++j, jf = __fadd_rn(jf, 1.0f)) {
            const float tj = __fmul_rn(jf, fc.step);
            Cell cl;
            cell_of<true>(__fmaf_rn(tj, d[0], q[0]), __fmaf_rn(tj, d[1], q[1]), __fmaf_rn(tj, d[2], q[2]), mx, my,
                          mz, cl);
            float v[8];
            fetch8<0>(src, cl.ix * gst.x + cl.iy * gst.y + cl.iz * gst.z, gst, v);
            if (MASK) mask_channels(v, cl.iz, b.org[2], fc.nz, fc.chmask, fc.vmin);
            DvrSample sm;
            interp_tf(v, cl, false, 1.0f, vmin, inv_range, lutmax, lmax, s_lut, sm);
            over(sm, c0, c1, c2, T);
            if (T <= thr) { ++j; break; }
        }
    }
    if (inrect) frags[b.frag_off + (long long)ry * rw + rx] = make_float4(c0, c1, c2, T);
    const unsigned int tot = __reduce_add_sync(0xffffffffu, (unsigned int)(hit ? j : 0));
    if (lane == 0 && tot > 0) {
        atomicAdd(&ctr->samples, (unsigned long long)tot);
        if (atomicExch(&b.sampled, 1) == 0) {
            atomicAdd(&ctr->bricks_sampled, 1ull);
            atomicAdd(&ctr->brick_bytes_sampled, (unsigned long long)b.bytes);
        }
    }
}

// ----------------------------------------------------------------------------------------------
// global early termination (occlusion skipping): one pass, each ray walking the bricks
// ----------------------------------------------------------------------------------------------
// Lattice index at which a ray crosses the plane {axis = face}: the binary32 operations of
// box_krange, clamped to +-2^30 before the conversion (far beyond any sampled index, which the
// host keeps below 2^28).  Because a correctly rounded division by step > 0 and the ceiling are
// monotone, a brick's [k0, k1) is the max / min of these indices over its faces, so walking the
// per-axis crossings reproduces every brick's segment exactly.
__device__ __forceinline__ int face_k(float face, float o, float d, float step) {
    const float t = __fdiv_rn(__fdiv_rn(__fsub_rn(face, o), d), step);
    return (int)ceilf(fminf(fmaxf(t, -1073741824.0f), 1073741824.0f));
}

// Sample index at which the ray enters (exit = false) or leaves cell c of an axis (planes
// min(c B, n) and min((c + 1) B, n)); a ray parallel to the axis never crosses.
__device__ __forceinline__ int cell_k(int c, bool exit, float o, float d, float B, float n, float step) {
    if (d == 0.0f) return exit ? 1073741824 : -1073741824;
    const float lo = fminf((float)c * B, n), hi = fminf((float)(c + 1) * B, n);
    const bool upper = (d > 0.0f) == exit;
    return face_k(upper ? hi : lo, o, d, step);
}

// Warps of a global-termination CTA: the CTA is a 32 x kMarchWarps (kMarchWarps x 32) tile of the
// frame, one warp per row (column) of 32 rays.
#ifndef VR_MARCH_WARPS
#define VR_MARCH_WARPS 8
#endif
constexpr int kMarchWarps = VR_MARCH_WARPS;
constexpr int kMarchThreads = 32 * kMarchWarps;

// A march CTA's walk state while its rays sample a segment: one int slot per thread for
// each of the three exits, the three cells, the ray's end, the segment's end, the step bound,
// the sample count, the ray's eye-space offset (two floats) and the pixel's index.  It sits in
// shared memory after the table.
enum MarchSlot { kWkX0, kWkC0 = kWkX0 + 3, kWkK1 = kWkC0 + 3, kWkEnd, kWkGuard, kWkSamp, kWkY0, kWkY1, kWkPix,
                 kWkSlots };
constexpr size_t kMarchStashBytes = (size_t)kWkSlots * kMarchThreads * sizeof(int);

// This thread's first stash slot.  The thread index is read with a volatile move so that the
// address is formed anew at each use instead of held in a register across the sample loop.
__device__ __forceinline__ volatile int *march_stash(float4 *s_lut, int nlut) {
    unsigned tid;
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    return reinterpret_cast<volatile int *>(s_lut + table_bytes(nlut) / sizeof(float4)) + tid;
}

// One CTA = a 32x8 (8x32) pixel tile of the frame.  Each ray is clipped to the cube (and the
// render window), then walks the brick grid front to back: its segment in brick b is
// [max(k, enter), min over axes of exit), sampled with the per-brick anchor and stencil of
// the fragment kernel (bit-identical samples), compositing into one running colour and
// transmittance; it stops once the transmittance reaches the threshold after a sample (global
// early termination), so bricks behind opaque pixels cost nothing.  Bricks whose values map
// only to zero opacity are walked through without sampling (their samples add nothing).
// Registers: the sample loop runs with the registers of the fragment kernel's loop plus the
// index clamps; the walk's state rests in shared memory meanwhile (volatile stores and loads
// around each segment, so no register holds it), the origin is rebuilt from the ray's two
// eye-space offsets where a brick or a crossing needs it, and the pixel's index waits in
// shared memory for the final write.
template <int S, int F, bool MASK>
__global__ void __launch_bounds__(kMarchThreads, VR_RAYMARCH_MIN_BLOCKS * 8 / kMarchWarps)
k_raymarch(const FrameConsts fc, const float4 *__restrict__ lut, DrawBrick *__restrict__ bricks,
           const MarchGrid g, const void *__restrict__ pool, float4 *__restrict__ out,
           Counters *__restrict__ ctr) {
    extern __shared__ float4 s_lut[];
    load_table(lut, fc.nlut, s_lut);
    __syncthreads();
    int nsamp = 0;
    float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, T = 1.0f;
    float y0 = 0.0f, y1 = 0.0f, d[3] = {0.0f, 0.0f, 0.0f};
    int K0 = 0, K1 = 0;
    int c[3] = {0, 0, 0}, kx[3] = {0, 0, 0};
    bool ok = false;
    {
        const int tw = fc.lanes_y ? kMarchWarps : kRcLong;
        const int ntx = (fc.cam.W + tw - 1) / tw;
        const int tx = (int)(blockIdx.x % ntx), ty = (int)(blockIdx.x / ntx);
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int px = fc.lanes_y ? tx * kMarchWarps + w : tx * kRcLong + lane;
        const int py = fc.lanes_y ? ty * kRcLong + lane : ty * kMarchWarps + w;
        const bool inframe = px < fc.cam.W && py < fc.cam.H;
        march_stash(s_lut, fc.nlut)[kWkPix * kMarchThreads] = inframe ? py * fc.cam.W + px : -1;      // frames hold < 2^31 pixels
        if (inframe) {
            ray_eye(fc.cam, px, py, y0, y1, d);
            float o[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) o[a] = ray_origin(fc.cam, a, y0, y1);
            ok = box_krange(o, d, g.clo, g.chi, fc.step, K0, K1);
            // per axis: the cell owning sample K0 and the index where the ray leaves it
#pragma unroll
            for (int a = 0; a < 3 && ok; ++a) {
                int ca;
                if (d[a] == 0.0f) {
                    // the slab test's own comparisons: the cell with lo <= o < hi
                    ca = clampi((int)floorf(__fmul_rn(o[a], g.invB[a])), 0, g.nb[a] - 1);
                    for (int r = 0; r < g.nb[a]; ++r) {
                        if (ca > 0 && o[a] < fminf((float)ca * g.B[a], g.n[a])) --ca;
                        else if (ca < g.nb[a] - 1 && o[a] >= fminf((float)(ca + 1) * g.B[a], g.n[a])) ++ca;
                        else break;
                    }
                    c[a] = ca;
                    kx[a] = cell_k(ca, true, o[a], d[a], g.B[a], g.n[a], fc.step);
                    ok = K0 < kx[a];
                } else {
                    // an estimate of the cell of sample K0 (any rounding), then settled on the cell
                    // whose [enter, exit) holds K0 by the exact crossings (a step or two at most;
                    // the moves only go one way, so the bound is never reached)
                    const float p = __fmaf_rn(__fmul_rn((float)K0, fc.step), d[a], o[a]);
                    ca = clampi((int)floorf(__fmul_rn(p, g.invB[a])), 0, g.nb[a] - 1);
                    const int step_dir = d[a] > 0.0f ? 1 : -1;
                    int ex = 0, en = 0;
                    bool settled = false;
                    for (int r = 0; r <= g.nb[a] && !settled; ++r) {
                        ex = cell_k(ca, true, o[a], d[a], g.B[a], g.n[a], fc.step);
                        if (ex <= K0 && (unsigned)(ca + step_dir) < (unsigned)g.nb[a]) { ca += step_dir; continue; }
                        en = cell_k(ca, false, o[a], d[a], g.B[a], g.n[a], fc.step);
                        if (en > K0 && (unsigned)(ca - step_dir) < (unsigned)g.nb[a]) { ca -= step_dir; continue; }
                        settled = true;
                    }
                    c[a] = ca;
                    kx[a] = ex;
                    ok = settled && en <= K0 && K0 < ex;
                }
            }
        }
    }
    int k = K0;
    // at most one segment per brick crossed (each step leaves a cell on some axis)
    for (int guard = ok ? g.nb[0] + g.nb[1] + g.nb[2] + 1 : 0; guard > 0 && k < K1; --guard) {
        int kend = min(min(kx[0], kx[1]), min(kx[2], K1));
        const long long bi = ((long long)c[2] * g.nb[1] + c[1]) * g.nb[0] + c[0];
        if (kend > k && !bricks[bi].skip) {
            const DrawBrick &b = bricks[bi];
            const void *src = static_cast<const char *>(pool) + b.data_off * (S == 0 ? 4 : 2);
            const Strides st{b.str[0], b.str[1], b.str[2]};
            const int mx = b.dim[0] - 2, my = b.dim[1] - 2, mz = b.dim[2] - 2;
            const float scale = S == 0 ? 1.0f : ldexpf(1.0f, b.exp2);
            const Atlas atl = gathers(F) ? atlas_of(b) : Atlas{};
            const float qx = anchor(ray_origin(fc.cam, 0, y0, y1), d[0], b.org_c[0], k, fc.step);
            const float qy = anchor(ray_origin(fc.cam, 1, y0, y1), d[1], b.org_c[1], k, fc.step);
            const float qz = anchor(ray_origin(fc.cam, 2, y0, y1), d[2], b.org_c[2], k, fc.step);
            const int n = kend - k;
            const float vcode = S == 0 ? fc.vmin : ldexpf(fc.vmin, -b.exp2);
            const int org_z = b.org[2];
            volatile int *wk = march_stash(s_lut, fc.nlut);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                wk[(kWkX0 + a) * kMarchThreads] = kx[a];
                wk[(kWkC0 + a) * kMarchThreads] = c[a];
            }
            wk[kWkK1 * kMarchThreads] = K1; wk[kWkEnd * kMarchThreads] = kend; wk[kWkGuard * kMarchThreads] = guard;
            wk[kWkSamp * kMarchThreads] = nsamp;
            wk[kWkY0 * kMarchThreads] = __float_as_int(y0); wk[kWkY1 * kMarchThreads] = __float_as_int(y1);
            const int j = dvr_segment<S, F, true, MASK, 1>(src, st, atl, mx, my, mz, scale, qx, qy, qz, d, n, fc,
                                                        s_lut, nullptr, org_z, vcode, c0, c1, c2, T);
            wk = march_stash(s_lut, fc.nlut);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                kx[a] = wk[(kWkX0 + a) * kMarchThreads];
                c[a] = wk[(kWkC0 + a) * kMarchThreads];
            }
            K1 = wk[kWkK1 * kMarchThreads]; kend = wk[kWkEnd * kMarchThreads]; guard = wk[kWkGuard * kMarchThreads];
            nsamp = wk[kWkSamp * kMarchThreads] + j;
            y0 = __int_as_float(wk[kWkY0 * kMarchThreads]); y1 = __int_as_float(wk[kWkY1 * kMarchThreads]);
            DrawBrick &bw = bricks[((long long)c[2] * g.nb[1] + c[1]) * g.nb[0] + c[0]];
            if (j > 0 && bw.sampled == 0 && atomicExch(&bw.sampled, 1) == 0) {
                atomicAdd(&ctr->bricks_sampled, 1ull);
                atomicAdd(&ctr->brick_bytes_sampled, (unsigned long long)bw.bytes);
            }
            if (T <= fc.thr) break;               // the whole ray is opaque
        }
        // leave the cells whose exit is here (several at an edge or corner)
        bool out_of_grid = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (kx[a] == kend && kend < K1) {
                c[a] += d[a] > 0.0f ? 1 : -1;
                if ((unsigned)c[a] >= (unsigned)g.nb[a]) out_of_grid = true;
                else kx[a] = cell_k(c[a], true, ray_origin(fc.cam, a, y0, y1), d[a], g.B[a], g.n[a], fc.step);
            }
        }
        if (out_of_grid) break;
        k = kend;
    }
    const int pix = march_stash(s_lut, fc.nlut)[kWkPix * kMarchThreads];
    if (pix >= 0) out[pix] = make_float4(c0, c1, c2, 1.0f - T);
    const unsigned int tot = __reduce_add_sync(0xffffffffu, (unsigned int)nsamp);
    if ((threadIdx.x & 31) == 0 && tot > 0) atomicAdd(&ctr->samples, (unsigned long long)tot);
}

// ----------------------------------------------------------------------------------------------
// compositing: one CTA = one 16x16 screen tile; each pixel blends the fragments of the bricks
// binned to its tile, in the work-list's front-to-back order (Section 2.5)
// ----------------------------------------------------------------------------------------------
// Bound by latency: the list, the bricks' rectangles and the fragments are one dependent load after the
// other.  The CTA therefore reads the entries of its tile once, side by side, into shared
// memory, and each pixel has four fragments on their way at a time; its launch overlaps the end of
// the ray cast (launch_composite) and waits for it before the first fragment.  512^2 frames 9.9 -> 7.8 us,
// HIPASS-scale 1024^2 29 -> 24, and about 4 us a frame less between the two kernels.
constexpr int kCompositeEntries = 128;
template <int MODE>
__global__ void __launch_bounds__(256)
k_composite(const FrameConsts fc, const DrawBrick *__restrict__ dbs, const int *__restrict__ tile_start,
            const int *__restrict__ tile_list, const void *frags, float *__restrict__ out) {
    __shared__ int s_rect[kCompositeEntries][4];
    __shared__ long long s_off[kCompositeEntries];
    const int px = blockIdx.x * kTile + (threadIdx.x & 15);
    const int py = blockIdx.y * kTile + (threadIdx.x >> 4);
    const bool inframe = px < fc.cam.W && py < fc.cam.H;
    const int t = blockIdx.y * gridDim.x + blockIdx.x;
    const int s0 = tile_start[t], s1 = tile_start[t + 1];
    float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, T = 1.0f, m = -INFINITY;
    for (int base = s0;; base += kCompositeEntries) {
        const int n = min(kCompositeEntries, s1 - base);
        if ((int)threadIdx.x < n) {
            const DrawBrick &b = dbs[tile_list[base + threadIdx.x]];
#pragma unroll
            for (int a = 0; a < 4; ++a) s_rect[threadIdx.x][a] = b.rect[a];
            s_off[threadIdx.x] = b.frag_off;
        }
        if (base == s0) cudaGridDependencySynchronize();     // (everything read so far was uploaded before the ray cast)
        __syncthreads();
        for (int e = 0; e < n; e += 4) {
            bool in[4];
            float4 f[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = min(e + u, n - 1);
                const int rx = px - s_rect[k][0], ry = py - s_rect[k][1];
                in[u] = inframe && e + u < n && (unsigned)rx < (unsigned)s_rect[k][2] && (unsigned)ry < (unsigned)s_rect[k][3];
                if (!in[u]) continue;
                const long long fi = s_off[k] + (long long)ry * s_rect[k][2] + rx;
                if (MODE == 0) f[u] = static_cast<const float4 *>(frags)[fi];
                else f[u].x = static_cast<const float *>(frags)[fi];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (!in[u]) continue;
                if (MODE == 0) {
                    c0 = __fmaf_rn(T, f[u].x, c0);
                    c1 = __fmaf_rn(T, f[u].y, c1);
                    c2 = __fmaf_rn(T, f[u].z, c2);
                    T = __fmul_rn(T, f[u].w);      // fragment .w holds the segment's transmittance
                } else {
                    m = f[u].x > m ? f[u].x : m;
                }
            }
        }
        if (base + kCompositeEntries >= s1) break;
        __syncthreads();
    }
    if (!inframe) return;
    const long long pix = (long long)py * fc.cam.W + px;
    if (MODE == 0) reinterpret_cast<float4 *>(out)[pix] = make_float4(c0, c1, c2, fc.sub ? T : 1.0f - T);
    else out[pix] = (m == -INFINITY && !fc.sub) ? fc.vmin : m;
}

// Sort-last second stage (Section 2.5): the sub-images of sibling parts, which are consecutive
// slabs of the cube along `axis`, blended per pixel front to back.  A ray crosses the slabs in
// increasing index order when its direction along the axis is positive, in decreasing order
// when negative; with a zero component it meets one slab only, and the others' (0, T = 1) leave
// the blend unchanged whatever the order.  The direction is the ray of that pixel in the
// fragment kernel's own FP32 arithmetic.
__global__ void __launch_bounds__(256)
k_composite_parts(const FrameConsts fc, int axis, int n, const float *__restrict__ subs, int row0, int rows,
                  int final_, float *__restrict__ out) {
    const long long npx = (long long)rows * fc.cam.W;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < npx;
         i += (long long)gridDim.x * blockDim.x) {
        if (fc.mode == 0) {
            const int x = (int)(i % fc.cam.W), y = row0 + (int)(i / fc.cam.W);
            float o[3], d[3];
            ray_for_pixel(fc.cam, x, y, o, d);
            const bool down = d[axis] < 0.0f;
            float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, T = 1.0f;
            for (int j = 0; j < n; ++j) {
                const int k = down ? n - 1 - j : j;
                const float4 f = reinterpret_cast<const float4 *>(subs)[(long long)k * npx + i];
                c0 = __fmaf_rn(T, f.x, c0);
                c1 = __fmaf_rn(T, f.y, c1);
                c2 = __fmaf_rn(T, f.z, c2);
                T = __fmul_rn(T, f.w);
            }
            reinterpret_cast<float4 *>(out)[i] = make_float4(c0, c1, c2, final_ ? 1.0f - T : T);
        } else {
            float m = -INFINITY;
            for (int k = 0; k < n; ++k) {
                const float f = subs[(long long)k * npx + i];
                m = f > m ? f : m;
            }
            out[i] = (m == -INFINITY && final_) ? fc.vmin : m;
        }
    }
}

// ----------------------------------------------------------------------------------------------
// backward pass
// ----------------------------------------------------------------------------------------------
// Composite backward: per pixel, fragments b = 1..B in front-to-back order with premultiplied
// colour C_b and transmittance T_b; C = sum_b P_b C_b, P_b = prod_{b'<b} T_b', output alpha
// A = 1 - prod_b T_b.  Then dL/dC_b = P_b gC and
// dL/dT_b = P_b (gC . Crest_b) - gA P_b Trest_b, with Crest_b / Trest_b the composite of the
// fragments behind b.  Pass 1 (front to back) parks P_b in gfrag.w; pass 2 (back to front)
// accumulates Crest/Trest and writes (dL/dC_b, dL/dT_b).
__global__ void __launch_bounds__(256)
k_composite_backward(const FrameConsts fc, const DrawBrick *__restrict__ dbs,
                     const int *__restrict__ tile_start, const int *__restrict__ tile_list,
                     const float4 *__restrict__ frags, const float4 *__restrict__ gout,
                     float4 *__restrict__ gfrag) {
    const int px = blockIdx.x * kTile + (threadIdx.x & 15);
    const int py = blockIdx.y * kTile + (threadIdx.x >> 4);
    if (px >= fc.cam.W || py >= fc.cam.H) return;
    const int t = blockIdx.y * gridDim.x + blockIdx.x;
    const int s0 = tile_start[t], s1 = tile_start[t + 1];
    const float4 g = gout[(long long)py * fc.cam.W + px];
    float P = 1.0f;
    for (int e = s0; e < s1; ++e) {
        const DrawBrick &b = dbs[tile_list[e]];
        const int rx = px - b.rect[0], ry = py - b.rect[1];
        if ((unsigned)rx < (unsigned)b.rect[2] && (unsigned)ry < (unsigned)b.rect[3]) {
            const long long fi = b.frag_off + (long long)ry * b.rect[2] + rx;
            gfrag[fi].w = P;
            P = __fmul_rn(P, frags[fi].w);
        }
    }
    float r0 = 0.0f, r1 = 0.0f, r2 = 0.0f, Tr = 1.0f;   // composite of the fragments behind
    for (int e = s1 - 1; e >= s0; --e) {
        const DrawBrick &b = dbs[tile_list[e]];
        const int rx = px - b.rect[0], ry = py - b.rect[1];
        if ((unsigned)rx < (unsigned)b.rect[2] && (unsigned)ry < (unsigned)b.rect[3]) {
            const long long fi = b.frag_off + (long long)ry * b.rect[2] + rx;
            const float Pb = gfrag[fi].w;
            const float4 f = frags[fi];
            const float gT = Pb * (g.x * r0 + g.y * r1 + g.z * r2 - g.w * Tr);
            gfrag[fi] = make_float4(Pb * g.x, Pb * g.y, Pb * g.z, gT);
            r0 = fmaf(f.w, r0, f.x);
            r1 = fmaf(f.w, r1, f.y);
            r2 = fmaf(f.w, r2, f.z);
            Tr *= f.w;
        }
    }
}

// A ray's cell accumulator after one step along axis SH (up: +1): the corners of the face both
// cells share move to their place in the new cell, the new far face starts empty.
template <int SH>
__device__ __forceinline__ void shift_face(float acc[8], bool up) {
    float nacc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const bool hi = (c >> SH) & 1;
        nacc[c] = up ? (hi ? 0.0f : acc[c ^ (1 << SH)]) : (hi ? acc[c ^ (1 << SH)] : 0.0f);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = nacc[c];
}

// Adds a ray's accumulated voxel gradients of cell (cx, cy, cz) (corner c = x + 2y + 4z) to the
// cube's gradient with one atomic per corner in `mask` (ghost copies map back to their source voxel).
__device__ __forceinline__ void flush_voxels(float *__restrict__ gvox, const float acc[8], unsigned mask, int cx, int cy, int cz,
                                             const DrawBrick &b, const FrameConsts &fc) {
    const int x0 = clampi(b.org[0] + cx, 0, fc.nx - 1), x1 = clampi(b.org[0] + cx + 1, 0, fc.nx - 1);
    const int y0 = clampi(b.org[1] + cy, 0, fc.ny - 1), y1 = clampi(b.org[1] + cy + 1, 0, fc.ny - 1);
    const int z0 = clampi(b.org[2] + cz, 0, fc.nz - 1), z1 = clampi(b.org[2] + cz + 1, 0, fc.nz - 1);
    // corner (0,0,0)'s address once, the other corners as 32-bit steps from it (a step along an
    // axis is one voxel's stride, or 0 where the cube's border clamps both corners together)
    float *p = gvox + ((long long)z0 * fc.ny + y0) * fc.nx + x0;
    const int dx = x1 - x0, dy = (y1 - y0) * fc.nx;
    const long long dz = (long long)(z1 - z0) * fc.nx * fc.ny;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (((mask >> c) & 1u) && acc[c] != 0.0f)
            atomicAdd(p + ((c & 1) ? dx : 0) + ((c & 2) ? dy : 0) + ((c & 4) ? dz : 0), acc[c]);
}

// The same into corner sums (k_corner_gather): the record of xy cell (x, y) in plane z holds the
// sums of its four corners, so a cell's eight corners are two vector atomics.  Cells run from -1 (the
// ghost copy below the cube) to n - 1, planes from -1 to n.
__device__ __forceinline__ void flush_corners(float4 *__restrict__ corners, const float acc[8], int cx, int cy, int cz,
                                              const DrawBrick &b, const FrameConsts &fc) {
    const int row = fc.nx + 1, plane = row * (fc.ny + 1);
    float4 *p = corners + ((long long)(b.org[2] + cz + 1) * plane + (b.org[1] + cy + 1) * row + (b.org[0] + cx + 1));
    atomicAdd(p, make_float4(acc[0], acc[1], acc[2], acc[3]));
    atomicAdd(p + plane, make_float4(acc[4], acc[5], acc[6], acc[7]));
}

// Adjoint ray cast (FP32 bricks).  Each (brick, pixel) segment is replayed front to back with
// the forward's arithmetic; from the stored segment colour C_b and transmittance T_b the
// gradient of every sample follows without per-sample storage:
//   dL/dc_j = gC T_{j-1} a_j
//   dL/da_j = T_{j-1} [ gC.c_j - (gC.(C_b - C_{<=j}) + gT T_b) / T_j ]   (T_j = T_{j-1}(1-a_j))
//   last composited sample: dL/da_j = T_{j-1} [ gC.c_j - gT ]
// Table gradients accumulate in partial rows in L2, each of a few CTAs (two float4 atomics per sample; eight
// float atomics per sample into shared-memory copies were 13 % slower per batch, their retries of
// contended adds and the copy-out included).
// Voxel gradients accumulate per ray for the 8 corners of its current cell and are added when the
// ray leaves the cell.  VOX 0: none; 1: one float atomic per corner into the cube's gradient, a step
// into an adjacent cell keeping the shared face's 4 sums; 2: two float4 atomics into corner
// sums that k_corner_gather adds up afterwards.
// Bound by L2's atomics (about 200 G 16-byte adds a second: without the table's adds, a timing copy,
// 9.8 instead of 12.7 ms a batch of 8 views; with half of them 10.7) above the replay's gathers.  With
// one atomic per corner it was bound by instruction issue: three variants of the flush, each run
// by the few lanes that needed it, 17.8 of 32 lanes active and 1.25 G warp instructions a view
// against 27.5 and 0.64 G (1.54 and 0.90 ms).
// Small launches are bound by the chain of samples: the next sample's gathers are issued ahead (one
// 256^2 view of 64^3 with the table's gradient alone 128 -> 117 us).  CTAs of half a work item, which
// hold their registers until their longest ray ends, and no spills (5 an SM, 91 registers): 117 -> 110.
// 256^3 cube, 8 views at 512^2, step 0.5, forward frames cast again: 18.5 -> 12.0 -> 11.2 ms with both
// gradients, 9.9 -> 8.9 -> 8.1 ms with the table's alone.
// ATLAS: the replay reads the stencils from the bricks' slice atlases (the forward's texels)
// instead of the linear copy; then no index is clamped (make_consts).  WRAP: fetch mode 3.
// THREADS: CTAs of half a work item up to so many table entries, as for the ray cast.  256^3, 2 views at
// 512^2, table gradient alone, us with halves / whole items: atlas 256 entries 2030 / 2255, 1024 2350 / 2394, 2048 2710 / 2493, 4096 6095 / 3656; linear 256
// 2905 / 3000, 640 3145 / 3148, 1024 4370 / 3270, 4096 8175 / 6028.
constexpr int kHalfTableAdj = 1024, kHalfTableAdjLinear = 640;
template <bool ATLAS, int VOX, bool WRAP, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 128 ? VR_ADJ_MIN_BLOCKS : 2)
k_adjoint(const FrameConsts fc, const float4 *__restrict__ lut, const DrawBrick *__restrict__ dbs,
          const TileItem *__restrict__ items, const float *__restrict__ pool,
          const float4 *__restrict__ frags, const float4 *__restrict__ gfrag,
          float *__restrict__ glut_partial, int rows, void *__restrict__ gvox) {
    extern __shared__ float4 s_lut[];
    load_table(lut, fc.nlut, s_lut);
    __syncthreads();
    constexpr int per = 256 / THREADS;           // CTAs of a work item
    const TileItem it = items[blockIdx.x / per];
    const DrawBrick &b = dbs[it.db];
    const int warp = (blockIdx.x % per) * (8 / per) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const bool odd = lane & 1;
    // the partial row of this CTA and of those rows apart (zeroed before the launch)
    float4 *g_row = reinterpret_cast<float4 *>(glut_partial) + (long long)(blockIdx.x % rows) * 2 * fc.nlut + (odd ? 1 : 0);
    // a warp's 32 rays are adjacent pixels along the image axis the brick layout follows
    int rx, ry;
    thread_pixel(fc.lanes_y, it, warp, lane, rx, ry);
    float4 gf = make_float4(0.0f, 0.0f, 0.0f, 0.0f), fr = gf;
    float o[3] = {0.0f, 0.0f, 0.0f}, d[3] = {0.0f, 0.0f, 0.0f};
    int k0 = 0, k1 = 0;
    bool live = rx < b.rect[2] && ry < b.rect[3];
    if (live) {
        const long long fi = b.frag_off + (long long)ry * b.rect[2] + rx;
        gf = gfrag[fi];
        fr = frags[fi];
        ray_for_pixel(fc.cam, b.rect[0] + rx, b.rect[1] + ry, o, d);
        live = (gf.x != 0.0f || gf.y != 0.0f || gf.z != 0.0f || gf.w != 0.0f) && box_krange(o, d, b.lo, b.hi, fc.step, k0, k1);
    }
    const float *src = pool + b.data_off;
    const Strides st{b.str[0], b.str[1], b.str[2]};
    const int mx = b.dim[0] - 2, my = b.dim[1] - 2, mz = b.dim[2] - 2;
    const float qx = anchor(o[0], d[0], b.org_c[0], k0, fc.step);
    const float qy = anchor(o[1], d[1], b.org_c[1], k0, fc.step);
    const float qz = anchor(o[2], d[2], b.org_c[2], k0, fc.step);
    const float nf = (float)(k1 - k0);         // at most 2^24 + 1, which rounds to 2^24
    const float dxdv = __fmul_rn(fc.lutmax, fc.inv_range);
    const float grest = gf.w * fr.w;
    float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, T = 1.0f;
    // voxel gradients of the ray's current cell, added to the cube when the ray leaves it
    float acc[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    CellF cc;
    cc.ixy = pair2(-4.0f, -4.0f);
    cc.iz = -4.0f;
    const Atlas atl = ATLAS ? atlas_of(b) : Atlas{};
    float jf = 0.0f;
    // sample j's cell; atlas bricks: its gathers are issued one sample ahead (the last one's again
    // at the end), so that their latency passes under a sample's arithmetic and atomics
    auto cell_at = [&](float j) {
        const float tj = __fmul_rn(j, fc.step);
        return cell_f(__ffma2_rn(pair2(tj, tj), pair2(d[0], d[1]), pair2(qx, qy)), __fmaf_rn(tj, d[2], qz));
    };
    CellF cn = cell_at(0.0f);
    float4 n0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), n1 = n0;
    if (ATLAS && live) gather_slices<0, WRAP>(atl, cn.ixy, cn.iz, n0, n1);
    while (__any_sync(0xffffffffu, live)) {
        int li = -1;
        float4 lo = make_float4(0.0f, 0.0f, 0.0f, 0.0f), hi = lo;    // the sample's adds to entries li and li + 1
        if (live) {
            CellF cl = cn;
            const float4 g0 = n0, g1 = n1;
            jf = __fadd_rn(jf, 1.0f);
            cn = cell_at(fminf(jf, nf - 1.0f));
            if (ATLAS) {
                gather_slices<0, WRAP>(atl, cn.ixy, cn.iz, n0, n1);
            } else {                               // indices clamped to the stored brick
                cl.ixy = pair2(fminf(fmaxf(cl.ixy.x, 0.0f), (float)mx), fminf(fmaxf(cl.ixy.y, 0.0f), (float)my));
                cl.iz = fminf(fmaxf(cl.iz, 0.0f), (float)mz);
            }
            const Cell ci{0, 0, 0, cl.fxy.x, cl.fxy.y, cl.fz};
            DvrSample sm;
            if (ATLAS && !fc.chmask) {
                interp_tf(lerp_z(g0, g1, cl.fz), ci, false, 1.0f, fc.vmin, fc.inv_range, fc.lutmax, fc.nlut - 2, s_lut, sm);
            } else {
                float v[8];
                const int iz = small_float_int(cl.iz);
                if (ATLAS) {
                    gathers_to_stencil(g0, g1, v);
                } else {
                    fetch8<0>(src, small_float_int(cl.ixy.x) * st.x + small_float_int(cl.ixy.y) * st.y + iz * st.z, st, v);
                }
                if (fc.chmask) mask_channels(v, iz, b.org[2], fc.nz, fc.chmask, fc.vmin);
                interp_tf(v, ci, false, 1.0f, fc.vmin, fc.inv_range, fc.lutmax, fc.nlut - 2, s_lut, sm);
            }
            const float Tb = T;
            over(sm, c0, c1, c2, T);
            const bool last = (T <= fc.thr) || !(jf < nf);
            const float gcdot = gf.x * sm.r + gf.y * sm.g + gf.z * sm.b;
            float ga;
            if (last) {
                ga = Tb * (gcdot - gf.w);
            } else {
                const float sdot = gf.x * (fr.x - c0) + gf.y * (fr.y - c1) + gf.z * (fr.z - c2);
                ga = Tb * (gcdot - (sdot + grest) / T);
            }
            const float wa = Tb * sm.a;
            const float gr = gf.x * wa, gg = gf.y * wa, gb = gf.z * wa;
            const float w1 = sm.lf, w0 = 1.0f - sm.lf;
            li = sm.li;
            lo = make_float4(w0 * gr, w0 * gg, w0 * gb, w0 * ga);
            hi = make_float4(w1 * gr, w1 * gg, w1 * gb, w1 * ga);
            if (VOX && sm.u > 0.0f && sm.u < 1.0f) {
                const float gx = gr * sm.D.x + gg * sm.D.y + gb * sm.D.z + ga * sm.D.w;
                const float gv = gx * dxdv;
                if (cl.ixy.x != cc.ixy.x || cl.ixy.y != cc.ixy.y || cl.iz != cc.iz) {
                    bool fresh = true;
                    if (cc.iz >= 0.0f) {
                        const int cx = small_float_int(cc.ixy.x), cy = small_float_int(cc.ixy.y), cz = small_float_int(cc.iz);
                        if (VOX == 2) {
                            flush_corners(static_cast<float4 *>(gvox), acc, cx, cy, cz, b, fc);
                        } else {
                            const float sx = cl.ixy.x - cc.ixy.x, sy = cl.ixy.y - cc.ixy.y, sz = cl.iz - cc.iz;
                            if (fabsf(sx) + fabsf(sy) + fabsf(sz) == 1.0f) {
                                // one step along one axis: the face both cells share keeps accumulating
                                const bool up = sx + sy + sz > 0.0f;
                                const unsigned lowf = sx != 0.0f ? 0x55u : (sy != 0.0f ? 0x33u : 0x0Fu);
                                flush_voxels(static_cast<float *>(gvox), acc, up ? lowf : (~lowf & 0xffu), cx, cy, cz, b, fc);
                                if (sx != 0.0f) shift_face<0>(acc, up);
                                else if (sy != 0.0f) shift_face<1>(acc, up);
                                else shift_face<2>(acc, up);
                                fresh = false;
                            } else {
                                flush_voxels(static_cast<float *>(gvox), acc, 0xffu, cx, cy, cz, b, fc);
                            }
                        }
                    }
                    if (fresh)
#pragma unroll
                        for (int c = 0; c < 8; ++c) acc[c] = 0.0f;
                    cc.ixy = cl.ixy;
                    cc.iz = cl.iz;
                }
                const float ux = sm.fx, uy = sm.fy;
                const float vx = 1.0f - ux, vy = 1.0f - uy;
                float uz = sm.fz, vz = 1.0f - sm.fz;
                if (fc.chmask) {
                    const int gz = b.org[2] + small_float_int(cl.iz);
                    if (!fc.chmask[clampi(gz + 1, 0, fc.nz - 1)]) uz = 0.0f;
                    if (!fc.chmask[clampi(gz, 0, fc.nz - 1)]) vz = 0.0f;
                }
                // trilinear weights of the 8 corners, factored by z, then y
                const float wz0 = gv * vz, wz1 = gv * uz;
                const float g00 = wz0 * vy, g10 = wz0 * uy, g01 = wz1 * vy, g11 = wz1 * uy;
                acc[0] = __fmaf_rn(g00, vx, acc[0]); acc[1] = __fmaf_rn(g00, ux, acc[1]);
                acc[2] = __fmaf_rn(g10, vx, acc[2]); acc[3] = __fmaf_rn(g10, ux, acc[3]);
                acc[4] = __fmaf_rn(g01, vx, acc[4]); acc[5] = __fmaf_rn(g01, ux, acc[5]);
                acc[6] = __fmaf_rn(g11, vx, acc[6]); acc[7] = __fmaf_rn(g11, ux, acc[7]);
            }
            live = !last;
        }
        // Table gradient: the record of an interval is 32 bytes, its adds to the lower entry and to the
        // upper one.  Two lanes add one sample's record together (even lanes the lower halves, odd
        // lanes the upper ones), so that a sample is one 32-byte request to L2 instead of two of 16.
        const float4 keep = odd ? hi : lo, send = odd ? lo : hi;
        const int lp = __shfl_xor_sync(0xffffffffu, li, 1);
        const float4 recv = make_float4(__shfl_xor_sync(0xffffffffu, send.x, 1), __shfl_xor_sync(0xffffffffu, send.y, 1),
                                        __shfl_xor_sync(0xffffffffu, send.z, 1), __shfl_xor_sync(0xffffffffu, send.w, 1));
        const int l1 = odd ? lp : li, l2 = odd ? li : lp;
        if (l1 >= 0) atomicAdd(g_row + 2 * l1, odd ? recv : keep);
        if (l2 >= 0) atomicAdd(g_row + 2 * l2, odd ? keep : recv);
    }
    if (VOX && cc.iz >= 0.0f) {
        const int cx = small_float_int(cc.ixy.x), cy = small_float_int(cc.ixy.y), cz = small_float_int(cc.iz);
        if (VOX == 2) flush_corners(static_cast<float4 *>(gvox), acc, cx, cy, cz, b, fc);
        else flush_voxels(static_cast<float *>(gvox), acc, 0xffu, cx, cy, cz, b, fc);
    }
}

// Corner sums -> voxel gradients: voxel (x, y, z) is the low corner of cell x, the high corner of cell
// x - 1 and, at the cube's border, the corner that the ghost copy beyond it stands for; likewise
// along y and z.  Bound by HBM: 16 B of sums read per voxel, the gradient read and written.
__global__ void __launch_bounds__(256)
k_corner_gather(const float4 *__restrict__ corners, int nx, int ny, int nz, float *__restrict__ gvox) {
    const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (x >= nx || y >= ny) return;
    const int row = nx + 1;
    const long long plane = (long long)row * (ny + 1);
    // the xy sums of a plane of corners at (x, y)
    auto xy_sum = [&](int p) {
        const float4 *q = corners + p * plane + (long long)y * row + x;    // record (x, y) is cell (x - 1, y - 1)
        float s = q[row + 1].x + q[row].y + q[1].z + q[0].w;
        // beyond the border: the ghost cell's far corner is this voxel too
        if (x == 0) s += q[row].x + q[0].z;
        if (x == nx - 1) s += q[row + 1].y + q[1].w;
        if (y == 0) s += q[1].x + q[0].y;
        if (y == ny - 1) s += q[row + 1].z + q[row].w;
        if (x == 0 && y == 0) s += q[0].x;
        if (x == nx - 1 && y == 0) s += q[1].y;
        if (x == 0 && y == ny - 1) s += q[row].z;
        if (x == nx - 1 && y == ny - 1) s += q[row + 1].w;
        return s;
    };
    for (int z = blockIdx.z; z < nz; z += gridDim.z) {
        float s = xy_sum(z + 1);
        if (z == 0) s += xy_sum(0);
        if (z == nz - 1) s += xy_sum(nz + 1);
        if (s != 0.0f) gvox[((long long)z * ny + y) * nx + x] += s;
    }
}

// Final reduction of the table-gradient partials, in FP64 and in two stages so that
// every entry's sum is spread over many threads yet formed in a fixed order: chunk y sums the
// partials of parts [y q, (y + 1) q) in part order, then the chunk sums are added in chunk order.
// A partial holds, per interval, 4 channels for its lower entry and 4 for its upper one: an
// entry is the sum of its own lower record and the upper one of the interval before it.
__global__ void k_lut_grad_chunks(const float *__restrict__ partial, int nparts, int n, double *__restrict__ chunks) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int q = (nparts + (int)gridDim.y - 1) / (int)gridDim.y;
    const int p0 = (int)blockIdx.y * q, p1 = min(nparts, p0 + q);
    const int lo = (i >> 2) * 8 + (i & 3);
    double a = 0.0;
    for (int p = p0; p < p1; ++p) {
        const float *r = partial + (long long)p * 2 * n;
        a += (double)r[lo];
        if (i >= 4) a += (double)r[lo - 4];
    }
    chunks[(long long)blockIdx.y * n + i] = a;
}

__global__ void k_lut_grad_reduce(const double *__restrict__ chunks, int nchunks, int n, float *__restrict__ glut) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double acc = 0.0;
    for (int y = 0; y < nchunks; ++y) acc += chunks[(long long)y * n + i];
    glut[i] = (float)acc;
}

// Several views' table gradients: each view's chunk sums are added to one FP64 accumulator
// (zeroed by the first view), which is rounded to FP32 once, after the last view.
__global__ void k_lut_grad_accumulate(const double *__restrict__ chunks, int nchunks, int n,
                                      double *__restrict__ acc, int first) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double a = first ? 0.0 : acc[i];
    for (int y = 0; y < nchunks; ++y) a += chunks[(long long)y * n + i];
    acc[i] = a;
}

__global__ void k_lut_grad_store(const double *__restrict__ acc, int n, float *__restrict__ glut) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) glut[i] = (float)acc[i];
}

// Function attributes (the dynamic shared-memory limit, the carveout) are set per device: a
// kernel's attributes on one GPU say nothing about another GPU of the same process.  Each
// launcher remembers what it set in one slot per device ordinal (devices beyond kAttrDevices
// are set on every launch).  Frames of the serving loop may launch from several host threads:
// the slots are atomics, and setting an attribute twice is harmless.
constexpr int kAttrDevices = 64;
struct DeviceAttrs {
    std::atomic<int> smem[kAttrDevices];     // dynamic shared-memory limit set (bytes), 0: not yet
    std::atomic<int> carve[kAttrDevices];    // carveout percentage set, -1: not yet
    DeviceAttrs() {
        for (int i = 0; i < kAttrDevices; ++i) { smem[i].store(0); carve[i].store(-1); }
    }
};

int current_device() {
    int d = -1;
    return cudaGetDevice(&d) == cudaSuccess ? d : -1;
}

// Raises the kernel's dynamic shared-memory limit to `bytes` on the current device (once).
cudaError_t ensure_smem_limit(const void *kernel, int bytes, DeviceAttrs &da) {
    const int dev = current_device();
    const bool cached = dev >= 0 && dev < kAttrDevices;
    if (cached && da.smem[dev].load(std::memory_order_acquire) >= bytes) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && cached) da.smem[dev].store(bytes, std::memory_order_release);
    return e;
}

// The unified L1 / shared memory of an SM serves the texture gathers as cache: ask for just the
// shared memory (the table) of the CTAs of `warps` warps the register file admits, leaving the
// rest to L1 (measured on HIPASS-scale frames at 5 CTAs: 25 % carveout 3.65 ms, the driver's
// default 3.75, 50 % 3.98).  Registers are allocated per warp in units of 256, 64 K per SM, at
// most 64 warps and 32 CTAs.  The kernel's current preference on this device is remembered in
// `da`.
cudaError_t set_carveout(const void *kernel, size_t smem_per_cta, DeviceAttrs &da, int warps) {
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    const int per_warp = (fa.numRegs * 32 + 255) / 256 * 256;
    const int ctas = std::max(1, std::min(32, std::min(64, 65536 / std::max(per_warp, 256)) / warps));
    const double need = ctas * (double)(smem_per_cta + 1024) / (228.0 * 1024.0);
    const int pct = std::min(100, std::max(0, (int)std::ceil(100.0 * need)));
    const int dev = current_device();
    const bool cached = dev >= 0 && dev < kAttrDevices;
    if (cached && da.carve[dev].load(std::memory_order_relaxed) == pct) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
    if (e == cudaSuccess && cached) da.carve[dev].store(pct, std::memory_order_relaxed);
    return e;
}

template <int S, int MODE, int F, bool MASK, bool HALF>
cudaError_t launch_rc_kernel(const FrameConsts &fc, const float4 *lut, const DrawBrick *db, const TileItem *items,
                      int nitems, const void *pool, void *frags, Counters *ctr, cudaStream_t s) {
    static DeviceAttrs da;
    constexpr int threads = HALF ? 128 : 256;
    const size_t smem = (MODE == 0 ? table_bytes(fc.nlut) : 0) + (MASK ? (size_t)fc.mask_planes : 0);
    const void *kern = reinterpret_cast<const void *>(k_raycast<S, MODE, F, MASK, HALF>);
    cudaError_t e = ensure_smem_limit(kern, (int)(2 * sizeof(float4) * kMaxLut) + kMaskPlanes, da);
    if (e != cudaSuccess) return e;
    if (MODE == 0) {
        e = set_carveout(kern, smem, da, threads / 32);
        if (e != cudaSuccess) return e;
    }
    k_raycast<S, MODE, F, MASK, HALF><<<nitems * (256 / threads), threads, smem, s>>>(fc, lut, const_cast<DrawBrick *>(db), items, pool, frags, ctr);
    return cudaGetLastError();
}
template <int S, int MODE, int F, bool MASK>
cudaError_t launch_rc(const FrameConsts &fc, const float4 *lut, const DrawBrick *db, const TileItem *items,
                      int nitems, const void *pool, void *frags, Counters *ctr, cudaStream_t s) {
    if constexpr (MODE == 0 && rc_halves<MODE, F>())
        if (fc.nlut > (straight(F) ? kHalfTableRows : kHalfTable))
            return launch_rc_kernel<S, MODE, F, MASK, false>(fc, lut, db, items, nitems, pool, frags, ctr, s);
    return launch_rc_kernel<S, MODE, F, MASK, rc_halves<MODE, F>()>(fc, lut, db, items, nitems, pool, frags, ctr, s);
}

template <bool MASK>
cudaError_t launch_staged(const FrameConsts &fc, const float4 *lut, const DrawBrick *db, const TileItem *items,
                          int nitems, const void *pool, void *frags, Counters *ctr, cudaStream_t s) {
    static DeviceAttrs da;
    const size_t smem = 2 * sizeof(float4) * (size_t)fc.nlut + 2 * sizeof(float) * (size_t)kStageFloats;
    const void *kern = reinterpret_cast<const void *>(k_raycast_staged<MASK>);
    cudaError_t e = ensure_smem_limit(kern, (int)(2 * sizeof(float4) * kMaxLut + 2 * sizeof(float) * kStageFloats), da);
    if (e != cudaSuccess) return e;
    k_raycast_staged<MASK><<<nitems, 256, smem, s>>>(fc, lut, const_cast<DrawBrick *>(db), items,
                                                     static_cast<const float *>(pool), static_cast<float4 *>(frags), ctr);
    return cudaGetLastError();
}

template <int S>
cudaError_t launch_rc_s(const FrameConsts &fc, const float4 *lut, const DrawBrick *db, const TileItem *items,
                        int nitems, const void *pool, void *frags, Counters *ctr, cudaStream_t s) {
    if (S == 0 && fc.fetch == 4 && fc.mode == 0)
        return fc.chmask ? launch_staged<true>(fc, lut, db, items, nitems, pool, frags, ctr, s)
                         : launch_staged<false>(fc, lut, db, items, nitems, pool, frags, ctr, s);
#define VR_RC(MODE, F, MASK) launch_rc<S, MODE, F, MASK>(fc, lut, db, items, nitems, pool, frags, ctr, s)
    if constexpr (S != 0) {           // pair atlases: 16-bit bricks only
        if (fc.fetch == 5) {
            if (fc.chmask) return fc.mode != 0 ? VR_RC(1, 5, true) : VR_RC(0, 5, true);
            return fc.mode != 0 ? VR_RC(1, 5, false) : VR_RC(0, 5, false);
        }
    }
#define VR_RC_MASKED(MODE, F) (fc.chmask ? VR_RC(MODE, F, true) : VR_RC(MODE, F, false))
#define VR_RC_MODE(F) (fc.mode != 0 ? VR_RC_MASKED(1, F) : VR_RC_MASKED(0, F))
    switch (fc.fetch) {
        case 1: return VR_RC(0, 1, false);      // (masked frames read rows)
        case 2: return VR_RC_MODE(2);
        case 3: return VR_RC_MODE(3);
        case 6: return VR_RC_MODE(6);
        case 7: return VR_RC_MODE(7);
        case 8: return VR_RC_MODE(8);
        default: return VR_RC_MODE(0);
    }
#undef VR_RC_MODE
#undef VR_RC_MASKED
#undef VR_RC
}

}  // namespace

cudaError_t launch_raycast(const FrameConsts &fc, const float4 *lut, const DrawBrick *db,
                           const TileItem *items, int nitems, const void *pool, void *frags,
                           Counters *ctr, cudaStream_t s) {
    if (nitems <= 0) return cudaSuccess;
    if (fc.storage == 0) return launch_rc_s<0>(fc, lut, db, items, nitems, pool, frags, ctr, s);
    if (fc.storage == 1) return launch_rc_s<1>(fc, lut, db, items, nitems, pool, frags, ctr, s);
    return launch_rc_s<2>(fc, lut, db, items, nitems, pool, frags, ctr, s);
}

template <int S, int F, bool MASK>
cudaError_t launch_march(const FrameConsts &fc, const float4 *lut, DrawBrick *bricks, const MarchGrid &g,
                         const void *pool, float4 *out, Counters *ctr, cudaStream_t s) {
    static DeviceAttrs da;
    const void *kern = reinterpret_cast<const void *>(k_raymarch<S, F, MASK>);
    cudaError_t e = ensure_smem_limit(kern, (int)(2 * sizeof(float4) * kMaxLut + kMarchStashBytes), da);
    const size_t smem = table_bytes(fc.nlut) + kMarchStashBytes;
    if (e == cudaSuccess) e = set_carveout(kern, smem, da, kMarchWarps);
    if (e != cudaSuccess) return e;
    const int tw = fc.lanes_y ? kMarchWarps : kRcLong, th = fc.lanes_y ? kRcLong : kMarchWarps;
    const long long ntiles = (long long)((fc.cam.W + tw - 1) / tw) * ((fc.cam.H + th - 1) / th);
    k_raymarch<S, F, MASK><<<(unsigned)ntiles, kMarchThreads, smem, s>>>(fc, lut, bricks, g, pool, out, ctr);
    return cudaGetLastError();
}

template <int S>
cudaError_t launch_march_s(const FrameConsts &fc, const float4 *lut, DrawBrick *bricks, const MarchGrid &g,
                           const void *pool, float4 *out, Counters *ctr, cudaStream_t s) {
    if constexpr (S != 0) {           // pair atlases: 16-bit bricks only
        if (fc.fetch == 5)
            return fc.chmask ? launch_march<S, 5, true>(fc, lut, bricks, g, pool, out, ctr, s)
                             : launch_march<S, 5, false>(fc, lut, bricks, g, pool, out, ctr, s);
    }
#define VR_MARCH(F) (fc.chmask ? launch_march<S, F, true>(fc, lut, bricks, g, pool, out, ctr, s) \
                               : launch_march<S, F, false>(fc, lut, bricks, g, pool, out, ctr, s))
    return fc.fetch == 2 ? VR_MARCH(2) : fc.fetch == 3 ? VR_MARCH(3) : VR_MARCH(0);
#undef VR_MARCH
}

cudaError_t launch_raymarch(const FrameConsts &fc, const float4 *lut, DrawBrick *bricks, const MarchGrid &g,
                            const void *pool, float4 *out, Counters *ctr, cudaStream_t s) {
    if (fc.storage == 0) return launch_march_s<0>(fc, lut, bricks, g, pool, out, ctr, s);
    if (fc.storage == 1) return launch_march_s<1>(fc, lut, bricks, g, pool, out, ctr, s);
    return launch_march_s<2>(fc, lut, bricks, g, pool, out, ctr, s);
}

cudaError_t launch_composite(const FrameConsts &fc, const DrawBrick *db, const int *tile_start,
                             const int *tile_list, const void *frags, float *out, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((fc.cam.W + kTile - 1) / kTile, (fc.cam.H + kTile - 1) / kTile);
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    // Right behind a ray cast the launch overlaps its end (a programmatic dependency; behind anything else
    // an ordinary one).  Captured launches keep plain edges, which every graph call understands.
    cudaLaunchAttribute pdl{};
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &pdl;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) cudaGetLastError();
    cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
    const cudaError_t e = fc.mode == 0 ? cudaLaunchKernelEx(&cfg, k_composite<0>, fc, db, tile_start, tile_list, frags, out)
                                       : cudaLaunchKernelEx(&cfg, k_composite<1>, fc, db, tile_start, tile_list, frags, out);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_composite_parts(const FrameConsts &fc, int axis, int n, const float *subs, int row0, int rows,
                                   int final_, float *out, cudaStream_t s) {
    const long long npx = (long long)rows * fc.cam.W;
    if (npx <= 0) return cudaSuccess;
    const int grid = (int)std::min<long long>((npx + 255) / 256, 152 * 8);
    k_composite_parts<<<grid, 256, 0, s>>>(fc, axis, n, subs, row0, rows, final_, out);
    return cudaGetLastError();
}

cudaError_t launch_composite_backward(const FrameConsts &fc, const DrawBrick *db,
                                      const int *tile_start, const int *tile_list,
                                      const float4 *frags, const float4 *gout, float4 *gfrag,
                                      cudaStream_t s) {
    dim3 grid((fc.cam.W + kTile - 1) / kTile, (fc.cam.H + kTile - 1) / kTile);
    k_composite_backward<<<grid, 256, 0, s>>>(fc, db, tile_start, tile_list, frags, gout, gfrag);
    return cudaGetLastError();
}

template <bool ATLAS, int VOX, bool WRAP, int THREADS>
static cudaError_t adjoint(const FrameConsts &fc, const float4 *lut, const DrawBrick *db, const TileItem *items, int nitems,
                           const float *pool, const float4 *frags, const float4 *gfrag, float *glut_partial, int rows, void *gvox,
                           cudaStream_t s) {
    static DeviceAttrs da;
    const auto kern = k_adjoint<ATLAS, VOX, WRAP, THREADS>;
    const cudaError_t e = ensure_smem_limit(reinterpret_cast<const void *>(kern), (int)(32 * kMaxLut), da);
    if (e != cudaSuccess) return e;
    kern<<<nitems * (256 / THREADS), THREADS, 32 * (size_t)fc.nlut, s>>>(fc, lut, db, items, pool, frags, gfrag, glut_partial, rows, gvox);
    return cudaGetLastError();
}

cudaError_t launch_adjoint(const FrameConsts &fc, const float4 *lut, const DrawBrick *db,
                           const TileItem *items, int nitems, const float *pool,
                           const float4 *frags, const float4 *gfrag, float *glut_partial, int rows,
                           float *gvox, float4 *corners, cudaStream_t s) {
    if (nitems <= 0) return cudaSuccess;
    const cudaError_t e = cudaMemsetAsync(glut_partial, 0, sizeof(float) * 8 * (size_t)fc.nlut * rows, s);
    if (e != cudaSuccess) return e;
#define VR_ADJ(A, V, W, G) (fc.nlut <= (A ? kHalfTableAdj : kHalfTableAdjLinear) ? adjoint<A, V, W, 128>(fc, lut, db, items, nitems, pool, frags, gfrag, glut_partial, rows, G, s) \
                                                     : adjoint<A, V, W, 256>(fc, lut, db, items, nitems, pool, frags, gfrag, glut_partial, rows, G, s))
#define VR_ADJ_VOX(A, W) (corners ? VR_ADJ(A, 2, W, corners) : gvox ? VR_ADJ(A, 1, W, gvox) : VR_ADJ(A, 0, W, nullptr))
    if (fc.fetch == 3) return VR_ADJ_VOX(true, true);
    return fc.fetch == 2 ? VR_ADJ_VOX(true, false) : VR_ADJ_VOX(false, false);
#undef VR_ADJ_VOX
#undef VR_ADJ
}

size_t corner_records(int nx, int ny, int nz) { return (size_t)(nz + 2) * (ny + 1) * (nx + 1); }

cudaError_t launch_corner_gather(const float4 *corners, int nx, int ny, int nz, float *gvox, cudaStream_t s) {
    const int gx = (nx + 31) / 32, gy = (ny + 7) / 8;
    const int gz = std::max(1, std::min(nz, 152 * 16 / std::max(1, gx * gy)));
    k_corner_gather<<<dim3(gx, gy, gz), 256, 0, s>>>(corners, nx, ny, nz, gvox);
    return cudaGetLastError();
}

static cudaError_t launch_lut_grad_chunks(const float *partial, int nparts, int n, double *chunks, cudaStream_t s) {
    dim3 grid((n + 255) / 256, kLutGradChunks);
    k_lut_grad_chunks<<<grid, 256, 0, s>>>(partial, nparts, n, chunks);
    return cudaGetLastError();
}

cudaError_t launch_lut_grad_reduce(const float *partial, int nparts, int nlut, double *chunks, float *glut,
                                   cudaStream_t s) {
    const int n = 4 * nlut;
    cudaError_t e = launch_lut_grad_chunks(partial, nparts, n, chunks, s);
    if (e != cudaSuccess) return e;
    k_lut_grad_reduce<<<(n + 255) / 256, 256, 0, s>>>(chunks, kLutGradChunks, n, glut);
    return cudaGetLastError();
}

cudaError_t launch_lut_grad_accumulate(const float *partial, int nparts, int nlut, double *chunks, double *acc,
                                       bool first, cudaStream_t s) {
    const int n = 4 * nlut;
    cudaError_t e = launch_lut_grad_chunks(partial, nparts, n, chunks, s);
    if (e != cudaSuccess) return e;
    k_lut_grad_accumulate<<<(n + 255) / 256, 256, 0, s>>>(chunks, kLutGradChunks, n, acc, first ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_lut_grad_store(const double *acc, int nlut, float *glut, cudaStream_t s) {
    const int n = 4 * nlut;
    k_lut_grad_store<<<(n + 255) / 256, 256, 0, s>>>(acc, n, glut);
    return cudaGetLastError();
}

}  // namespace vr
