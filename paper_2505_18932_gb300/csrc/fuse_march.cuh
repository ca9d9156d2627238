// Device code shared by the fusion kernels (forward, batched, backward):
// map and depth loads, the nearest-pixel contract, the per-sample TSDF sum,
// the warp-bundle march with its slab tests, and the kernel-variant dispatch.
#pragma once

#include <cuda_fp16.h>
#include <math.h>

#include "bounds_check.cuh"
#include "gvs_internal.cuh"

namespace gvs {
namespace {

#define kInf __int_as_float(0x7f800000)

__device__ __forceinline__ bool valid_depth(float d) { return isfinite(d) && d > 0.0f; }

// Depth element load (FP32 or FP16) widened to FP32.
__device__ __forceinline__ float load_depth(const float *p) { return __ldg(p); }
__device__ __forceinline__ float load_depth(const __half *p) { return __half2float(__ldg(p)); }

// The depth as the map stores it: exact for float2, rounded to half for half2.
__device__ __forceinline__ float as_stored(float d, float2 *) { return d; }
__device__ __forceinline__ float as_stored(float d, __half2 *) { return __half2float(__float2half_rn(d)); }

__device__ __forceinline__ void store_map(float2 *p, float d, float w) { *p = make_float2(d, w); }
__device__ __forceinline__ void store_map(__half2 *p, float d, float w) { *p = __floats2half2_rn(d, w); }

__device__ __forceinline__ float2 load_map(const float2 *p) { return __ldg(p); }
__device__ __forceinline__ float2 load_map(const __half2 *p) { return __half22float2(__ldg(p)); }

// Nearest integers (ties to even) of the exact real quotients hx/hz, hy/hz.
// With q = h * fast_rcp(hz) (within 3e-7 |q| of the quotient) and n = rint(q), the
// residual h - n hz, rounded once, is below |hz| / 2 in magnitude only if the exact one is
// (rounding is monotone), and then n is the answer.  Otherwise (q within its error of
// a half-integer: a lane in several thousand; or |q| >= 2^22, whose shifted n is off) the
// decision is re-taken from the signs of the exact residuals h - (n +/- 0.5) hz (one
// rounding each in the FMA, which never changes a sign).  The fix-up leaves n
// unchanged when q is not near a half-integer, so it runs for both coordinates
// under one branch.
__device__ __forceinline__ float exact_nearest_fixup(float num, float den, float n) {
    if (fabsf(n) < 4194304.0f) {
        const float hi = __fmaf_rn(-(n + 0.5f), den, num);
        const float lo = __fmaf_rn(-(n - 0.5f), den, num);
        const bool odd = (__float2int_rz(n) & 1) != 0;
        if (hi > 0.0f || (hi == 0.0f && odd)) n += 1.0f;
        else if (lo < 0.0f || (lo == 0.0f && odd)) n -= 1.0f;
    }
    return n;
}

// The candidate (u, v) and whether the residuals prove it.  An infinite q leaves a shifted
// index far outside any image and a residual that proves nothing.
__device__ __forceinline__ bool nearest_pixel_fast(float hx, float hy, float hz, int &u, int &v) {
    const float r = fast_rcp(hz);
    const float nx = shift_round(hx * r, u), ny = shift_round(hy * r, v);
    const float rx = __fmaf_rn(-nx, hz, hx), ry = __fmaf_rn(-ny, hz, hy);
    return fmaxf(fabsf(rx), fabsf(ry)) < 0.5f * fabsf(hz);
}

__device__ __forceinline__ void nearest_pixel_exact(float hx, float hy, float hz, int &u, int &v) {
    const float r = fast_rcp(hz);
    u = __float2int_rz(exact_nearest_fixup(hx, hz, rintf(hx * r)));
    v = __float2int_rz(exact_nearest_fixup(hy, hz, rintf(hy * r)));
}

__device__ __forceinline__ void nearest_pixel(float hx, float hy, float hz, int &u, int &v) {
    if (!nearest_pixel_fast(hx, hy, hz, u, v)) nearest_pixel_exact(hx, hy, hz, u, v);
}

#ifndef GVS_FUSE_WARPS
#define GVS_FUSE_WARPS 4        // warps (bundles) per fusion block
#endif
constexpr int FZ_WARPS = GVS_FUSE_WARPS;
// Samples evaluated after both slab tests fail, before testing again: the failing short
// segment and the sample after it (8 x 1080p, 16 x 1080p with a half2 map: 2: 293 and 570 us,
// 3: 274 and 557, 4: 293 and 554, at 9 resident blocks).
constexpr int SKIP_COOL = 3;

// Bundle shape and slab-test lengths of the march.  Every variant computes the
// same result; they differ only in speed, and the autotuner picks one per
// workload (gvs_fuse_params.variant; shaped_variant gives the tile's number).
//   bx x by : target pixels one warp marches together (bx * by = 32)
//   llong   : samples per segment in the first slab test
//   lshort  : samples per segment in the second test when the first fails
//   full    : the call has exactly KMAX views, so the per-view guard k < K
//             compiles away and the unrolled views form one block of code
//   spt     : samples each lane evaluates at once in a run of evaluations
//             (1 or 2: two keep twice the gathers in flight)
//   warp    : the mapping.  false: lane per ray (a bundle of bx x by = 32 rays per
//             warp); true: warp per ray (bx = by = 1), its lanes split into
//             views x samples, so a step evaluates 32 / KMAX consecutive samples
//             of the one ray at once and its slab tests hold for that ray alone
template <int BX_, int BY_, int LLONG_, int LSHORT_, bool FULL_ = false, int SPT_ = 1, bool WARP_ = false>
struct Tile {
    static constexpr int bx = BX_, by = BY_, llong = LLONG_, lshort = LSHORT_, spt = SPT_;
    static constexpr bool full = FULL_, warp = WARP_;
    static_assert(warp ? (bx == 1 && by == 1 && spt == 1) : bx * by == 32, "a bundle is one warp, or one ray");
    static_assert(llong >= 1 && lshort >= 1, "skip lengths must advance the march");
    static_assert(spt == 1 || spt == 2, "one or two samples at once");
};
template <typename T>
struct FullTile;
template <int BX_, int BY_, int LLONG_, int LSHORT_, bool FULL_, int SPT_, bool WARP_>
struct FullTile<Tile<BX_, BY_, LLONG_, LSHORT_, FULL_, SPT_, WARP_>> {
    using type = Tile<BX_, BY_, LLONG_, LSHORT_, true, SPT_, WARP_>;
};
using Tile0 = Tile<8, 4, 8, 2>;
using Tile1 = Tile<8, 4, 16, 4>;
using Tile2 = Tile<16, 2, 8, 2>;
using Tile3 = Tile<4, 8, 8, 2>;
using Tile4 = Tile<4, 8, 8, 2, false, 2>;
using Tile5 = Tile<8, 4, 8, 2, false, 2>;
using Tile6 = Tile<1, 1, 8, 2, false, 1, true>;
constexpr int kFuseVariants = 7;

// Resident blocks per SM asked of the register allocator, measured over 5 to 12 (us):
//   8 or 16 views, all of them present: 12 (40 registers; the rays spill to L1 and the warps
//     hide it): 8 x 1080p 254 against 274 at 9 and 301 at 7; 16 x 1080p, half2 map, 507
//     against 557 and 621 (one view per step; two: 236 and 467 at 12);
//   up to 4 views: 7 (72 registers), for small targets are one wave of bundles whose time is
//     one bundle's chain of tests and samples: 4 x 320x240 26.8 against 28.8 at 9;
//   otherwise (exactly 5 to 7 views, a guard per view, the temporal input, 32 views): 9
//     (56 registers): 5 views at 961x541 49.6 against 51.0 at 12.
template <int KMAX, typename T, bool TMP>
constexpr int fuse_min_blocks() {
    return KMAX <= 4 ? 7 : (T::full && !T::warp && !TMP && KMAX >= 8 && KMAX <= 16) ? 12 : 9;
}

struct Ray {
    float ax, ay, az;
};

// Where segment q of a slab test begins, in units of the test's segment length: one after
// another, but with only two segments (9 to 16 views) the second is twice as long.
// 16 x 1080p: 467 us with equal segments, 450 with 1 + 2, 461 with 1 + 3; four
// segments are best equal (8 x 1080p: 236 us, 254 with 1 + 1 + 1 + 3, 285 with 1 + 1 + 2 + 4).
template <int NSEG>
__device__ __forceinline__ constexpr int seg_begin(int q) {
    return NSEG == 2 && q == 2 ? 3 : q;
}

// The rays of a bundle seen from one view: the ranges of the ray coefficients
// (ax, ay, az) over the bundle's pixels and the view's offset b.  Each coefficient
// is fma(M0, i, fma(M1, j, M2)), monotone in i and in j also after rounding, so its
// extremes are those of the four corner pixels, exactly.
struct SlabRays {
    float axlo, axhi, aylo, ayhi, azlo, azhi, b0, b1, b2;
};

__device__ __forceinline__ SlabRays slab_rays(const ViewXform &xf, int i0, int i1, int j0, int j1) {
    const float ilo = (float)i0, ihi = (float)i1, jlo = (float)j0, jhi = (float)j1;
    float lo[3], hi[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const float *M = xf.M + 3 * r;
        const float t0 = __fmaf_rn(M[1], jlo, M[2]), t1 = __fmaf_rn(M[1], jhi, M[2]);
        const float c0 = __fmaf_rn(M[0], ilo, t0), c1 = __fmaf_rn(M[0], ihi, t0);
        const float c2 = __fmaf_rn(M[0], ilo, t1), c3 = __fmaf_rn(M[0], ihi, t1);
        lo[r] = fminf(fminf(c0, c1), fminf(c2, c3));
        hi[r] = fmaxf(fmaxf(c0, c1), fmaxf(c2, c3));
    }
    SlabRays s;
    s.axlo = lo[0]; s.axhi = hi[0];
    s.aylo = lo[1]; s.ayhi = hi[1];
    s.azlo = lo[2]; s.azhi = hi[2];
    s.b0 = xf.b[0]; s.b1 = xf.b[1]; s.b2 = xf.b[2];
    return s;
}

// Where a view's bound tiles of each level begin, counted in bounds from a.ob[0],
// and their row pitch; entry [kBoundLevels] is the whole view (pitch 0).  Kept in
// shared memory ([level * KMAX + view]): the lanes of a slab test want different
// views and levels, which constant loads would serialise and branches would diverge on.
template <int KMAX>
__device__ __forceinline__ void fill_slab_table(const FuseArgs &a, int2 *tab, int tid, int threads) {
    for (int e = tid; e < (kBoundLevels + 1) * KMAX; e += threads) {
        const int l = e / KMAX, k = e % KMAX;
        int2 t = make_int2(0, 0);
        if (k < a.K) {
            if (l < kBoundLevels) t = make_int2((int)(a.ob[l] - a.ob[0]) + k * a.th[l] * a.tw[l], a.tw[l]);
            else t = make_int2((int)(a.tg - a.ob[0]) + k, 0);
        }
        tab[e] = t;
    }
}

// The bundle's rays between depths z0 and z1, 0 < z0 < z1, seen from view k.  At one
// depth z a ray's homogeneous coordinates lie in [z alo + b, z ahi + b] each, so its
// projection lies in the quotient of those intervals (positive depths); along a ray
// the projection is monotone in z, so over the slab it lies between its ranges at z0
// and z1.  That box is as tight as the hull of the 8 projected corners where az does
// not vary over the bundle (views that look along the target's axis) and wider by
// x (azhi - azlo) / az elsewhere (below a pixel or two for bundles of 32 pixels), and
// takes 4 reciprocals and 8 products in place of 8 projections: the 8 x 1080p fusion
// kernel 375 -> 315 us.  (FP32 rounding of the
// samples is covered by a 1 pixel and 1e-6 relative margin.)  A pixel
// of depth d can make a sample at projected depth z end a crossing only if
// d <= z (sdf <= 0) and d >= z - mu (not cut off), so the view is free over
// the slab when no valid depth in the pixel box lies in
// [zlo - 1.0001 mu, zhi] (every term positive or cut off), or the box is
// outside the image, or the slab is behind the camera.  One bound load: the
// finest tile level whose overlapping 2x2 block covers the box, else the whole
// view.  The bound's range decides first; failing that, its mask of occupied
// depth bins (a clear bin holds no depth; see DepthBound), which separates the
// surfaces of a tile that straddles a depth discontinuity.  When every view is free over the
// slab, no sample of it can end a crossing (S > 0 wherever W > 0).
// AHEAD: free means that no valid depth lies in [zlo - 1.0001 mu, zhi + 1.0001 mu]: every
// term is not only positive or cut off but saturated (sdf >= 1) or cut off.
template <int KMAX, bool AHEAD = false>
__device__ __forceinline__ bool slab_view_free(const FuseArgs &a, const int2 *tab, int k, const SlabRays &r, float z0,
                                               float z1) {
    const float h0lo = __fmaf_rn(z0, r.azlo, r.b2), h0hi = __fmaf_rn(z0, r.azhi, r.b2);
    const float h1lo = __fmaf_rn(z1, r.azlo, r.b2), h1hi = __fmaf_rn(z1, r.azhi, r.b2);
    float zlo = fminf(h0lo, h1lo), zhi = fmaxf(h0hi, h1hi);
    const bool front = h0lo > 1e-6f && h1lo > 1e-6f;  // false for NaN
    zhi += 1e-6f * fabsf(zhi);
    zlo -= 1e-6f * fabsf(zlo);
    if (zhi <= 1e-6f) return true;  // behind the camera throughout
    if (!front) return false;       // crosses the camera plane: do not try
    if (AHEAD) zhi = __fadd_ru(zhi, a.behind);
    const float q0hi = fast_rcp(h0lo), q0lo = fast_rcp(h0hi), q1hi = fast_rcp(h1lo), q1lo = fast_rcp(h1hi);
    const auto low = [](float h, float qlo, float qhi) { return h * (h < 0.0f ? qhi : qlo); };
    const auto high = [](float h, float qlo, float qhi) { return h * (h < 0.0f ? qlo : qhi); };
    float xlo = fminf(low(__fmaf_rn(z0, r.axlo, r.b0), q0lo, q0hi), low(__fmaf_rn(z1, r.axlo, r.b0), q1lo, q1hi));
    float xhi = fmaxf(high(__fmaf_rn(z0, r.axhi, r.b0), q0lo, q0hi), high(__fmaf_rn(z1, r.axhi, r.b0), q1lo, q1hi));
    float ylo = fminf(low(__fmaf_rn(z0, r.aylo, r.b1), q0lo, q0hi), low(__fmaf_rn(z1, r.aylo, r.b1), q1lo, q1hi));
    float yhi = fmaxf(high(__fmaf_rn(z0, r.ayhi, r.b1), q0lo, q0hi), high(__fmaf_rn(z1, r.ayhi, r.b1), q1lo, q1hi));
    xlo -= 1.0f; xhi += 1.0f; ylo -= 1.0f; yhi += 1.0f;
    if (!(xlo <= xhi && ylo <= yhi)) return false;  // NaN
    const float wmax = (float)(a.W - 1), hmax = (float)(a.H - 1);
    if (xhi < 0.0f || yhi < 0.0f || xlo > wmax || ylo > hmax) return true;  // outside
    // the pixels floor(lo) .. ceil(hi) within the image, from the low bits of a sum with
    // 2^23 rounded down or up (the values lie in [0, 2^14))
    const int bx0 = __float_as_int(__fadd_rd(fmaxf(xlo, 0.0f), 8388608.0f)) - 0x4B000000;
    const int bx1 = __float_as_int(__fadd_ru(fminf(xhi, wmax), 8388608.0f)) - 0x4B000000;
    const int by0 = __float_as_int(__fadd_rd(fmaxf(ylo, 0.0f), 8388608.0f)) - 0x4B000000;
    const int by1 = __float_as_int(__fadd_ru(fminf(yhi, hmax), 8388608.0f)) - 0x4B000000;
    // a box spanning fewer than 2^l pixels per axis covers at most 2x2 tiles of level l
    const int span = max(bx1 - bx0, by1 - by0);
    const int l = max(32 - __clz(span) - kBoundShift0, 0);
    const int2 t = tab[min(l, kBoundLevels) * KMAX + k];
    const int sh = l < kBoundLevels ? l + kBoundShift0 : 31;  // 31: the whole view's one entry
    const int e = t.x + (by0 >> sh) * t.y + (bx0 >> sh);
    if (!GVS_IN_BOUNDS(e, (a.tg + a.K) - a.ob[0], GVS_SITE_FUSE_BOUNDS)) return false;
    const uint4 b = __ldg(reinterpret_cast<const uint4 *>(a.ob[0] + e));
    const float lo = __uint_as_float(b.x), hi = __uint_as_float(b.y);
    const float qlo = __fsub_rn(zlo, a.behind);
    if (zhi < lo || qlo > hi) return true;
    // here lo <= zhi, so 0 <= m1, and m0 <= m1 (the bins are monotone)
    const int base = depth_bin(lo);
    const int m0 = min(max(depth_bin(fmaxf(qlo, 0.0f)) - base, 0), kDepthBins - 1);
    const int m1 = min(depth_bin(zhi) - base, kDepthBins - 1);
    const unsigned long long occupied = ((unsigned long long)b.w << 32) | b.z;
    return (occupied & (~0ull << m0) & (~0ull >> (kDepthBins - 1 - m1))) == 0ull;
}

// S and W of one sample over the input views (Supplement A.1), before the
// temporal term and the optional normalisation, exactly as the march computes them.
// A view whose sample lies behind its camera or off its image, or in front of
// the surface by more than mu, enters with weight 0 (a predicated gather, no
// branch): adding 0 * x leaves S and W as they were.
// FULL: the call has exactly KMAX views (no per-view guard).  View k's map plane is
// a.vb[k], a constant-bank read of the kernel's parameters.
//
// With every view present, two views at a time (four of four) go through the same three
// steps (pixels, gathers, sums) with one branch, for the rare pixel that needs the exact
// decision: the group's gathers are in flight together.  8 x 1080p fusion kernel, in groups
// of 1, 2, 4 and 8: 250, 236, 265 and 286 us (the larger ones spill); the sphere march
// of 4 views 113, 105 and 101 us.
template <int KMAX, typename MT, bool FULL = false>
__device__ __forceinline__ void evaluate_sample(const FuseArgs &a, const Ray (&ray)[KMAX], float zs, float &S,
                                                float &Wsum) {
    constexpr int G = !FULL ? 1 : KMAX <= 4 ? KMAX : 2;
    const size_t plane = (size_t)a.W * a.H;
    S = 0.0f;
    Wsum = 0.0f;
#pragma unroll
    for (int k0 = 0; k0 < KMAX; k0 += G) {
        if (FULL || k0 < a.K) {
            float hz[G];
            int u[G], v[G];
            bool sure = true;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int k = k0 + g;
                if (k >= KMAX) continue;
                hz[g] = __fmaf_rn(zs, ray[k].az, a.xf[k].b[2]);
                const float hx = __fmaf_rn(zs, ray[k].ax, a.xf[k].b[0]);
                const float hy = __fmaf_rn(zs, ray[k].ay, a.xf[k].b[1]);
                sure = nearest_pixel_fast(hx, hy, hz[g], u[g], v[g]) && sure;
            }
            if (!sure) {
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    const int k = k0 + g;
                    if (k >= KMAX) continue;
                    nearest_pixel_exact(__fmaf_rn(zs, ray[k].ax, a.xf[k].b[0]),
                                        __fmaf_rn(zs, ray[k].ay, a.xf[k].b[1]), hz[g], u[g], v[g]);
                }
            }
            float2 p[G];
            bool in[G];
#pragma unroll
            for (int g = 0; g < G; ++g) {
                const int k = k0 + g;
                if (k >= KMAX) continue;
                in[g] = hz[g] > 1e-6f && (unsigned)u[g] < (unsigned)a.W && (unsigned)v[g] < (unsigned)a.H &&
                        GVS_IN_BOUNDS((size_t)k * plane + (size_t)v[g] * a.W + u[g], (size_t)a.K * plane,
                                      GVS_SITE_FUSE_MAP);
                p[g] = make_float2(0.0f, 0.0f);
                if (in[g]) {
                    const MT *plane_k = reinterpret_cast<const MT *>(a.vb[k]);
                    p[g] = load_map(plane_k + (v[g] * a.W + u[g]));  // v W + u < 2^28
                }
            }
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if (k0 + g >= KMAX) continue;
                const float sdf = (p[g].x - hz[g]) * a.inv_mu;
                const float w = (in[g] && sdf >= -1.0f) ? p[g].y : 0.0f;
                S = fmaf(w, fminf(sdf, 1.0f), S);
                Wsum += w;
            }
        }
    }
}

// Samples zs0 and zs1 at once (each exactly as evaluate_sample computes it): the
// two samples' gathers of a view are independent, so a lane keeps both in flight.
template <int KMAX, typename MT, bool FULL = false>
__device__ __forceinline__ void evaluate_sample2(const FuseArgs &a, const Ray (&ray)[KMAX], float zs0, float zs1,
                                                 float &S0, float &W0, float &S1, float &W1) {
    const size_t plane = (size_t)a.W * a.H;
    S0 = W0 = S1 = W1 = 0.0f;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        if (FULL || k < a.K) {
            const MT *plane_k = reinterpret_cast<const MT *>(a.vb[k]);
            float hz[2], pd[2], pw[2];
            bool in[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float zs = j ? zs1 : zs0;
                hz[j] = __fmaf_rn(zs, ray[k].az, a.xf[k].b[2]);
                const float hx = __fmaf_rn(zs, ray[k].ax, a.xf[k].b[0]);
                const float hy = __fmaf_rn(zs, ray[k].ay, a.xf[k].b[1]);
                int u, v;
                nearest_pixel(hx, hy, hz[j], u, v);
                in[j] = hz[j] > 1e-6f && (unsigned)u < (unsigned)a.W && (unsigned)v < (unsigned)a.H &&
                        GVS_IN_BOUNDS((size_t)k * plane + (size_t)v * a.W + u, (size_t)a.K * plane,
                                      GVS_SITE_FUSE_MAP);
                float2 p = make_float2(0.0f, 0.0f);
                if (in[j]) p = load_map(plane_k + (v * a.W + u));
                pd[j] = p.x;
                pw[j] = p.y;
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float sdf = (pd[j] - hz[j]) * a.inv_mu;
                const float w = (in[j] && sdf >= -1.0f) ? pw[j] : 0.0f;
                float &S = j ? S1 : S0;
                float &Wsum = j ? W1 : W0;
                S = fmaf(w, fminf(sdf, 1.0f), S);
                Wsum += w;
            }
        }
    }
}

// One warp per bundle of BX x BY target pixels.  The warp marches one sample
// index s for all its rays: cooperative slab tests (lane = view x segment,
// 32 / KMAX consecutive segments at once, `tab` from fill_slab_table) skip runs of samples that hold no
// crossing end for any ray of the bundle; otherwise every ray still marching
// evaluates sample s (all KMAX views unrolled, one 8-byte gather each) and
// checks its own crossing.  The result equals the full uniform march.
// TMP: the temporal input (previous output depth and weight) and the views'
// weight at the crossing are compiled in only where they are used.
template <int KMAX, typename MT, typename T, bool TMP = false>
__device__ __forceinline__ void march_rays(const FuseArgs &a, const int2 *tab, int bundle, int lane) {
    constexpr int BX = T::bx, BY = T::by, SKIP_LONG = T::llong, SKIP_SHORT = T::lshort;
    constexpr int NSEG = 32 / KMAX;
    constexpr unsigned SEGMASK = KMAX == 32 ? 0xffffffffu : ((1u << KMAX) - 1u);
    const int nbx = (a.Wt + BX - 1) / BX;
    const int i0 = (bundle % nbx) * BX, j0 = (bundle / nbx) * BY;
    const int i1 = min(i0 + BX - 1, a.Wt - 1), j1 = min(j0 + BY - 1, a.Ht - 1);
    const int i = i0 + (lane % BX), j = j0 + (lane / BX);
    const bool inside = i < a.Wt && j < a.Ht;
    const float fi = (float)min(i, a.Wt - 1), fj = (float)min(j, a.Ht - 1);
    Ray ray[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        if (T::full || k < a.K) {
            const float *M = a.xf[k].M;
            ray[k].ax = __fmaf_rn(M[0], fi, __fmaf_rn(M[1], fj, M[2]));
            ray[k].ay = __fmaf_rn(M[3], fi, __fmaf_rn(M[4], fj, M[5]));
            ray[k].az = __fmaf_rn(M[6], fi, __fmaf_rn(M[7], fj, M[8]));
        }
    }
    // this lane's role in the slab tests: view tk of segment tseg
    const int tk = lane % KMAX, tseg = lane / KMAX;
    const bool tview = tk < a.K;
    const SlabRays slab = slab_rays(a.xf[tview ? tk : 0], i0, i1, j0, j1);
    // temporal input at this ray's pixel
    float td = 0.0f, tw = 0.0f;
    if (TMP && a.tmp_depth && inside) {
        const size_t o = (size_t)j * a.Wt + i;
        const float d = a.tmp_depth[o], w = a.tmp_weight[o];
        if (valid_depth(d) && w > 0.0f) {
            td = d;
            tw = w;
        }
    }
    float S_prev = 0.0f, W_prev = 0.0f, z_prev = 0.0f, Wv_prev = 0.0f;
    float wview = 0.0f;
    bool have_prev = false;  // sample s-1 was evaluated (uniform across the warp)
    bool done = !inside;
    float out = 0.0f;
    int idx = -1;
    int s = 0;
    int cool = 0;
    bool shorter = false;
    while (s < a.D) {
        if (__all_sync(0xffffffffu, done)) break;
        if (cool == 0 && s < a.D - 1) {
            const int L = shorter ? SKIP_SHORT : SKIP_LONG;
            const int sa = s + seg_begin<NSEG>(tseg) * L;
            bool f = false;
            if (sa < a.D - 1) {
                const int sb = min(s + seg_begin<NSEG>(tseg + 1) * L, a.D - 1);
                const float z0 = __fmaf_rn((float)sa, a.dz, a.zn), z1 = __fmaf_rn((float)sb, a.dz, a.zn);
                f = !tview || slab_view_free<KMAX>(a, tab, tk, slab, z0, z1);
            }
            const unsigned ball = __ballot_sync(0xffffffffu, f);
            int nfree = 0;
#pragma unroll
            for (int g = 0; g < NSEG; ++g) {
                bool free_g = ((ball >> (g * KMAX)) & SEGMASK) == SEGMASK;
                if (TMP) {
                    // the temporal input sits at the ray's own pixel, so its projected depth is the
                    // sample's: ray by ray, and only where the ray still marches (the range of
                    // td over the bundle, in its place, kept every sample between the two surfaces of
                    // a depth edge: 8 x 720p 233 us against 161)
                    const float z0 = __fmaf_rn((float)(s + seg_begin<NSEG>(g) * L), a.dz, a.zn);
                    const float z1 = __fmaf_rn((float)min(s + seg_begin<NSEG>(g + 1) * L, a.D - 1), a.dz, a.zn);
                    const bool hit = !done && tw > 0.0f && !(z1 < td || z0 > td + a.behind);
                    free_g = !__any_sync(0xffffffffu, hit) && free_g;
                }
                if (nfree == g && free_g) ++nfree;
            }
            if (nfree > 0) {
                s = min(s + seg_begin<NSEG>(nfree) * L, a.D - 1);  // samples up to s are not crossing ends; s is evaluated next
                if (s == a.D - 1) break;           // ... unless it is the last: nothing follows it
                have_prev = false;
                if (nfree == NSEG) {
                    shorter = false;
                    continue;
                }
            }
            // the segment of length L at s is not free: only shorter ones there can be
            if (!shorter && SKIP_SHORT < SKIP_LONG) {
                shorter = true;
                continue;
            }
            shorter = SKIP_SHORT < SKIP_LONG;  // more often than not the surface is still near
            cool = SKIP_COOL;
        }
        // every lane evaluates (the warp issues the sample anyway); lanes still marching record it
        const int nev = (T::spt == 2 && cool >= 2 && s + 1 < a.D) ? 2 : 1;
        const float zs0 = __fmaf_rn((float)s, a.dz, a.zn);
        float Se[2], We[2], ze[2];
        ze[0] = zs0;
        if (T::spt == 2 && nev == 2) {
            ze[1] = __fmaf_rn((float)(s + 1), a.dz, a.zn);
            evaluate_sample2<KMAX, MT, T::full>(a, ray, ze[0], ze[1], Se[0], We[0], Se[1], We[1]);
        } else {
            evaluate_sample<KMAX, MT, T::full>(a, ray, zs0, Se[0], We[0]);
        }
#pragma unroll
        for (int e = 0; e < T::spt; ++e) {
            if (e < nev) {
                const float zs = ze[e];
                float S = Se[e], Wsum = We[e];
                if (!done) {
                    const float Wv = Wsum;
                    if (TMP && tw > 0.0f) {
                        const float sdf = (td - zs) * a.inv_mu;
                        if (sdf >= -1.0f) {
                            S = fmaf(tw, fminf(sdf, 1.0f), S);
                            Wsum += tw;
                        }
                    }
                    if (a.normalize && Wsum > 0.0f) S = S / Wsum;
                    if (have_prev && W_prev > 0.0f && Wsum > 0.0f && S_prev > 0.0f && S <= 0.0f) {
                        const float t = S_prev / (S_prev - S);
                        out = z_prev + (zs - z_prev) * t;
                        if (TMP) wview = Wv_prev + t * (Wv - Wv_prev);
                        idx = s - 1;
                        done = true;
                    }
                    S_prev = S;
                    W_prev = Wsum;
                    Wv_prev = Wv;
                    z_prev = zs;
                }
                have_prev = true;
                ++s;
                if (cool > 0) --cool;
            }
        }
    }
    if (inside) {
        const size_t o = (size_t)j * a.Wt + i;
        a.fused[o] = out;
        if (a.crossing) a.crossing[o] = (int16_t)idx;
        if (TMP && a.wview) a.wview[o] = wview;
    }
}

// One warp per target ray (the warp-per-pixel mapping; `pixel` < Wt * Ht).  Lane
// (q, k) = (lane / KMAX, lane % KMAX) takes view k: in a slab test, segment q of
// the ray's own slab (its four corner rays are the ray itself); in a run of
// evaluations, sample s + q.  Each sample's S and W are summed over the views in
// view order from the lanes' terms, exactly as evaluate_sample sums them, and the
// samples are then scanned in order, so the crossing, its index and its depth are
// bit for bit those of march_rays (and of the full uniform march).  No temporal
// input.
template <int KMAX, typename MT, typename T>
__device__ __forceinline__ void march_ray_warp(const FuseArgs &a, const int2 *tab, int pixel, int lane) {
    constexpr int NQ = 32 / KMAX;  // samples per step = segments per slab test
    constexpr unsigned SEGMASK = KMAX == 32 ? 0xffffffffu : ((1u << KMAX) - 1u);
    constexpr int SKIP_LONG = T::llong, SKIP_SHORT = T::lshort;
    const int i = pixel % a.Wt, j = pixel / a.Wt;
    const int tk = lane % KMAX, tq = lane / KMAX;
    const bool tview = T::full || tk < a.K;
    const int kk = tview ? tk : 0;
    const size_t plane = (size_t)a.W * a.H;
    // the slab of one ray: every range is a point
    const SlabRays slab = slab_rays(a.xf[kk], i, i, j, j);
    const Ray ray = {slab.axlo, slab.aylo, slab.azlo};
    const float tb0 = slab.b0, tb1 = slab.b1, tb2 = slab.b2;
    const MT *plane_k = reinterpret_cast<const MT *>(a.vb[kk]);
    float S_prev = 0.0f, W_prev = 0.0f, z_prev = 0.0f;
    bool have_prev = false;
    float out = 0.0f;
    int idx = -1;
    int s = 0, cool = 0;
    bool shorter = false;
    while (s < a.D) {
        if (cool == 0 && s < a.D - 1) {
            const int L = shorter ? SKIP_SHORT : SKIP_LONG;
            const int sa = s + tq * L;
            bool f = false;
            if (sa < a.D - 1) {
                const int sb = min(sa + L, a.D - 1);
                const float z0 = __fmaf_rn((float)sa, a.dz, a.zn), z1 = __fmaf_rn((float)sb, a.dz, a.zn);
                f = !tview || slab_view_free<KMAX>(a, tab, tk, slab, z0, z1);
            }
            const unsigned ball = __ballot_sync(0xffffffffu, f);
            int nfree = 0;
#pragma unroll
            for (int g = 0; g < NQ; ++g) {
                if (nfree == g && ((ball >> (g * KMAX)) & SEGMASK) == SEGMASK) ++nfree;
            }
            if (nfree > 0) {
                s = min(s + nfree * L, a.D - 1);
                if (s == a.D - 1) break;
                have_prev = false;
                if (nfree == NQ) {
                    shorter = false;
                    continue;
                }
            }
            if (!shorter && SKIP_SHORT < SKIP_LONG) {
                shorter = true;
                continue;
            }
            shorter = SKIP_SHORT < SKIP_LONG;  // more often than not the surface is still near
            cool = SKIP_COOL;
        }
        // this lane's term of sample s + tq in view tk, as evaluate_sample forms it
        float w = 0.0f, t = 0.0f;
        if (s + tq < a.D && tview) {
            const float zs = __fmaf_rn((float)(s + tq), a.dz, a.zn);
            const float hz = __fmaf_rn(zs, ray.az, tb2);
            const float hx = __fmaf_rn(zs, ray.ax, tb0);
            const float hy = __fmaf_rn(zs, ray.ay, tb1);
            int u, v;
            nearest_pixel(hx, hy, hz, u, v);
            const bool in = hz > 1e-6f && (unsigned)u < (unsigned)a.W && (unsigned)v < (unsigned)a.H &&
                            GVS_IN_BOUNDS((size_t)kk * plane + (size_t)v * a.W + u, (size_t)a.K * plane,
                                          GVS_SITE_FUSE_MAP);
            float2 p = make_float2(0.0f, 0.0f);
            if (in) p = load_map(plane_k + (v * a.W + u));  // v W + u < 2^28
            const float sdf = (p.x - hz) * a.inv_mu;
            w = (in && sdf >= -1.0f) ? p.y : 0.0f;
            t = fminf(sdf, 1.0f);
        }
        // S and W of sample s + tq: its group's terms in view order
        float S = 0.0f, Wsum = 0.0f;
#pragma unroll
        for (int k = 0; k < KMAX; ++k) {
            const float wk = __shfl_sync(0xffffffffu, w, tq * KMAX + k);
            const float tk_ = __shfl_sync(0xffffffffu, t, tq * KMAX + k);
            if (T::full || k < a.K) {
                S = fmaf(wk, tk_, S);
                Wsum += wk;
            }
        }
        // the step's samples in order
        bool done = false;
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            float Sq = __shfl_sync(0xffffffffu, S, q * KMAX);
            const float Wq = __shfl_sync(0xffffffffu, Wsum, q * KMAX);
            if (!done && s < a.D) {
                const float zs = __fmaf_rn((float)s, a.dz, a.zn);
                if (a.normalize && Wq > 0.0f) Sq = Sq / Wq;
                if (have_prev && W_prev > 0.0f && Wq > 0.0f && S_prev > 0.0f && Sq <= 0.0f) {
                    const float tt = S_prev / (S_prev - Sq);
                    out = z_prev + (zs - z_prev) * tt;
                    idx = s - 1;
                    done = true;
                }
                S_prev = Sq;
                W_prev = Wq;
                z_prev = zs;
                have_prev = true;
                ++s;
                if (cool > 0) --cool;
            }
        }
        if (done) break;
    }
    if (lane == 0) {
        const size_t o = (size_t)j * a.Wt + i;
        a.fused[o] = out;
        if (a.crossing) a.crossing[o] = (int16_t)idx;
    }
}

template <int KMAX, typename MT, typename T, bool TMP = false>
__device__ __forceinline__ void march_bundle(const FuseArgs &a, const int2 *tab, int bundle, int lane) {
    if constexpr (T::warp) {
        static_assert(!TMP, "the warp-per-ray march takes no temporal input");
        march_ray_warp<KMAX, MT, T>(a, tab, bundle, lane);
    } else {
        march_rays<KMAX, MT, T, TMP>(a, tab, bundle, lane);
    }
}

// Calls F<Tile_i>::run(...) for the variant, with the full form of the tile
// when the call has exactly KMAX views.  The 8- and 16-view kernels (5 to 16 views)
// have every tile; up to 4 views the two plain ones (0 and 3) are built, for 17 to
// 32 views the default and the warp-per-ray one (fewer instantiations to build).
template <int KMAX, typename MT, template <int, typename, typename> class F, typename T, typename... Args>
void full_or_not(int K, Args... args) {
    if (K == KMAX) F<KMAX, MT, typename FullTile<T>::type>::run(args...);
    else F<KMAX, MT, T>::run(args...);
}

template <int KMAX, typename MT, template <int, typename, typename> class F, typename... Args>
void by_variant(int K, int variant, Args... args) {
    if constexpr (KMAX >= 8) {  // the warp-per-ray mapping: 8, 16 and 32-view kernels
        if (variant == 6) {
            full_or_not<KMAX, MT, F, Tile6>(K, args...);
            return;
        }
    }
    if (KMAX == 8 || KMAX == 16) {
        switch (variant) {
            case 1: full_or_not<KMAX, MT, F, Tile1>(K, args...); return;
            case 2: full_or_not<KMAX, MT, F, Tile2>(K, args...); return;
            case 3: full_or_not<KMAX, MT, F, Tile3>(K, args...); return;
            case 4: full_or_not<KMAX, MT, F, Tile4>(K, args...); return;
            case 5: full_or_not<KMAX, MT, F, Tile5>(K, args...); return;
            default: break;
        }
    }
    if (KMAX == 4 && variant == 3) {
        full_or_not<KMAX, MT, F, Tile3>(K, args...);
        return;
    }
    full_or_not<KMAX, MT, F, Tile0>(K, args...);
}

// View counts below 8 that are not a power of two: kernels for exactly K views (4 x 8
// bundles).  A slab test takes 32 / K segments of K lanes, and no view has a guard:
// 5 x 961x541 63 -> 50 us, 7 x 720p arc 109 -> 98 (9 blocks per SM; 12: 51 and 99).
template <typename MT, template <int, typename, typename> class F, typename... Args>
bool by_exact_k(int K, int variant, Args... args) {
    if (variant != 3) return false;
    using T = typename FullTile<Tile3>::type;
    switch (K) {
        case 2: F<2, MT, T>::run(args...); return true;
        case 3: F<3, MT, T>::run(args...); return true;
        case 5: F<5, MT, T>::run(args...); return true;
        case 6: F<6, MT, T>::run(args...); return true;
        case 7: F<7, MT, T>::run(args...); return true;
        default: return false;
    }
}

template <template <int, typename, typename> class F, typename... Args>
void by_kmax(int K, int map_dtype, int variant, Args... args) {
    if (map_dtype == GVS_F16) {
        if (by_exact_k<__half2, F>(K, variant, args...)) return;
        if (K <= 4) by_variant<4, __half2, F>(K, variant, args...);
        else if (K <= 8) by_variant<8, __half2, F>(K, variant, args...);
        else if (K <= 16) by_variant<16, __half2, F>(K, variant, args...);
        else by_variant<32, __half2, F>(K, variant, args...);
    } else {
        if (by_exact_k<float2, F>(K, variant, args...)) return;
        if (K <= 4) by_variant<4, float2, F>(K, variant, args...);
        else if (K <= 8) by_variant<8, float2, F>(K, variant, args...);
        else if (K <= 16) by_variant<16, float2, F>(K, variant, args...);
        else by_variant<32, float2, F>(K, variant, args...);
    }
}

// The same for kernels built with the default variant's tiles only (variant 3: the 4 x 8 one).
template <int KMAX, typename MT, template <int, typename, typename> class F, typename... Args>
void by_shape(int K, int variant, Args... args) {
    if (KMAX <= 8 && variant == 3) full_or_not<KMAX, MT, F, Tile3>(K, args...);
    else full_or_not<KMAX, MT, F, Tile0>(K, args...);
}

template <template <int, typename, typename> class F, typename... Args>
void by_kmax_tile0(int K, int map_dtype, int variant, Args... args) {
    if (map_dtype != GVS_F16 && by_exact_k<float2, F>(K, variant, args...)) return;
    if (map_dtype == GVS_F16) {
        if (K <= 4) by_shape<4, __half2, F>(K, variant, args...);
        else if (K <= 8) by_shape<8, __half2, F>(K, variant, args...);
        else if (K <= 16) by_shape<16, __half2, F>(K, variant, args...);
        else by_shape<32, __half2, F>(K, variant, args...);
    } else {
        if (K <= 4) by_shape<4, float2, F>(K, variant, args...);
        else if (K <= 8) by_shape<8, float2, F>(K, variant, args...);
        else if (K <= 16) by_shape<16, float2, F>(K, variant, args...);
        else by_shape<32, float2, F>(K, variant, args...);
    }
}

}  // namespace
}  // namespace gvs
