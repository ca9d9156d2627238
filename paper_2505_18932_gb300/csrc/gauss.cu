// Pixel-sized Gaussian forward render (Sec. 3.1, Supplement A.3), each input
// view separately, with the rasterisation rules of 3D Gaussian splatting
// (Kerbl et al. 2023) restated for isotropic, fully opaque Gaussians:
//   prep   : one thread per source pixel.  Splat contract for the mean
//            (x, y) and depth z; EWA covariance
//              Sigma = (scale rho)^2 [[1 + a^2, q a b], [q a b, q^2 (1 + b^2)]] + 0.3 I
//            (rho = f (d / z), a = (x - cx) / fx, b = (y - cy) / fy, q = fy / fx);
//            radius r = min(ceil(3 sqrt(lambda_max)), max_radius), narrowed
//            to where alpha can reach 1/255 (see GaussRec); the record
//            (x, y, z, half-widths | conic, colour); one counter increment per
//            16 x 16 target tile its box meets (warp-aggregated atomics).
//   scan   : exclusive scan of the tile counters -> list offsets.
//   fill   : each Gaussian writes its key (bits(z) << 32 | source index) into
//            the list of every tile it meets.
//   render : one block per tile.  The list is sorted ascending (bitonic, in
//            shared memory up to GS_SORT_CAP keys, longer ones by such chunks
//            and merges), then every thread composites its pixel front to back:
//            alpha = min(0.99, exp(power)), skipped below 1/255, stop before
//            a Gaussian that would take T below 1e-4.
// The radius, the box and the key are integer decisions taken with explicitly
// rounded FP32 operations (no contraction), exactly as the header states them.
#include <cuda_fp16.h>
#include <math.h>

#include "bounds_check.cuh"
#include "gauss_internal.cuh"

namespace gvs {
namespace {

constexpr int GS_THREADS = GS_TILE * GS_TILE;

__device__ __forceinline__ bool valid_depth(float d) { return isfinite(d) && d > 0.0f; }
__device__ __forceinline__ float load_depth(const float *p) { return __ldg(p); }
__device__ __forceinline__ float load_depth(const __half *p) { return __half2float(__ldg(p)); }

// a.w holds the half-widths (hx, hy) of the Gaussian's box as a half2 (bits 0:
// no Gaussian): the contract radius r, tightened to the extent of the ellipse
// where alpha can reach 1/255, sqrt(2 ln 255 Sigma_xx) (and yy), widened by
// 0.1 % + 1e-3 px and rounded up.  A pixel between that box and the contract's
// [x - r, x + r] box has alpha below 1/255 by more than 1 % and is skipped by
// both, so the narrower box changes no result; it only shortens the lists.
struct GaussRec {
    float4 a;  // x, y, z, half2 (hx, hy)
    float4 b;  // -conic_xx / 2, -conic_xy, -conic_yy / 2, colour bits
};

__device__ __forceinline__ float2 half_widths(float w) {
    const unsigned bits = __float_as_uint(w);
    return __half22float2(*reinterpret_cast<const __half2 *>(&bits));
}

// Warp-aggregated atomicAdd of 1 on ctr[t]: lanes adding to the same counter
// share one atomic; each gets a distinct old value.
__device__ __forceinline__ unsigned agg_increment(unsigned *ctr, int t) {
    const unsigned peers = __match_any_sync(__activemask(), t);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(&ctr[t], (unsigned)__popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + __popc(peers & ((1u << lane) - 1u));
}

__device__ __forceinline__ GaussRec *recs(const GaussArgs &g) {
    return reinterpret_cast<GaussRec *>(g.ws + g.L.off_rec);
}

// Target pixels of a record's box: [ceil(x - hx), floor(x + hx)] clipped (and y alike).
__device__ __forceinline__ bool box_of(const GaussArgs &g, float4 a, int &i0, int &i1, int &j0, int &j1) {
    if (__float_as_uint(a.w) == 0u) return false;
    const float2 h = half_widths(a.w);
    float lx = ceilf(__fsub_rn(a.x, h.x)), hx = floorf(__fadd_rn(a.x, h.x));
    float ly = ceilf(__fsub_rn(a.y, h.y)), hy = floorf(__fadd_rn(a.y, h.y));
    if (lx < 0.0f) lx = 0.0f;
    if (ly < 0.0f) ly = 0.0f;
    if (hx > (float)(g.Wt - 1)) hx = (float)(g.Wt - 1);
    if (hy > (float)(g.Ht - 1)) hy = (float)(g.Ht - 1);
    if (!(lx <= hx) || !(ly <= hy)) return false;
    i0 = (int)lx; i1 = (int)hx; j0 = (int)ly; j1 = (int)hy;
    return true;
}

template <typename DT>
__global__ void __launch_bounds__(256) gauss_prep(const GaussArgs g, int k) {
    const int u = blockIdx.x * 32 + threadIdx.x;
    const int v = blockIdx.y * 8 + threadIdx.y;
    if (u >= g.W || v >= g.H) return;
    const int src = v * g.W + u;
    const size_t HW = (size_t)g.W * g.H;
    const float d = load_depth(reinterpret_cast<const DT *>(g.depth) + (size_t)k * HW + src);
    GaussRec r;
    r.a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    r.b = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (valid_depth(d)) {
        const float *A = g.xf[k].M, *c = g.xf[k].b;
        const float fu = (float)u, fv = (float)v;
        const float m0 = __fmaf_rn(A[0], fu, __fmaf_rn(A[1], fv, A[2]));
        const float m1 = __fmaf_rn(A[3], fu, __fmaf_rn(A[4], fv, A[5]));
        const float m2 = __fmaf_rn(A[6], fu, __fmaf_rn(A[7], fv, A[8]));
        const float h0 = __fmaf_rn(d, m0, c[0]);
        const float h1 = __fmaf_rn(d, m1, c[1]);
        const float h2 = __fmaf_rn(d, m2, c[2]);
        if (h2 > 1e-6f) {
            const float x = __fdiv_rn(h0, h2), y = __fdiv_rn(h1, h2);
            const float rho = __fmul_rn(g.f_ratio[k], __fdiv_rn(d, h2));
            const float t = __fmul_rn(g.scale_px, rho);
            const float s2 = __fmul_rn(t, t);
            const float ea = __fdiv_rn(__fsub_rn(x, g.in32[2]), g.in32[0]);
            const float eb = __fdiv_rn(__fsub_rn(y, g.in32[3]), g.in32[1]);
            const float q = g.in32[4];
            const float aa = __fmul_rn(ea, ea), bb = __fmul_rn(eb, eb), ab = __fmul_rn(ea, eb);
            const float qq = __fmul_rn(q, q);
            const float sxx = __fadd_rn(__fmul_rn(s2, __fadd_rn(1.0f, aa)), 0.3f);
            const float sxy = __fmul_rn(s2, __fmul_rn(q, ab));
            const float syy = __fadd_rn(__fmul_rn(s2, __fmul_rn(qq, __fadd_rn(1.0f, bb))), 0.3f);
            const float det = __fsub_rn(__fmul_rn(sxx, syy), __fmul_rn(sxy, sxy));
            if (det > 0.0f) {
                const float mid = __fmul_rn(0.5f, __fadd_rn(sxx, syy));
                float disc = __fsub_rn(__fmul_rn(mid, mid), det);
                disc = disc > 0.1f ? disc : 0.1f;
                const float lam = __fadd_rn(mid, __fsqrt_rn(disc));
                float rr = ceilf(__fmul_rn(3.0f, __fsqrt_rn(lam)));
                if (!(rr <= (float)g.max_radius)) rr = (float)g.max_radius;
                const float ex = fmaf(sqrtf(11.0825271f * sxx), 1.001f, 1e-3f);  // 2 ln 255 = 11.0825271
                const float ey = fmaf(sqrtf(11.0825271f * syy), 1.001f, 1e-3f);
                const __half2 hw = __halves2half2(__float2half_ru(fminf(ex, rr)), __float2half_ru(fminf(ey, rr)));
                r.a = make_float4(x, y, h2, __uint_as_float(*reinterpret_cast<const unsigned *>(&hw)));
                const float inv = 1.0f / det;
                r.b = make_float4(-0.5f * syy * inv, sxy * inv, -0.5f * sxx * inv,
                                  __uint_as_float(__ldg(&g.rgba[(size_t)k * HW + src])));
            }
        }
    }
    int i0, i1, j0, j1;
    const bool any = box_of(g, r.a, i0, i1, j0, j1);
    if (!any) r.a.w = 0.0f;
    recs(g)[src] = r;
    if (any) {
        unsigned *count = reinterpret_cast<unsigned *>(g.ws + g.L.off_count);
        for (int ty = j0 / GS_TILE; ty <= j1 / GS_TILE; ++ty)
            for (int tx = i0 / GS_TILE; tx <= i1 / GS_TILE; ++tx) agg_increment(count, ty * g.L.tiles_x + tx);
    }
}

// Single block: exclusive scan of the tile counters into 64-bit offsets
// (offset[nt] = total); the counters are reset to serve as fill cursors.
__global__ void __launch_bounds__(1024) gauss_scan(GaussArgs g) {
    const int nt = g.L.tiles_x * g.L.tiles_y;
    unsigned *count = reinterpret_cast<unsigned *>(g.ws + g.L.off_count);
    unsigned long long *off = reinterpret_cast<unsigned long long *>(g.ws + g.L.off_offset);
    __shared__ unsigned long long warp_sum[32];
    const int tid = threadIdx.x;
    const int per = (nt + 1023) / 1024;
    const int b0 = tid * per, b1 = min(b0 + per, nt);
    unsigned long long s = 0;
    for (int t = b0; t < b1; ++t) s += count[t];
    // inclusive scan of s over the block
    unsigned long long x = s;
    const int lane = tid & 31, w = tid >> 5;
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, m);
        if (lane >= m) x += y;
    }
    if (lane == 31) warp_sum[w] = x;
    __syncthreads();
    if (w == 0) {
        unsigned long long z = warp_sum[lane];
#pragma unroll
        for (int m = 1; m < 32; m <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, z, m);
            if (lane >= m) z += y;
        }
        warp_sum[lane] = z;
    }
    __syncthreads();
    unsigned long long run = x - s + (w > 0 ? warp_sum[w - 1] : 0ull);
    for (int t = b0; t < b1; ++t) {
        off[t] = run;
        run += count[t];
        count[t] = 0u;
    }
    if (tid == 1023) off[nt] = run;
}

__global__ void __launch_bounds__(256) gauss_fill(const GaussArgs g) {
    const int u = blockIdx.x * 32 + threadIdx.x;
    const int v = blockIdx.y * 8 + threadIdx.y;
    if (u >= g.W || v >= g.H) return;
    const int src = v * g.W + u;
    const float4 a = recs(g)[src].a;
    int i0, i1, j0, j1;
    if (!box_of(g, a, i0, i1, j0, j1)) return;
    unsigned *cursor = reinterpret_cast<unsigned *>(g.ws + g.L.off_count);
    const unsigned long long *off = reinterpret_cast<const unsigned long long *>(g.ws + g.L.off_offset);
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(g.ws + g.L.off_keys);
    const unsigned long long key = ((unsigned long long)__float_as_uint(a.z) << 32) | (unsigned)src;
    const int tx0 = i0 / GS_TILE, tx1 = i1 / GS_TILE, ty0 = j0 / GS_TILE, ty1 = j1 / GS_TILE;
    if (__all_sync(__activemask(), tx1 - tx0 <= 1 && ty1 - ty0 <= 1)) {
        // the usual boxes: at most 2 x 2 tiles, whose counters answer together (4 views at 720p:
        // 57 -> 52 us).  A warp with a larger box takes all of its boxes tile by tile, as going both
        // ways costs more than either (1 view of 720p, Gaussians of 4 pixels: 39 us so, 34 now).
        unsigned base[4], peers[4];
        unsigned long long first[4];
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int tx = tx0 + (e & 1), ty = ty0 + (e >> 1);
            peers[e] = 0u;
            if (tx <= tx1 && ty <= ty1) {
                const int t = ty * g.L.tiles_x + tx;
                peers[e] = __match_any_sync(__activemask(), t);
                base[e] = 0u;
                first[e] = off[t];
                if (lane == __ffs(peers[e]) - 1) base[e] = atomicAdd(&cursor[t], (unsigned)__popc(peers[e]));
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (peers[e]) {
                const unsigned b = __shfl_sync(peers[e], base[e], __ffs(peers[e]) - 1);
                const unsigned long long pos = first[e] + b + __popc(peers[e] & ((1u << lane) - 1u));
                if (GVS_IN_BOUNDS(pos, g.L.n_keys, GVS_SITE_GAUSS_KEY)) keys[pos] = key;
            }
        }
        return;
    }
    for (int ty = ty0; ty <= ty1; ++ty)
        for (int tx = tx0; tx <= tx1; ++tx) {
            const int t = ty * g.L.tiles_x + tx;
            const unsigned long long pos = off[t] + agg_increment(cursor, t);
            if (GVS_IN_BOUNDS(pos, g.L.n_keys, GVS_SITE_GAUSS_KEY)) keys[pos] = key;
        }
}

// Ascending bitonic sort of key[0, n) by the block; positions n.. act as +inf
// padding up to the next power of two and are never touched (every compare
// puts the smaller key at the lower index).
// Pair i of a step lies, for strides up to 32, within the 64 keys at 64 (i / 32), which
// the same warp handles in each of those steps: they only need the warp in step, and
// the block waits where a longer stride comes before or after (6 of the 45 steps of 512 keys).
__device__ void block_sort(unsigned long long *key, int n) {
    int N = 1, lg = 0;
    while (N < n) { N <<= 1; ++lg; }
    for (int lk = 1; lk <= lg; ++lk) {
        const int hk = 1 << (lk - 1);
        if (hk > 32) __syncthreads();
        // first step of the merge: compare mirrored positions of each block of 2 hk
        for (int i = threadIdx.x; i < N / 2; i += blockDim.x) {
            const int blk = i >> (lk - 1), p = i & (hk - 1);
            const int x = (blk << lk) + p, y = (blk << lk) + (2 * hk - 1 - p);
            if (y < n) {
                const unsigned long long kx = key[x], ky = key[y];
                if (kx > ky) { key[x] = ky; key[y] = kx; }
            }
        }
        if (hk > 32) __syncthreads();
        else __syncwarp();
        for (int lj = lk - 2; lj >= 0; --lj) {
            const int j = 1 << lj;
            for (int i = threadIdx.x; i < N / 2; i += blockDim.x) {
                const int x = ((i >> lj) << (lj + 1)) + (i & (j - 1)), y = x + j;
                if (y < n) {
                    const unsigned long long kx = key[x], ky = key[y];
                    if (kx > ky) { key[x] = ky; key[y] = kx; }
                }
            }
            if (j > 32) __syncthreads();
            else __syncwarp();
        }
    }
    __syncthreads();
}

// The same for n <= 2 GS_THREADS (the usual list has 441): one pair per thread and step and
// every stride a constant, about half the instructions a step.  4 views at 720p: render
// 612 -> 519 us.
__device__ __forceinline__ void block_sort_small(unsigned long long *key, int n) {
    const int i = threadIdx.x;
    const auto step = [&](int x, int y) {
        if (y < n) {
            const unsigned long long kx = key[x], ky = key[y];
            if (kx > ky) { key[x] = ky; key[y] = kx; }
        }
    };
    static_assert(GS_THREADS == 256, "2^9 keys, one pair per thread");
#pragma unroll
    for (int lk = 1; lk <= 9; ++lk) {
        const int hk = 1 << (lk - 1);
        if (hk >= n) break;  // sorted (the whole block leaves together)
        if (hk > 32) __syncthreads();
        const int x = i + (i & ~(hk - 1));  // a 0 bit inserted into i at hk
        step(x, x ^ (2 * hk - 1));
        if (hk > 32) __syncthreads();
        else __syncwarp();
#pragma unroll
        for (int lj = lk - 2; lj >= 0; --lj) {
            const int j = 1 << lj;
            const int xj = i + (i & ~(j - 1));
            step(xj, xj + j);
            if (j > 32) __syncthreads();
            else __syncwarp();
        }
    }
    __syncthreads();
}

// A list longer than the shared array (a target much coarser than the view), in place in
// global memory: chunks of GS_SORT_CAP keys are sorted in shared memory, and every merge
// of longer runs takes only its strides of a chunk or more in global memory; the shorter ones
// are taken chunk by chunk in shared memory again.  4 views of 1280x720 into 320x180 (about 5000
// keys a tile) 3.34 -> 1.82 ms, into 160x90 12.1 -> 6.3.
__device__ void block_sort_long(unsigned long long *key, unsigned long long *chunk, int n) {
    constexpr int LC = 11;
    static_assert(GS_SORT_CAP == 1 << LC, "a chunk is a power of two");
    const int chunks = (n + GS_SORT_CAP - 1) / GS_SORT_CAP;
    const auto load = [&](int c) {
        for (int e = threadIdx.x; e < GS_SORT_CAP; e += GS_THREADS) {
            const int q = c * GS_SORT_CAP + e;
            chunk[e] = q < n ? key[q] : ~0ull;
        }
        __syncthreads();
    };
    const auto store = [&](int c) {
        __syncthreads();
        for (int e = threadIdx.x; e < GS_SORT_CAP; e += GS_THREADS) {
            const int q = c * GS_SORT_CAP + e;
            if (q < n) key[q] = chunk[e];
        }
        __syncthreads();
    };
    for (int c = 0; c < chunks; ++c) {
        load(c);
        block_sort(chunk, min(GS_SORT_CAP, n - c * GS_SORT_CAP));
        store(c);
    }
    int lg = LC;
    while ((1 << lg) < n) ++lg;
    const auto order = [&](unsigned long long *k, int x, int y) {
        const unsigned long long kx = k[x], ky = k[y];
        if (kx > ky) { k[x] = ky; k[y] = kx; }
    };
    for (int lk = LC + 1; lk <= lg; ++lk) {
        const int hk = 1 << (lk - 1), pairs = 1 << (lg - 1);
        for (int i = threadIdx.x; i < pairs; i += GS_THREADS) {
            const int x = i + (i & ~(hk - 1)), y = x ^ (2 * hk - 1);  // mirrored positions
            if (y < n) order(key, x, y);
        }
        __syncthreads();
        for (int lj = lk - 2; lj >= LC; --lj) {
            const int j = 1 << lj;
            for (int i = threadIdx.x; i < pairs; i += GS_THREADS) {
                const int x = i + (i & ~(j - 1));
                if (x + j < n) order(key, x, x + j);
            }
            __syncthreads();
        }
        for (int c = 0; c < chunks; ++c) {
            load(c);
            for (int lj = LC - 1; lj >= 0; --lj) {
                const int j = 1 << lj;
                for (int i = threadIdx.x; i < GS_SORT_CAP / 2; i += GS_THREADS) {
                    const int x = i + (i & ~(j - 1));
                    order(chunk, x, x + j);
                }
                if (j > 32) __syncthreads();
                else __syncwarp();
            }
            store(c);
        }
    }
}

// Transposes a 32 x 32 bit matrix held one row per lane: afterwards bit q of lane p is
// what bit p of lane q was.  Five exchanges of half-blocks.
__device__ __forceinline__ unsigned transpose_bits(unsigned x, int lane) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        const unsigned low = m == 16 ? 0x0000ffffu : m == 8 ? 0x00ff00ffu : m == 4 ? 0x0f0f0f0fu
                                     : m == 2 ? 0x33333333u : 0x55555555u;  // the low half of each block
        const unsigned y = __shfl_xor_sync(0xffffffffu, x, m);
        x = (lane & m) ? ((x & ~low) | ((y >> m) & low)) : ((x & low) | ((y << m) & ~low));
    }
    return x;
}

// The set bits lo .. hi of a 16-bit mask, clipped to the tile (0: none).
__device__ __forceinline__ unsigned span_mask(float lo, float hi) {
    const int l = (int)fmaxf(lo, 0.0f), h = (int)fminf(hi, (float)(GS_TILE - 1));
    return l <= h && hi >= 0.0f ? ((2u << h) - 1u) & ~((1u << l) - 1u) : 0u;
}

// Threads of a block: 8 warps, each an 8 x 4 rectangle of the 16 x 16 tile
// (2 across, 4 down), one pixel per lane.  A pixel-sized Gaussian meets about 25 of the
// tile's 256 pixels, so a lane must not look at every one: each Gaussian of a batch of
// 256 sorted ones gets a mask of the tile's columns and one of its rows it covers, and a
// warp turns 32 of them at a time (one per lane, the mask of its rectangle's pixels) into
// one 32-bit word per pixel of the Gaussians that cover it.  Every lane then walks the
// set bits of its own words, in order.  (Walking, per warp, the Gaussians that meet its
// rectangle, 117 of them for 25 that count, and a barrier after each of the sort's 45
// steps, took 245 us a view at 720p; this takes 153.)
__global__ void __launch_bounds__(GS_THREADS) gauss_render(const GaussArgs g, int k) {
    constexpr int WORDS = GS_THREADS / 32;
    __shared__ unsigned long long skeys[GS_SORT_CAP];
    __shared__ float4 sa[GS_THREADS], sb[GS_THREADS];  // (x, y, z, colour), (conic)
    __shared__ unsigned scover[GS_THREADS];            // columns | rows << 16 of the tile
    __shared__ unsigned sword[GS_THREADS / 32][WORDS][32];
    const int t = blockIdx.y * g.L.tiles_x + blockIdx.x;
    const unsigned long long *off = reinterpret_cast<const unsigned long long *>(g.ws + g.L.off_offset);
    unsigned long long *gkeys = reinterpret_cast<unsigned long long *>(g.ws + g.L.off_keys) + off[t];
    const int n = (int)(off[t + 1] - off[t]);
    unsigned long long *keys = gkeys;
    if (n <= GS_SORT_CAP) {
        for (int e = threadIdx.x; e < n; e += GS_THREADS) skeys[e] = gkeys[e];
        keys = skeys;
    }
    __syncthreads();
    if (n <= 2 * GS_THREADS) block_sort_small(skeys, n);
    else if (n <= GS_SORT_CAP) block_sort(skeys, n);
    else block_sort_long(gkeys, skeys, n);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cx = (warp & 1) * 8, cy = (warp >> 1) * 4;  // the warp's rectangle within the tile
    const int i = blockIdx.x * GS_TILE + cx + (lane & 7);
    const int j = blockIdx.y * GS_TILE + cy + (lane >> 3);
    const bool inside = i < g.Wt && j < g.Ht;
    const float tx0 = (float)(blockIdx.x * GS_TILE), ty0 = (float)(blockIdx.y * GS_TILE);
    const float fi = (float)i, fj = (float)j;
    bool done = !inside;
    float T = 1.0f, cr = 0.0f, cg = 0.0f, cb = 0.0f, zs = 0.0f, ws = 0.0f;
    const GaussRec *rec = recs(g);
    for (int b0 = 0; b0 < n; b0 += GS_THREADS) {
        if (__syncthreads_count(!done) == 0) break;  // also orders the reuse of sa / sb / scover
        const int e = b0 + threadIdx.x;
        unsigned cover = 0;
        if (e < n) {
            unsigned src = (unsigned)(keys[e] & 0xffffffffull);
            if (!GVS_IN_BOUNDS(src, (size_t)g.W * g.H, GVS_SITE_GAUSS_REC)) src = 0;
            const GaussRec r = rec[src];
            sa[threadIdx.x] = make_float4(r.a.x, r.a.y, r.a.z, r.b.w);
            sb[threadIdx.x] = r.b;
            const float2 h = half_widths(r.a.w);
            cover = span_mask(ceilf(__fsub_rn(r.a.x, h.x)) - tx0, floorf(__fadd_rn(r.a.x, h.x)) - tx0) |
                    (span_mask(ceilf(__fsub_rn(r.a.y, h.y)) - ty0, floorf(__fadd_rn(r.a.y, h.y)) - ty0) << 16);
        }
        scover[threadIdx.x] = cover;
        __syncthreads();
        const int words = (min(GS_THREADS, n - b0) + 31) / 32;
        int nw = 0;                // this pixel's non-empty words,
        unsigned which = 0;        // and which ones they are (4 bits each)
        for (int w = 0; w < words; ++w) {
            const unsigned c = scover[w * 32 + lane];
            const unsigned cols = (c >> cx) & 0xffu, rows = (c >> (16 + cy)) & 0xfu;
            // bit 8 r + c of the rectangle: the columns once per covered row
            unsigned m = cols * ((rows & 1u) | ((rows & 2u) << 7) | ((rows & 4u) << 14) | ((rows & 8u) << 21));
            if (!__any_sync(0xffffffffu, m != 0u)) continue;
            m = transpose_bits(m, lane);
            if (m != 0u) {
                sword[warp][nw][lane] = m;
                which |= (unsigned)w << (4 * nw);
                ++nw;
            }
        }
        unsigned cur = 0;
        const unsigned *word = &sword[warp][0][lane];
        int q0 = 0;
        while (!done) {
            if (cur == 0u) {
                if (nw == 0) break;
                --nw;
                cur = *word;
                word += 32;
                q0 = (int)(which & 15u) * 32;
                which >>= 4;
            }
            const int q = q0 + __ffs((int)cur) - 1;
            cur &= cur - 1u;
            const float4 a = sa[q];
            const float4 c = sb[q];
            const float dx = a.x - fi, dy = a.y - fj;
            const float power = fmaf(dx, fmaf(c.x, dx, c.y * dy), c.z * dy * dy);
            // exp(-5.6) < 1/255 whatever the rounding of the exponential: skip without it
            const float al = fminf(0.99f, __expf(power));
            const bool use = !(power > 0.0f || power < -5.6f) && !(al < 1.0f / 255.0f);
            const float Tn = T * (1.0f - al);
            done = use && Tn < 1e-4f;
            if (use && !done) {
                const float wgt = __fmul_rn(al, T);
                const unsigned col = __float_as_uint(a.w);
                cr = fmaf((float)(col & 0xffu) * (1.0f / 255.0f), wgt, cr);
                cg = fmaf((float)((col >> 8) & 0xffu) * (1.0f / 255.0f), wgt, cg);
                cb = fmaf((float)((col >> 16) & 0xffu) * (1.0f / 255.0f), wgt, cb);
                zs = fmaf(a.z, wgt, zs);
                ws = __fadd_rn(ws, wgt);
                T = Tn;
            }
        }
    }
    if (inside) {
        const size_t o = (size_t)k * g.Wt * g.Ht + (size_t)j * g.Wt + i;
        g.color[o] = make_float4(cr, cg, cb, 1.0f - T);
        g.depth_out[o] = ws > 0.0f ? zs / ws : 0.0f;
    }
}

}  // namespace

cudaError_t launch_gauss_splat(const GaussArgs &a, int K, cudaStream_t st) {
    const GaussLayout &L = a.L;
    const dim3 pg((unsigned)((a.W + 31) / 32), (unsigned)((a.H + 7) / 8)), pb(32, 8);
    const dim3 rg((unsigned)L.tiles_x, (unsigned)L.tiles_y);
    const size_t nt = (size_t)L.tiles_x * L.tiles_y;
    for (int k = 0; k < K; ++k) {
        cudaError_t e = cudaMemsetAsync(a.ws + L.off_count, 0, nt * 4, st);
        if (e != cudaSuccess) return e;
        if (a.depth_dtype == GVS_F16) gauss_prep<__half><<<pg, pb, 0, st>>>(a, k);
        else gauss_prep<float><<<pg, pb, 0, st>>>(a, k);
        gauss_scan<<<1, 1024, 0, st>>>(a);
        gauss_fill<<<pg, pb, 0, st>>>(a);
        gauss_render<<<rg, GS_THREADS, 0, st>>>(a, k);
    }
    return cudaGetLastError();
}

GVS_BOUNDS_TAKE_FN(bounds_take_gauss)

}  // namespace gvs
