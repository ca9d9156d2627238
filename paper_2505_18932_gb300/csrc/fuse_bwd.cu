// Adjoint of the image-based TSDF fusion (Supplement A.1, Eq. 3 differentiated).
#include "fuse_march.cuh"

namespace gvs {
namespace {

// ---------------------------------------------------------------------------
// Adjoint of the fused depth (normalize = 0), in two passes.
//
// D = z_s + dz S_s / (S_s - S_{s+1}) depends on the inputs only through the
// two bracketing samples.  For a view contributing at one of them with
// clamped distance c, weight omega and signed distance sdf at input pixel q:
//   dD/dd(q) += g_S omega [-1 < sdf < 1] / mu                 (the clamp)
//   dD/dd(n) += g_S c domega(q)/dd(n)   for q's window entries n (the weight)
// with g_S = dD/dS of that sample.  The weight's derivative is linear in
// g_S c, so pass 1 (a lane per target pixel and view) accumulates, per sampled
// input pixel q, A(q) = sum g_S c and B(q) = sum g_S omega [...] / mu with one
// float2 atomic per (sample, view); pass 2 (per input pixel x)
// applies domega/dnu and the window:
//   grad(x) = B(x) + P(x) sum_{entries n of x} 2 (d_x - d_n) [|d_x - d_n| < mu]
//           + sum_{c whose window holds x, with multiplicity}
//                 P(c) (-2) (d_c - d_x) [|d_c - d_x| < mu]
// where P(c) = A(c) domega/dnu(c) (0 when the weight is saturated or c is
// invalid).  With omega = w_c (nu / w^2)^(-1/2) unsaturated, domega/dnu =
// -0.5 omega / nu = -0.5 omega^3 / (w^2 w_c^2), so a float2 map gives P(c)
// from its stored omega without re-summing the window; for a half2 map (omega
// rounded to half) nu is re-summed from the depths.  Nothing of size D x H x W
// is stored; the bracketing samples are recomputed with the forward's operations in
// the forward's order (evaluate_sample), so S is the same bits.
// ---------------------------------------------------------------------------

// Pass 1.  Only target pixels with a crossing (and a non-zero upstream
// gradient) have work, about a third of them on the 8 x 1080p frame; so each
// block of 128 threads first lists the pixels with work among its 16 x 32 tile
// (in raster order, through a block-wide prefix count of warp ballots) and then
// deals the list out, a group of KMAX lanes to a pixel and a lane to a view: the lane
// keeps its view's coefficients, gathers the map at both samples, adds the
// group's terms to S_s and S_{s+1} in view order (the forward's own order and
// operations, so the same bits) and, with its terms still in registers, issues its two
// atomics.  8 x 1080p: 121 -> 107 us against a thread to a pixel, which recomputed every
// term after the sums; resident blocks 8 (64 registers), 12, 16: 107, 115, 112 us.  The list
// carries each pixel's sample and gradient, one load less in the chain: 96 us.
constexpr int BS_TX = 16, BS_TY = 32, BS_THREADS = 128, BS_BLOCKS = 8;
template <int KMAX, typename MT>
__global__ void __launch_bounds__(BS_THREADS, BS_BLOCKS) fuse_bwd_scatter(const __grid_constant__ FuseArgs a,
                                                                         const int16_t *__restrict__ crossing,
                                                                         const float *__restrict__ grad_fused,
                                                                         float2 *__restrict__ acc) {
    constexpr int PER = BS_TX * BS_TY / BS_THREADS;  // pixels per thread in the listing pass
    constexpr int GROUPS = BS_THREADS / KMAX;        // pixels at a time
    __shared__ int2 s_list[BS_TX * BS_TY];  // (tile-local raster index | sample << 16, upstream gradient)
    __shared__ int s_warp[BS_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int base = 0;
#pragma unroll
    for (int r = 0; r < PER; ++r) {
        const int e = r * BS_THREADS + tid;  // tile-local raster index
        const int i = blockIdx.x * BS_TX + (e % BS_TX), j = blockIdx.y * BS_TY + (e / BS_TX);
        int s = -1;
        float G = 0.0f;
        if (i < a.Wt && j < a.Ht) {
            const size_t o = (size_t)j * a.Wt + i;
            s = crossing[o];
            G = grad_fused[o];
        }
        const bool work = s >= 0 && s + 1 < a.D && G != 0.0f;
        const unsigned ball = __ballot_sync(0xffffffffu, work);
        if (lane == 0) s_warp[warp] = __popc(ball);
        __syncthreads();
        int before = base;
        for (int w = 0; w < warp; ++w) before += s_warp[w];
        int total = base;
        for (int w = 0; w < BS_THREADS / 32; ++w) total += s_warp[w];
        if (work)  // a sample index has 15 bits, a tile index 9
            s_list[before + __popc(ball & ((1u << lane) - 1u))] = make_int2(e | (s << 16), __float_as_int(G));
        __syncthreads();  // s_warp is rewritten by the next round
        base = total;
    }
    const int k = tid % KMAX, first = lane - lane % KMAX;  // this lane's view; its group's first lane
    const ViewXform xf = a.xf[k < a.K ? k : 0];
    const size_t plane = (size_t)a.W * a.H;
    const MT *map = reinterpret_cast<const MT *>(a.dw) + (k < a.K ? (size_t)k * plane : 0);
    float2 *acc_k = acc + (k < a.K ? (size_t)k * plane : 0);
    for (int q0 = warp * (32 / KMAX); q0 < base; q0 += GROUPS) {  // the same for the whole warp
        const int q = q0 + lane / KMAX;
        const bool on = q < base;
        const int2 l = s_list[on ? q : q0];
        const int e = l.x & 0xffff, s = l.x >> 16;
        const float G = __int_as_float(l.y);
        const int i = blockIdx.x * BS_TX + (e % BS_TX), j = blockIdx.y * BS_TY + (e / BS_TX);
        const float fi = (float)i, fj = (float)j;
        const float ax = __fmaf_rn(xf.M[0], fi, __fmaf_rn(xf.M[1], fj, xf.M[2]));
        const float ay = __fmaf_rn(xf.M[3], fi, __fmaf_rn(xf.M[4], fj, xf.M[5]));
        const float az = __fmaf_rn(xf.M[6], fi, __fmaf_rn(xf.M[7], fj, xf.M[8]));
        float zs[2], w[2], c[2], inband[2];
        int at[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            zs[t] = __fmaf_rn((float)(s + t), a.dz, a.zn);
            const float hz = __fmaf_rn(zs[t], az, xf.b[2]);
            const float hx = __fmaf_rn(zs[t], ax, xf.b[0]);
            const float hy = __fmaf_rn(zs[t], ay, xf.b[1]);
            int u, v;
            nearest_pixel(hx, hy, hz, u, v);
            const bool in = k < a.K && hz > 1e-6f && (unsigned)u < (unsigned)a.W && (unsigned)v < (unsigned)a.H &&
                            GVS_IN_BOUNDS((size_t)k * plane + (size_t)v * a.W + u, (size_t)a.K * plane,
                                          GVS_SITE_FUSE_MAP);
            at[t] = in ? v * a.W + u : 0;
            float2 p = make_float2(0.0f, 0.0f);
            if (in) p = load_map(map + at[t]);
            const float sdf = (p.x - hz) * a.inv_mu;
            w[t] = (in && sdf >= -1.0f) ? p.y : 0.0f;
            c[t] = w[t] != 0.0f ? fminf(sdf, 1.0f) : 0.0f;
            inband[t] = (sdf > -1.0f && sdf < 1.0f) ? a.inv_mu : 0.0f;
        }
        float S0 = 0.0f, S1 = 0.0f;
#pragma unroll
        for (int g = 0; g < KMAX; ++g) {
            S0 = fmaf(__shfl_sync(0xffffffffu, w[0], first + g), __shfl_sync(0xffffffffu, c[0], first + g), S0);
            S1 = fmaf(__shfl_sync(0xffffffffu, w[1], first + g), __shfl_sync(0xffffffffu, c[1], first + g), S1);
        }
        const float den = (S0 - S1) * (S0 - S1);
        const float gS[2] = {G * (zs[1] - zs[0]) * (-S1) / den, G * (zs[1] - zs[0]) * S0 / den};
#pragma unroll
        for (int t = 0; t < 2; ++t)
            if (on && w[t] > 0.0f)
                atomicAdd(&acc_k[at[t]], make_float2(gS[t] * c[t], gS[t] * w[t] * inband[t]));
    }
}

template <int KMAX, typename MT>
void bwd_scatter_k(const FuseArgs &a, const int16_t *crossing, const float *grad_fused, float2 *acc,
                   cudaStream_t st) {
    const dim3 grid((a.Wt + BS_TX - 1) / BS_TX, (a.Ht + BS_TY - 1) / BS_TY), block(BS_THREADS);
    fuse_bwd_scatter<KMAX, MT><<<grid, block, 0, st>>>(a, crossing, grad_fused, acc);
}

// Entries e in [-R, R] of a clamp-to-edge window centred at c that land on x
// (one axis, image extent n).
__device__ __forceinline__ int window_multiplicity(int c, int x, int n, int R) {
    if (c < 0 || c >= n) return 0;
    if (n == 1) return 2 * R + 1;
    if (x == 0) return max(0, R - c + 1);
    if (x == n - 1) return max(0, c - (n - 1) + R + 1);
    return abs(c - x) <= R ? 1 : 0;
}

#ifndef GVS_GATHER_ROWS
#define GVS_GATHER_ROWS 4
#endif
constexpr int GB_TX = 32;                 // block of 32 x 32 input pixels: 32 x (32 / GB_ROWS) threads,
constexpr int GB_TY = 32;                 // each thread GB_ROWS consecutive rows
constexpr int GB_ROWS = GVS_GATHER_ROWS;
static_assert(GB_TY % GB_ROWS == 0, "the rows split evenly among the thread rows");

// P(c) from A(c) (0 outside the image), the weight omega and the depth d (NaN: invalid).
__device__ __forceinline__ float adjoint_p(float A, float om, float d, float inv_w2, float wconst) {
    return (A != 0.0f && d == d && om < 1.0f) ? A * (-0.5f * om * om * om * (inv_w2 / (wconst * wconst))) : 0.0f;
}

// The same without a stored FP32 weight: nu is summed again from the depth tile dt, whose
// element [0][ox] is the corner of c's window.
template <int R, int DW>
__device__ __forceinline__ float adjoint_p_resum(float A, float d, const float (*dt)[DW], int ox, float mu,
                                                 float wconst, float inv_w2) {
    if (!(A != 0.0f && d == d)) return 0.0f;
    float nu = 0.0f;
    for (int dy = 0; dy <= 2 * R; ++dy)
        for (int dx = 0; dx <= 2 * R; ++dx) {
            const float t = fminf(fabsf(d - dt[dy][ox + dx]), mu);
            nu = fmaf(t, t, nu);
        }
    const float unclamped = nu > 0.0f ? wconst * rsqrtf(nu * inv_w2) : 2.0f;
    return unclamped < 1.0f ? A * (-0.5f * unclamped / nu) : 0.0f;
}

// MAP: depths and weights come from the forward's float2 (d, omega) planes; otherwise from
// `depth`, the weights' nu summed again.
// The shared tile holds (-d, 2 P) of the outputs and an R halo, depths replicated past the
// image's borders (NaN: invalid) and P = 0 there.  For a pixel x off the image's edge rows
// and columns, entry n of its window and the window centre c = n coincide, so its gradient is
// one pass over the tile: (d_x - d_n) (2 P(x) + 2 P(n)) where |d_x - d_n| < mu (false for an
// invalid n or x).  The factor 2 of the square's derivative sits in the tile, exactly.  One
// packed addition gives both factors of a term, the depth test predicates its one FMA, and
// a thread's GB_ROWS outputs share the values of their window rows.  On an edge
// row or column the clamped entries of other windows land on x too: those pixels, and
// only those, add the remaining multiplicity of each window that holds them.  A tile
// whose P are all 0 (no crossing was sampled there, or every weight is saturated) has
// grad = B.  8 x 1080p: 278 -> 159 us, 4 x 640x360: 39.7 -> 18.6 us (from separate depth and P
// tiles, a packed pair's work in two additions, and every block at the border on a
// scalar path of two windows a pixel).
template <int R, typename DT, bool MAP>
__global__ void __launch_bounds__(GB_TX *(GB_TY / GB_ROWS)) fuse_bwd_gather(const DT *__restrict__ depth,
                                                                const float2 *__restrict__ wmap,
                                                                const float2 *__restrict__ acc,
                                                                float *__restrict__ grad, int W, int H, float mu,
                                                                float wconst, float inv_w2) {
    constexpr int DW = GB_TX + 4 * R, DH = GB_TY + 4 * R;   // depths for the re-sum: outputs + 2R halo
    constexpr int PW = GB_TX + 2 * R, PH = GB_TY + 2 * R;   // (-d, 2 P): outputs + R halo
    constexpr int THREADS = GB_TX * (GB_TY / GB_ROWS);
    __shared__ float dt[MAP ? 1 : DH][DW];
    __shared__ float2 ct[PH][PW];
    const int k = blockIdx.z;
    const size_t plane = (size_t)k * W * H;
    const float2 *ak = acc + plane;
    const int bx = blockIdx.x * GB_TX, by = blockIdx.y * GB_TY;
    const int tid = threadIdx.x;
    if (!MAP) {
        for (int e = tid; e < DH * DW; e += THREADS) {
            const int sy = e / DW, sx = e - sy * DW;
            const int gx = min(max(bx - 2 * R + sx, 0), W - 1), gy = min(max(by - 2 * R + sy, 0), H - 1);
            const float d = load_depth(&depth[plane + (size_t)gy * W + gx]);
            dt[sy][sx] = valid_depth(d) ? d : __int_as_float(0x7fc00000);  // NaN marks invalid
        }
        __syncthreads();
    }
    bool any = false;
    constexpr int NL = (PH * PW + THREADS - 1) / THREADS;
#pragma unroll(MAP ? 3 : 1)
    for (int n = 0; n < NL; ++n) {
        const int e = tid + n * THREADS;
        if (e < PH * PW) {
            const int py = e / PW, px = e - py * PW;
            const int cx = bx - R + px, cy = by - R + py;
            const int gx = min(max(cx, 0), W - 1), gy = min(max(cy, 0), H - 1);
            const int o = gy * W + gx;
            const float A = (gx == cx && gy == cy) ? __ldg(&ak[o]).x : 0.0f;
            float d, P;
            if (MAP) {
                const float2 m = __ldg(&wmap[plane + o]);
                d = m.x > 0.0f ? m.x : __int_as_float(0x7fc00000);
                P = adjoint_p(A, m.y, d, inv_w2, wconst);
            } else {
                d = dt[py + R][px + R];
                P = adjoint_p_resum<R, DW>(A, d, dt + py, px, mu, wconst, inv_w2);
            }
            any |= P != 0.0f;
            ct[py][px] = make_float2(-d, 2.0f * P);
        }
    }
    const bool work = __syncthreads_or(any);
    const int lx = tid % GB_TX, x = bx + lx;
    const int ly0 = (tid / GB_TX) * GB_ROWS;  // this thread's GB_ROWS consecutive rows
    if (x >= W || by + ly0 >= H) return;
    float2 own[GB_ROWS];  // (d_x, 2 P(x))
    float g[GB_ROWS];
#pragma unroll
    for (int p = 0; p < GB_ROWS; ++p) g[p] = by + ly0 + p < H ? __ldg(&ak[(size_t)(by + ly0 + p) * W + x]).y : 0.0f;  // B(x)
    if (work) {
#pragma unroll
        for (int p = 0; p < GB_ROWS; ++p) {
            const float2 c = ct[ly0 + p + R][lx + R];
            own[p] = make_float2(-c.x, c.y);
        }
#pragma unroll
        for (int r = 0; r < GB_ROWS + 2 * R; ++r) {
#pragma unroll
            for (int ox = 0; ox <= 2 * R; ++ox) {
                const float2 c = ct[ly0 + r][lx + ox];
#pragma unroll
                for (int p = 0; p < GB_ROWS; ++p) {
                    if (r - p < 0 || r - p > 2 * R) continue;  // a row outside the window
                    const float2 t = __fadd2_rn(own[p], c);    // (d_x - d_n, 2 P(x) + 2 P(n))
                    if (fabsf(t.x) < mu) g[p] = fmaf(t.x, t.y, g[p]);
                }
            }
        }
        if (x == 0 || x == W - 1 || by + ly0 == 0 || by + ly0 + GB_ROWS >= H) {
#pragma unroll 1
            for (int p = 0; p < GB_ROWS; ++p) {
                const int y = by + ly0 + p;
                if (y >= H || !(x == 0 || x == W - 1 || y == 0 || y == H - 1)) continue;
                const float dx = -ct[ly0 + p + R][lx + R].x;
                float more = 0.0f;
                for (int oy = -R; oy <= R; ++oy) {
                    const int my = window_multiplicity(y + oy, y, H, R);
                    for (int ox = -R; ox <= R; ++ox) {
                        const int m = my * window_multiplicity(x + ox, x, W, R);
                        const float2 c = ct[ly0 + p + R + oy][lx + R + ox];
                        const float diff = dx + c.x;
                        if (m > 1 && fabsf(diff) < mu) more = fmaf((float)(m - 1) * c.y, diff, more);
                    }
                }
#pragma unroll
                for (int q = 0; q < GB_ROWS; ++q)
                    if (q == p) g[q] += more;  // (no dynamic index into registers)
            }
        }
    }
#pragma unroll
    for (int p = 0; p < GB_ROWS; ++p)
        if (by + ly0 + p < H) grad[plane + (size_t)(by + ly0 + p) * W + x] = g[p];
}

template <int R, typename DT>
cudaError_t launch_bwd_gather_r(const void *depth, const float2 *wmap, const float2 *acc, float *grad, int K, int W,
                                int H, float mu, float wconst, float inv_w2, cudaStream_t st) {
    dim3 grid((W + GB_TX - 1) / GB_TX, (H + GB_TY - 1) / GB_TY, K);
    constexpr int threads = GB_TX * (GB_TY / GB_ROWS);
    const DT *d = reinterpret_cast<const DT *>(depth);
    if (wmap) fuse_bwd_gather<R, DT, true><<<grid, threads, 0, st>>>(d, wmap, acc, grad, W, H, mu, wconst, inv_w2);
    else fuse_bwd_gather<R, DT, false><<<grid, threads, 0, st>>>(d, wmap, acc, grad, W, H, mu, wconst, inv_w2);
    return cudaGetLastError();
}

template <typename DT>
cudaError_t launch_bwd_gather(const void *depth, const float2 *wmap, const float2 *acc, float *grad, int K, int W,
                              int H, float mu, float wconst, int window, cudaStream_t st) {
    const float inv_w2 = (float)(1.0 / ((double)window * (double)window));
    switch (window / 2) {
        case 0: return launch_bwd_gather_r<0, DT>(depth, wmap, acc, grad, K, W, H, mu, wconst, inv_w2, st);
        case 1: return launch_bwd_gather_r<1, DT>(depth, wmap, acc, grad, K, W, H, mu, wconst, inv_w2, st);
        case 2: return launch_bwd_gather_r<2, DT>(depth, wmap, acc, grad, K, W, H, mu, wconst, inv_w2, st);
        case 3: return launch_bwd_gather_r<3, DT>(depth, wmap, acc, grad, K, W, H, mu, wconst, inv_w2, st);
        case 4: return launch_bwd_gather_r<4, DT>(depth, wmap, acc, grad, K, W, H, mu, wconst, inv_w2, st);
        case 5: return launch_bwd_gather_r<5, DT>(depth, wmap, acc, grad, K, W, H, mu, wconst, inv_w2, st);
        case 6: return launch_bwd_gather_r<6, DT>(depth, wmap, acc, grad, K, W, H, mu, wconst, inv_w2, st);
        case 7: return launch_bwd_gather_r<7, DT>(depth, wmap, acc, grad, K, W, H, mu, wconst, inv_w2, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_fuse_backward(const FuseArgs &a, const void *depth, int depth_dtype, const int16_t *crossing,
                                 const float *grad_fused, float *grad_depths, float2 *acc, float mu, float wconst,
                                 int window, cudaStream_t st) {
    if (a.K == 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(acc, 0, (size_t)a.K * a.W * a.H * sizeof(float2), st);
    if (e != cudaSuccess) return e;
    if (a.map_dtype == GVS_F16) {
        if (a.K <= 4) bwd_scatter_k<4, __half2>(a, crossing, grad_fused, acc, st);
        else if (a.K <= 8) bwd_scatter_k<8, __half2>(a, crossing, grad_fused, acc, st);
        else if (a.K <= 16) bwd_scatter_k<16, __half2>(a, crossing, grad_fused, acc, st);
        else bwd_scatter_k<32, __half2>(a, crossing, grad_fused, acc, st);
    } else {
        if (a.K <= 4) bwd_scatter_k<4, float2>(a, crossing, grad_fused, acc, st);
        else if (a.K <= 8) bwd_scatter_k<8, float2>(a, crossing, grad_fused, acc, st);
        else if (a.K <= 16) bwd_scatter_k<16, float2>(a, crossing, grad_fused, acc, st);
        else bwd_scatter_k<32, float2>(a, crossing, grad_fused, acc, st);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const float2 *wmap = a.map_dtype == GVS_F16 ? nullptr : reinterpret_cast<const float2 *>(a.dw);
    return depth_dtype == GVS_F16
               ? launch_bwd_gather<__half>(depth, wmap, acc, grad_depths, a.K, a.W, a.H, mu, wconst, window, st)
               : launch_bwd_gather<float>(depth, wmap, acc, grad_depths, a.K, a.W, a.H, mu, wconst, window, st);
}

GVS_BOUNDS_TAKE_FN(bounds_take_fuse_bwd)

}  // namespace gvs
