// The paper's own raymarch for the image-based TSDF (Supplement A.1): from
// z_near, advance by 0.8 s until s changes sign, then three bisection steps.
// One lane per target ray, in bundles of a warp that prove free space together; the
// per-view ray coefficients, the sample evaluation, the nearest-pixel contract and the
// slab test are those of the uniform march (fuse_march.cuh).  Every operation that moves the march is an explicitly
// rounded FP32 operation and the weights come from the correctly rounded map,
// so the trajectory, the evaluation count and the depth are reproducible bit
// for bit on the host (see gvs_fuse_depth_sphere in gvs.h).
#include "fuse_march.cuh"
#include "sphere_internal.cuh"

namespace gvs {
namespace {

// evaluate_sample of the uniform march with a branch per view in place of the
// predicated gather: the same S and W.  Used when the call has fewer views than
// KMAX (the per-view guard already splits the code there, and the branches let
// lanes at unrelated depths skip work); with exactly KMAX views the predicated
// form, one block of code over all views, is faster (3.80 against 4.38 ms at
// 8 x 1080p).
template <int KMAX>
__device__ __forceinline__ void sphere_sample(const FuseArgs &a, const Ray (&ray)[KMAX], float zs, float &S,
                                              float &Wsum) {
    const float2 *map = reinterpret_cast<const float2 *>(a.dw);
    const size_t plane = (size_t)a.W * a.H;
    S = 0.0f;
    Wsum = 0.0f;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        if (k < a.K) {
            const float hz = __fmaf_rn(zs, ray[k].az, a.xf[k].b[2]);
            if (hz > 1e-6f) {
                const float hx = __fmaf_rn(zs, ray[k].ax, a.xf[k].b[0]);
                const float hy = __fmaf_rn(zs, ray[k].ay, a.xf[k].b[1]);
                int u, v;
                nearest_pixel(hx, hy, hz, u, v);
                if ((unsigned)u < (unsigned)a.W && (unsigned)v < (unsigned)a.H &&
                    GVS_IN_BOUNDS((size_t)k * plane + (size_t)v * a.W + u, (size_t)a.K * plane, GVS_SITE_FUSE_MAP)) {
                    const float2 p = __ldg(&map[(size_t)k * plane + (size_t)v * a.W + u]);
                    const float sdf = (p.x - hz) * a.inv_mu;
                    if (sdf >= -1.0f) {
                        S = fmaf(p.y, fminf(sdf, 1.0f), S);
                        Wsum += p.y;
                    }
                }
            }
        }
    }
}

template <int KMAX, bool FULL>
__device__ __forceinline__ void sphere_eval(const FuseArgs &a, const Ray (&ray)[KMAX], float z, float &S, float &W) {
    if (FULL) evaluate_sample<KMAX, float2, true>(a, ray, z, S, W);
    else sphere_sample<KMAX>(a, ray, z, S, W);
}

// Steps of 0.8 mu per segment of the free-space test: the long form first, the short one
// where it fails, then SP_COOL + 1 samples of every ray before the next test (4 views at
// 960x540, us: 8 / 2 / 6 98, 8 / 2 / 4 101, 8 / 2 / 2 107, 16 / 2 / 4 99, 8 / 4 / 4 106).
constexpr int SP_LONG = 8, SP_SHORT = 2, SP_COOL = 6;
constexpr int SP_BX = 4, SP_BY = 8, SP_WARPS = 4;  // 8 x 4: 98.7 against 96.8 us

// One warp per 4x8 bundle of target pixels, one ray per lane.  Most samples of the march
// lie in free space, where every view's term is saturated (sdf >= 1) or cut off: there
// S = W, summed alike, so the step is exactly 0.8 mu (also where W = 0) and no crossing
// ends.  The warp proves that for whole stretches of its rays, from the rearmost one on,
// with the uniform march's slab test (lanes = views x segments); a ray inside a proven
// stretch takes its steps, the same rounded additions, without evaluating them.  The last
// sample in the stretch is evaluated: the next one needs its S and W.  The three
// bisections are iterations of the same loop, so that rays which cross at different
// samples do not hold up the rest of the bundle.  4 views at 960x540: 483 -> 114 us (one
// ray of a 32 x 1 strip per thread, every sample evaluated, before).  FULL: the call has exactly KMAX views.
template <int KMAX, bool FULL>
__global__ void __launch_bounds__(32 * SP_WARPS) sphere_kernel(const __grid_constant__ SphereArgs s) {
    __shared__ int2 tab[(kBoundLevels + 1) * KMAX];
    constexpr int NSEG = 32 / KMAX;
    constexpr unsigned SEGMASK = KMAX == 32 ? 0xffffffffu : ((1u << KMAX) - 1u);
    const FuseArgs &a = s.f;
    fill_slab_table<KMAX>(a, tab, threadIdx.x, 32 * SP_WARPS);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int bundle = blockIdx.x * SP_WARPS + (threadIdx.x >> 5);
    const int nbx = (a.Wt + SP_BX - 1) / SP_BX;
    const int i0 = (bundle % nbx) * SP_BX, j0 = (bundle / nbx) * SP_BY;
    if (j0 >= a.Ht) return;  // the whole warp leaves together
    const int i1 = min(i0 + SP_BX - 1, a.Wt - 1), j1 = min(j0 + SP_BY - 1, a.Ht - 1);
    const int i = i0 + (lane % SP_BX), j = j0 + (lane / SP_BX);
    const bool inside = i < a.Wt && j < a.Ht;
    const float fi = (float)min(i, a.Wt - 1), fj = (float)min(j, a.Ht - 1);
    Ray ray[KMAX];
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        if (FULL || k < a.K) {
            const float *M = a.xf[k].M;
            ray[k].ax = __fmaf_rn(M[0], fi, __fmaf_rn(M[1], fj, M[2]));
            ray[k].ay = __fmaf_rn(M[3], fi, __fmaf_rn(M[4], fj, M[5]));
            ray[k].az = __fmaf_rn(M[6], fi, __fmaf_rn(M[7], fj, M[8]));
        }
    }
    const int tk = lane % KMAX, tseg = lane / KMAX;  // this lane's role in the tests
    const bool tview = tk < a.K;
    const SlabRays slab = slab_rays(a.xf[tview ? tk : 0], i0, i1, j0, j1);
    float z = a.zn, z_prev = 0.0f, S_prev = 0.0f, W_prev = 0.0f, out = 0.0f;
    float lo = 0.0f, hi = 0.0f;
    bool have_prev = false;
    int bisect = 0;  // bisections left
    int it = 0, extra = 0;
    int cool = 0;
    bool shorter = false;
    for (;;) {
        const bool marching = inside && bisect == 0 && it < s.max_steps && z <= s.zf;
        if (!__any_sync(0xffffffffu, marching || bisect > 0)) break;
        if (cool == 0) {
            // the rearmost marching ray; depths are positive, so they order like their bits
            const float zmin = __uint_as_float(__reduce_min_sync(0xffffffffu, marching ? __float_as_uint(z) : 0x7f800000u));
            if (zmin < kInf) {
                const float L = (float)(shorter ? SP_SHORT : SP_LONG) * s.c08mu;
                const float z0 = __fmaf_rn((float)tseg, L, zmin), z1 = __fmaf_rn((float)(tseg + 1), L, zmin);
                const bool f = !tview || z0 > s.zf || (z0 < z1 && z1 < 1e30f && slab_view_free<KMAX, true>(a, tab, tk, slab, z0, z1));
                const unsigned ball = __ballot_sync(0xffffffffu, f);
                int nfree = 0;
#pragma unroll
                for (int g = 0; g < NSEG; ++g) {
                    if (nfree == g && ((ball >> (g * KMAX)) & SEGMASK) == SEGMASK) ++nfree;
                }
                if (nfree > 0) {
                    const float zend = __fmaf_rn((float)nfree, L, zmin);
                    if (marching) {
                        while (it < s.max_steps) {
                            const float zn = __fadd_rn(z, s.c08mu);
                            // the next sample lies beyond the stretch, or the march ends there
                            if (!(zn <= zend)) break;
                            z = zn;
                            ++it;
                            have_prev = false;
                            if (!(z <= s.zf)) break;
                        }
                    }
                    if (nfree == NSEG) {
                        shorter = false;
                        continue;
                    }
                }
                if (!shorter) {
                    shorter = true;
                    continue;
                }
                cool = SP_COOL;
            }
        } else {
            --cool;
        }
        if (inside && (bisect > 0 || (it < s.max_steps && z <= s.zf))) {
            const bool b = bisect > 0;
            const float zs = b ? __fmul_rn(0.5f, __fadd_rn(lo, hi)) : z;
            float S, W;
            sphere_eval<KMAX, FULL>(a, ray, zs, S, W);
            if (b) {
                ++extra;
                if (W > 0.0f && S > 0.0f) lo = zs;
                else hi = zs;
                if (--bisect == 0) {
                    out = __fmul_rn(0.5f, __fadd_rn(lo, hi));
                    z = kInf;  // done
                }
            } else {
                ++it;
                if (have_prev && W_prev > 0.0f && W > 0.0f && S_prev > 0.0f && S <= 0.0f) {
                    lo = z_prev;
                    hi = z;
                    bisect = 3;
                } else {
                    float stepn = 1.0f;
                    if (W > 0.0f) {
                        const float sn = __fdiv_rn(S, W);
                        stepn = sn > s.min_frac ? sn : s.min_frac;
                    }
                    S_prev = S;
                    W_prev = W;
                    z_prev = z;
                    have_prev = true;
                    z = __fadd_rn(z, __fmul_rn(s.c08mu, stepn));
                }
            }
        }
    }
    if (inside) {
        const size_t o = (size_t)j * a.Wt + i;
        a.fused[o] = out;
        if (s.evals) s.evals[o] = it + extra;
    }
}

template <int KMAX>
void launch_k(const SphereArgs &s, cudaStream_t st) {
    const int64_t nb = (int64_t)((s.f.Wt + SP_BX - 1) / SP_BX) * ((s.f.Ht + SP_BY - 1) / SP_BY);
    const unsigned grid = (unsigned)((nb + SP_WARPS - 1) / SP_WARPS), block = 32 * SP_WARPS;
    if (s.f.K == KMAX) sphere_kernel<KMAX, true><<<grid, block, 0, st>>>(s);
    else sphere_kernel<KMAX, false><<<grid, block, 0, st>>>(s);
}

}  // namespace

cudaError_t launch_sphere(const SphereArgs &s, cudaStream_t st) {
    if (s.f.K <= 4) launch_k<4>(s, st);
    else if (s.f.K <= 8) launch_k<8>(s, st);
    else if (s.f.K <= 16) launch_k<16>(s, st);
    else launch_k<32>(s, st);
    return cudaGetLastError();
}

GVS_BOUNDS_TAKE_FN(bounds_take_sphere)

}  // namespace gvs
