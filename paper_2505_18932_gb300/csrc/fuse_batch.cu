// Batched fusion: many (frame, target) items per launch.
#include "fuse_march.cuh"

namespace gvs {
namespace {

// Up to kBatchArgs (frame, target) items in one launch: each item's blocks follow the
// previous one's, so an item's last bundles overlap the next item's first.  The items'
// arguments are the kernel's parameters: the march reads them from the constant bank, as
// the single-item kernel does.  2 x 4 targets of 8 views: 1.16 ms as one persistent launch
// with the arguments in shared memory, 1.10 as one launch per item, 1.04 so.
constexpr int kBatchArgs = GVS_BATCH_LAUNCH_ITEMS;
struct BatchArgs {
    FuseArgs item[kBatchArgs];
    unsigned first_block[kBatchArgs];
    int n;
};
static_assert(sizeof(BatchArgs) <= 32764, "the parameter space");

template <int KMAX, typename MT, typename T>
__global__ void __launch_bounds__(32 * FZ_WARPS, fuse_min_blocks<KMAX, T, false>()) fuse_batch_kernel(const __grid_constant__ BatchArgs b) {
    __shared__ int2 tab[(kBoundLevels + 1) * KMAX];
    int n = 0;
    while (n + 1 < b.n && blockIdx.x >= b.first_block[n + 1]) ++n;
    const FuseArgs &a = b.item[n];
    fill_slab_table<KMAX>(a, tab, threadIdx.x, 32 * FZ_WARPS);
    __syncthreads();
    const int nbundles = ((a.Wt + T::bx - 1) / T::bx) * ((a.Ht + T::by - 1) / T::by);
    const int bundle = (int)(blockIdx.x - b.first_block[n]) * FZ_WARPS + (threadIdx.x >> 5);
    if (bundle >= nbundles) return;  // the whole warp leaves together
    march_bundle<KMAX, MT, T>(a, tab, bundle, threadIdx.x & 31);
}

template <int KMAX, typename MT, typename T>
struct BatchLaunch {
    static void run(const FuseArgs *items, int n_items, cudaStream_t st) {
        BatchArgs b;
        for (int i0 = 0; i0 < n_items; i0 += kBatchArgs) {
            b.n = n_items - i0 < kBatchArgs ? n_items - i0 : kBatchArgs;
            unsigned blocks = 0;
            for (int i = 0; i < b.n; ++i) {
                const FuseArgs &a = items[i0 + i];
                b.item[i] = a;
                b.first_block[i] = blocks;
                const int64_t nb = (int64_t)((a.Wt + T::bx - 1) / T::bx) * ((a.Ht + T::by - 1) / T::by);
                blocks += (unsigned)((nb + FZ_WARPS - 1) / FZ_WARPS);
            }
            fuse_batch_kernel<KMAX, MT, T><<<blocks, 32 * FZ_WARPS, 0, st>>>(b);
        }
    }
};

}  // namespace

cudaError_t launch_fuse_batch(const FuseArgs *items, int n_items, int K, int map_dtype, int variant, cudaStream_t st) {
    // one bundle shape for the launch: the one that suits the items' mean size
    int64_t pixels = 0;
    for (int i = 0; i < n_items; ++i) pixels += (int64_t)items[i].Wt * items[i].Ht;
    variant = shaped_variant(variant, K, pixels, (int64_t)n_items * items[0].W * items[0].H);
    by_kmax<BatchLaunch>(K, map_dtype, variant, items, n_items, st);
    return cudaGetLastError();
}
GVS_BOUNDS_TAKE_FN(bounds_take_fuse_batch)

}  // namespace gvs
