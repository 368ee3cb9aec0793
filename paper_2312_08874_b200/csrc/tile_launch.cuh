// Launch of one instantiation family of the register-tiled kernels (a translation unit per head size keeps the build
// parallel).
#pragma once
#include "tile_fwd.cuh"

#include <atomic>

namespace aa {

enum TileKernel { kTileAggregate, kTileBroadcast, kTileSlab };
struct TileLaunch {
    dim3 grid;
    int threads, cluster;
    size_t smem;
    bool dependent;          // may start while its predecessor in the stream drains (programmatic dependent launch)
    cudaStream_t stream;
};

// Raises a kernel's dynamic shared-memory limit once per device.
template <typename K> inline cudaError_t tile_allow_smem(K kern, std::atomic<unsigned long long>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
}

template <typename K> inline cudaError_t tile_launch(K kern, std::atomic<unsigned long long>& done, const TileArgs& a, const TileLaunch& l) {
    cudaError_t e = tile_allow_smem(kern, done);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = l.grid;
    cfg.blockDim = dim3(l.threads);
    cfg.dynamicSmemBytes = l.smem;
    cfg.stream = l.stream;
    cudaLaunchAttribute at[2];
    int na = 0;
    if (l.cluster > 0) {
        at[na].id = cudaLaunchAttributeClusterDimension;
        at[na].val.clusterDim.x = l.cluster; at[na].val.clusterDim.y = 1; at[na].val.clusterDim.z = 1;
        ++na;
    }
    if (l.dependent) {
        at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = at;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// BIAS: 0 none, 1 rows of 16-byte pieces, 2 any alignment
template <typename T, int DK, int KG, int BIAS> cudaError_t tile_dispatch_kg(TileKernel k, const TileArgs& a, const TileLaunch& l) {
    static std::atomic<unsigned long long> done[3];
    if (k == kTileAggregate) return tile_launch(tile_aggregate_kernel<T, DK, KG, BIAS>, done[0], a, l);
    if (KG == 1 && l.threads == 256) return tile_launch(tile_slab_kernel<T, DK, 1, 8, BIAS>, done[1], a, l);
    return tile_launch(tile_slab_kernel<T, DK, KG, 4, BIAS>, done[2], a, l);
}
template <typename T, int DK, int BIAS> cudaError_t tile_dispatch_b(TileKernel k, const TileArgs& a, const TileLaunch& l) {
    static std::atomic<unsigned long long> done;
    if (k == kTileBroadcast) return tile_launch(tile_broadcast_kernel<T, DK, BIAS>, done, a, l);
    return a.kg == 1   ? tile_dispatch_kg<T, DK, 1, BIAS>(k, a, l)
           : a.kg == 2 ? tile_dispatch_kg<T, DK, 2, BIAS>(k, a, l)
                       : tile_dispatch_kg<T, DK, 4, BIAS>(k, a, l);
}
template <int DK> cudaError_t tile_dispatch_dk(TileKernel k, int dtype, int bias, const TileArgs& a, const TileLaunch& l) {
    if (dtype == kBF16)
        return bias == 0   ? tile_dispatch_b<__nv_bfloat16, DK, 0>(k, a, l)
               : bias == 1 ? tile_dispatch_b<__nv_bfloat16, DK, 1>(k, a, l)
                           : tile_dispatch_b<__nv_bfloat16, DK, 2>(k, a, l);
    return bias == 0   ? tile_dispatch_b<__half, DK, 0>(k, a, l)
           : bias == 1 ? tile_dispatch_b<__half, DK, 1>(k, a, l)
                       : tile_dispatch_b<__half, DK, 2>(k, a, l);
}
#define AA_TILE_DECLARE(DK) cudaError_t tile_dispatch_##DK(TileKernel k, int dtype, int bias, const TileArgs& a, const TileLaunch& l)
AA_TILE_DECLARE(32); AA_TILE_DECLARE(48); AA_TILE_DECLARE(64); AA_TILE_DECLARE(80); AA_TILE_DECLARE(96); AA_TILE_DECLARE(128);

}  // namespace aa
