// Forward pass on register tiles (16-bit types, up to 256 agents, head_dim up to 128, any grid and strides): pooling,
// aggregation with its cluster merge, broadcast with the depthwise term.  Each phase is a device function, used by a kernel of
// its own (long grids) and by one kernel that runs all three per slab (short grids).
#pragma once
#include "tile_bc.cuh"
#include "tile_pool.cuh"

namespace aa {

// --------------------------------------------------------------------------------------------------------- kernels
template <typename T>
__device__ __forceinline__ AggCta<T> agg_cta(const TileArgs& p, int slab, int part, int rb) {
    AggCta<T> c;
    const int head = slab % p.heads;
    c.a = static_cast<const T*>(p.a) + (size_t)slab * p.n * p.d;
    const long long off = tok_offset(p.lin, slab, p.heads, 0);
    c.k = static_cast<const T*>(p.k) + off;
    c.v = static_cast<const T*>(p.v) + off;
    c.b1 = p.b1 ? static_cast<const T*>(p.b1) + (size_t)head * p.n * p.N : nullptr;
    c.b1_end = p.b1 ? static_cast<const T*>(p.b1) + (size_t)p.heads * p.n * p.N : nullptr;
    c.va = static_cast<T*>(p.va) + (size_t)slab * p.n * p.d;
    c.kst = p.lin.st;
    c.N = p.N; c.n = p.n; c.d = p.d;
    c.t0 = min(p.N, part * p.agg_tokens);
    c.t1 = min(p.N, c.t0 + p.agg_tokens);
    c.rg = p.rg;
    c.row0 = rb * p.rg * 16;
    c.c1 = p.scale1 * kLog2e;
    return c;
}
template <typename T>
__device__ __forceinline__ BcCta<T> bc_cta(const TileArgs& p, int slab, int part, int tokens) {
    BcCta<T> c;
    const int head = slab % p.heads;
    const long long off = tok_offset(p.lin, slab, p.heads, 0);
    c.q = static_cast<const T*>(p.q) + off;
    c.v = p.wd ? static_cast<const T*>(p.v) + off : nullptr;
    c.a = static_cast<const T*>(p.a) + (size_t)slab * p.n * p.d;
    c.va = static_cast<const T*>(p.va) + (size_t)slab * p.n * p.d;
    c.b2 = p.b2 ? static_cast<const T*>(p.b2) + (size_t)head * p.N * p.n : nullptr;
    c.b2_end = p.b2 ? static_cast<const T*>(p.b2) + (size_t)p.heads * p.N * p.n : nullptr;
    c.wd = p.wd ? static_cast<const T*>(p.wd) + (size_t)head * p.d * 9 : nullptr;
    c.out = static_cast<T*>(p.out) + tok_offset(p.lout, slab, p.heads, 0);
    c.qst = p.lin.st; c.ost = p.lout.st;
    c.N = p.N; c.n = p.n; c.d = p.d; c.H = p.H; c.W = p.W;
    c.t0 = min(p.N, part * tokens);
    c.t1 = min(p.N, c.t0 + tokens);
    c.c1 = p.scale2 * kLog2e;
    return c;
}

// grid (cluster of token parts, row blocks, slabs)
template <typename T, int DK, int KG, int BIAS>
__global__ void __launch_bounds__(256, 2) tile_aggregate_kernel(const __grid_constant__ TileArgs p) {
    extern __shared__ __align__(128) unsigned char smem[];
    pdl_release_next();
    const AggCta<T> c = agg_cta<T>(p, blockIdx.z, blockIdx.x, blockIdx.y);
    agg_phase<T, DK, KG, 8, BIAS>(c, smem, [] { pdl_wait_prior(); });
    cluster_sync_all(gridDim.x);
    agg_merge<T, DK, KG, 8>(c, smem, blockIdx.x, gridDim.x);
    if (gridDim.x > 1) cluster_sync_all();                                // siblings still read this block's shared memory
}

// grid (token parts, slabs)
template <typename T, int DK, int BIAS>
__global__ void __launch_bounds__(512, 1) tile_broadcast_kernel(const __grid_constant__ TileArgs p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const BcCta<T> c = bc_cta<T>(p, blockIdx.y, blockIdx.x, p.bc_tokens);
    pdl_wait_prior();
    bc_fill<T, DK>(c, smem);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    bc_phase<T, DK, BIAS>(c, smem, blockDim.x >> 5);
}

// Short grids: a cluster of blocks per slab runs the three phases, tied by cluster barriers.  grid (cluster, slabs)
template <typename T, int DK, int KG, int NW, int BIAS>
__global__ void __launch_bounds__(NW * 32, 16 / NW) tile_slab_kernel(const __grid_constant__ TileArgs p) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int slab = blockIdx.y, crank = blockIdx.x, csize = gridDim.x, warp = threadIdx.x >> 5;
    pdl_wait_prior();           // (no early release: blocks of the next call would take the slots that balance this one)
    const AggCta<T> c = agg_cta<T>(p, slab, crank, 0);
    agg_phase<T, DK, KG, NW, BIAS>(c, smem, [&] {
        if (p.pool) {
            const T* q = static_cast<const T*>(p.q) + tok_offset(p.lin, slab, p.heads, 0);
            T* a = const_cast<T*>(c.a);
            if (p.H * p.W <= 32 * p.n) {                 // small windows: a thread per 16 bytes of an agent
                const int cpt = p.d >> 3, items = (p.n - crank + csize - 1) / csize * cpt;
                for (int i = threadIdx.x; i < items; i += NW * 32) {
                    const int agent = crank + i / cpt * csize, ch = i % cpt;
                    pool_chunk<T>(q + ch * 8, p.lin.st, p.H, p.W, p.pool, p.pool, agent,
                                  [&](const float (&f)[8]) { *reinterpret_cast<uint4*>(a + (size_t)agent * p.d + ch * 8) = pack16<T>(f); });
                }
            } else {
                for (int i = crank + warp * csize; i < p.n; i += csize * (NW))
                    pool_window<T>(q, p.lin.st, p.H, p.W, p.pool, p.pool, i, p.d,
                                   [&](int ch, const float (&f)[8]) { *reinterpret_cast<uint4*>(a + (size_t)i * p.d + ch * 8) = pack16<T>(f); });
            }
            cluster_sync_all(csize);
        }
    });
    cluster_sync_all(csize);
    agg_merge<T, DK, KG, NW>(c, smem, crank, csize);
    cluster_sync_all(csize);
    const BcCta<T> b = bc_cta<T>(p, slab, crank, p.agg_tokens);
    bc_fill<T, DK>(b, smem);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    bc_phase<T, DK, BIAS>(b, smem, NW);
}

// WIDE: the eight warps of a block share a window
template <typename T, bool WIDE>
__global__ void __launch_bounds__(256) tile_pool_kernel(const __grid_constant__ TileArgs p) {
    pdl_wait_prior();
    pdl_release_next();
    const int warp = threadIdx.x >> 5;
    const long long cell = WIDE ? blockIdx.x : (long long)blockIdx.x * 8 + warp;
    if (cell >= (long long)p.slabs * p.n) return;
    const int slab = (int)(cell / p.n), agent = (int)(cell - (long long)slab * p.n);
    T* a = static_cast<T*>(const_cast<void*>(p.a)) + (size_t)cell * p.d;
    const T* q = static_cast<const T*>(p.q) + tok_offset(p.lin, slab, p.heads, 0);
    if constexpr (WIDE) {
        __shared__ __align__(16) float part[8][128];
        pool_window<T>(q, p.lin.st, p.H, p.W, p.pool, p.pool, agent, p.d, [&](int ch, const float (&f)[8]) {
#pragma unroll
            for (int i = 0; i < 8; ++i) part[warp][ch * 8 + i] = f[i];
        }, warp, 8);
        __syncthreads();
        if ((int)threadIdx.x < p.d / 2) {
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int w = 0; w < 8; ++w) s = fadd2(s, *reinterpret_cast<const float2*>(&part[w][2 * threadIdx.x]));
            *reinterpret_cast<uint32_t*>(a + 2 * threadIdx.x) = pack2<T>(s.x, s.y);
        }
    } else {
        pool_window<T>(q, p.lin.st, p.H, p.W, p.pool, p.pool, agent, p.d,
                       [&](int ch, const float (&f)[8]) { *reinterpret_cast<uint4*>(a + ch * 8) = pack16<T>(f); });
    }
}

}  // namespace aa
