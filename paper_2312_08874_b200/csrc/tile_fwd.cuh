// Forward pass on register tiles (16-bit types, up to 256 agents, head_dim up to 128, any grid and strides): pooling,
// aggregation with its cluster merge, broadcast with the depthwise term.  Each phase is a device function, used by a kernel of
// its own (long grids) and by one kernel that runs all three per slab (short grids).
#pragma once
#include "tile_bc.cuh"

namespace aa {

// --------------------------------------------------------------------------------------------------------- pooling
// One warp: mean of the window of agent (ay, ax) -> d elements at `out` (fixed order, fp32).
template <typename T>
__device__ __forceinline__ void pool_window(const T* q, long long qst, int H, int W, int p, int agent, int d, T* out) {
    const int lane = threadIdx.x & 31;
    const int ay = agent / p, ax = agent - ay * p;
    const int y0 = (ay * H) / p, y1 = ((ay + 1) * H + p - 1) / p, x0 = (ax * W) / p, x1 = ((ax + 1) * W + p - 1) / p;
    const int ww = x1 - x0, cnt = (y1 - y0) * ww;
    // lanes = (token sub-lane, 16-byte chunk): a power of two of chunks, so that shuffles reduce over the sub-lanes
    const int cpt = d / 8, cp2 = cpt <= 1 ? 1 : cpt <= 2 ? 2 : cpt <= 4 ? 4 : cpt <= 8 ? 8 : 16, tpl = 32 / cp2;
    const int ch = lane & (cp2 - 1), ts = lane / cp2;
    float2 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = make_float2(0.f, 0.f);
    int wy = ts / ww, wx = ts - wy * ww;
    const T* base = q + ((size_t)y0 * W + x0) * qst + ch * 8;
    for (int i = ts; i < cnt; i += 8 * tpl) {
        uint4 raw[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            raw[u] = make_uint4(0u, 0u, 0u, 0u);
            if (i + u * tpl < cnt && ch < cpt) raw[u] = __ldg(reinterpret_cast<const uint4*>(base + ((size_t)wy * W + wx) * qst));
            wx += tpl;
            while (wx >= ww) { wx -= ww; ++wy; }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            acc[0] = fadd2(acc[0], unpack2<T>(raw[u].x));
            acc[1] = fadd2(acc[1], unpack2<T>(raw[u].y));
            acc[2] = fadd2(acc[2], unpack2<T>(raw[u].z));
            acc[3] = fadd2(acc[3], unpack2<T>(raw[u].w));
        }
    }
    for (int o = cp2; o < 32; o <<= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            acc[k].x += __shfl_xor_sync(0xffffffffu, acc[k].x, o);
            acc[k].y += __shfl_xor_sync(0xffffffffu, acc[k].y, o);
        }
    if (ts == 0 && ch < cpt) {
        const float inv = 1.f / (float)cnt;
        const float f[8] = {acc[0].x * inv, acc[0].y * inv, acc[1].x * inv, acc[1].y * inv,
                            acc[2].x * inv, acc[2].y * inv, acc[3].x * inv, acc[3].y * inv};
        *reinterpret_cast<uint4*>(out + ch * 8) = pack16<T>(f);
    }
}

// One thread: eight channels of one agent, for small windows (independent loads, no shuffles; fixed order, fp32).
template <typename T>
__device__ __forceinline__ void pool_chunk(const T* q, long long qst, int H, int W, int p, int agent, T* out) {
    const int ay = agent / p, ax = agent - ay * p;
    const int y0 = (ay * H) / p, y1 = ((ay + 1) * H + p - 1) / p, x0 = (ax * W) / p, x1 = ((ax + 1) * W + p - 1) / p;
    float2 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = make_float2(0.f, 0.f);
    for (int y = y0; y < y1; ++y) {
        const T* row = q + (long long)(y * W) * qst;
#pragma unroll 4
        for (int x = x0; x < x1; ++x) {
            const uint4 raw = __ldg(reinterpret_cast<const uint4*>(row + x * qst));
            acc[0] = fadd2(acc[0], unpack2<T>(raw.x));
            acc[1] = fadd2(acc[1], unpack2<T>(raw.y));
            acc[2] = fadd2(acc[2], unpack2<T>(raw.z));
            acc[3] = fadd2(acc[3], unpack2<T>(raw.w));
        }
    }
    const float inv = 1.f / (float)((y1 - y0) * (x1 - x0));
    const float f[8] = {acc[0].x * inv, acc[0].y * inv, acc[1].x * inv, acc[1].y * inv,
                        acc[2].x * inv, acc[2].y * inv, acc[3].x * inv, acc[3].y * inv};
    *reinterpret_cast<uint4*>(out) = pack16<T>(f);
}

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
    const AggCta<T> c = agg_cta<T>(p, slab, crank, 0);
    agg_phase<T, DK, KG, NW, BIAS>(c, smem, [&] {
        if (p.pool) {
            const T* q = static_cast<const T*>(p.q) + tok_offset(p.lin, slab, p.heads, 0);
            T* a = const_cast<T*>(c.a);
            if (p.H * p.W <= 32 * p.n) {                 // small windows: a thread per 16 bytes of an agent
                const int cpt = p.d >> 3, items = (p.n - crank + csize - 1) / csize * cpt;
                for (int i = threadIdx.x; i < items; i += NW * 32) {
                    const int agent = crank + i / cpt * csize, ch = i % cpt;
                    pool_chunk<T>(q + ch * 8, p.lin.st, p.H, p.W, p.pool, agent, a + (size_t)agent * p.d + ch * 8);
                }
            } else {
                for (int i = crank + warp * csize; i < p.n; i += csize * (NW))
                    pool_window<T>(q, p.lin.st, p.H, p.W, p.pool, i, p.d, a + (size_t)i * p.d);
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

template <typename T>
__global__ void __launch_bounds__(256) tile_pool_kernel(const __grid_constant__ TileArgs p) {
    pdl_release_next();
    const long long cell = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (cell >= (long long)p.slabs * p.n) return;
    const int slab = (int)(cell / p.n), agent = (int)(cell - (long long)slab * p.n);
    pool_window<T>(static_cast<const T*>(p.q) + tok_offset(p.lin, slab, p.heads, 0), p.lin.st, p.H, p.W, p.pool, agent, p.d,
                   static_cast<T*>(const_cast<void*>(p.a)) + (size_t)cell * p.d);
}

}  // namespace aa
