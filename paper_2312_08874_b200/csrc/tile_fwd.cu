// Launch plans of the register-tiled forward kernels.
#include "tile_launch.cuh"

#include <algorithm>

namespace aa {

namespace {

int dk_of(int d) { return d <= 32 ? 32 : d <= 48 ? 48 : d <= 64 ? 64 : d <= 80 ? 80 : d <= 96 ? 96 : 128; }
cudaError_t dispatch(TileKernel k, int dtype, int dk, int bias, const TileArgs& a, const TileLaunch& l) {
    switch (dk) {
        case 32: return tile_dispatch_32(k, dtype, bias, a, l);
        case 48: return tile_dispatch_48(k, dtype, bias, a, l);
        case 64: return tile_dispatch_64(k, dtype, bias, a, l);
        case 80: return tile_dispatch_80(k, dtype, bias, a, l);
        case 96: return tile_dispatch_96(k, dtype, bias, a, l);
        default: return tile_dispatch_128(k, dtype, bias, a, l);
    }
}
template <int DK> int agg_smem_dk(int kg, int warps) {
    if (warps == 8) return kg == 1 ? AggShape<DK, 1, 8>::kSmem : kg == 2 ? AggShape<DK, 2, 8>::kSmem : AggShape<DK, 4, 8>::kSmem;
    return kg == 1 ? AggShape<DK, 1, 4>::kSmem : kg == 2 ? AggShape<DK, 2, 4>::kSmem : AggShape<DK, 4, 4>::kSmem;
}
int agg_smem(int dk, int kg, int warps) {
    switch (dk) {
        case 32: return agg_smem_dk<32>(kg, warps);
        case 48: return agg_smem_dk<48>(kg, warps);
        case 64: return agg_smem_dk<64>(kg, warps);
        case 80: return agg_smem_dk<80>(kg, warps);
        case 96: return agg_smem_dk<96>(kg, warps);
        default: return agg_smem_dk<128>(kg, warps);
    }
}
int bc_smem(int dk, const TileArgs& a, int warps) {
    const bool dwc = a.wd != nullptr;
    switch (dk) {
        case 32: return BcShape<32>::smem_bytes(a.n, warps, a.W, dwc);
        case 48: return BcShape<48>::smem_bytes(a.n, warps, a.W, dwc);
        case 64: return BcShape<64>::smem_bytes(a.n, warps, a.W, dwc);
        case 80: return BcShape<80>::smem_bytes(a.n, warps, a.W, dwc);
        case 96: return BcShape<96>::smem_bytes(a.n, warps, a.W, dwc);
        default: return BcShape<128>::smem_bytes(a.n, warps, a.W, dwc);
    }
}
int bias_align(int row) { return row % 8 == 0 ? 8 : 1; }
int bias_kind(const void* b, int align) { return !b ? 0 : align == 8 ? 1 : 2; }
int up32(int x) { return (x + 31) & ~31; }

// The one-kernel path: blocks of four warps (up to 64 agents; eight warps have rows for 128), registers for sixteen warps an SM either way.
struct SlabPlan {
    int warps, rg, kg, smem;
    long long slots;               // blocks resident at once
};
SlabPlan slab_plan(const TileArgs& a, int sm_count) {
    const int dk = dk_of(a.d);
    SlabPlan s;
    s.warps = a.n <= 64 ? 4 : 8;
    s.rg = (a.n + 15) / 16;
    s.kg = s.warps == 8 || s.rg > 2 ? 1 : s.rg == 2 ? 2 : 4;
    s.smem = std::max(agg_smem(dk, s.kg, s.warps), bc_smem(dk, a, s.warps));
    s.slots = std::min<long long>(16 / s.warps, 227 * 1024 / (s.smem + 1024)) * sm_count;
    return s;
}
// Row and key groups of an aggregation block: at most eight warps, all of them with rows.
int agg_rows(const TileArgs& a, TileArgs* out) {
    const int rb = (a.n + 8 * 16 - 1) / (8 * 16);
    out->rg = ((a.n + rb - 1) / rb + 16 - 1) / 16;
    out->kg = out->rg <= 2 ? 4 : out->rg <= 4 ? 2 : 1;
    return rb;
}

}  // namespace

cudaError_t launch_tile_aggregate(int dtype, TileArgs a, int sm_count, bool dependent, cudaStream_t st) {
    const int dk = dk_of(a.d);
    const int rb = agg_rows(a, &a);
    a.b2 = nullptr;
    // Parts of the token axis (one block each, a cluster per slab).  Two blocks share an SM and hide each other's
    // latencies, so the best split is the one with the shortest blocks in the fewest waves; a block's start and merge count as
    // 128 tokens.  A cluster of sixteen asks for eight SMs of one GPC (two blocks share an SM): fourteen of them are resident at once, the
    // fifteenth waits for one to end (49 agents, whole forward pass, eights against sixteens: 14 slabs of 8775 tokens 83 and 69 us, 16 slabs
    // 85 and 92 us; 16640 tokens 115 and 98, 124 and 125 us; 2800 tokens 37 and 35, 38 and 44 us).
    int best = 1;
    long long best_cost = 0;
    const int smem = agg_smem(dk, a.kg, 8);
    for (int c = 1; c <= 16; c *= 2) {
        const int tokens = up32((a.N + c - 1) / c);
        if (c > 1 && (tokens < 64 || c * a.kg > 32)) break;
        if (c == 16 && (a.slabs * rb > 14 || smem > 112 * 1024)) break;
        const long long blocks = (long long)a.slabs * rb * c;
        const long long cost = ((blocks + 2LL * sm_count - 1) / (2LL * sm_count)) * (tokens + 128LL);
        if (c == 1 || cost < best_cost) { best = c; best_cost = cost; }
    }
    a.agg_tokens = up32((a.N + best - 1) / best);
    TileLaunch l;
    l.grid = dim3(best, rb, a.slabs);
    l.threads = 256;
    l.cluster = best;
    l.smem = smem;
    l.dependent = dependent;
    l.stream = st;
    return dispatch(kTileAggregate, dtype, dk, bias_kind(a.b1, bias_align(a.N)), a, l);
}

cudaError_t launch_tile_broadcast(int dtype, TileArgs a, int sm_count, bool dependent, cudaStream_t st) {
    const int dk = dk_of(a.d);
    a.b1 = nullptr;
    // Small agent counts: blocks of eight warps, two to an SM.  Large ones: the agents and their features fill a third of
    // the shared memory or more, so one block of sixteen warps shares them.
    const bool pair = bc_smem(dk, a, 8) <= 113 * 1024;
    int warps = pair ? 8 : 16;
    while (bc_smem(dk, a, warps) > 227 * 1024) warps -= 4;      // (256 agents of 128 channels: 8; four always fit)
    const int slots = pair ? 2 * sm_count : sm_count;
    const int pass = warps * 16;                       // tokens of one pass of a block
    int best = 1;
    double best_cost = 0;
    for (int k = 1; k <= 16; ++k) {
        const long long blocks = (long long)a.slabs * ((a.N + (long long)pass * k - 1) / ((long long)pass * k));
        const double cost = (double)((blocks + slots - 1) / slots) * (k + 0.4);
        if (k == 1 || cost < best_cost) { best = k; best_cost = cost; }
        if ((long long)pass * k >= a.N) break;
    }
    a.bc_tokens = pass * best;
    TileLaunch l;
    l.grid = dim3((a.N + a.bc_tokens - 1) / a.bc_tokens, a.slabs);
    l.threads = warps * 32;
    l.cluster = 0;
    l.smem = bc_smem(dk, a, warps);
    l.dependent = dependent;
    l.stream = st;
    return dispatch(kTileBroadcast, dtype, dk, bias_kind(a.b2, bias_align(a.n)), a, l);
}

// It saves two launches and the agents' way through memory; a slab's chain runs in at most eight blocks, so the longer the grid, the less it
// saves (three kernels against one, 49 agents of 64 channels, 1 to 384 slabs: 196 tokens 1.18 to 1.32 times its time, 400 tokens 0.89 to
// 1.07, 784 tokens 0.77 to 1.04; 64 agents, 784 tokens 0.88 to 1.23).  Slabs beyond the resident blocks start when others end, which only the
// shortest chains can afford (384 slabs on 296 slots: 49 agents of 128 channels, 49 tokens 1.23, 100 tokens 0.77, 196 tokens 0.73; 81
// agents of 64 channels, 100 tokens 1.28, 196 tokens 1.02, 256 tokens 0.88).
bool tile_one_kernel(const TileArgs& a, int sm_count) {
    if (a.N > 1024 || a.n > 128) return false;
    const SlabPlan s = slab_plan(a, sm_count);
    return bc_smem(dk_of(a.d), a, s.warps) <= 113 * 1024 && (a.slabs <= s.slots || a.N <= (a.n > 64 ? 196 : 64));
}

cudaError_t launch_tile_forward(int dtype, TileArgs a, int sm_count, bool one_kernel, cudaStream_t st, int* launches) {
    if (one_kernel) {
        const SlabPlan s = slab_plan(a, sm_count);
        a.rg = s.rg;
        a.kg = s.kg;
        TileLaunch l;
        l.smem = s.smem;
        // blocks per slab: as many as are resident at once
        int c = 1;
        while (c < 8 && a.slabs * 2LL * c <= s.slots && a.N > 32 * c) c *= 2;
        a.agg_tokens = up32((a.N + c - 1) / c);
        l.grid = dim3(c, a.slabs);
        l.threads = s.warps * 32;
        l.cluster = c;
        l.dependent = true;
        l.stream = st;
        *launches += 1;
        return dispatch(kTileSlab, dtype, dk_of(a.d), !a.b1 && !a.b2 ? 0 : a.b1 && a.b2 && a.N % 8 == 0 && a.n % 8 == 0 ? 1 : 2, a, l);
    }
    if (a.pool) {
        // a warp per window, or (few windows, more than 32 tokens each) a block per window
        const long long cells = (long long)a.slabs * a.n;
        const bool wide = cells < 8LL * sm_count && a.N > 32 * a.n;
        const unsigned blocks = (unsigned)(wide ? cells : (cells + 7) / 8);
        cudaError_t e = dtype == kBF16 ? launch_dependent(wide ? tile_pool_kernel<__nv_bfloat16, true> : tile_pool_kernel<__nv_bfloat16, false>, dim3(blocks), 256, 0, st, a)
                                       : launch_dependent(wide ? tile_pool_kernel<__half, true> : tile_pool_kernel<__half, false>, dim3(blocks), 256, 0, st, a);
        if (e != cudaSuccess) return e;
        *launches += 1;
    }
    cudaError_t e = launch_tile_aggregate(dtype, a, sm_count, a.pool != 0, st);
    if (e != cudaSuccess) return e;
    e = launch_tile_broadcast(dtype, a, sm_count, true, st);
    *launches += 2;
    return e;
}

}  // namespace aa
