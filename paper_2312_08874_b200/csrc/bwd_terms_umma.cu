// Backward pass with fp32 accuracy on the 5th-generation tensor cores: the two gradient stages for bf16 tensors of up to 64 channels, and
// the token statistics of the first.
//
// Statistics (X = Q, Y = dO, M = V_A):        S = X A^T, dP = Y M^T; lse[token] = log-sum-exp of S, dot[token] = its softmax . dP
// Broadcast stage (X = Q, Y = dO, M = V_A):   S = X A^T, dP = Y M^T, P = exp(S - lse[token]), dS = P o (dP - dot[token]);
//     dQ += scale dS A,  dV_A += P^T Y,  dA += scale dS^T X,  dB2 += dS.
// Aggregation stage (X = K, Y = V, M = dV_A): S = X A^T, dP = Y M^T, P = exp(S - lse[agent]), dS = P o (dP - D[agent]);
//     dK += scale dS A,  dV += P M,  dA += scale dS^T X,  dB1 += dS.
// A, M, P and dS are sums of three bf16 terms, a product keeps the six pairs of order below three (bwd_terms.cuh).
//
// Unit of work: 64 agents of a slab x 128 tokens.  One block per SM takes a contiguous run of the (slab, tile) sequence for its 64 agents;
// blocks for the other agents of a slab run beside it, so that X and Y come from DRAM once.  The terms of A and M stay in shared memory.  Roles as in bwd_umma.cu: eight row warps (thread = token, half of the agents), four
// output warps, a TMA warp, an issuer of S and dP, an issuer of the products of P and dS.  P and dS are in fp32 registers while the
// products of the tile before run, and are split into terms once those have read theirs: 96 KB of term tiles fit once, not twice.
//
// Accuracy: an accumulation in tensor memory does not round to nearest, so a chain drifts with its length (see term_sum).  The small pairs
// of S and dP therefore have accumulators of their own and those of the other products come first, sums over tokens leave tensor memory after every tile and join in fp32 registers, and the agents' share of a
// token's gradient leaves after 64 of them.  Probabilities add up to one only where logits and statistics drift alike: the statistics above
// come from the same instructions as the broadcast stage's logits, and the aggregation's logits are one chain, small pairs first, where
// bwd_values_umma.cu made the statistics.  (With the pairs apart there, and a common part of 8 in the logits, dV of four slabs of 64 x 64 tokens,
// 81 agents, was 3.8e-7 too large; 5e-8 in one chain.  With statistics from bwd_sums_kernel it is the other way round: 4e-8 and 4.5e-7.)
//
// What bounds it: the products, whose operands are read from shared memory again for every pair of terms (3900 to 4700 cycles of the tensor pipe a tile),
// beside splitting and storing terms (2000), and fp32 reductions (a tile adds 32 KB of bias gradients and 32 or 64 KB of rows): see
// backward_terms_umma_order.  16 slabs of a 128 x 128 grid, 256 agents, biases: broadcast 355 us, aggregation 447 us with nothing cleared before them
// (342 and 420 after 107 us of clearing), statistics 87 + 6 us; on mma.sync (bwd_sums_kernel, bwd_rows_kernel) 828, 1010 and 242 us.  192 slabs of
// 14 x 14, 81 agents, whole pass: 313 -> 187 us; one slab of 40 x 23, 49 agents of 32 channels: 62 -> 51 us.
#include "bwd_terms_launch.cuh"
#include "stream_common.cuh"

#include <algorithm>
#include <cstring>

namespace aa {

namespace {

constexpr int kTok = 128;                    // tokens per tile
constexpr int kTile = kTok * 128;            // bytes of a swizzled [128][64] tile of 16-bit elements
constexpr int kMat = 64 * 128;               // bytes of a [64][64] tile
constexpr int kStages = 2, kTerms = 3;
constexpr int kStage = 2 * kTile;            // X | Y
constexpr int kRowThreads = 256, kThreads = kRowThreads + 128 + 96;

// shared memory (bytes from a 1024-aligned base; mbarriers and two words of the block at its start)
constexpr int OFF_DEAD = 128, OFF_TMEM = 132;
constexpr int OFF_RING = 1024;
constexpr int OFF_AM = OFF_RING + kStages * kStage;          // terms of A, terms of M
constexpr int OFF_P = OFF_AM + 2 * kTerms * kMat;            // per term: P | dS
constexpr int OFF_BIAS = OFF_P + 2 * kTerms * kTile;         // [128 tokens][64 agents], or twice [64 agents][64 tokens]
constexpr int OFF_STAT = OFF_BIAS + kTile;                   // aggregation: [2][64] (lse, D)
constexpr int OFF_EX = OFF_P;                                // statistics: [2 tiles][2 halves][128] (max, sum, dot)
constexpr int kSmemBytes = OFF_STAT + 2 * 64 * 8 + 1024;
static_assert(kSmemBytes <= 232448 && kSmemBytes > 116 * 1024, "one block per SM");

// mbarriers                        count             waiter
constexpr int BAR_FULL = 0;   // [2] tx               issuer of S and dP
constexpr int BAR_AM = 2;     //     tx               the same
constexpr int BAR_S = 3;      //     commit           row warps: S and dP of a tile
constexpr int BAR_READ = 4;   //     row warps        issuer of S and dP: they have been read
constexpr int BAR_P = 5;      //     row warps        issuer of the products: P and dS written
constexpr int BAR_DONE = 6;   // [2] commit           row warps, output warps: every product of a tile (producer: the last tile of a slab)
constexpr int BAR_OUT = 8;    //     output warps     issuer of the products: outputs and sums read
constexpr int BAR_DRAIN = 10; // [2] commit           each issuer, once, at its end
constexpr int BAR_BIAS = 12;  //     tx               row warps
constexpr int BAR_BREAD = 13; //     row warps        producer: the biases have been read
constexpr int BAR_FREE = 14;  // [2] commit           producer: the sums of a tile (statistics: S and dP), the last to read its X and Y
constexpr int kBars = 16;
static_assert(8 * kBars <= OFF_DEAD, "mbarriers");
constexpr int kTimeoutTile = 3, kTimeoutRole = 6;

// tensor memory columns: leading and small pairs of S, of dP; then (broadcast) sums of P^T [X | Y] and dS^T [X | Y] | dQ, (aggregation)
// dK | dV | sums of dS^T X
constexpr uint32_t TM_S = 0, TM_DP = 128, TM_BUF = 256;

enum Mode { kStats, kBcast, kAgg };

struct Args {
    const float2* stats;      // broadcast: (log2-sum-exp, row dot) [slabs][N]; aggregation: (log2-sum-exp, D) [slabs][n]
    float2* tok_stats;        // statistics: the former, where one block holds all agents,
    float4* partial;          // else (max, sum, dot) [blocks][slabs][N]
    float *outer0, *outer1;   // fp32 [slabs][n][d]: dV_A (broadcast) and dA (added)
    float *row0, *row1;       // fp32 [slabs][N][d]: dQ, or dK and dV (added where there are several blocks of agents)
    float* dbias;             // fp32 [heads][N][n] (broadcast) or [heads][n][N] (added; stored where the batch has one entry), or null
    int* status;
    int slabs, heads, N, n, d, tiles, blocks;
    int bias;                 // 0: none; 1: tiles of token rows; 2: tiles of agent rows
    int chain;                // aggregation: all pairs of S in one accumulator, as where `stats` come from bwd_values_umma_kernel
    int owned;                // tiles of a stretch whose batch entries a block takes one after another (0: the sequence in its natural order)
    int all;                  // and all blocks of agents of each
    float scale;
    alignas(64) CUtensorMap tm_x, tm_y, tm_a, tm_m, tm_b;
};

__device__ __forceinline__ void load_pairs(uint32_t taddr, float2 (&v)[16]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float a[16];
        tmem_ld16(taddr + 16 * h, a);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 8; ++j) v[8 * h + j] = make_float2(a[2 * j], a[2 * j + 1]);
    }
}
// 32 columns of leading pairs and of small ones (64 columns on), joined
__device__ __forceinline__ void load_joined(uint32_t taddr, float2 (&v)[16]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float a[16], b[16];
        tmem_ld16(taddr + 16 * h, a);
        tmem_ld16(taddr + 64 + 16 * h, b);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 8; ++j) v[8 * h + j] = fadd2(make_float2(a[2 * j], a[2 * j + 1]), make_float2(b[2 * j], b[2 * j + 1]));
    }
}
__device__ __forceinline__ void st_shared4(uint32_t addr, const uint32_t (&v)[4]) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
// OWN: in one of the orders that p.owned says (the natural one has instantiations of its own, up to 6 % faster without their bookkeeping)
template <int MODE, bool OWN>
__global__ void __launch_bounds__(kThreads, 1) bwd_terms_umma_kernel(const __grid_constant__ Args p) {
    constexpr bool BCAST = MODE == kBcast, AGG = MODE == kAgg, STATS = MODE == kStats;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = p.N, n = p.n, d = p.d;
    // Natural order: a run of the (slab, tile) sequence for one block of 64 agents.  Owned: a run of the (head, tile) sequence, cut into stretches of
    // up to p.owned tiles of a head, all batch entries of a stretch in turn; p.all: of each, all blocks of agents in turn.
    const bool all = OWN && p.all;
    const int side = all ? 1 : p.blocks, lanes = gridDim.x / side, me = blockIdx.x / side;            // blocks of agents side by side; runs of the sequence
    const int batch = OWN ? p.slabs / p.heads : 1;
    const long long total = (long long)p.slabs / batch * p.tiles, first = total * me / lanes, end = total * (me + 1) / lanes;
    const int count = (int)(end - first) * batch * (all ? p.blocks : 1);
    int slab = (int)(first / p.tiles), tile = (int)(first - (long long)slab * p.tiles), ab = all ? 0 : blockIdx.x % side;      // of the role's current tile
    long long at = first;                        // start of its current segment: tiles of one slab that follow one another, for one block of agents
    int entry = 0, left = 0, length = 0;         // its batch entry, how many of its tiles are left
    bool fresh = true;                           // the first tile of a segment
    auto segment = [&] {
        slab = (int)(at / p.tiles);
        tile = (int)(at - (long long)slab * p.tiles);
        left = length = min((int)min(end - at, (long long)(p.tiles - tile)), p.owned);
        slab += entry * p.heads;
    };
    if (OWN) segment();
    auto is_fresh = [&](int i) { return OWN ? fresh : i == 0 || tile == 0; };
    auto is_last = [&](int i) { return OWN ? left == 1 : tile == p.tiles - 1 || i == count - 1; };
    const uint32_t base = smem_u32(smem);

    Pipe pp;
    pp.status = p.status;
    pp.dead = reinterpret_cast<int*>(smem + OFF_DEAD);
    pp.bars = base;
    if (tid == 0) {
        *pp.dead = 0;
        for (int i = 0; i < kBars; ++i) mbar_init(pp.bars + 8 * i, i == BAR_READ || i == BAR_P || i == BAR_BREAD ? 8u : i == BAR_OUT ? 4u : 1u);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc<512>(base + OFF_TMEM);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pp.tmem = *reinterpret_cast<const volatile uint32_t*>(smem + OFF_TMEM);
    pdl_wait_prior();
    pdl_release_next();
    auto advance = [&] {
        ++tile;
        if (!OWN) {
            if (tile == p.tiles) { tile = 0; ++slab; }
            return;
        }
        fresh = --left == 0;
        if (!fresh) return;
        if (!all || ++ab == p.blocks) {
            if (all) ab = 0;
            if (++entry == batch) { entry = 0; at += length; }
        }
        segment();
    };

    if (warp == 12) {
        // ------------------------------------------------------------------ producer
        if (lane == 0) {
            for (int i = 0; i < count && !pipe_dead(pp); ++i, advance()) {
                const int b = i & 1;
                if (i >= 2) wait_spin(pp, BAR_FREE + b, (i >> 1) - 1, kTimeoutRole);
                const uint32_t bar = pipe_bar(pp, BAR_FULL + b), dst = base + OFF_RING + b * kStage;
                mbar_arrive_expect_tx(bar, kStage);
                tma_load_3d(dst, &p.tm_x, 0, tile * kTok, slab, bar);
                tma_load_3d(dst + kTile, &p.tm_y, 0, tile * kTok, slab, bar);
                if (p.bias) {
                    if (i > 0) wait_spin(pp, BAR_BREAD, i - 1, kTimeoutRole);
                    const uint32_t bb = pipe_bar(pp, BAR_BIAS), to = base + OFF_BIAS;
                    const int head = slab % p.heads;
                    mbar_arrive_expect_tx(bb, kTile);
                    if (p.bias == 1) {
                        tma_load_3d(to, &p.tm_b, ab * 64, tile * kTok, head, bb);
                    } else {
                        tma_load_3d(to, &p.tm_b, tile * kTok, ab * 64, head, bb);
                        tma_load_3d(to + kMat, &p.tm_b, tile * kTok + 64, ab * 64, head, bb);
                    }
                }
                if (is_fresh(i)) {
                    if (i > 0) wait_spin(pp, (STATS ? BAR_FREE : BAR_DONE) + (b ^ 1), (i - 1) >> 1, kTimeoutRole);  // the last tile of the segment before
                    const uint32_t bam = pipe_bar(pp, BAR_AM), am = base + OFF_AM;
                    mbar_arrive_expect_tx(bam, 2 * kTerms * kMat);
                    for (int t = 0; t < kTerms; ++t) {
                        tma_load_3d(am + t * kMat, &p.tm_a, 0, ab * 64, t * p.slabs + slab, bam);
                        tma_load_3d(am + (kTerms + t) * kMat, &p.tm_m, 0, ab * 64, t * p.slabs + slab, bam);
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 13) {
        // ------------------------------------------------------------------ S and dP
        const uint32_t id = umma_idesc(1, 128, 64, 0), ts = pp.tmem + TM_S;
        const uint64_t da = umma_desc_sw128(base + OFF_AM);
        int groups = 0;
        for (int i = 0; i < count && !pipe_dead(pp); ++i, advance()) {
            const int b = i & 1;
            if (is_fresh(i)) wait_spin(pp, BAR_AM, groups++, kTimeoutTile);
            wait_spin(pp, BAR_FULL + b, i >> 1, kTimeoutTile);
            if (i > 0) wait_spin(pp, BAR_READ, i - 1, kTimeoutRole);
            tc_fence_after_sync();
            const uint64_t dx = umma_desc_sw128(base + OFF_RING + b * kStage);
            // descriptor start addresses count 16-byte units: + 2 per k step of a K-major operand (32 bytes)
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                const bool chain = AGG && which == 0 && p.chain;
#pragma unroll
                for (int t = kTerms - 1; t >= 0; --t)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        umma_ss_w(ts + (TM_DP - TM_S) * which + (chain || t == 0 ? 0 : 64), dx + which * (kTile >> 4) + 2 * k, da + (which * kTerms + t) * (kMat >> 4) + 2 * k, id,
                                  k > 0 || (chain ? t < kTerms - 1 : t == 1));
            }
            if (STATS) umma_commit_w(pipe_bar(pp, BAR_FREE + b));
            umma_commit_w(pipe_bar(pp, BAR_S));
        }
        umma_drain_w(pp, BAR_DRAIN);
        __syncwarp();
    } else if (warp == 14) {
        if (!STATS) {
        // ------------------------------------------------------------------ products of P and dS
        const uint32_t id_out = umma_idesc(1, 128, 64, 1), id_sum = umma_idesc(1, 128, BCAST ? 128 : 64, 1) | (1u << 15);
        const uint64_t dp = umma_desc_sw128(base + OFF_P), da = umma_desc_sw128(base + OFF_AM), dps = desc_mn(base + OFF_P, kTile);
        for (int i = 0; i < count && !pipe_dead(pp); ++i) {
            const int b = i & 1;
            wait_spin(pp, BAR_P, i, kTimeoutRole);
            if (i > 0) wait_spin(pp, BAR_OUT, i - 1, kTimeoutRole);
            tc_fence_after_sync();
            const uint64_t dxy = desc_mn(base + OFF_RING + b * kStage, kTile);
            const uint32_t tb = pp.tmem + TM_BUF;
            // + 128 per k step of an MN-major operand (16 rows of 128 bytes)
#pragma unroll
            for (int t = kTerms - 1; t >= 0; --t)
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    umma_ss_w(tb + (BCAST ? 0 : 128), dps + t * (2 * kTile >> 4) + 128 * k, dxy + 128 * k, id_sum, t < kTerms - 1 || k > 0);
            umma_commit_w(pipe_bar(pp, BAR_FREE + b));
            // pairs of terms (t of dS or P, u of A or M), the smallest first
#pragma unroll
            for (int which = 0; which < (BCAST ? 1 : 2); ++which)
#pragma unroll
                for (int order = kTerms - 1; order >= 0; --order)
#pragma unroll
                    for (int t = 0; t <= order; ++t)
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            umma_ss_w(tb + (BCAST ? 128 : 64 * which), dp + (2 * t + 1 - which) * (kTile >> 4) + 2 * k,
                                      da + (which * kTerms + order - t) * (kMat >> 4) + 128 * k, id_out, order < kTerms - 1 || t > 0 || k > 0);
            umma_commit_w(pipe_bar(pp, BAR_DONE + b));
        }
        umma_drain_w(pp, BAR_DRAIN + 1);
        }
        __syncwarp();
    } else if (warp >= 8) {
        if (!STATS) {
        // ------------------------------------------------------------------ outputs
        const int q = warp & 3, g = lane >> 2, t = lane & 3;
        const bool second = q >= 2, sums = BCAST || second;            // lanes 64 ..: rows of dS
        float acc[2][32];                                              // rows 16 f + g + 8 h of the warp's 32
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
            for (int k = 0; k < 32; ++k) acc[f][k] = 0.f;
        for (int i = 0; i < count; ++i, advance()) {
            const int b = i & 1;
            const uint32_t rows = pp.tmem + TM_BUF + ((uint32_t)(32 * q) << 16);
            wait_par(pp, BAR_DONE + b, i >> 1, kTimeoutTile);
            tc_fence_after_sync();
            float o[32];
            if (sums)
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    tmem_ld_16x256b_x8(rows + (BCAST ? (second ? 0u : 64u) : 128u) + ((uint32_t)(16 * f) << 16), o);
                    tmem_ld_wait();
#pragma unroll
                    for (int k = 0; k < 32; k += 2) {
                        const float2 v = fadd2(make_float2(acc[f][k], acc[f][k + 1]), make_float2(o[k], o[k + 1]));
                        acc[f][k] = v.x;
                        acc[f][k + 1] = v.y;
                    }
                }
            const int tok0 = tile * kTok + 32 * q + g;
#pragma unroll
            for (int which = 0; which < (BCAST ? 1 : 2); ++which) {
                float* dst = which == 0 ? p.row0 : p.row1;
                const float scale = which == 0 ? p.scale : 1.f;
#pragma unroll
                for (int f = 0; f < 2; ++f) {
                    tmem_ld_16x256b_x8(rows + (BCAST ? 128u : 64u * which) + ((uint32_t)(16 * f) << 16), o);
                    tmem_ld_wait();
                    if (which == (BCAST ? 0 : 1) && f == 1) {          // everything is in registers: hand the buffer back before the stores
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) pipe_arrive(pp, BAR_OUT);
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int tok = tok0 + 16 * f + 8 * h;
                        if (tok >= N) continue;
                        float* r = dst + ((size_t)slab * N + tok) * d + 2 * t;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            if (8 * j >= d) break;
                            const float2 v = make_float2(scale * o[4 * j + 2 * h], scale * o[4 * j + 2 * h + 1]);
                            if (p.blocks == 1 || (all && ab == 0)) *reinterpret_cast<float2*>(r + 8 * j) = v;      // (the others follow from the same thread)
                            else red_add2(r + 8 * j, v.x, v.y);
                        }
                    }
                }
            }
            if (sums && is_last(i)) {                                  // the last tile of the segment
                float* dst = second ? p.outer1 : p.outer0;
                const float scale = second ? p.scale : 1.f;
#pragma unroll
                for (int f = 0; f < 2; ++f)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int r = ab * 64 + 32 * (q & 1) + 16 * f + 8 * h + g;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            if (r < n && 8 * j < d) red_add2(dst + ((size_t)slab * n + r) * d + 8 * j + 2 * t, scale * acc[f][4 * j + 2 * h], scale * acc[f][4 * j + 2 * h + 1]);
                            acc[f][4 * j + 2 * h] = acc[f][4 * j + 2 * h + 1] = 0.f;
                        }
                    }
            }
        }
        }
    } else {
        // ------------------------------------------------------------------ row warps
        const int q = warp & 3, half = warp >> 2, r = 32 * q + lane;
        const uint32_t ts = pp.tmem + TM_S + ((uint32_t)(32 * q) << 16) + 32 * half;
        const float c1 = p.scale * kLog2e;
        float2* s_stat = reinterpret_cast<float2*>(smem + OFF_STAT);
        int parity = 0;
        const float2 none = make_float2(INFINITY, 0.f);                // (a token or an agent that does not exist: its probabilities are zero)
        float2 next = none;
        if (BCAST && tile * kTok + r < N) next = __ldg(p.stats + (size_t)slab * N + tile * kTok + r);
        uint32_t bw[16];                                               // 32 biases as pairs, read a tile ahead
        auto load_bias = [&](int i) {
            if (p.bias) wait_par(pp, BAR_BIAS, i, kTimeoutTile);
            if (!AGG || p.bias != 2) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint4 w = make_uint4(0u, 0u, 0u, 0u);
                    if (p.bias) w = *reinterpret_cast<const uint4*>(smem + OFF_BIAS + r * 128 + (((4 * half + c) ^ (r & 7)) << 4));
                    bw[4 * c] = w.x; bw[4 * c + 1] = w.y; bw[4 * c + 2] = w.z; bw[4 * c + 3] = w.w;
                }
            } else {
                const unsigned char* src = smem + OFF_BIAS + (r >> 6) * kMat + (32 * half) * 128 + (r & 7) * 2;
                const int ch = (r & 63) >> 3;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const uint32_t lo = *reinterpret_cast<const unsigned short*>(src + 2 * j * 128 + ((ch ^ (2 * j & 7)) << 4));
                    const uint32_t hi = *reinterpret_cast<const unsigned short*>(src + (2 * j + 1) * 128 + ((ch ^ ((2 * j + 1) & 7)) << 4));
                    bw[j] = lo | hi << 16;
                }
            }
            // Every lane's words must be in registers before the buffer is handed back: loads that queue behind reductions were overtaken by
            // the arrival and then by the next tile.  So the arriving lane is chosen by a vote on the words themselves.
            uint32_t x = bw[0];
#pragma unroll
            for (int j = 1; j < 16; ++j) x ^= bw[j];
            if (p.bias && lane == (__all_sync(0xffffffffu, x == 0x5bd1e995u) ? 31 : 0)) pipe_arrive(pp, BAR_BREAD);
        };
        load_bias(0);
        for (int i = 0; i < count; ++i) {
            const int now = slab, at_tile = tile, block = ab;          // this tile; the role's state goes on to the next
            const int c0 = block * 64 + 32 * half, lim = n - c0;       // columns of this half that exist
            const bool first_tile = is_fresh(i);
            if (i + 1 < count) advance();
            const int b = i & 1, tok = at_tile * kTok + r, head = now % p.heads;
            const bool ok = tok < N, store = p.slabs == p.heads || (OWN && now < p.heads);      // a head's first batch entry, here before the others
            const float2 st = next;
            if (BCAST) {
                next = none;
                if (i + 1 < count && tile * kTok + r < N) next = __ldg(p.stats + (size_t)slab * N + tile * kTok + r);
            } else if (AGG && first_tile) {                                 // another segment: its statistics
                parity ^= 1;
                if (tid < 64) s_stat[parity * 64 + tid] = block * 64 + tid < n ? __ldg(p.stats + (size_t)now * n + block * 64 + tid) : none;
                bar_named(1, kRowThreads);
            }
            wait_par(pp, BAR_S, i, kTimeoutTile);
            tc_fence_after_sync();
            float2 pr[16], ds[16];
            if (AGG && p.chain) load_pairs(ts, pr);
            else load_joined(ts, pr);
            load_joined(ts + (TM_DP - TM_S), ds);
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) pipe_arrive(pp, BAR_READ);
            // logits in log2 units
#pragma unroll
            for (int j = 0; j < 16; ++j) pr[j] = ffma2(pr[j], make_float2(c1, c1), fmul2(unpack2<__nv_bfloat16>(bw[j]), make_float2(kLog2e, kLog2e)));
            if constexpr (STATS) {
                if (lim < 32)
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (2 * j >= lim) pr[j].x = -INFINITY;
                        if (2 * j + 1 >= lim) pr[j].y = -INFINITY;
                    }
                float m = fmaxf(pr[0].x, pr[0].y);
#pragma unroll
                for (int j = 1; j < 16; ++j) m = max3(m, pr[j].x, pr[j].y);
                const float mb = m == -INFINITY ? 0.f : -m;            // (every agent of this half may be masked)
                float2 l2 = make_float2(0.f, 0.f), d2 = l2;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float2 x = fadd2(pr[j], make_float2(mb, mb));
                    pr[j] = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                    l2 = fadd2(l2, pr[j]);
                    d2 = ffma2(pr[j], ds[j], d2);
                }
                const float l = l2.x + l2.y, dot = d2.x + d2.y;
                float4* ex = reinterpret_cast<float4*>(smem + OFF_EX) + b * 256;
                if (half) ex[r] = make_float4(m, l, dot, 0.f);
                bar_named(2 + q, 64);
                if (!half && ok) {
                    const float4 o = ex[r];
                    const float mm = fmaxf(m, o.x), f = m == -INFINITY ? 0.f : exp2f(m - mm), fo = o.x == -INFINITY ? 0.f : exp2f(o.x - mm);
                    const float tot = fmaf(l, f, o.y * fo), dt = fmaf(dot, f, o.z * fo);
                    if (p.blocks == 1) p.tok_stats[(size_t)now * N + tok] = make_float2(mm + log2f(tot), dt / tot);
                    else p.partial[((size_t)block * p.slabs + now) * N + tok] = make_float4(mm, tot, dt, 0.f);
                }
                if (i + 1 < count) load_bias(i + 1);
                continue;
            }
            // probabilities and logit gradients
            const float4* sst = reinterpret_cast<const float4*>(s_stat + parity * 64 + 32 * half);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                float4 v = make_float4(st.x, st.y, st.x, st.y);
                if (AGG) v = sst[j];                                   // (lse, D) of two agents
                const float2 x = fadd2(pr[j], make_float2(-v.x, -v.z));
                pr[j] = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                if (BCAST && 2 * j >= lim) pr[j].x = 0.f;
                if (BCAST && 2 * j + 1 >= lim) pr[j].y = 0.f;
                if (AGG && !ok) pr[j] = make_float2(0.f, 0.f);
                ds[j] = fmul2(pr[j], fadd2(ds[j], make_float2(-v.y, -v.w)));
            }
            // as operands, once the products of the tile before have read theirs
            if (i > 0) wait_par(pp, BAR_DONE + (b ^ 1), (i - 1) >> 1, kTimeoutTile);
            const uint32_t prow = base + OFF_P + r * 128;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t off = prow + (((4 * half + c) ^ (r & 7)) << 4);
                uint32_t u[kTerms][4], v[kTerms][4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    uint32_t w[kTerms];
                    split_pair<__nv_bfloat16, kTerms>(pr[4 * c + k], w);
#pragma unroll
                    for (int t = 0; t < kTerms; ++t) u[t][k] = w[t];
                    split_pair<__nv_bfloat16, kTerms>(ds[4 * c + k], w);
#pragma unroll
                    for (int t = 0; t < kTerms; ++t) v[t][k] = w[t];
                }
#pragma unroll
                for (int t = 0; t < kTerms; ++t) {
                    st_shared4(off + 2 * t * kTile, u[t]);
                    st_shared4(off + (2 * t + 1) * kTile, v[t]);
                }
            }
            tc_fence_before_sync();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) pipe_arrive(pp, BAR_P);
            if (p.dbias && lim > 0) {
                if (BCAST) {
                    // [token][agent]: this warp's terms of dS, read back so that neighbouring lanes add to neighbouring agents
                    const int t0 = at_tile * kTok + 32 * q;
                    float* g = p.dbias + ((size_t)head * N + t0) * n + c0;
                    const unsigned char* src = smem + OFF_P + kTile + 32 * q * 128;
                    if (n % 4 == 0) {
                        const int cc = lane >> 3;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int rr = 8 * k + (lane & 7);
                            float2 v[4];
#pragma unroll
                            for (int t = kTerms - 1; t >= 0; --t) {
                                const uint4 w = *reinterpret_cast<const uint4*>(src + 2 * t * kTile + rr * 128 + (((4 * half + cc) ^ (rr & 7)) << 4));
                                const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                                for (int e = 0; e < 4; ++e) v[e] = t == kTerms - 1 ? unpack2<__nv_bfloat16>(u[e]) : fadd2(v[e], unpack2<__nv_bfloat16>(u[e]));
                            }
                            if (t0 + rr < N) put_dbias8(g + (size_t)rr * n + 8 * cc, reinterpret_cast<const float*>(v), lim - 8 * cc, true, store);
                        }
                    } else if (lane < lim) {
                        const int left = min(32, N - t0), ch = 4 * half + (lane >> 3);
                        for (int rr = 0; rr < left; ++rr) {
                            const unsigned char* e = src + rr * 128 + ((ch ^ (rr & 7)) << 4) + (lane & 7) * 2;
                            float v = 0.f;
#pragma unroll
                            for (int t = kTerms - 1; t >= 0; --t) v += __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(e + 2 * t * kTile));
                            if (store) g[(size_t)rr * n + lane] = v;
                            else atomicAdd(g + (size_t)rr * n + lane, v);
                        }
                    }
                    __syncwarp();
                } else if (ok) {
                    float* g = p.dbias + ((size_t)head * n + c0) * N + tok;
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float v = j & 1 ? ds[j >> 1].y : ds[j >> 1].x;
                        if (j >= lim) break;
                        if (store) g[(size_t)j * N] = v;
                        else atomicAdd(g + (size_t)j * N, v);
                    }
                }
            }
            if (i + 1 < count) load_bias(i + 1);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc<512>(pp.tmem);
}

// Token statistics from those of every block of agents
__global__ void __launch_bounds__(256) bwd_stats_merge_kernel(const float4* partial, float2* stats, long long tokens, int blocks) {
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    pdl_wait_prior();
    pdl_release_next();
    if (i >= tokens) return;
    float m = -INFINITY, l = 0.f, dot = 0.f;
    for (int k = 0; k < blocks; ++k) {
        const float4 v = partial[k * tokens + i];
        const float mm = fmaxf(m, v.x), f = m == -INFINITY ? 0.f : exp2f(m - mm), fo = v.x == -INFINITY ? 0.f : exp2f(v.x - mm);
        l = fmaf(l, f, v.y * fo);
        dot = fmaf(dot, f, v.z * fo);
        m = mm;
    }
    stats[i] = make_float2(m + log2f(l), dot / l);
}

template <int MODE, bool OWN> cudaError_t launch(const Args& a, int sm_count, cudaStream_t st) {
    static std::atomic<unsigned long long> done;
    cudaError_t e = allow_smem(bwd_terms_umma_kernel<MODE, OWN>, done, kSmemBytes);
    if (e != cudaSuccess) return e;
    const int side = a.all ? 1 : a.blocks;
    const long long total = (long long)(OWN ? a.heads : a.slabs) * a.tiles, lanes = std::min<long long>(total, std::max(1, sm_count / side));
    return launch_dependent(bwd_terms_umma_kernel<MODE, OWN>, dim3((unsigned)(lanes * side)), kThreads, kSmemBytes, st, a);
}

}  // namespace

// One agent or one token: a softmax over it has no gradient, which the recomputed products give exactly only where both passes agree.
// A unit costs 64 agents of 64 channels whatever there are.  More than 32 agents are faster here than on mma.sync (some hundred shapes of 49
// to 16384 tokens, whole pass: 0.33 to 1.05 times as long, the latter at 49 tokens).  Up to 32, one block of agents there, they are where
// agents or channels fill the unit and tokens the chip, or where the token axis is long, or (lines of few agents) a large batch has short
// slabs.  mma.sync -> here: 16 slabs of 196 tokens, 25 agents of 32 channels 42 -> 47 us, 48 slabs of 3136, 16 agents of 40 channels 214 -> 242;
// but 192 slabs of 196, 25 agents of 40 channels 122 -> 104, one slab of 16384, 9 agents of 40 channels 129 -> 116, 16 slabs of 1023, 25 agents
// of 56 channels 74 -> 66.
bool backward_terms_umma_eligible(int dtype, int slabs, int n, int N, int d) {
    if (dtype != kBF16 || d > 64 || d % 8 || n < 2 || n > 256 || N < 2) return false;
    if (n > 32) return true;
    const long long tokens = (long long)slabs * N;
    if (d > 48) return n > 16 ? N >= 196 || tokens >= 9000 : N >= 1024 || tokens >= 16000;
    if (d > 32) return n > 16 ? N >= 1024 || tokens >= 28000 : N >= 8192 || (N <= 512 && tokens >= 28000);
    return n > 16 && (N >= 8192 || (N <= 256 && tokens >= 28000));
}

// Order of the work (see the kernel).  A block that has all batch entries of its tiles stores the first one's bias gradients and adds the others' to them:
// nothing is cleared, and what is added to is still in L2 (a reduction of 32 KB on every SM: 1650 cycles where L2 holds the sums, 3400 where it
// does not).  The same goes for the rows of dQ, dK and dV and a block that has all blocks of agents.  A stretch ends with a change of A and M, so
// runs have to be long and even.  Whole pass in us, 148 SMs, natural order / all batch entries, stretches of 4, 8 and 16 tiles / all agents, too,
// stretches of 2, 4 and 8:
//   two batch entries of 8 heads, 128 x 128 tokens, 256 agents (6.9 tiles a block)   1248 / 1147 1149 1173 / 1064 1083 1188
//   one of 8 heads, 128 x 128, 256                                                    602 /  596  597  603 /  563  568  626
//   two of 8 heads, 92 x 151, 81 (5.9)                                                667 /  640  641  652 /  604  605  606
//   two of 8 heads, 75 x 117, 144 (3.7)                                               600 /  591  595  601 /  555  591  589
//   one of 8 heads, 92 x 151, 81 to 196 agents: 349 to 332, 468 to 459, 616 to 608 (stretches of 2); 256 agents 570 to 588
//   one of 8 heads, 75 x 117, 256 agents of 40 channels (3.7)                         393 /  398  397  392 /  416  425  427
//   eight of 2 heads, 128 x 128, 196 agents of 40 channels (6.9 a run of four)       1152 / 1115 1197 1202
//   fourteen of 2 heads, 75 x 117, 144 agents of 40 channels (2.8 a run of three)     864 /  995
//   four of 4 heads, 128 x 128, 144 agents of 40 channels (10.4 a run of three)       887 /  931
//   one of 8 heads, 92 x 151, 256 agents of 40 channels (5.9)                         549 /   -              /  584
UmmaOrder backward_terms_umma_order(int slabs, int heads, int n, int N, int d, int sm_count) {
    const long long tiles = (long long)heads * ((N + kTok - 1) / kTok), blocks = (n + 63) / 64, lanes = std::max<long long>(1, sm_count / blocks);
    // blocks have whole tiles of the axis, one more for some than for others: at most an eighth above the average
    auto even = [&](long long runs) { return (tiles + runs - 1) / runs * runs * 8 <= tiles * 9; };
    const bool wide = d > 48;                                           // (narrow rows: less to clear)
    if (blocks > 1 && tiles >= (slabs != heads ? 3 : n % 64 ? 5 : 6) * (long long)sm_count && even(sm_count) && (wide || slabs != heads)) return {2, 1};
    if (wide && slabs != heads && tiles >= 4 * lanes && even(lanes) && 4LL * heads * n * N >= 24 << 20) return {4, 0};
    return {0, 0};
}

size_t backward_terms_umma_bytes(int slabs, int heads, int n, int N) {
    return (N % 8 ? padded_bias_bytes(heads, n, N) : 0) + (n % 8 ? padded_bias_bytes(heads, n, N) : 0) + (n > 64 ? (size_t)((n + 63) / 64) * slabs * N * 16 : 0);
}
void backward_terms_umma_padded(int heads, int n, int N, void* ws, void** b1, void** b2, void** partial) {
    char* w = static_cast<char*>(ws);
    *b1 = N % 8 ? w : nullptr;
    if (N % 8) w += padded_bias_bytes(heads, n, N);
    *b2 = n % 8 ? w : nullptr;
    if (n % 8) w += padded_bias_bytes(heads, n, N);
    *partial = w;
}

cudaError_t launch_backward_terms_umma(BwdTermsUmma stage, const BwdCall& c, const void* a_t, const void* m_t, float2* stats, const void* padded, void* partial, cudaStream_t st) {
    Args a;
    memset(&a, 0, sizeof(a));
    const int N = c.H * c.W;
    const bool queries = stage != kUmmaAggregate;
    a.slabs = c.slabs; a.heads = c.heads; a.N = N; a.n = c.n; a.d = c.d; a.tiles = (N + kTok - 1) / kTok; a.blocks = (c.n + 63) / 64;
    a.status = c.status;
    a.stats = stats; a.tok_stats = stats; a.partial = static_cast<float4*>(partial);
    const void* bias = queries ? c.b2 : c.b1;
    a.bias = !bias ? 0 : queries || padded ? 1 : 2;
    a.outer0 = c.ws_dva; a.outer1 = c.ws_da;
    a.row0 = queries ? c.dq : c.dk; a.row1 = c.dv;
    a.dbias = queries ? c.db2 : c.db1;
    a.chain = backward_values_eligible(c.slabs, c.n, N);
    const UmmaOrder order = backward_terms_umma_order(c.slabs, c.heads, c.n, N, c.d, c.sm_count);
    if (stage != kUmmaStats) { a.owned = order.stretch; a.all = order.all_agents; }
    a.scale = queries ? c.scale2 : c.scale1;
    if (!make_map_3d_u16(&a.tm_x, queries ? c.q : c.k, c.slabs, N, c.d, kTok) || !make_map_3d_u16(&a.tm_y, queries ? c.d_out : c.v, c.slabs, N, c.d, kTok) ||
        !make_map_3d_u16(&a.tm_a, a_t, (uint64_t)kTerms * c.slabs, c.n, c.d, 64) || !make_map_3d_u16(&a.tm_m, m_t, (uint64_t)kTerms * c.slabs, c.n, c.d, 64))
        return cudaErrorInvalidValue;
    if (bias && !(padded ? make_map_3d_u16(&a.tm_b, padded, c.heads, N, bias_width(c.n), kTok)
                  : queries ? make_map_3d_u16(&a.tm_b, bias, c.heads, N, c.n, kTok) : make_map_3d_u16(&a.tm_b, bias, c.heads, c.n, N, 64)))
        return cudaErrorInvalidValue;
    if (stage == kUmmaBroadcast) return a.owned ? launch<kBcast, true>(a, c.sm_count, st) : launch<kBcast, false>(a, c.sm_count, st);
    if (stage == kUmmaAggregate) return a.owned ? launch<kAgg, true>(a, c.sm_count, st) : launch<kAgg, false>(a, c.sm_count, st);
    cudaError_t e = launch<kStats, false>(a, c.sm_count, st);
    if (e != cudaSuccess || a.blocks == 1) return e;
    const long long tokens = (long long)c.slabs * N;
    return launch_dependent(bwd_stats_merge_kernel, dim3((unsigned)((tokens + 255) / 256)), 256, 0, st, (const float4*)a.partial, stats, tokens, a.blocks);
}

}  // namespace aa
