// Backward pass of the agent-attention module (Eq. 6): the two gradient stages on the 5th-generation tensor cores for n <= 64 agents and
// d = 64 channels of 16-bit types.
//
// Broadcast stage (X = Q, Y = dO, M = V_A):   S = X A^T, dP = Y M^T, P = softmax_agents, dS = P o (dP - rowdot);
//     dQ = scale dS A,  dV_A += P^T Y,  dA += scale dS^T X,  dB2 += dS.
// Aggregation stage (X = K, Y = V, M = dV_A): S = X A^T, dP = Y M^T, P = exp(S - lse), dS = P o (dP - D);
//     dK = scale dS A,  dV = P M,  dA += scale dS^T X,  dB1 += dS.
// A, M, P and dS are rounded to the element type to serve as operands; dP feeds the difference dP - rowdot, which cancels the part that
// the agents have in common (rows of V_A are close to the mean of V), so there M is carried as two 16-bit terms.
//
// One block per SM takes a contiguous run of the (slab, tile of 128 tokens) sequence, so that no SM has more than one tile above the
// average; A and M of the next slab arrive with its first tile.  Roles:
//   warps 0-7   "row warps": thread = (token, half of the agents).  Logits and dP from tensor memory, bias from the ring stage; P and dS as
//               swizzled rows of 64 agents in shared memory: the same bytes are the K-major operand of the products per token and the
//               MN-major operand of the sums over tokens, so nothing is transposed.  Then the bias gradient: staged in fp32 and added by one bulk
//               reduction a tile, which runs beside the next tile (rows that are no multiple of 16 bytes: by coalesced reductions of the warps).
//   warps 8-11  outputs: per-token products from tensor memory to global memory; at the end of a slab its sums.  Aggregation: a slab ahead,
//               D and the terms of dV_A.
//   warp 12     TMA: X, Y and the bias as token rows, two stages of 48 KB.
//   warp 13, 14 issue S and dP (a tile ahead), and the products of P and dS.
// Broadcast: the sums of both halves are one 128-row operand [P | dS] against [X | Y], eight instructions of 128 columns, of whose four
// blocks two are used; as two products of 64 x 64 they would be sixteen.  (Aggregation: against X alone, 64 columns.)
//
// What bounds it: the chain load -> logits -> softmax -> products -> stage free through two stages, and HBM: 64 slabs of a 56 x 56 grid, 49
// agents: broadcast 5500 cycles a tile (softmax 2000, probabilities as operands 670, waits 1500), aggregation 6500; 103 MB, 16 us at the copy
// bandwidth, and 154 MB, 24 us.  Bias gradients by reductions of the row warps took them 1700 to 2500 cycles a tile; staged for the bulk
// reduction 600: whole pass 184.9 -> 177.6 us, 384 slabs of 196 tokens 109.9 -> 106.5.
// With mma.sync, 64-token tiles and scalar bias loads and reductions the two took 96 and 93 us.
#include "bwd_terms.cuh"
#include "stream_common.cuh"

#include <cstring>

namespace aa {

namespace {

constexpr int kTok = 128;                    // tokens per tile
constexpr int kTile = kTok * 128;            // bytes of a swizzled [128][64] tile of 16-bit elements
constexpr int kStages = 2;
constexpr int kStage = 3 * kTile;            // X | Y | bias
constexpr int kMat = 64 * 128;               // bytes of a [64][64] tile
constexpr int kRowThreads = 256, kThreads = kRowThreads + 128 + 96;
constexpr int kPatch = 33;                   // row pitch of a warp's patch of logit gradients (floats)

// shared memory (bytes from a 1024-aligned base)
constexpr int OFF_RING = 1024;
constexpr int OFF_AM = OFF_RING + kStages * kStage;          // two buffers of A | M | M's residual
constexpr int OFF_P = OFF_AM + 2 * 3 * kMat;                 // P | dS
constexpr int OFF_PATCH = OFF_P + 2 * kTile;                 // broadcast: logit gradients, staged (below) or as [8 warps][32][kPatch] floats;
                                                             // aggregation: [2][64] (lse, D), then the stage
// Stage of logit gradients for the bulk reduction.  Aggregation: [n][128 tokens].  Broadcast: n a multiple of four: twice [128 tokens][32 agents],
// 128-byte swizzle; n odd: [128 tokens][n] (a thread's stores of one agent go to different banks).
constexpr int kStageBytes = 128 * 64 * 4, kStatBytes = 2 * 64 * 8;
static_assert(OFF_PATCH % 1024 == 0 && kStatBytes + kStageBytes <= 8 * 32 * kPatch * 4, "stage");
constexpr int OFF_EX = OFF_PATCH + 8 * 32 * kPatch * 4;      // broadcast: [2 tiles][2 halves][128] (max, sum, dot)
constexpr int kSmemBytes = OFF_EX + 2 * 256 * 16 + 1024;
static_assert(kSmemBytes <= 232448 && kSmemBytes > 116 * 1024, "one block per SM");

// mbarriers                        count             waiter
constexpr int BAR_FULL = 0;   // [2] tx               logits issuer, row warps
constexpr int BAR_S = 2;      // [2] commit           row warps: S and dP of a tile
constexpr int BAR_P = 4;      // [2] row warps        both issuers: P and dS written, S and dP read
constexpr int BAR_DONE = 6;   // [2] commit           producer, row warps, output warps: every product of a tile
constexpr int BAR_OUT = 8;    //     output warps     products issuer: outputs (and a finished slab's sums) read
constexpr int BAR_DRAIN = 9;  // [2] commit           each issuer, once, at its end
constexpr int BAR_M = 11;     // [2] output warps     logits issuer, row warps: terms of dV_A and statistics of a slab (aggregation)
constexpr int kBars = 13;
constexpr int kTimeoutTile = 3, kTimeoutRole = 6;

// tensor memory columns: S | dP, twice; outputs; sums
constexpr uint32_t TM_S = 0, TM_OUT = 256, TM_SUM = 384;

struct UmmaArgs {
    const float2* stats;      // aggregation: .x = log2-sum-exp [slabs][n]
    const float *va, *dva;    // aggregation: V_A and dV_A, fp32 [slabs][n][64]
    float *outer0, *outer1;   // fp32 [slabs][n][64]: dV_A (broadcast) and dA (added)
    float *row0, *row1;       // fp32 [slabs][N][64]: dQ, or dK and dV
    float* dbias;             // fp32, B2's layout [heads][N][n] or B1's [heads][n][N] (added), or null
    int* status;
    int slabs, heads, N, n, tiles, bias;
    int bulk;                 // bias gradients by bulk reductions
    float scale;
    alignas(64) CUtensorMap tm_x, tm_y, tm_a, tm_m, tm_b, tm_db;
};

__device__ __forceinline__ void st_shared_f32(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(addr), "f"(v) : "memory"); }
// One bulk reduction (fp32 additions in L2) of a staged box; what lies outside the tensor is left out.
__device__ __forceinline__ void reduce_add_3d(const CUtensorMap* map, int x, int y, int z, uint32_t src) {
    asm volatile("cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2, %3}], [%4];\n"
                 ::"l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(src) : "memory");
}

template <typename T, bool BCAST>
__global__ void __launch_bounds__(kThreads, 1) bwd_umma_kernel(const __grid_constant__ UmmaArgs p) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ int s_dead;
    __shared__ uint32_t s_tmem;
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int fmt = Elem<T>::kIsBf16 ? 1 : 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = p.N, n = p.n;
    const long long total = (long long)p.slabs * p.tiles;
    const long long first = total * blockIdx.x / gridDim.x;
    const int count = (int)(total * (blockIdx.x + 1) / gridDim.x - first);
    int slab = (int)(first / p.tiles), tile = (int)(first - (long long)slab * p.tiles);     // of the role's current tile
    const uint32_t base = smem_u32(smem);

    Pipe pp;
    pp.status = p.status;
    pp.dead = &s_dead;
    pp.bars = base;
    if (tid == 0) {
        s_dead = 0;
        for (int i = 0; i < kBars; ++i) mbar_init(pp.bars + 8 * i, i >= BAR_P && i < BAR_DONE ? 8u : i == BAR_OUT || i >= BAR_M ? 4u : 1u);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc<512>(smem_u32(&s_tmem));
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pp.tmem = s_tmem;
    pdl_wait_prior();
    pdl_release_next();
    auto advance = [&] {
        if (++tile == p.tiles) { tile = 0; ++slab; }
    };

    if (warp == 12) {
        // ------------------------------------------------------------------ producer
        if (lane == 0) {
            int buf = 0;
            for (int i = 0; i < count && !pipe_dead(pp); ++i, advance()) {
                const int b = i & 1;
                // the products of tile i - 2 are the last to read this stage, and A and M of a slab before the previous one
                if (i >= 2) wait_spin(pp, BAR_DONE + b, (i >> 1) - 1, kTimeoutRole);
                const bool fresh = i == 0 || tile == 0;
                const uint32_t bar = pipe_bar(pp, BAR_FULL + b), dst = base + OFF_RING + b * kStage;
                mbar_arrive_expect_tx(bar, (p.bias ? 3u : 2u) * kTile + (fresh ? (BCAST ? 3u : 1u) * kMat : 0u));
                if (fresh) {
                    const uint32_t am = base + OFF_AM + buf * 3 * kMat;
                    buf ^= 1;
                    tma_load_3d(am, &p.tm_a, 0, 0, slab, bar);
                    if (BCAST) {
                        tma_load_3d(am + kMat, &p.tm_m, 0, 0, slab, bar);
                        tma_load_3d(am + 2 * kMat, &p.tm_m, 0, 0, p.slabs + slab, bar);
                    }
                }
                tma_load_3d(dst, &p.tm_x, 0, tile * kTok, slab, bar);
                tma_load_3d(dst + kTile, &p.tm_y, 0, tile * kTok, slab, bar);
                if (p.bias) tma_load_3d(dst + 2 * kTile, &p.tm_b, 0, tile * kTok, slab % p.heads, bar);
            }
        }
        __syncwarp();
    } else if (warp == 13) {
        // ------------------------------------------------------------------ S and dP, a tile ahead
        const uint32_t id = umma_idesc(fmt, 128, 64, 0);
        int buf = 1, order = 0;
        for (int i = 0; i < count && !pipe_dead(pp); ++i, advance()) {
            const int b = i & 1;
            if (i == 0 || tile == 0) {
                buf ^= 1;
                if (!BCAST) wait_spin(pp, BAR_M + buf, order++ >> 1, kTimeoutRole);
            }
            if (i >= 2) wait_spin(pp, BAR_P + b, (i >> 1) - 1, kTimeoutRole);          // tile i - 2 has been read out of tensor memory
            wait_spin(pp, BAR_FULL + b, i >> 1, kTimeoutTile);
            tc_fence_after_sync();
            const uint64_t dx = umma_desc_sw128(base + OFF_RING + b * kStage), dy = dx + (kTile >> 4);
            const uint64_t da = umma_desc_sw128(base + OFF_AM + buf * 3 * kMat), dm = da + (kMat >> 4), dr = dm + (kMat >> 4);
            const uint32_t ts = pp.tmem + TM_S + 128 * b;
            // descriptor start addresses count 16-byte units: + 2 per k step of a K-major operand (32 bytes)
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_ss_w(ts, dx + 2 * k, da + 2 * k, id, k > 0);
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_ss_w(ts + 64, dy + 2 * k, dr + 2 * k, id, k > 0);
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_ss_w(ts + 64, dy + 2 * k, dm + 2 * k, id, 1u);
            umma_commit_w(pipe_bar(pp, BAR_S + b));
        }
        umma_drain_w(pp, BAR_DRAIN);
        __syncwarp();
    } else if (warp == 14) {
        // ------------------------------------------------------------------ products of P and dS
        const uint32_t id_out = umma_idesc(fmt, 128, 64, 1), id_sum = umma_idesc(fmt, 128, BCAST ? 128 : 64, 1) | (1u << 15);
        const uint64_t dp = umma_desc_sw128(base + OFF_P), ds = dp + (kTile >> 4), dps = desc_mn(base + OFF_P, kTile);
        int buf = 1;
        for (int i = 0; i < count && !pipe_dead(pp); ++i, advance()) {
            const int b = i & 1;
            const bool fresh = i == 0 || tile == 0;
            if (fresh) buf ^= 1;
            wait_spin(pp, BAR_P + b, i >> 1, kTimeoutRole);
            if (fresh && i > 0) wait_spin(pp, BAR_OUT, i - 1, kTimeoutRole);           // the slab before: its sums have been read
            tc_fence_after_sync();
            const uint64_t dxy = desc_mn(base + OFF_RING + b * kStage, kTile);
            const uint64_t da = umma_desc_sw128(base + OFF_AM + buf * 3 * kMat), dm = da + (kMat >> 4);
            // + 128 per k step of an MN-major operand (16 rows of 128 bytes)
#pragma unroll
            for (int k = 0; k < 8; ++k) umma_ss_w(pp.tmem + TM_SUM, dps + 128 * k, dxy + 128 * k, id_sum, fresh ? k > 0 : 1u);
            if (!fresh) { wait_spin(pp, BAR_OUT, i - 1, kTimeoutRole); tc_fence_after_sync(); }
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_ss_w(pp.tmem + TM_OUT, ds + 2 * k, da + 128 * k, id_out, k > 0);
            if (!BCAST)
#pragma unroll
                for (int k = 0; k < 4; ++k) umma_ss_w(pp.tmem + TM_OUT + 64, dp + 2 * k, dm + 128 * k, id_out, k > 0);
            umma_commit_w(pipe_bar(pp, BAR_DONE + b));
        }
        umma_drain_w(pp, BAR_DRAIN + 1);
        __syncwarp();
    } else if (warp >= 8) {
        // ------------------------------------------------------------------ outputs
        const int q = warp & 3, g = lane >> 2, t = lane & 3;
        const uint32_t rows = pp.tmem + ((uint32_t)(32 * q) << 16);
        // M of a slab for the aggregation: the two terms of dV_A, and (log2-sum-exp, D = dV_A . V_A) of its agents
        auto prepare = [&](int of, int buf) {
            const int c = lane & 7, r0 = 16 * q + (lane >> 3);         // rows r0 + 4 k, channels 8 c ..
            float4 dva[4][2], va[4][2];
            float lse[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool have = r0 + 4 * k < n;
                const size_t row = (size_t)of * n + r0 + 4 * k;
                lse[k] = INFINITY;                                 // (an agent that does not exist: its probabilities are zero)
                if (have) lse[k] = __ldcg(&p.stats[row].x);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    dva[k][h] = va[k][h] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (have) dva[k][h] = __ldcg(reinterpret_cast<const float4*>(p.dva + row * 64 + 8 * c + 4 * h));
                    if (have) va[k][h] = __ldcg(reinterpret_cast<const float4*>(p.va + row * 64 + 8 * c + 4 * h));
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int r = r0 + 4 * k;
                uint32_t hi[4], lo[4];
                float dot = 0.f;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 a = dva[k][h], v = va[k][h];
                    dot = fmaf(a.x, v.x, fmaf(a.y, v.y, fmaf(a.z, v.z, fmaf(a.w, v.w, dot))));
                    uint32_t w[2];
                    split_pair<T, 2>(a.x, a.y, w);
                    hi[2 * h] = w[0]; lo[2 * h] = w[1];
                    split_pair<T, 2>(a.z, a.w, w);
                    hi[2 * h + 1] = w[0]; lo[2 * h + 1] = w[1];
                }
                const uint32_t at = base + OFF_AM + (3 * buf + 1) * kMat + r * 128 + ((c ^ (r & 7)) << 4);
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(at), "r"(hi[0]), "r"(hi[1]), "r"(hi[2]), "r"(hi[3]) : "memory");
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(at + kMat), "r"(lo[0]), "r"(lo[1]), "r"(lo[2]), "r"(lo[3]) : "memory");
#pragma unroll
                for (int o = 4; o; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
                if (c == 0) reinterpret_cast<float2*>(smem + OFF_PATCH)[64 * buf + r] = make_float2(lse[k], dot);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) pipe_arrive(pp, BAR_M + buf);
        };
        int prepared = 0, order = -1;                              // slabs of the run, in their order
        for (int i = 0; i < count; ++i, advance()) {
            const int b = i & 1;
            if (!BCAST && (i == 0 || tile == 0)) {
                // a slab ahead: every tile of the slab before this one is done, and with them the buffer of the next
                ++order;
                const int last = p.tiles - tile < count - i ? order + 1 : order;
#pragma unroll 1
                for (; prepared <= last; ++prepared) prepare(slab + prepared - order, prepared & 1);
            }
            wait_par(pp, BAR_DONE + b, i >> 1, kTimeoutTile);
            tc_fence_after_sync();
            float o[2][32];                                        // rows 16 f + g + 8 h of the warp's 32
            const int tok0 = tile * kTok + 32 * q + g;
            auto store = [&](float* dst, float scale) {
#pragma unroll
                for (int f = 0; f < 2; ++f)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int tok = tok0 + 16 * f + 8 * h;
                        if (tok >= N) continue;
                        float* d = dst + ((size_t)slab * N + tok) * 64 + 2 * t;
#pragma unroll
                        for (int j = 0; j < 8; ++j) *reinterpret_cast<float2*>(d + 8 * j) = make_float2(scale * o[f][4 * j + 2 * h], scale * o[f][4 * j + 2 * h + 1]);
                    }
            };
            if (tile == p.tiles - 1 || i == count - 1) {           // the last tile of the slab in this block: its sums
                const bool second = q >= 2;                        // lanes 64 ..: rows of dS
                if (BCAST || second) {
#pragma unroll
                    for (int f = 0; f < 2; ++f) tmem_ld_16x256b_x8(rows + TM_SUM + (second ? 0u : 64u) + ((uint32_t)(16 * f) << 16), o[f]);
                    tmem_ld_wait();
                    float* dst = second ? p.outer1 : p.outer0;
                    const float scale = second ? p.scale : 1.f;
#pragma unroll
                    for (int f = 0; f < 2; ++f)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int r = 32 * (q & 1) + 16 * f + 8 * h + g;
                            if (r >= n) continue;
                            float* d = dst + ((size_t)slab * n + r) * 64 + 2 * t;
#pragma unroll
                            for (int j = 0; j < 8; ++j) red_add2(d + 8 * j, scale * o[f][4 * j + 2 * h], scale * o[f][4 * j + 2 * h + 1]);
                        }
                }
            }
#pragma unroll
            for (int which = 0; which < (BCAST ? 1 : 2); ++which) {
#pragma unroll
                for (int f = 0; f < 2; ++f) tmem_ld_16x256b_x8(rows + TM_OUT + 64 * which + ((uint32_t)(16 * f) << 16), o[f]);
                tmem_ld_wait();
                if (which == (BCAST ? 0 : 1)) {                    // everything is in registers: hand the buffers back before the stores
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) pipe_arrive(pp, BAR_OUT);
                }
                store(which == 0 ? p.row0 : p.row1, which == 0 ? p.scale : 1.f);
            }
        }
    } else {
        // ------------------------------------------------------------------ row warps
        const int q = warp & 3, half = warp >> 2, r = 32 * q + lane, c0 = 32 * half;
        const int lim = n - c0;                                    // columns of this half that exist (uniform; may be <= 0)
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        const float c1 = p.scale * kLog2e;
        float2* s_stat = reinterpret_cast<float2*>(smem + OFF_PATCH);
        float* patch = reinterpret_cast<float*>(smem + OFF_PATCH) + warp * 32 * kPatch;
        float4* ex = reinterpret_cast<float4*>(smem + OFF_EX);
        int order = -1;                                            // slab of the run
        for (int i = 0; i < count; ++i, advance()) {
            const int b = i & 1, tok = tile * kTok + r;
            const bool ok = tok < N;
            if (!BCAST && (i == 0 || tile == 0)) {                 // another slab: its statistics
                ++order;
                wait_par(pp, BAR_M + (order & 1), order >> 1, kTimeoutTile);
            }
            wait_par(pp, BAR_FULL + b, i >> 1, kTimeoutTile);
            wait_par(pp, BAR_S + b, i >> 1, kTimeoutTile);
            tc_fence_after_sync();
            const uint32_t ts = pp.tmem + TM_S + 128 * b + lane_base + c0;
            uint32_t sr[32], dr[32];
            tmem_ld32(ts, sr);
            tmem_ld_wait();
            tmem_ld32(ts + 64, dr);
            // logits in log2 units
            float2 s[16];
            const uint32_t brow = base + OFF_RING + b * kStage + 2 * kTile + r * 128;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint4 w = make_uint4(0u, 0u, 0u, 0u);
                if (p.bias) asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w) : "r"(brow + (((4 * half + c) ^ (r & 7)) << 4)));
                const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int j = 4 * c + k;
                    s[j] = ffma2(unpack2<T>(u[k]), make_float2(kLog2e, kLog2e),
                                 fmul2(make_float2(__uint_as_float(sr[2 * j]), __uint_as_float(sr[2 * j + 1])), make_float2(c1, c1)));
                }
            }
            float2 dp[16];
            if (BCAST) {
                if (lim < 32)
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (2 * j >= lim) s[j].x = -INFINITY;
                        if (2 * j + 1 >= lim) s[j].y = -INFINITY;
                    }
                float m = fmaxf(s[0].x, s[0].y);
#pragma unroll
                for (int j = 1; j < 16; ++j) m = max3(m, s[j].x, s[j].y);
                const float mb = m == -INFINITY ? 0.f : -m;        // (every column of this half may be removed)
                float2 l2 = make_float2(0.f, 0.f), d2 = l2;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float2 x = fadd2(s[j], make_float2(mb, mb));
                    s[j] = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                    l2 = fadd2(l2, s[j]);
                }
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    dp[j] = make_float2(__uint_as_float(dr[2 * j]), __uint_as_float(dr[2 * j + 1]));
                    d2 = ffma2(s[j], dp[j], d2);
                }
                // the other half of the agents: maximum, sum, dot product
                const float l = l2.x + l2.y, d = d2.x + d2.y;
                ex[b * 256 + half * 128 + r] = make_float4(m, l, d, 0.f);
                bar_named(2 + q, 64);
                const float4 o = ex[b * 256 + (half ^ 1) * 128 + r];
                const float mm = fmaxf(m, o.x), f = fast_exp2(m - mm), fo = fast_exp2(o.x - mm);
                const float inv = 1.f / (l * f + o.y * fo), dot = (d * f + o.z * fo) * inv, w = ok ? f * inv : 0.f;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    s[j] = fmul2(s[j], make_float2(w, w));
                    dp[j] = fmul2(s[j], fadd2(dp[j], make_float2(-dot, -dot)));
                }
            } else {
                tmem_ld_wait();
                const float4* st = reinterpret_cast<const float4*>(s_stat + (order & 1) * 64 + c0);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float4 v = st[j];                        // (lse, D) of two agents
                    s[j] = fadd2(s[j], make_float2(-v.x, -v.z));
                    s[j] = make_float2(fast_exp2(s[j].x), fast_exp2(s[j].y));
                    if (!ok) s[j] = make_float2(0.f, 0.f);
                    // (a softmax over one token has no gradient; the two roundings of its dot product need not agree)
                    dp[j] = N == 1 ? make_float2(0.f, 0.f)
                                   : fmul2(s[j], fadd2(make_float2(__uint_as_float(dr[2 * j]), __uint_as_float(dr[2 * j + 1])), make_float2(-v.y, -v.w)));
                }
            }
            // as operands, once the products of the tile before have read theirs
            if (i > 0) wait_par(pp, BAR_DONE + (b ^ 1), (i - 1) >> 1, kTimeoutTile);
            const uint32_t prow = base + OFF_P + r * 128;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t off = prow + (((4 * half + c) ^ (r & 7)) << 4);
                uint32_t u[4], v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    u[k] = pack2<T>(s[4 * c + k].x, s[4 * c + k].y);
                    v[k] = pack2<T>(dp[4 * c + k].x, dp[4 * c + k].y);
                }
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(off), "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]) : "memory");
                asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(off + kTile), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
            }
            tc_fence_before_sync();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) pipe_arrive(pp, BAR_P + b);
            if (p.dbias && p.bulk) {
                const int head = slab % p.heads;
                const uint32_t stage = base + OFF_PATCH + (BCAST ? 0 : kStatBytes);
                // the reduction of the tile before has read the stage
                if (tid == 0) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
                bar_named(1, kRowThreads);
                if (!BCAST) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < lim) st_shared_f32(stage + ((c0 + j) * 128 + r) * 4, j & 1 ? dp[j >> 1].y : dp[j >> 1].x);
                } else if (n % 4 == 0) {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        if (4 * c < lim)
                            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(stage + half * (kStageBytes / 2) + r * 128 + ((c ^ (r & 7)) << 4)),
                                         "f"(dp[2 * c].x), "f"(dp[2 * c].y), "f"(dp[2 * c + 1].x), "f"(dp[2 * c + 1].y) : "memory");
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < lim) st_shared_f32(stage + (r * n + c0 + j) * 4, j & 1 ? dp[j >> 1].y : dp[j >> 1].x);
                }
                fence_proxy_async();
                bar_named(1, kRowThreads);
                if (tid == 0) {
                    if (!BCAST) reduce_add_3d(&p.tm_db, tile * kTok, 0, head, stage);
                    else if (n % 4 == 0) {
                        reduce_add_3d(&p.tm_db, 0, tile * kTok, head, stage);
                        if (n > 32) reduce_add_3d(&p.tm_db, 32, tile * kTok, head, stage + kStageBytes / 2);
                    } else
                        asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;\n"
                                     ::"l"(p.dbias + ((size_t)head * N + (size_t)tile * kTok) * n), "r"(stage), "r"(min(kTok, N - tile * kTok) * n * 4) : "memory");
                    asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
                }
            } else if (p.dbias && lim > 0) {
                const int head = slab % p.heads;
                if (BCAST) {
                    // [token][agent]: through the warp's patch, so that the lanes of a reduction are neighbouring agents
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        patch[lane * kPatch + 2 * j] = dp[j].x;
                        patch[lane * kPatch + 2 * j + 1] = dp[j].y;
                    }
                    __syncwarp();
                    const int t0 = tile * kTok + 32 * q, left = min(32, N - t0);
                    float* g = p.dbias + ((size_t)head * N + t0) * n + c0 + lane;
                    if (lane < lim)
#pragma unroll 8
                        for (int k = 0; k < left; ++k) atomicAdd(g + (size_t)k * n, patch[k * kPatch + lane]);
                    __syncwarp();
                } else if (ok) {
                    float* g = p.dbias + ((size_t)head * n + c0) * N + tok;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (2 * j < lim) atomicAdd(g + (size_t)(2 * j) * N, dp[j].x);
                        if (2 * j + 1 < lim) atomicAdd(g + (size_t)(2 * j + 1) * N, dp[j].y);
                    }
                }
            }
        }
        if (p.bulk && tid == 0) asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc<512>(pp.tmem);
}

template <typename T, bool BCAST> cudaError_t launch(const UmmaArgs& a, int sm_count, cudaStream_t st) {
    static std::atomic<unsigned long long> done;
    cudaError_t e = allow_smem(bwd_umma_kernel<T, BCAST>, done, kSmemBytes);
    if (e != cudaSuccess) return e;
    const long long total = (long long)a.slabs * a.tiles;
    return launch_dependent(bwd_umma_kernel<T, BCAST>, dim3((unsigned)(total < sm_count ? total : sm_count)), kThreads, kSmemBytes, st, a);
}

}  // namespace

// Map of a bias gradient, fp32 [heads][rows][cols], for reduce_add_3d.
static bool make_map_grad(CUtensorMap* out, void* base, uint64_t heads, uint64_t rows, uint64_t cols, uint32_t box_rows, uint32_t box_cols, bool swizzle) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn || (reinterpret_cast<uintptr_t>(base) & 15u) || cols % 4) return false;
    const cuuint64_t dims[3] = {cols, rows, heads}, strides[2] = {4 * cols, 4 * rows * cols};
    const cuuint32_t box[3] = {box_cols, box_rows, 1}, estr[3] = {1, 1, 1};
    return fn(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool backward_umma_eligible(int dtype, int n, int d) { return (dtype == kBF16 || dtype == kF16) && n <= 64 && d == 64; }

cudaError_t launch_backward_umma(int dtype, bool broadcast_stage, const BwdCall& c, cudaStream_t st) {
    UmmaArgs a;
    memset(&a, 0, sizeof(a));
    const int N = c.H * c.W;
    const void* bias = broadcast_stage ? c.b2 : c.b1;
    a.slabs = c.slabs; a.heads = c.heads; a.N = N; a.n = c.n; a.tiles = (N + kTok - 1) / kTok; a.bias = bias != nullptr;
    a.status = c.status;
    a.stats = reinterpret_cast<const float2*>(c.ws_lse);
    a.va = c.ws_va; a.dva = c.ws_dva;
    a.outer0 = c.ws_dva; a.outer1 = c.ws_da;
    a.row0 = broadcast_stage ? c.dq : c.dk; a.row1 = c.dv;
    a.dbias = broadcast_stage ? c.db2 : c.db1;
    a.scale = broadcast_stage ? c.scale2 : c.scale1;
    const void* rows = !broadcast_stage ? c.ws_mixed : c.n % 8 ? static_cast<const char*>(c.ws_mixed) + padded_bias_bytes(c.heads, c.n, N) : c.b2;       // (B2 as it is where TMA takes it)
    if (!make_map_rows3d_u16(&a.tm_x, broadcast_stage ? c.q : c.k, c.slabs, N, kTok, true) || !make_map_rows3d_u16(&a.tm_y, broadcast_stage ? c.d_out : c.v, c.slabs, N, kTok, true) ||
        !make_map_rows3d_u16(&a.tm_a, c.ws_a, c.slabs, c.n, 64, true) || (broadcast_stage && !make_map_rows3d_u16(&a.tm_m, c.ws_part, 2 * (uint64_t)c.slabs, c.n, 64, true)) ||
        (bias && !make_map_3d_u16(&a.tm_b, rows, c.heads, N, bias_width(c.n), kTok)))
        return cudaErrorInvalidValue;
    // Rows of 16 bytes: tokens a multiple of four, and agents a multiple of four or odd (token rows that follow one another, 128 at a time).
    a.bulk = a.dbias && N % 4 == 0 && (!broadcast_stage || c.n % 4 == 0 || c.n % 2);
    if (a.bulk && !broadcast_stage && !make_map_grad(&a.tm_db, a.dbias, c.heads, c.n, N, c.n, kTok, false)) return cudaErrorInvalidValue;
    if (a.bulk && broadcast_stage && c.n % 4 == 0 && !make_map_grad(&a.tm_db, a.dbias, c.heads, N, c.n, kTok, 32, true)) return cudaErrorInvalidValue;
    if (dtype == kBF16) return broadcast_stage ? launch<__nv_bfloat16, true>(a, c.sm_count, st) : launch<__nv_bfloat16, false>(a, c.sm_count, st);
    if (dtype == kF16) return broadcast_stage ? launch<__half, true>(a, c.sm_count, st) : launch<__half, false>(a, c.sm_count, st);
    return cudaErrorInvalidValue;
}

size_t backward_umma_bytes(int heads, int n, int N) { return (n % 8 ? 2 : 1) * padded_bias_bytes(heads, n, N); }

}  // namespace aa
