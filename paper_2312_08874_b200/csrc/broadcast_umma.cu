// Agent broadcast O = softmax(scale2 * Q A^T + B2) V_A + DWC(V) (Eq. 3, Eq. 5, Eq. 6) for large agent
// counts (64 < n <= 256, d <= 64, 16-bit elements) on the 5th-generation tensor cores.
//
// Grid: (splits, slabs), one block per SM.  The slab's agents A and agent features V_A stay resident in shared memory; a block walks its
// share of the slab's tiles, patches of 8 x 16 tokens of the grid (a window with its halo is 180 tokens there, 390 for 128 tokens of a row, and
// zeros outside the grid are what TMA fills in) or, on grids that do not fill patches, runs of 128 tokens.  Two teams of eight warps work on a
// tile each (even and odd ones); per tile the agents are taken in steps of 64, whose logits alternate between two buffers: while the softmax of one step runs, the other buffer's
// products and next logits are under way.
//   warps 0-15 "row warps", a team each eight: thread (query row, half of a step's agents): online softmax over the steps with its own running
//                         maximum, sum and accumulator O_h in tensor memory (no reduction crosses threads); the probabilities go back
//                         to tensor memory over the logits just read, as the A operand of P V_A.
//   warps 16-23 "output warps": 32 rows x 32 channels of every tile in mma.sync accumulator layout: the depthwise 3x3 term (dwc_diag.cuh), then
//                         the two halves' accumulators, weighted by the row's (max, sum) of both; rounded once and stored.
//   warps 24, 25 "producers": one lane each issues its team's TMA copies (Q tiles, B2 tiles); warp 26 those of the V tokens.
//   warps 27, 28 "MMA issuers", one per team: the products of a step once its probabilities are written, then the logits two steps on over them
//                         (instructions of one thread run in their order).
// Every wait is bounded (pipe.cuh).  No TMA multicast, no clusters.
//
// What bounds it: the row warps' instructions (issue 64 % on the 256 x 256 grid), then exponentials (2048 cycles a tile at the special-function rate, of
// 7200) and HBM.  With one team of sixteen row warps that wrote probabilities to shared memory and took the depthwise term themselves, everything
// in step, 16 slabs of a 256 x 256 grid with 256 agents took 343 us; two teams 283; logits in two buffers and output warps of their own 209.
#include "dwc_diag.cuh"
#include "stream_common.cuh"

#include <cstring>

namespace aa {

namespace {
constexpr int TH = 8, TW = 16, QT = TH * TW;             // tile
constexpr int NROW = 512, NOUT = 256;                    // threads: two teams of 256, output warps
constexpr int NT = NROW + NOUT + 256;                    // + five warps of roles (three idle: register splits go by four warps)
constexpr int kRowRegs = 72, kOutRegs = 80, kRoleRegs = 32;        // of 64 at launch
static_assert(NROW * kRowRegs + NOUT * kOutRegs + 256 * kRoleRegs <= NT * 64, "register split");
constexpr int kTile = 64 * 128;                          // swizzled [64][64] tile of 16-bit elements
constexpr float kTau = 5.5f;
constexpr int kTimeoutTile = 3, kTimeoutLoads = 4, kTimeoutRole = 6;

// shared memory (bytes from a 1024-aligned base)
constexpr int OFF_BAR = 0, OFF_DEAD = 512, OFF_TMEM = 516;
constexpr int OFF_ML = 1024;                             // [team][parity of its tile][half][128 rows] (max, sum)
constexpr int OFF_ZEROS = OFF_ML + 8 * 128 * 8;          // zeros, as many as the filter
constexpr int OFF_TAB = OFF_ZEROS + kFilterWords * 4;    // filter
constexpr int OFF_A = 15 * 1024;                         // agents [256][128 B]
constexpr int OFF_VA = OFF_A + 4 * kTile;                // agent features [256][128 B]
constexpr int OFF_Q = OFF_VA + 4 * kTile;                // a query tile [128][128 B] per team
constexpr int OFF_B2 = OFF_Q + 4 * kTile;                // biases of a step [128][128 B], two per team
constexpr int kHaloRows = (TH + 2) * (TW + 2), kHaloBytes = kHaloRows * 128, kHalo = (kHaloBytes + 1023) / 1024 * 1024;
constexpr int OFF_H = OFF_B2 + 4 * 2 * kTile;            // two windows of V tokens [10][18][128 B]; runs: one [3][136][128 B]
constexpr int kRunRows = (QT + 2 + 7) / 8 * 8;           // (eight rows: a period of the swizzle)
constexpr int smem_bytes(bool run) { return OFF_H + (run ? 3 * kRunRows * 128 : 2 * kHalo) + 1024; }
static_assert(OFF_ZEROS % 128 == 0 && OFF_TAB + kFilterWords * 4 <= OFF_A, "small buffers");
static_assert(smem_bytes(true) <= 232448 && smem_bytes(false) <= 232448 && smem_bytes(false) > 116 * 1024, "one block per SM");

// mbarriers (t: + team; ts: + 2 team + step parity; i: + tile parity)   count       waiter
constexpr int BAR_AG = 0;          //             tx          row warps
constexpr int BAR_PREP = 1;        //             1           MMA issuers, output warps      V_A pad rows zeroed, filter
constexpr int BAR_Q_FULL = 2;      // t           tx          MMA issuer
constexpr int BAR_Q_EMPTY = 4;     // t           commit      producer
constexpr int BAR_B_FULL = 6;      // ts          tx          row warps
constexpr int BAR_B_EMPTY = 10;    // ts          8 warps     producer
constexpr int BAR_S_FULL = 14;     // ts          commit      row warps
constexpr int BAR_P_FULL = 18;     // ts          8 warps     MMA issuer      (logits read as well)
constexpr int BAR_PV = 22;         // ts          commit      row warps       products of a step (only where a reference moves)
constexpr int BAR_O_FULL = 26;     // t           commit      output warps    every product of a tile
constexpr int BAR_O_EMPTY = 28;    // t           8 warps     MMA issuer, row warps    accumulators and (max, sum) read
constexpr int BAR_ML = 30;         // t           8 warps     output warps
constexpr int BAR_H_FULL = 32;     // i           tx          output warps    V tokens of the tile's depthwise window (runs: of index 0 only)
constexpr int BAR_H_EMPTY = 34;    // i           8 warps     their producer
constexpr int BAR_DRAIN = 36;      // t           commit      MMA issuer, once, at its end
constexpr int kBars = 38;
static_assert(8 * kBars <= OFF_DEAD, "mbarriers");

// tensor memory, columns of a team: logits (then probabilities) of two steps 64 each, accumulators of two halves 64 each
constexpr uint32_t TM_TEAM = 256, TM_O = 128;

struct UmmaBcArgs {
    AttnArgs a;
    int steps, tps, tiles, tiles_x;    // steps of 64 agents; tiles per split, of a slab, of a row of them
    int hf;                            // dimension order of the Q and V maps (tma_load_grid)
    alignas(64) CUtensorMap tm_q, tm_a, tm_va, tm_b, tm_h;
};
}  // namespace

// RUN: a tile is a run of 128 tokens; ROUNDED: see umma_sums_rounded
template <typename T, bool RUN, bool ROUNDED>
__global__ void __launch_bounds__(NT, 1) broadcast_umma_kernel(const __grid_constant__ UmmaBcArgs g) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int fmt = Elem<T>::kIsBf16 ? 1 : 0;
    constexpr int th = RUN ? 1 : TH, tw = RUN ? QT : TW;       // (runs: the grid is one row to the maps of Q, B2 and V)
    const AttnArgs& p = g.a;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int split = blockIdx.x, slab = blockIdx.y;
    const int head = slab % p.heads;
    const int n = p.cols, steps = g.steps;
    const bool has_b2 = p.bias != nullptr, has_dwc = p.dwc_w != nullptr;
    const int i0 = split * g.tps, tiles = min(g.tiles, i0 + g.tps) - i0;      // >= 1 by the plan

    Pipe pp;
    pp.status = p.status;
    pp.dead = reinterpret_cast<int*>(smem + OFF_DEAD);
    pp.bars = smem_u32(smem + OFF_BAR);
    if (tid == 0) {
        *pp.dead = 0;
        for (int i = 0; i < kBars; ++i) {
            const bool warps = (i >= BAR_B_EMPTY && i < BAR_S_FULL) || (i >= BAR_P_FULL && i < BAR_PV) || (i >= BAR_O_EMPTY && i < BAR_H_FULL) || (i >= BAR_H_EMPTY && i < BAR_DRAIN);
            mbar_init(pp.bars + 8 * i, warps ? 8u : 1u);
        }
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc<512>(smem_u32(smem + OFF_TMEM));
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pp.tmem = *reinterpret_cast<const volatile uint32_t*>(smem + OFF_TMEM);
    pdl_wait_prior();                                     // A and V_A come from the preceding kernels
    pdl_release_next();

    const uint32_t sA = smem_u32(smem + OFF_A), sVA = smem_u32(smem + OFF_VA), sQ = smem_u32(smem + OFF_Q);
    const uint32_t sB2 = smem_u32(smem + OFF_B2), sH = smem_u32(smem + OFF_H);

    if (warp >= 24) {
        set_regs_dec<kRoleRegs>();
        if (warp <= 25) {
            // ------------------------------------------------------------------ producer of a team
            const int team = warp - 24;
            if (lane == 0) {
                if (team == 0) {
                    const int blocks = (steps + 1) >> 1;               // of 128 agents
                    mbar_arrive_expect_tx(pipe_bar(pp, BAR_AG), (uint32_t)blocks * 4 * kTile);
                    for (int mb = 0; mb < blocks; ++mb) {
                        tma_load_2d(sA + mb * 2 * kTile, &g.tm_a, 0, slab * n + 128 * mb, pipe_bar(pp, BAR_AG));
                        tma_load_2d(sVA + mb * 2 * kTile, &g.tm_va, 0, slab * n + 128 * mb, pipe_bar(pp, BAR_AG));
                    }
                }
                int j = 0;
                for (int i = team; i < tiles; i += 2) {
                    const int ty = (i0 + i) / g.tiles_x, y = th * ty, x = tw * (i0 + i - ty * g.tiles_x);
                    if (i >= 2) wait_spin(pp, BAR_Q_EMPTY + team, (i >> 1) - 1, kTimeoutRole);
                    const uint32_t qb = pipe_bar(pp, BAR_Q_FULL + team);
                    mbar_arrive_expect_tx(qb, 2 * kTile);
                    tma_load_grid(sQ + team * 2 * kTile, &g.tm_q, g.hf, x, y, head, slab / p.heads, qb);
                    if (has_b2)
                        for (int a = 0; a < steps; ++a, ++j) {
                            const int b = 2 * team + (j & 1);
                            if (j >= 2) wait_spin(pp, BAR_B_EMPTY + b, (j >> 1) - 1, kTimeoutRole);
                            const uint32_t bar = pipe_bar(pp, BAR_B_FULL + b);
                            mbar_arrive_expect_tx(bar, 2 * kTile);
                            tma_load_4d(sB2 + b * 2 * kTile, &g.tm_b, 64 * a, x, y, head, bar);
                        }
                    if (pipe_dead(pp)) break;
                }
            }
            __syncwarp();
        } else if (warp == 26) {
            // ------------------------------------------------------------------ producer of the V tokens
            if (has_dwc && lane == 0)
                for (int i = 0; i < tiles && !pipe_dead(pp); ++i) {
                    const int ty = (i0 + i) / g.tiles_x, y = th * ty, x = tw * (i0 + i - ty * g.tiles_x);
                    if (RUN) {                                         // the rows above, of and below the run
                        const uint32_t bar = pipe_bar(pp, BAR_H_FULL);
                        if (i >= 1) wait_spin(pp, BAR_H_EMPTY, i - 1, kTimeoutRole);
                        mbar_arrive_expect_tx(bar, 3 * kRunRows * 128);
                        for (int u = 0; u < 3; ++u) tma_load_grid(sH + u * kRunRows * 128, &g.tm_h, g.hf, x - 1 + (u - 1) * p.W, 0, head, slab / p.heads, bar);
                        continue;
                    }
                    const uint32_t bar = pipe_bar(pp, BAR_H_FULL + (i & 1));
                    if (i >= 2) wait_spin(pp, BAR_H_EMPTY + (i & 1), (i >> 1) - 1, kTimeoutRole);
                    mbar_arrive_expect_tx(bar, kHaloBytes);
                    tma_load_grid(sH + (i & 1) * kHalo, &g.tm_h, g.hf, x - 1, y - 1, head, slab / p.heads, bar);
                }
            __syncwarp();
        } else if (warp <= 28) {
            // ------------------------------------------------------------------ MMA issuer of a team (the whole warp runs the loop; one elected lane issues)
            const int team = warp - 27, count = (tiles - team + 1) / 2 * steps;
            if (count > 0) {
                const uint32_t idS = umma_idesc(fmt, 128, 64, 0), idMN = umma_idesc(fmt, 128, 64, 1);
                const uint64_t dA = umma_desc_sw128(sA), dQ = umma_desc_sw128(sQ) + 1024 * team, dVA = umma_desc_sw128(sVA);
                const uint32_t ts = pp.tmem + TM_TEAM * team;
                // descriptor start addresses count 16-byte units: + 2 per K-step of a K-major operand (32 bytes), + 128 per K-step of an
                // MN-major operand (16 rows of 128 bytes), + 512 per 64 rows; + 8 columns per K-step of an operand in tensor memory
                int sa = 0, sk = 0;                                    // step and tile of the logits to come
                auto logits = [&](int b) {
                    if (sa == 0) wait_spin(pp, BAR_Q_FULL + team, sk, kTimeoutLoads);
                    tc_fence_after_sync();
                    const uint64_t db = dA + 512 * sa;
#pragma unroll
                    for (int k = 0; k < 4; ++k) umma_ss_w(ts + 64 * b, dQ + 2 * k, db + 2 * k, idS, k > 0);
                    umma_commit_w(pipe_bar(pp, BAR_S_FULL + 2 * team + b));
                    if (++sa == steps) { sa = 0; ++sk; umma_commit_w(pipe_bar(pp, BAR_Q_EMPTY + team)); }
                };
                wait_spin(pp, BAR_PREP, 0, kTimeoutLoads);
                logits(0);
                if (count > 1) logits(1);
                int a = 0, tile = 0;                                   // step and tile of the products
                for (int j = 0; j < count && !pipe_dead(pp); ++j) {
                    const int b = j & 1;
                    wait_spin(pp, BAR_P_FULL + 2 * team + b, j >> 1, kTimeoutRole);
                    if (a == 0 && tile > 0) wait_spin(pp, BAR_O_EMPTY + team, tile - 1, kTimeoutRole);
                    tc_fence_after_sync();
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        if (64 * a + 32 * h < n) {
                            const uint32_t od = ts + TM_O + 64 * h, oa = ts + 64 * b + 32 * h;
                            const uint64_t ob = dVA + 128 * (4 * a + 2 * h);
                            umma_ts_w(od, oa, ob, idMN, a > 0);
                            umma_ts_w(od, oa + 8, ob + 128, idMN, 1u);
                        }
                    umma_commit_w(pipe_bar(pp, BAR_PV + 2 * team + b));
                    if (++a == steps) { a = 0; ++tile; umma_commit_w(pipe_bar(pp, BAR_O_FULL + team)); }
                    if (j + 2 < count) logits(b);
                }
                umma_drain_w(pp, BAR_DRAIN + team);
            }
            __syncwarp();
        }
    } else if (warp >= 16) {
        // ------------------------------------------------------------------ output warps
        set_regs_inc<kOutRegs>();
        const int q = warp & 3, half = (warp >> 2) & 1, c0 = 32 * half, lg = lane >> 2;
        const uint32_t* tab = filter_lane(reinterpret_cast<const uint32_t*>(smem + OFF_TAB) + c0, reinterpret_cast<const uint32_t*>(smem + OFF_ZEROS), lane);
        uint32_t at[6];
        if (!RUN) patch_offsets<TW + 2>(at, 2 * q * (TW + 2), 64 * half, lane);
        T* gO = static_cast<T*>(p.out) + tok_offset(p.lout, slab, p.heads, 0);
        const size_t so = (size_t)p.lout.st;
        wait_par(pp, BAR_PREP, 0, kTimeoutLoads);
        for (int i = 0; i < tiles; ++i) {
            const int team = i & 1, k = i >> 1;
            float o[2][4][4];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int jj = 0; jj < 4; ++jj)
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[mt][jj][e] = 0.f;
            if (has_dwc) {
                const int ib = RUN ? 0 : team;
                wait_par(pp, BAR_H_FULL + ib, RUN ? i : k, kTimeoutLoads);
                if constexpr (RUN) {
                    uint32_t in[2];
#pragma unroll
                    for (int mt = 0; mt < 2; ++mt) {               // (past the last token: anything, not stored)
                        const int t = QT * (i0 + i) + 32 * q + 16 * mt + (lane & 15), y = t / p.W;
                        in[mt] = grid_taps(t - y * p.W, y, p.H, p.W, lane);
                    }
                    dwc_rows<T>(o, sH, 32 * q + (lane & 15), 64 * half, in, smem_u32(smem + OFF_ZEROS), tab, lane, [](int u, int v) { return u * kRunRows + v; });
                } else {
                    dwc_patch<T>(o, at, sH + team * kHalo, tab);
                }
                // The window goes back to TMA: an arrival overtakes loads that are still queued, so the arriving lane hangs on the products of
                // what was loaded.
                uint32_t x = 0u;
#pragma unroll
                for (int k = 0; k < 8; ++k) x ^= __float_as_uint(o[k >> 2][k & 3][0]);
                if (lane == (__all_sync(0xffffffffu, x == 0x5bd1e995u) ? 31 : 0)) pipe_arrive(pp, BAR_H_EMPTY + ib);
            }
            wait_par(pp, BAR_ML + team, k, kTimeoutTile);
            float w0, w1;                                      // weights of row 32 q + lane's two accumulators
            {
                const float2* sML = reinterpret_cast<const float2*>(smem + OFF_ML) + (team * 2 + (k & 1)) * 256 + 32 * q + lane;
                const float2 a0 = sML[0], a1 = sML[128];
                const float mm = fmaxf(a0.x, a1.x), e0 = fast_exp2((a0.x - mm) * kLog2e), e1 = fast_exp2((a1.x - mm) * kLog2e);
                const float inv = 1.f / fmaf(e0, a0.y, e1 * a1.y);
                w0 = e0 * inv; w1 = e1 * inv;
            }
            wait_par(pp, BAR_O_FULL + team, k, kTimeoutTile);
            tc_fence_after_sync();
            const uint32_t tO = pp.tmem + TM_TEAM * team + TM_O + c0 + ((uint32_t)(32 * q) << 16);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                float wr[2][2];                                // [half][row g, row g + 8]
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    wr[0][hh] = __shfl_sync(0xffffffffu, w0, 16 * mt + 8 * hh + lg);
                    wr[1][hh] = __shfl_sync(0xffffffffu, w1, 16 * mt + 8 * hh + lg);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float ra[16];
                    tmem_ld_16x256b_x4(tO + 64 * h + (16u * mt << 16), ra);
                    tmem_ld_wait();
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj)
#pragma unroll
                        for (int e = 0; e < 4; ++e) o[mt][jj][e] = fmaf(wr[h][e >> 1], ra[4 * jj + e], o[mt][jj][e]);
                }
            }
            tc_fence_before_sync();
            pipe_arrive_warp(pp, BAR_O_EMPTY + team, lane);
            if constexpr (RUN) {
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    const int t = QT * (i0 + i) + 32 * q + 16 * mt;
                    const bool ok[2] = {t + lg < p.rows, t + 8 + lg < p.rows};
                    store_rows<T>(o[mt], gO + (size_t)t * so, so, c0, p.d, ok, lane);
                }
                continue;
            }
            const int ty = (i0 + i) / g.tiles_x, y = TH * ty + 2 * q, x = TW * (i0 + i - ty * g.tiles_x);
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const bool ok[2] = {y + mt < p.H && x + lg < p.W, y + mt < p.H && x + 8 + lg < p.W};
                store_rows<T>(o[mt], gO + ((size_t)(y + mt) * p.W + x) * so, so, c0, p.d, ok, lane);
            }
        }
    } else {
        // ------------------------------------------------------------------ row warps
        set_regs_inc<kRowRegs>();
        const int team = warp >> 3, half = (warp >> 2) & 1;    // 32 agents of every step
        const int q = warp & 3, row = 32 * q + lane;           // query row of the tile = tensor-memory lane
        const uint32_t lane_base = ((uint32_t)(32 * q)) << 16;
        const uint32_t tS = pp.tmem + TM_TEAM * team + 32 * half + lane_base;      // logits, then probabilities (the first 16 columns)
        const uint32_t tO = pp.tmem + TM_TEAM * team + TM_O + 64 * half + lane_base;
        // set-up: filter taps, zero rows of V_A past the last agent (0 * NaN is not 0)
        if (has_dwc) fill_filter(reinterpret_cast<uint32_t*>(smem + OFF_TAB), p.dwc_w, head, p.d, tid, NROW);
        for (int e = tid; e < kFilterWords; e += NROW) reinterpret_cast<uint32_t*>(smem + OFF_ZEROS)[e] = 0u;
        wait_par(pp, BAR_AG, 0, kTimeoutLoads);
        for (int e = tid; e < (64 * steps - n) * 8; e += NROW)
            *(reinterpret_cast<uint4*>(smem + OFF_VA + (n + (e >> 3)) * 128) + (e & 7)) = make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async();
        asm volatile("bar.sync 1, %0;\n" ::"n"(NROW) : "memory");
        if (tid == 0) pipe_arrive(pp, BAR_PREP);

        int j = 0;                                             // steps so far
        for (int i = team; i < tiles; i += 2) {
            float m_ref = kRefFloor, l = 0.f;
            for (int a = 0; a < steps; ++a, ++j) {
                const int b = j & 1, bar = 2 * team + b;
                const int valid = min(32, n - (64 * a + 32 * half));    // agents of this thread in the step (uniform; may be <= 0)
                wait_par(pp, BAR_S_FULL + bar, j >> 1, kTimeoutTile);
                tc_fence_after_sync();
                float sv[32];
                tmem_ld32(tS + 64 * b, *reinterpret_cast<uint32_t(*)[32]>(sv));
                if (has_b2) wait_par(pp, BAR_B_FULL + bar, j >> 1, kTimeoutLoads);
                tmem_ld_wait();
                if (has_b2) {                                // logits in natural units: scale2 * q.a + b2
                    const unsigned char* sB = smem + OFF_B2 + bar * 2 * kTile + row * 128;
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) {
                        const uint4 raw = *reinterpret_cast<const uint4*>(sB + (((4 * half + jj) ^ (row & 7)) << 4));
                        const uint32_t w4[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {        // packed pairs: one instruction per two logits
                            const float2 r2 = ffma2(make_float2(sv[8 * jj + 2 * k], sv[8 * jj + 2 * k + 1]), make_float2(p.scale, p.scale), unpack2<T>(w4[k]));
                            sv[8 * jj + 2 * k] = r2.x; sv[8 * jj + 2 * k + 1] = r2.y;
                        }
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const float2 r2 = fmul2(make_float2(sv[2 * k], sv[2 * k + 1]), make_float2(p.scale, p.scale));
                        sv[2 * k] = r2.x; sv[2 * k + 1] = r2.y;
                    }
                }
                if (valid < 32) {
#pragma unroll
                    for (int k = 0; k < 32; ++k) if (k >= valid) sv[k] = -INFINITY;
                }
                float mx0 = fmaxf(sv[0], sv[1]), mx1 = fmaxf(sv[2], sv[3]);
#pragma unroll
                for (int k = 4; k < 32; k += 4) { mx0 = max3(mx0, sv[k], sv[k + 1]); mx1 = max3(mx1, sv[k + 2], sv[k + 3]); }
                const float mx = fmaxf(mx0, mx1);
                float corr = 1.f;
                const bool moved = mx > m_ref + kTau;          // also the first step with an open agent (m_ref = kRefFloor)
                if (moved) {
                    corr = fast_exp2((m_ref - mx) * kLog2e);
                    m_ref = mx;
                    l *= corr;
                }
                const bool any_moved = __any_sync(0xffffffffu, moved);
                // Every lane's biases are in registers once the vote on their maxima is known: the arriving lane depends on it.
                if (has_b2 && lane == (any_moved ? 31 : 0)) pipe_arrive(pp, BAR_B_EMPTY + bar);
                uint32_t pk[16];
                {
                    const float nb = -m_ref * kLog2e;
                    float2 s01 = make_float2(0.f, 0.f), s23 = make_float2(0.f, 0.f);
                    const float2 l2e = make_float2(kLog2e, kLog2e), nb2 = make_float2(nb, nb);
#pragma unroll
                    for (int k = 0; k < 16; k += 2) {
                        const float2 a0 = ffma2(make_float2(sv[2 * k], sv[2 * k + 1]), l2e, nb2);
                        const float2 a1 = ffma2(make_float2(sv[2 * k + 2], sv[2 * k + 3]), l2e, nb2);
                        const float2 p01 = make_float2(fast_exp2(a0.x), fast_exp2(a0.y));     // exp2(-inf) = 0 past the last agent
                        const float2 p23 = make_float2(fast_exp2(a1.x), fast_exp2(a1.y));
                        pk[k] = pack2<T>(p01.x, p01.y);
                        pk[k + 1] = pack2<T>(p23.x, p23.y);
                        if (ROUNDED) { add_pair<T>(s01, pk[k]); add_pair<T>(s23, pk[k + 1]); }
                        else { s01 = fadd2(s01, p01); s23 = fadd2(s23, p23); }
                    }
                    l += (s01.x + s01.y) + (s23.x + s23.y);
                }
                tmem_st16(tS + 64 * b, pk);
                if (a > 0 && any_moved) {                      // rare: the accumulator follows, once the products of the step before are done
                    wait_par(pp, BAR_PV + 2 * team + (b ^ 1), (j - 1) >> 1, kTimeoutTile);
                    tc_fence_after_sync();
#pragma unroll
                    for (int hh = 0; hh < 4; ++hh) {
                        float ra[16];
                        uint32_t wa[16];
                        tmem_ld16(tO + 16 * hh, ra);
                        tmem_ld_wait();
#pragma unroll
                        for (int k = 0; k < 16; ++k) wa[k] = __float_as_uint(ra[k] * corr);
                        tmem_st16(tO + 16 * hh, wa);
                    }
                }
                if (a == steps - 1) {
                    // (with two steps nothing else holds the (max, sum) of this tile back until those of the tile before have been read)
                    if (steps == 2 && i >= 2) wait_par(pp, BAR_O_EMPTY + team, (i >> 1) - 1, kTimeoutRole);
                    reinterpret_cast<float2*>(smem + OFF_ML)[(team * 2 + ((i >> 1) & 1)) * 256 + half * 128 + row] = make_float2(m_ref, l);
                    pipe_arrive_warp(pp, BAR_ML + team, lane);
                }
                tmem_st_wait();
                tc_fence_before_sync();
                pipe_arrive_warp(pp, BAR_P_FULL + bar, lane);
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc<512>(pp.tmem);
}

// ------------------------------------------------------------------------------------- host
bool broadcast_umma_eligible(int dtype, int n_agents, int n_tokens, int d) {
    if (dtype != kBF16 && dtype != kF16) return false;
    if (n_agents <= 64 || n_agents > 256 || n_agents % 8 != 0 || d > 64 || d % 8 != 0 || n_tokens < QT) return false;
    return encode_tiled_fn() != nullptr;
}

template <typename T, bool RUN, bool ROUNDED>
static cudaError_t launch_bc_umma_t(const UmmaBcArgs& g, int splits, cudaStream_t st) {
    static std::atomic<unsigned long long> done;
    cudaError_t e = allow_smem(broadcast_umma_kernel<T, RUN, ROUNDED>, done, smem_bytes(RUN));
    if (e != cudaSuccess) return e;
    return launch_dependent(broadcast_umma_kernel<T, RUN, ROUNDED>, dim3(splits, g.a.slabs), NT, smem_bytes(RUN), st, g);
}

// Map of B2 [heads][H][W][n] with boxes of 64 agents x a tile of tokens.
static bool make_map_b2(CUtensorMap* out, const void* base, uint64_t heads, uint64_t H, uint64_t W, uint64_t n, uint32_t th, uint32_t tw) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn || (reinterpret_cast<uintptr_t>(base) & 15u) || n % 8) return false;
    const cuuint64_t dims[4] = {n, W, H, heads}, strides[3] = {2 * n, 2 * n * W, 2 * n * W * H};
    const cuuint32_t box[4] = {64, tw, th, 1}, estr[4] = {1, 1, 1, 1};
    return fn(out, CU_TENSOR_MAP_DATA_TYPE_UINT16, 4, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// cudaErrorNotSupported: a tensor map could not be encoded.
cudaError_t launch_broadcast_umma(int dtype, const AttnArgs& p, int sm_count, cudaStream_t st) {
    UmmaBcArgs g;
    memset(&g, 0, sizeof(g));
    g.a = p;
    g.steps = (p.cols + 63) / 64;
    const uint64_t S = p.slabs, n = p.cols;
    const int batch = p.slabs / p.heads, patches = ((p.W + TW - 1) / TW) * ((p.H + TH - 1) / TH), runs = (p.rows + QT - 1) / QT;
    unsigned long long dims[2], strides[3];
    bool hf;
    if (!tok_map_dims(p.lin, batch, p.heads, (long long)p.rows, &hf, dims, strides)) return cudaErrorNotSupported;
    g.hf = hf;
    auto maps = [&](bool run) {
        const uint64_t H = run ? 1 : p.H, W = run ? p.rows : p.W;
        const uint32_t th = run ? 1 : TH, tw = run ? QT : TW;
        g.tiles_x = run ? runs : (p.W + TW - 1) / TW;
        g.tiles = run ? runs : patches;
        return make_map_grid5d_u16(&g.tm_q, hf, p.qm, p.lin, batch, p.heads, H, W, th, tw, p.d) && (!p.bias || make_map_b2(&g.tm_b, p.bias, p.heads, H, W, n, th, tw)) &&
               (!p.dwc_w || make_map_grid5d_u16(&g.tm_h, hf, p.dwc_v, p.lin, batch, p.heads, H, W, run ? 1 : TH + 2, run ? kRunRows : TW + 2, p.d));
    };
    if (!make_map_2d_u16(&g.tm_a, p.km, S * n, p.d, 128, 64)) return cudaErrorNotSupported;
    if (!make_map_2d_u16(&g.tm_va, p.vm, S * n, p.d, 128, 64)) return cudaErrorNotSupported;
    // Whole pass on patches over that on runs (256 and 144 agents, 1 and 16 slabs): as many patches as runs 0.95 to 1.02 (16 slabs of 128 x 128, 144
    // agents 95.5 and 100 us), 1.05 times as many 0.97 to 1.02, 1.2 times 1.00 to 1.12, 1.4 times 1.10 to 1.16, twice 1.10 to 1.45, sixteen times
    // 2.5 to 8 (16 slabs of 16384 x 1, 256 agents 852 and 105 us).  Strides that express patches alone: those.
    const bool run = 8LL * patches > 9LL * runs && maps(true);
    if (!run && !maps(false)) return cudaErrorNotSupported;
    int splits = sm_count / p.slabs;                        // one block per SM, one wave
    if (splits < 1) splits = 1;
    if (splits > g.tiles) splits = g.tiles;
    g.tps = (g.tiles + splits - 1) / splits;
    splits = (g.tiles + g.tps - 1) / g.tps;
    auto go = [&](auto t) {
        using T = decltype(t);
        const bool rounded = umma_sums_rounded(p.rows, p.d);
        return run ? rounded ? launch_bc_umma_t<T, true, true>(g, splits, st) : launch_bc_umma_t<T, true, false>(g, splits, st)
                   : rounded ? launch_bc_umma_t<T, false, true>(g, splits, st) : launch_bc_umma_t<T, false, false>(g, splits, st);
    };
    if (dtype == kBF16) return go(__nv_bfloat16{});
    if (dtype == kF16) return go(__half{});
    return cudaErrorInvalidValue;
}

}  // namespace aa
