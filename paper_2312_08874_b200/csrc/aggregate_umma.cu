// Agent aggregation V_A = softmax(scale1 * A K^T + B1) V (Eq. 3, Eq. 5) for large agent counts
// (64 < n <= 256, d <= 64, 16-bit elements) on the 5th-generation tensor cores.
//
// Grid: (splits, slabs), one block of 19 warps per SM.  A block keeps the slab's agents resident (up to
// two 128-row operand blocks) and streams its share of the slab's 64-token tiles (K, V and the matching
// B1 columns) through a four-stage TMA ring.  Two chains of eight row warps work beside one another: agents 0-127 and 128-255 of every
// tile, or (up to 128 agents) the even and the odd tiles.  A chain's logits alternate between two buffers in tensor memory: while the
// softmax of one tile runs, the products of the one before and the logits of the next are under way.
//   warp 16 "producer":  one lane issues every TMA copy, ahead of the others through full/empty mbarriers.
//   warps 17, 18 "MMA issuers", one per chain: the products P V of a tile once its probabilities are written, then the logits
//                        S = A_block K^T two tiles on over them (instructions of one thread run in their order).
//   warps 0-15 "row warps": thread (agent row, token half): reads its 32 logits of the tile from tensor
//                        memory, adds scale and bias, keeps its own running maximum / sum (no reduction
//                        crosses threads: each token half has its own accumulator in tensor memory),
//                        writes the probabilities back over them as the A operand of P V.
//                        A row's reference maximum moves only when exceeded by a margin; only then does the thread wait for products, and
//                        rescales its accumulator row in tensor memory.
// At the end the two token halves of a row, and the chains of up to 128 agents, meet in shared memory and the block writes one partial state;
// a second small kernel merges the slab's partials in a fixed order, spread over many blocks (a merge by
// the slab's last block alone took longer than the streaming part).
// Every wait is bounded (pipe.cuh).  No TMA multicast, no clusters.
//
// What bounds it: the row warps' instructions and exponentials (half of the time at the special-function rate), then HBM.  With probabilities through shared
// memory, a wait for the products of the tile before in every tile and arrivals of single threads, 16 slabs of a 256 x 256 grid with 256
// agents took 177 us; this way 133.  (A state per chain of up to 128 agents gave the merge twice as much to read: one slab of 128 x 128 tokens, 128 agents,
// whole pass 21.5 us; joined in the block 18.8.)
#include "merge.cuh"
#include "stream_common.cuh"

#include <cstring>

namespace aa {

namespace {
constexpr int KT = 64;                 // tokens per tile
constexpr int NROW = 512;              // row-warp threads
constexpr int NT = NROW + 96;          // + producer warp + two MMA issuer warps (logits, products)
constexpr int STAGES = 4;
constexpr int kTile = 64 * 128;        // swizzled [64][64] tile of 16-bit elements
constexpr float kTau = 5.5f;           // margin (natural units) before a row's reference maximum moves
constexpr int kTimeoutTile = 3, kTimeoutLoads = 4, kTimeoutRole = 6;

// shared memory (bytes from a 1024-aligned base)
constexpr int OFF_BAR = 0;                               // mbarriers
constexpr int OFF_A = 1024;                              // agents [256][128 B]
constexpr int OFF_RING = OFF_A + 4 * kTile;              // STAGES x (K | V | B1 [256][128 B], later the probabilities)
constexpr int kStage = 2 * kTile + 4 * kTile;
constexpr int kSmemBytes = OFF_RING + STAGES * kStage + 1024;
static_assert(kSmemBytes <= 232448 && kSmemBytes > 116 * 1024, "one block per SM");

// mbarriers (cb: + 2 chain + parity of the chain's tile)   count            waiter
constexpr int BAR_FULL = 0;       // [STAGES]        tx             MMA issuers
constexpr int BAR_EMPTY = 4;      // [STAGES]        one commit per chain that takes the tile     producer
constexpr int BAR_S_FULL = 8;     // cb              commit         the chain's row warps
constexpr int BAR_P_FULL = 12;    // cb              8 warps        the chain's MMA issuer        (logits and biases read as well)
constexpr int BAR_PV = 16;        // cb              commit         the chain's row warps (where a reference moves, and at the end)
constexpr int BAR_AG = 20;        //                 tx             both MMA issuers
constexpr int BAR_DRAIN = 21;     // [chain]         commit         MMA issuer, once, at its end
constexpr int kBars = 23;

// tensor memory, columns of a chain: logits (then probabilities) of two tiles 64 each, accumulators of two token halves 64 each
constexpr uint32_t TM_CHAIN = 256, TM_O = 128;

struct UmmaAggArgs {
    AttnArgs a;
    int rows_pad, tps;                 // padded agent rows (128 or 256), tiles per split
    int hf_k, hf_v;                    // dimension order of the K and V maps (tma_load_tok)
    alignas(64) CUtensorMap tm_a, tm_k, tm_v, tm_b;
};
}  // namespace

// ROUNDED: see umma_sums_rounded; MB: 128-row agent blocks
template <typename T, bool ROUNDED, int MB>
__global__ void __launch_bounds__(NT, 1) aggregate_umma_kernel(const __grid_constant__ UmmaAggArgs g) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ int s_dead;
    __shared__ uint32_t s_tmem;
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int fmt = Elem<T>::kIsBf16 ? 1 : 0;
    const AttnArgs& p = g.a;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int split = blockIdx.x, slab = blockIdx.y;
    const int head = slab % p.heads;
    const int n = p.rows, N = p.cols;
    constexpr int rows_pad = 128 * MB;
    const bool has_bias = p.bias != nullptr;
    const int tiles_all = (N + KT - 1) / KT;
    const int t0 = split * g.tps, t1 = min(tiles_all, t0 + g.tps);
    const int tiles = t1 - t0;                            // >= 1 by the plan

    Pipe pp;
    pp.status = p.status;
    pp.dead = &s_dead;
    pp.bars = smem_u32(smem + OFF_BAR);
    if (tid == 0) {
        s_dead = 0;
        for (int i = 0; i < kBars; ++i)
            mbar_init(pp.bars + 8 * i, (i >= BAR_P_FULL && i < BAR_PV) ? 8u : (i >= BAR_EMPTY && i < BAR_S_FULL) ? (uint32_t)MB : 1u);
        mbar_fence_init();
    }
    if (warp == 0) tmem_alloc<512>(smem_u32(&s_tmem));
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pp.tmem = s_tmem;
    pdl_wait_prior();                                     // the agents come from the preceding kernel
    pdl_release_next();

    const uint32_t sA = smem_u32(smem + OFF_A), ring = smem_u32(smem + OFF_RING);
    const size_t pf = partial_floats(rows_pad, 64);
    float* part = p.partials + ((size_t)slab * gridDim.x + split) * pf;

    if (warp == 16) {
        // ------------------------------------------------------------------ producer
        if (lane == 0) {
            mbar_arrive_expect_tx(pipe_bar(pp, BAR_AG), (uint32_t)MB * 2 * kTile);
            for (int mb = 0; mb < MB; ++mb) tma_load_2d(sA + mb * 2 * kTile, &g.tm_a, 0, slab * n + 128 * mb, pipe_bar(pp, BAR_AG));
            const uint32_t tx = 2 * kTile + (has_bias ? (uint32_t)MB * 2 * kTile : 0u);
            for (int t = 0; t < tiles && !pipe_dead(pp); ++t) {
                const int s = t % STAGES, c0 = (t0 + t) * KT;
                if (t >= STAGES) wait_spin(pp, BAR_EMPTY + s, t / STAGES - 1, kTimeoutRole);
                const uint32_t bar = pipe_bar(pp, BAR_FULL + s), dst = ring + s * kStage;
                mbar_arrive_expect_tx(bar, tx);
                tma_load_tok(dst, &g.tm_k, g.hf_k, c0, head, slab / p.heads, bar);
                tma_load_tok(dst + kTile, &g.tm_v, g.hf_v, c0, head, slab / p.heads, bar);
                if (has_bias)
                    for (int mb = 0; mb < MB; ++mb) tma_load_2d(dst + 2 * kTile + mb * 2 * kTile, &g.tm_b, c0, head * n + 128 * mb, bar);
            }
        }
        __syncwarp();
    } else if (warp >= 17) {
        // ------------------------------------------------------------------ MMA issuer of a chain (the whole warp runs the loop; one elected lane issues)
        const int m = warp - 17, first = MB == 1 ? m : 0, step = MB == 1 ? 2 : 1, count = (tiles - first + step - 1) / step;
        if (count > 0) {
            const uint32_t idK = umma_idesc(fmt, 128, 64, 0), idMN = umma_idesc(fmt, 128, 64, 1);
            const uint64_t dA = umma_desc_sw128(sA) + (MB == 1 ? 0 : 1024 * m), dRing = umma_desc_sw128(ring);
            const uint32_t tc = pp.tmem + TM_CHAIN * m;
            // descriptor start addresses count 16-byte units: + 2 per K-step of a K-major operand (32 bytes), + 128 per K-step of an MN-major
            // operand (16 rows of 128 bytes), + 1024 per 128-row block; + 8 columns per K-step of an operand in tensor memory
            auto logits = [&](int k) {
                const int t = first + step * k, s = t % STAGES, b = k & 1;
                wait_spin(pp, BAR_FULL + s, t / STAGES, kTimeoutTile);
                tc_fence_after_sync();
                const uint64_t dK = dRing + (uint64_t)(s * (kStage >> 4));
#pragma unroll
                for (int i = 0; i < 4; ++i) umma_ss_w(tc + 64 * b, dA + 2 * i, dK + 2 * i, idK, i > 0);
                umma_commit_w(pipe_bar(pp, BAR_S_FULL + 2 * m + b));
            };
            wait_spin(pp, BAR_AG, 0, kTimeoutLoads);
            logits(0);
            if (count > 1) logits(1);
            for (int k = 0; k < count && !pipe_dead(pp); ++k) {
                const int t = first + step * k, s = t % STAGES, b = k & 1;
                wait_spin(pp, BAR_P_FULL + 2 * m + b, k >> 1, kTimeoutRole);
                tc_fence_after_sync();
                const int ntok = min(KT, N - (t0 + t) * KT);
                const uint64_t dV = dRing + (uint64_t)(s * (kStage >> 4)) + (uint64_t)(kTile >> 4);
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    if (32 * c < ntok) {
                        const uint32_t od = tc + TM_O + 64 * c, oa = tc + 64 * b + 32 * c;
                        umma_ts_w(od, oa, dV + 256 * c, idMN, k > 0);
                        umma_ts_w(od, oa + 8, dV + 256 * c + 128, idMN, 1u);
                    }
                umma_commit_w(pipe_bar(pp, BAR_EMPTY + s));
                umma_commit_w(pipe_bar(pp, BAR_PV + 2 * m + b));
                if (k + 2 < count) logits(k + 2);
            }
            umma_drain_w(pp, BAR_DRAIN + m);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ row warps
        const int m = (warp >> 2) & 1, c = warp >> 3, mb = MB == 1 ? 0 : m;    // chain, token half, agent block
        const int first = MB == 1 ? m : 0, step = MB == 1 ? 2 : 1, count = (tiles - first + step - 1) / step;
        const int row = 128 * mb + 32 * (warp & 3) + lane;     // agent row (padded)
        const uint32_t lane_base = ((uint32_t)(32 * (warp & 3))) << 16;
        const uint32_t tS = pp.tmem + TM_CHAIN * m + 32 * c + lane_base, tO = pp.tmem + TM_CHAIN * m + TM_O + 64 * c + lane_base;
        float m_ref = kRefFloor, l = 0.f;
        bool started = false;
        for (int k = 0; k < count; ++k) {
            const int t = first + step * k, b = k & 1, s = t % STAGES;
            const int valid = min(32, N - ((t0 + t) * KT + 32 * c));      // tokens of this thread's half (uniform; may be <= 0)
            wait_par(pp, BAR_S_FULL + 2 * m + b, k >> 1, kTimeoutTile);
            tc_fence_after_sync();
            if (valid > 0) {
                float sv[32];
                tmem_ld32(tS + 64 * b, *reinterpret_cast<uint32_t(*)[32]>(sv));
                tmem_ld_wait();
                if (has_bias) {                              // logits in natural units: scale1 * a.k + b1
                    const unsigned char* sB = smem + OFF_RING + s * kStage + 2 * kTile + row * 128;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint4 raw = *reinterpret_cast<const uint4*>(sB + (((4 * c + j) ^ (row & 7)) << 4));
                        const uint32_t w4[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {            // packed pairs: one instruction per two logits
                            const float2 r2 = ffma2(make_float2(sv[8 * j + 2 * i], sv[8 * j + 2 * i + 1]), make_float2(p.scale, p.scale), unpack2<T>(w4[i]));
                            sv[8 * j + 2 * i] = r2.x; sv[8 * j + 2 * i + 1] = r2.y;
                        }
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float2 r2 = fmul2(make_float2(sv[2 * i], sv[2 * i + 1]), make_float2(p.scale, p.scale));
                        sv[2 * i] = r2.x; sv[2 * i + 1] = r2.y;
                    }
                }
                if (valid < 32) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) if (i >= valid) sv[i] = -INFINITY;
                }
                float mx0 = fmaxf(sv[0], sv[1]), mx1 = fmaxf(sv[2], sv[3]);
#pragma unroll
                for (int i = 4; i < 32; i += 4) { mx0 = max3(mx0, sv[i], sv[i + 1]); mx1 = max3(mx1, sv[i + 2], sv[i + 3]); }
                const float mx = fmaxf(mx0, mx1);
                float corr = 1.f;
                const bool moved = mx > m_ref + kTau;          // also the first tile with an open key (m_ref = kRefFloor)
                if (moved) {
                    corr = fast_exp2((m_ref - mx) * kLog2e);
                    m_ref = mx;
                    l *= corr;
                }
                uint32_t pk[16];
                {
                    const float nb = -m_ref * kLog2e;
                    float2 s01 = make_float2(0.f, 0.f), s23 = make_float2(0.f, 0.f);
                    const float2 l2e = make_float2(kLog2e, kLog2e), nb2 = make_float2(nb, nb);
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const float2 a0 = ffma2(make_float2(sv[2 * i], sv[2 * i + 1]), l2e, nb2);
                        const float2 a1 = ffma2(make_float2(sv[2 * i + 2], sv[2 * i + 3]), l2e, nb2);
                        const float2 p01 = make_float2(fast_exp2(a0.x), fast_exp2(a0.y));     // exp2(-inf) = 0 past the range
                        const float2 p23 = make_float2(fast_exp2(a1.x), fast_exp2(a1.y));
                        pk[i] = pack2<T>(p01.x, p01.y);
                        pk[i + 1] = pack2<T>(p23.x, p23.y);
                        if (ROUNDED) { add_pair<T>(s01, pk[i]); add_pair<T>(s23, pk[i + 1]); }
                        else { s01 = fadd2(s01, p01); s23 = fadd2(s23, p23); }
                    }
                    l += (s01.x + s01.y) + (s23.x + s23.y);
                }
                tmem_st16(tS + 64 * b, pk);
                if (started && __any_sync(0xffffffffu, moved)) {   // rare: the accumulator follows, once the products of the tile before are done
                    wait_par(pp, BAR_PV + 2 * m + (b ^ 1), (k - 1) >> 1, kTimeoutTile);
                    tc_fence_after_sync();
#pragma unroll
                    for (int hh = 0; hh < 4; ++hh) {
                        float ra[16];
                        uint32_t wa[16];
                        tmem_ld16(tO + 16 * hh, ra);
                        tmem_ld_wait();
#pragma unroll
                        for (int i = 0; i < 16; ++i) wa[i] = __float_as_uint(ra[i] * corr);
                        tmem_st16(tO + 16 * hh, wa);
                    }
                }
                started = true;
                tmem_st_wait();
            }
            tc_fence_before_sync();
            pipe_arrive_warp(pp, BAR_P_FULL + 2 * m + b, lane);
        }
        if (count > 0) {
            wait_par(pp, BAR_PV + 2 * m + ((count - 1) & 1), (count - 1) >> 1, kTimeoutTile);
            tc_fence_after_sync();
        }
        // both chains are through with the ring before its memory is reused for the exchange below
        asm volatile("bar.sync 3, %0;\n" ::"n"(NROW) : "memory");
        // the two token halves of a row meet in shared memory (the ring is drained: every product is done)
        float o[64];
        {
            uint32_t ra[32], rb[32];
            tmem_ld32(tO, ra);
            tmem_ld32(tO + 32, rb);
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 32; ++k) {
                o[k] = started ? __uint_as_float(ra[k]) : 0.f;
                o[32 + k] = started ? __uint_as_float(rb[k]) : 0.f;
            }
        }
        tc_fence_before_sync();
        float* sX = reinterpret_cast<float*>(smem + OFF_RING) + (size_t)(128 * m + (row & 127)) * 68;      // [256][68]: row, m, l
        if (c == 1) {
#pragma unroll
            for (int k = 0; k < 16; ++k) *reinterpret_cast<float4*>(sX + 4 * k) = make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
            sX[64] = m_ref; sX[65] = started ? l : 0.f;
        }
        asm volatile("bar.sync %0, 256;\n" ::"r"(1 + m) : "memory");       // the chain's own barrier
        if (c == 0) {
            // state of the row: (reference, sum, products), joined with another one in shared memory
            float mm = m_ref, ls = started ? l : 0.f;
            auto join = [&](const float* x) {
                const float om = x[64], mn = fmaxf(mm, om), bs = (mn == -INFINITY) ? 0.f : mn;
                const float wa = fast_exp2((mm - bs) * kLog2e), wb = fast_exp2((om - bs) * kLog2e);
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const float4 v = *reinterpret_cast<const float4*>(x + 4 * k);
                    o[4 * k] = o[4 * k] * wa + v.x * wb; o[4 * k + 1] = o[4 * k + 1] * wa + v.y * wb;
                    o[4 * k + 2] = o[4 * k + 2] * wa + v.z * wb; o[4 * k + 3] = o[4 * k + 3] * wa + v.w * wb;
                }
                ls = ls * wa + x[65] * wb;
                mm = mn;
            };
            auto put = [&](float* x) {
#pragma unroll
                for (int k = 0; k < 16; ++k) *reinterpret_cast<float4*>(x + 4 * k) = make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
            };
            join(sX);
            if (MB == 1) {                                 // and the other chain's (its tiles of the same agents)
                if (m == 1) { put(sX); sX[64] = mm; sX[65] = ls; }
                asm volatile("bar.sync 4, 256;\n" ::: "memory");
                if (m == 0) join(sX + 128 * 68);
            }
            if (MB == 2 || m == 0) {
                part[row] = mm * kLog2e;                   // the merge works in log2 units
                part[rows_pad + row] = ls;
                put(part + 2 * rows_pad + row * 64);
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc<512>(pp.tmem);
}

// Merge of the slab's partial states into V_A: grid (rows, slabs); a thread takes a row's four channels and every SHARES-th part, its
// loads in flight together; the shares meet in shared memory (fixed order: bit-reproducible).  One share for up to sixteen parts; one slab
// in 60 parts: 34 us with one share, 5.3 us with four.
template <typename T, int SHARES>
__global__ void __launch_bounds__(256) merge_umma_kernel(const float* __restrict__ partials, int parts, int rows_pad,
                                                         int n, int d, T* __restrict__ out) {
    constexpr int kRows = 16 / SHARES;
    __shared__ float4 s_num[SHARES][kRows][16];
    __shared__ float2 s_ml[SHARES][kRows];
    const int slab = blockIdx.y;
    pdl_wait_prior();
    pdl_release_next();
    const size_t pf = partial_floats(rows_pad, 64);
    const float* base = partials + (size_t)slab * parts * pf;
    const int cg = threadIdx.x & 15, ri = (threadIdx.x >> 4) % kRows, share = threadIdx.x / (16 * kRows);
    const int r = blockIdx.x * kRows + ri, rr = min(r, n - 1);
    float mx = -INFINITY, den = 0.f;
    float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q0 = share; q0 < parts; q0 += 8 * SHARES) {
        float m[8], l[8];
        float4 a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int q = q0 + SHARES * i;
            m[i] = -INFINITY;
            if (q < parts) {
                const float* pq = base + q * pf;
                m[i] = __ldcg(pq + rr);
                l[i] = __ldcg(pq + rows_pad + rr);
                a[i] = __ldcg(reinterpret_cast<const float4*>(pq + 2 * (size_t)rows_pad + (size_t)rr * 64 + 4 * cg));
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (q0 + SHARES * i >= parts) break;
            const float mn = fmaxf(mx, m[i]), bs = (mn == -INFINITY) ? 0.f : mn;
            const float c0 = exp2f(mx - bs), c1 = exp2f(m[i] - bs);
            den = den * c0 + l[i] * c1;
            num.x = num.x * c0 + a[i].x * c1; num.y = num.y * c0 + a[i].y * c1;
            num.z = num.z * c0 + a[i].z * c1; num.w = num.w * c0 + a[i].w * c1;
            mx = mn;
        }
    }
    s_num[share][ri][cg] = num;
    if (cg == 0) s_ml[share][ri] = make_float2(mx, den);
    __syncthreads();
    if (share != 0 || r >= n || cg >= d >> 2) return;
    float mm = -INFINITY;
#pragma unroll
    for (int q = 0; q < SHARES; ++q) mm = fmaxf(mm, s_ml[q][ri].x);
    const float bs = (mm == -INFINITY) ? 0.f : mm;
    den = 0.f;
    num = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < SHARES; ++q) {
        const float c = exp2f(s_ml[q][ri].x - bs);
        const float4 a = s_num[q][ri][cg];
        den += s_ml[q][ri].y * c;
        num.x = fmaf(a.x, c, num.x); num.y = fmaf(a.y, c, num.y);
        num.z = fmaf(a.z, c, num.z); num.w = fmaf(a.w, c, num.w);
    }
    const float inv = 1.f / den;
    uint2 o;
    o.x = pack2<T>(num.x * inv, num.y * inv);
    o.y = pack2<T>(num.z * inv, num.w * inv);
    *reinterpret_cast<uint2*>(out + ((size_t)slab * n + r) * d + 4 * cg) = o;
}

// ------------------------------------------------------------------------------------- host
bool aggregate_umma_eligible(int dtype, int n_agents, int n_tokens, int d, bool has_bias) {
    if (dtype != kBF16 && dtype != kF16) return false;
    if (n_agents <= 64 || n_agents > 256 || d > 64 || d % 8 != 0 || n_tokens < KT) return false;
    if (has_bias && n_tokens % 8 != 0) return false;        // TMA needs 16-byte aligned bias rows
    return encode_tiled_fn() != nullptr;
}

AggPlan plan_aggregate_umma(int slabs, int n_agents, int n_tokens, int d, int sm_count) {
    (void)d;
    AggPlan pl;
    pl.rows_pad = n_agents <= 128 ? 128 : 256;
    pl.dpad = 64;
    pl.row_blocks = 1;
    const int tiles = (n_tokens + KT - 1) / KT;
    int splits = sm_count / slabs;                          // one block per SM, one wave
    if (splits < 1) splits = 1;
    if (splits > (tiles + 3) / 4) splits = (tiles + 3) / 4; // at least four tiles per block
    if (splits < 1) splits = 1;
    if (splits > 64) splits = 64;
    const int tps = (tiles + splits - 1) / splits;
    pl.splits = (tiles + tps - 1) / tps;
    pl.parts = pl.splits;
    return pl;
}

template <typename T>
static cudaError_t launch_umma_t(const UmmaAggArgs& g, cudaStream_t st) {
    const bool one = g.rows_pad == 128;
    auto kern = umma_sums_rounded(g.a.cols, g.a.d) ? (one ? aggregate_umma_kernel<T, true, 1> : aggregate_umma_kernel<T, true, 2>)
                                                   : (one ? aggregate_umma_kernel<T, false, 1> : aggregate_umma_kernel<T, false, 2>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    dim3 grid(g.a.splits, g.a.slabs);
    e = launch_dependent(kern, grid, NT, kSmemBytes, st, g);
    if (e != cudaSuccess) return e;
    const int parts = g.a.splits;
    const bool few = parts <= 16;
    const int rows = few ? 16 : 4;
    return launch_dependent(few ? merge_umma_kernel<T, 1> : merge_umma_kernel<T, 4>, dim3((g.a.rows + rows - 1) / rows, g.a.slabs), 256, 0, st,
                            (const float*)g.a.partials, parts, g.rows_pad, g.a.rows, g.a.d, static_cast<T*>(g.a.out));
}

// cudaErrorNotSupported: a tensor map could not be encoded.
cudaError_t launch_aggregate_umma(int dtype, const AttnArgs& p, const AggPlan& plan, cudaStream_t st) {
    UmmaAggArgs g;
    memset(&g, 0, sizeof(g));
    g.a = p;
    g.a.splits = plan.splits;
    g.rows_pad = plan.rows_pad;
    const int tiles = (p.cols + KT - 1) / KT;
    g.tps = (tiles + plan.splits - 1) / plan.splits;
    const uint64_t S = p.slabs, N = p.cols, n = p.rows;
    if (!make_map_2d_u16(&g.tm_a, p.qm, S * n, p.d, 128, 64)) return cudaErrorNotSupported;
    const int batch = p.slabs / p.heads;
    if (!make_map_tok_u16(&g.tm_k, &g.hf_k, p.km, p.lin, batch, p.heads, (long long)N, p.d, 64, true)) return cudaErrorNotSupported;
    if (!make_map_tok_u16(&g.tm_v, &g.hf_v, p.vm, p.lin, batch, p.heads, (long long)N, p.d, 64, true)) return cudaErrorNotSupported;
    if (p.bias && !make_map_2d_u16(&g.tm_b, p.bias, (uint64_t)p.heads * n, N, 128, 64)) return cudaErrorNotSupported;
    if (dtype == kBF16) return launch_umma_t<__nv_bfloat16>(g, st);
    if (dtype == kF16) return launch_umma_t<__half>(g, st);
    return cudaErrorInvalidValue;
}

}  // namespace aa
