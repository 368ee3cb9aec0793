// Backward pass of the agent-attention module: the agent values V_A = softmax(scale A K^T + B1) V in fp32 and as 16-bit terms, and the row
// statistics, on the 5th-generation tensor cores (16-bit tensors of up to 64 channels).
//
// Rows = agents, so that a softmax row belongs to a thread pair and the probabilities go back to tensor memory as the A operand of P V
// without a transpose.  Two precisions: mixed (A one term, P two) and full (bf16, A and P three terms; see bwd_terms.cuh).  Two row
// layouts: a block of 128 agents, or (STACK, up to 64 agents) the agents twice, lanes 0 .. 63 with the first 64 tokens of a tile and lanes
// 64 .. 127 with the others; the probabilities of the other half are zeros that are written once.
//
// One block per SM takes a contiguous run of the (slab, tile of 128 tokens) sequence.  Roles:
//   warps 0-7   row warps: two threads per row share its columns and meet over the row's maximum; P goes to tensor memory as terms
//   warps 8-11  thread = row: the product of every tile joins the running sum in fp32 registers (term_sum says why), so nothing is rescaled
//               in tensor memory
//   warp 12     TMA: K and V, three stages; the biases, two
//   warp 13, 14 issue the logits (a tile ahead) and P V
// Runs that hold part of a slab leave partial states; bwd_values_merge_kernel joins them, one warp per row.
//
// What bounds it: full, the splits and the row warps' waits (16 slabs of a 128 x 128 grid, 256 agents: 104 + 8 us, 495 TFLOP/s of term
// pairs, a third of the bf16 rate; bwd_sums_kernel 317 us); mixed, the start of the kernel (about 12 of 27 us at 64 slabs of 56 x 56).
#include "bwd_terms_launch.cuh"
#include "stream_common.cuh"

#include <algorithm>
#include <cstring>

namespace aa {

namespace {

constexpr int kTok = 128;                    // tokens per tile
constexpr int kTile = kTok * 128;            // bytes of a swizzled [128][64] tile of 16-bit elements
constexpr int kMat = 64 * 128;
constexpr int kStages = 3, kBiasStages = 2;
constexpr int kRowThreads = 256, kThreads = kRowThreads + 128 + 96;
constexpr int kState = 128 * 64 + 128 * 4;   // floats of a partial state: sums [128][64], then (reference, sum of half the columns) [128][2]

// shared memory (bytes from a 1024-aligned base)
constexpr int OFF_DEAD = 256, OFF_TMEM = 260;
constexpr int OFF_RING = 1024;                                // K | V
constexpr int OFF_BIAS = OFF_RING + kStages * 2 * kTile;      // two boxes of [rows][64 tokens], or two of [128 tokens][64 agents]
constexpr int OFF_F = OFF_BIAS + kBiasStages * 2 * kTile;     // [4 tiles][128] factor of the sums so far
constexpr int OFF_EX = OFF_F + 4 * 128 * 4;                   // [2 tiles][2 halves][128] maxima
constexpr int OFF_A = OFF_EX + 2 * 2 * 128 * 4;               // terms of A, 128 rows each
__host__ __device__ constexpr int a_buffers(int ta) { return ta == 1 ? 2 : 1; }          // (three terms: no room for a second slab's)
template <int TA> constexpr int kSmem = OFF_A + a_buffers(TA) * TA * kTile + 1024;
static_assert(OFF_A % 1024 == 0 && kSmem<3> <= 232448 && kSmem<1> > 116 * 1024, "one block per SM");

// mbarriers                        count             waiter
constexpr int BAR_FULL = 0;    // [3] tx              issuer of the logits
constexpr int BAR_BIAS = 3;    // [2] tx              row warps
constexpr int BAR_BREAD = 5;   // [2] row warps       producer: the biases have been read
constexpr int BAR_A = 7;       // [2] tx              issuer of the logits
constexpr int BAR_S = 9;       // [2] commit          row warps
constexpr int BAR_READ = 11;   // [2] row warps       issuer of the logits: they have been read
constexpr int BAR_P = 13;      //     row warps       issuer of P V: the probabilities are in tensor memory
constexpr int BAR_DONE = 14;   // [2] commit          row warps, output warps: P V of a tile
constexpr int BAR_OUT = 16;    // [2] output warps    issuer of P V: its result has been read
constexpr int BAR_DRAIN = 18;  // [2] commit          each issuer, once, at its end
constexpr int BAR_FREE = 20;   // [3] commit          producer: P V of the tile in this stage, the last to read it
constexpr int kBars = 23;
static_assert(8 * kBars <= OFF_DEAD, "mbarriers");
// A producer that is late must not find the barrier it waits on two phases further: the next phase of a stage's own barrier needs the
// very load that the producer is about to issue.
static_assert(kBars - BAR_FREE == kStages, "one release barrier per stage");
constexpr int kTimeoutTile = 3, kTimeoutRole = 6;

// tensor memory columns: logits, twice; terms of P (128 tokens = 64 columns each); products (twice where there is room)
constexpr uint32_t TM_S = 0, TM_P = 256;

struct Args {
    float* state;             // partial states [slabs][parts][row blocks][kState]
    int* status;
    int slabs, heads, N, n, d, tiles, blocks, parts;
    int bias;                 // 0: none; 1: tiles of token rows; 2: tiles of agent rows
    float scale;
    alignas(64) CUtensorMap tm_k, tm_v, tm_a, tm_b;
};
// run (of `lanes`) that holds tile x of `total`
__host__ __device__ inline int owner(long long x, long long lanes, long long total) {
    const unsigned long long v = (unsigned long long)(x + 1) * lanes - 1;
    return (v | (unsigned long long)total) >> 32 ? (int)(v / total) : (int)((uint32_t)v / (uint32_t)total);
}

// 8 consecutive columns of this thread's tensor-memory row <- registers
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
                 "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
template <typename T, int TA, int TP, bool STACK>
__global__ void __launch_bounds__(kThreads, 1) bwd_values_umma_kernel(const __grid_constant__ Args p) {
    constexpr int kFmt = Elem<T>::kIsBf16 ? 1 : 0, kCols = STACK ? 32 : 64, kD = TP == 2 ? 2 : 1;
    constexpr uint32_t TM_D = TM_P + TP * 64;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int N = p.N, n = p.n;
    const int rb = blockIdx.x % p.blocks, lanes = gridDim.x / p.blocks, me = blockIdx.x / p.blocks;      // block of agents; runs of its sequence
    const long long total = (long long)p.slabs * p.tiles, first = total * me / lanes;
    const int count = (int)(total * (me + 1) / lanes - first);
    int slab = (int)(first / p.tiles), tile = (int)(first - (long long)slab * p.tiles);     // of the role's current tile
    const uint32_t base = smem_u32(smem);
    float* f_s = reinterpret_cast<float*>(smem + OFF_F);

    Pipe pp;
    pp.status = p.status;
    pp.dead = reinterpret_cast<int*>(smem + OFF_DEAD);
    pp.bars = base;
    if (tid == 0) {
        *pp.dead = 0;
        for (int i = 0; i < kBars; ++i)
            mbar_init(pp.bars + 8 * i, (i >= BAR_BREAD && i < BAR_A) || (i >= BAR_READ && i <= BAR_P) ? 8u : i >= BAR_OUT && i < BAR_DRAIN ? 4u : 1u);
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
        if (++tile == p.tiles) { tile = 0; ++slab; }
    };
    // partial state of the current slab
    auto state = [&] { return p.state + (((size_t)slab * p.parts + (me - owner((long long)slab * p.tiles, lanes, total))) * p.blocks + rb) * kState; };

    if (warp == 12) {
        // ------------------------------------------------------------------ producer
        if (lane == 0) {
            int buf = 0;
            for (int i = 0; i < count && !pipe_dead(pp); ++i, advance()) {
                const int s = i % kStages, b = i & 1;
                if (i >= kStages) wait_spin(pp, BAR_FREE + s, i / kStages - 1, kTimeoutRole);
                const uint32_t bar = pipe_bar(pp, BAR_FULL + s), dst = base + OFF_RING + s * 2 * kTile;
                mbar_arrive_expect_tx(bar, 2 * kTile);
                tma_load_3d(dst, &p.tm_k, 0, tile * kTok, slab, bar);
                tma_load_3d(dst + kTile, &p.tm_v, 0, tile * kTok, slab, bar);
                if (i == 0 || tile == 0) {
                    // the last logits of the slab whose A this buffer holds: the slab before, or the one before that
                    constexpr int kBack = a_buffers(TA);
                    if (i >= kBack) wait_spin(pp, BAR_S + ((i - kBack) & 1), (i - kBack) >> 1, kTimeoutRole);
                    const uint32_t ba = pipe_bar(pp, BAR_A + buf);
                    mbar_arrive_expect_tx(ba, TA * kTile);
                    for (int t = 0; t < TA; ++t)
                        for (int h = 0; h < 2; ++h) tma_load_3d(base + OFF_A + (buf * TA + t) * kTile + h * kMat, &p.tm_a, 0, STACK ? 0 : rb * 128 + h * 64, t * p.slabs + slab, ba);
                    buf = (buf + 1) % kBack;
                }
                if (p.bias) {
                    if (i >= 2) wait_spin(pp, BAR_BREAD + b, (i >> 1) - 1, kTimeoutRole);
                    const uint32_t bb = pipe_bar(pp, BAR_BIAS + b), to = base + OFF_BIAS + b * 2 * kTile;
                    const int head = slab % p.heads;
                    mbar_arrive_expect_tx(bb, STACK ? kTile : 2 * kTile);
                    if (p.bias == 2) {
                        for (int h = 0; h < 2; ++h) tma_load_3d(to + h * (STACK ? kMat : kTile), &p.tm_b, tile * kTok + 64 * h, rb * 128, head, bb);
                    } else {
                        for (int h = 0; h < (STACK ? 1 : 2); ++h) tma_load_3d(to + h * kTile, &p.tm_b, rb * 128 + 64 * h, tile * kTok, head, bb);
                    }
                }
            }
        }
        __syncwarp();
    } else if (warp == 13) {
        // ------------------------------------------------------------------ logits, a tile ahead
        const uint32_t id = umma_idesc(kFmt, 128, 128, 0);
        uint64_t da = umma_desc_sw128(base + OFF_A);
        int slabs = 0;
        for (int i = 0; i < count && !pipe_dead(pp); ++i, advance()) {
            const int s = i % kStages, b = i & 1;
            if (i == 0 || tile == 0) {
                da = umma_desc_sw128(base + OFF_A + slabs % a_buffers(TA) * TA * kTile);
                wait_spin(pp, BAR_A + slabs % a_buffers(TA), slabs / a_buffers(TA), kTimeoutTile);
                ++slabs;
            }
            wait_spin(pp, BAR_FULL + s, i / kStages, kTimeoutTile);
            if (i >= 2) wait_spin(pp, BAR_READ + b, (i >> 1) - 1, kTimeoutRole);
            tc_fence_after_sync();
            const uint64_t dk = umma_desc_sw128(base + OFF_RING + s * 2 * kTile);
#pragma unroll
            for (int t = TA - 1; t >= 0; --t)
#pragma unroll
                for (int k = 0; k < 4; ++k) umma_ss_w(pp.tmem + TM_S + 128 * b, da + t * (kTile >> 4) + 2 * k, dk + 2 * k, id, t < TA - 1 || k > 0);
            umma_commit_w(pipe_bar(pp, BAR_S + b));
        }
        umma_drain_w(pp, BAR_DRAIN);
        __syncwarp();
    } else if (warp == 14) {
        // ------------------------------------------------------------------ P V
        const uint32_t id = umma_idesc(kFmt, 128, 64, 1);
        for (int i = 0; i < count && !pipe_dead(pp); ++i) {
            const int s = i % kStages, b = i & 1, db = i % kD;
            wait_spin(pp, BAR_P, i, kTimeoutRole);
            if (i >= kD) wait_spin(pp, BAR_OUT + db, i / kD - 1, kTimeoutRole);
            tc_fence_after_sync();
            const uint64_t dv = umma_desc_sw128(base + OFF_RING + s * 2 * kTile + kTile);
#pragma unroll
            for (int t = TP - 1; t >= 0; --t)
#pragma unroll
                for (int k = 0; k < 8; ++k) umma_ts_w(pp.tmem + TM_D + 64 * db, pp.tmem + TM_P + 64 * t + 8 * k, dv + 128 * k, id, t < TP - 1 || k > 0);
            umma_commit_w(pipe_bar(pp, BAR_FREE + s));
            umma_commit_w(pipe_bar(pp, BAR_DONE + b));
        }
        umma_drain_w(pp, BAR_DRAIN + 1);
        __syncwarp();
    } else if (warp >= 8) {
        // ------------------------------------------------------------------ sums
        const int q = warp & 3, r = 32 * q + lane;
        float2 acc[32];
        for (int i = 0; i < count; ++i, advance()) {
            const int b = i & 1, db = i % kD;
            wait_par(pp, BAR_DONE + b, i >> 1, kTimeoutTile);
            tc_fence_after_sync();
            const bool fresh = i == 0 || tile == 0;
            const float f = f_s[(i & 3) * 128 + r];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t o[32];
                tmem_ld32(pp.tmem + TM_D + 64 * db + ((uint32_t)(32 * q) << 16) + 32 * h, o);
                tmem_ld_wait();
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const float2 v = make_float2(__uint_as_float(o[2 * k]), __uint_as_float(o[2 * k + 1]));
                    float2& a = acc[16 * h + k];
                    a = fresh ? v : ffma2(a, make_float2(f, f), v);
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) pipe_arrive(pp, BAR_OUT + db);
            if (tile == p.tiles - 1 || i == count - 1) {               // the last tile of the slab in this block
                float4* dst = reinterpret_cast<float4*>(state() + r * 64);
                if ((STACK ? r & 63 : rb * 128 + r) < n)
#pragma unroll
                    for (int k = 0; k < 16; ++k) dst[k] = make_float4(acc[2 * k].x, acc[2 * k].y, acc[2 * k + 1].x, acc[2 * k + 1].y);
            }
        }
    } else {
        // ------------------------------------------------------------------ row warps
        const int q = warp & 3, half = warp >> 2, r = 32 * q + lane;
        const int col0 = STACK ? 64 * (q >> 1) + 32 * half : 64 * half;      // this thread's tokens of a tile
        const uint32_t lane_base = (uint32_t)(32 * q) << 16, tp = pp.tmem + TM_P + lane_base;
        const float c1 = p.scale * kLog2e;
        float* ex = reinterpret_cast<float*>(smem + OFF_EX);
        float ref = -INFINITY, sum = 0.f;
        if (STACK) {
            const uint32_t zero[8] = {};
#pragma unroll
            for (int t = 0; t < TP; ++t)
#pragma unroll
                for (int k = 0; k < 2; ++k) tmem_st8(tp + 64 * t + ((col0 ^ 64) >> 1) + 8 * k, zero);
            tmem_st_wait();
        }
        for (int i = 0; i < count; ++i, advance()) {
            const int b = i & 1, left = N - tile * kTok - col0;        // columns of this thread that exist
            if (p.bias) wait_par(pp, BAR_BIAS + b, i >> 1, kTimeoutTile);
            wait_par(pp, BAR_S + b, i >> 1, kTimeoutTile);
            tc_fence_after_sync();
            if (i == 0 || tile == 0) { ref = -INFINITY; sum = 0.f; }
            // logits in log2 units
            float2 s[kCols / 2];
            const unsigned char* bs = smem + OFF_BIAS + b * 2 * kTile;
#pragma unroll
            for (int h = 0; h < kCols / 32; ++h) {
                uint32_t o[32];
                tmem_ld32(pp.tmem + TM_S + 128 * b + lane_base + col0 + 32 * h, o);
                tmem_ld_wait();
                const int c = col0 + 32 * h;
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    uint32_t u[4] = {0u, 0u, 0u, 0u};
                    if (p.bias == 2) {
                        const int row = STACK ? r & 63 : r;
                        const uint4 w = *reinterpret_cast<const uint4*>(bs + (c >> 6) * (STACK ? kMat : kTile) + row * 128 + (((((c & 63) >> 3) + g) ^ (row & 7)) << 4));
                        u[0] = w.x; u[1] = w.y; u[2] = w.z; u[3] = w.w;
                    } else if (p.bias == 1) {
                        const int a = STACK ? r & 63 : r;
                        const unsigned char* col = bs + (a >> 6) * kTile + (a & 7) * 2;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int t0 = c + 8 * g + 2 * k;          // (c and g are multiples of 8)
                            const uint32_t lo = *reinterpret_cast<const unsigned short*>(col + t0 * 128 + ((((a & 63) >> 3) ^ (2 * k)) << 4));
                            const uint32_t hi = *reinterpret_cast<const unsigned short*>(col + (t0 + 1) * 128 + ((((a & 63) >> 3) ^ (2 * k + 1)) << 4));
                            u[k] = lo | hi << 16;
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int j = 4 * g + k;
                        s[16 * h + j] = ffma2(unpack2<T>(u[k]), make_float2(kLog2e, kLog2e),
                                              fmul2(make_float2(__uint_as_float(o[2 * j]), __uint_as_float(o[2 * j + 1])), make_float2(c1, c1)));
                    }
                }
            }
            if (left < kCols)
#pragma unroll
                for (int j = 0; j < kCols / 2; ++j) {
                    if (2 * j >= left) s[j].x = -INFINITY;
                    if (2 * j + 1 >= left) s[j].y = -INFINITY;
                }
            float m = fmaxf(s[0].x, s[0].y);
#pragma unroll
            for (int j = 1; j < kCols / 2; ++j) m = max3(m, s[j].x, s[j].y);
            tc_fence_before_sync();
            ex[(b * 2 + half) * 128 + r] = m;
            bar_named(1 + q, 64);
            if (lane == 0) {                                           // (every lane's loads have been consumed before the barrier)
                pipe_arrive(pp, BAR_READ + b);
                if (p.bias) pipe_arrive(pp, BAR_BREAD + b);
            }
            const float nr = fmaxf(ref, fmaxf(m, ex[(b * 2 + (half ^ 1)) * 128 + r]));
            const float base_r = nr == -INFINITY ? 0.f : nr, f = ref == -INFINITY ? 0.f : fast_exp2(ref - base_r);      // (every key so far may be masked)
            ref = nr;
            float2 l2 = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < kCols / 2; ++j) {
                const float2 x = fadd2(s[j], make_float2(-base_r, -base_r));
                s[j] = make_float2(fast_exp2(x.x), fast_exp2(x.y));
                l2 = fadd2(l2, s[j]);
            }
            sum = fmaf(sum, f, l2.x + l2.y);
            // to tensor memory, once P V of the tile before has read its own
            if (i > 0) wait_par(pp, BAR_DONE + (b ^ 1), (i - 1) >> 1, kTimeoutTile);
            tc_fence_after_sync();
            if (half == 0) f_s[(i & 3) * 128 + r] = f;
#pragma unroll
            for (int g = 0; g < kCols / 16; ++g) {
                uint32_t u[TP][8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    uint32_t w[TP];
                    split_pair<T, TP, false>(s[8 * g + k], w);              // (at most one, or NaN)
#pragma unroll
                    for (int t = 0; t < TP; ++t) u[t][k] = w[t];
                }
#pragma unroll
                for (int t = 0; t < TP; ++t) tmem_st8(tp + 64 * t + (col0 >> 1) + 8 * g, u[t]);
            }
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) pipe_arrive(pp, BAR_P);
            if (tile == p.tiles - 1 || i == count - 1)                 // the last tile of the slab in this block
                *reinterpret_cast<float2*>(state() + 128 * 64 + (r * 2 + half) * 2) = make_float2(ref, sum);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc<512>(pp.tmem);
}

// V_A from the partial states, in fp32 and as TM terms, and the log2-sum-exp of its row: one warp per (slab, agent), or (WARPS = 8) a block,
// whose warps take the states in turn.
template <typename T, int TM, int WARPS>
__global__ void __launch_bounds__(256) bwd_values_merge_kernel(const float* states, float* va, T* terms, float2* stats, int slabs, int n, int d, int tiles, int blocks, int parts, int lanes, int stack) {
    __shared__ float s_max[WARPS], s_tot[WARPS];
    __shared__ float2 s_sum[WARPS][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, w0 = WARPS > 1 ? warp : 0;
    const int row = WARPS > 1 ? blockIdx.x : blockIdx.x * 8 + warp;
    pdl_wait_prior();
    pdl_release_next();
    if (row >= slabs * n) return;
    const int slab = row / n, a = row - slab * n, rb = stack ? 0 : a >> 7, r = stack ? a : a & 127;
    const long long total = (long long)slabs * tiles, t0 = (long long)slab * tiles;
    const int have = owner(t0 + tiles - 1, lanes, total) - owner(t0, lanes, total) + 1, subs = stack ? 2 : 1;
    // partial states of the row, the warp's own: a lane each, 32 at a time
    const int cnt = (have * subs - w0 + WARPS - 1) / WARPS;
    const float* st = states + ((size_t)slab * parts * blocks + rb) * kState;
    auto at = [&](int q) { return st + (size_t)(stack ? (q * WARPS + w0) >> 1 : q * WARPS + w0) * blocks * kState; };
    auto sub_row = [&](int q) { return stack ? r + 64 * ((q * WARPS + w0) & 1) : r; };
    auto head = [&](int q) {                                           // (reference, sum); nothing counts: (-inf, 0)
        float2 v = make_float2(-INFINITY, 0.f);
        if (q < cnt) {
            const float4 w = *reinterpret_cast<const float4*>(at(q) + 128 * 64 + sub_row(q) * 4);
            v = make_float2(w.x, w.y + w.w);
        }
        return v;
    };
    float2 v = head(lane);
    float mm = v.y > 0.f ? v.x : -INFINITY;
    for (int q = 32; q < cnt; q += 32) {
        const float2 u = head(q + lane);
        if (u.y > 0.f) mm = fmaxf(mm, u.x);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o));
    if (WARPS > 1) {
        s_max[w0] = mm;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < WARPS; ++w) mm = fmaxf(mm, s_max[w]);
    }
    float tot = 0.f;
    float2 o = make_float2(0.f, 0.f);
    for (int q0 = 0; q0 < cnt; q0 += 32) {
        if (q0 > 0) v = head(q0 + lane);
        const float f = v.y > 0.f ? exp2f(v.x - mm) : v.y;             // (NaN stays, an empty one has no weight)
        tot = fmaf(v.y, f, tot);
#pragma unroll 4
        for (int q = q0; q < min(cnt, q0 + 32); ++q) {
            const float g = __shfl_sync(0xffffffffu, f, q - q0);
            const float2 w = *reinterpret_cast<const float2*>(at(q) + sub_row(q) * 64 + 2 * lane);
            if (g != 0.f) o = make_float2(fmaf(w.x, g, o.x), fmaf(w.y, g, o.y));
        }
    }
#pragma unroll
    for (int k = 16; k; k >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, k);
    if (WARPS > 1) {
        s_tot[w0] = tot;
        s_sum[w0][lane] = o;
        __syncthreads();
        if (w0 > 0) return;
#pragma unroll
        for (int w = 1; w < WARPS; ++w) {
            tot += s_tot[w];
            o = fadd2(o, s_sum[w][lane]);
        }
    }
    const float inv = 1.f / tot;
    if (lane == 0) stats[row].x = mm + log2f(tot);
    if (2 * lane >= d) return;
    o.x *= inv; o.y *= inv;
    const size_t off = (size_t)row * d + 2 * lane;
    *reinterpret_cast<float2*>(va + off) = o;
    uint32_t w[TM];
    split_pair<T, TM>(o.x, o.y, w);
#pragma unroll
    for (int k = 0; k < TM; ++k) *reinterpret_cast<uint32_t*>(terms + (size_t)k * slabs * n * d + off) = w[k];
}

struct Plan {
    int stack, blocks, tiles, lanes, parts;
};
Plan plan(int slabs, int n, int N, int sm_count) {
    Plan v;
    v.stack = n <= 64;
    v.blocks = (n + 127) / 128;
    v.tiles = (N + kTok - 1) / kTok;
    const long long total = (long long)slabs * v.tiles;
    v.lanes = (int)std::min<long long>(total, std::max(1, sm_count / v.blocks));
    const int run = (int)std::min<long long>(total / v.lanes, v.tiles);      // every run has at least so many tiles
    v.parts = (v.tiles + run - 2) / run + 1;
    return v;
}

template <typename T, int TA, int TP, bool STACK> cudaError_t launch(const Args& a, int grid, cudaStream_t st) {
    static std::atomic<unsigned long long> done;
    cudaError_t e = allow_smem(bwd_values_umma_kernel<T, TA, TP, STACK>, done, kSmem<TA>);
    if (e != cudaSuccess) return e;
    return launch_dependent(bwd_values_umma_kernel<T, TA, TP, STACK>, dim3(grid), kThreads, kSmem<TA>, st, a);
}
// A warp goes through about five states in a microsecond, so a block takes a row that may have more than sixteen (whole pass, 49 agents of
// 64 channels, one slab: of 16384 tokens 127 -> 61 us, of 3136 tokens 47 -> 34; two slabs of 1640: 40.5 -> 34).
template <typename T, int TM> cudaError_t merge(const Args& a, const Plan& v, float* va, void* terms, float2* stats, cudaStream_t st) {
    const bool wide = (v.parts << v.stack) > 16;
    const int rows = a.slabs * a.n;
    return launch_dependent(wide ? bwd_values_merge_kernel<T, TM, 8> : bwd_values_merge_kernel<T, TM, 1>, dim3(wide ? rows : (rows + 7) / 8), 256, 0, st, (const float*)a.state, va, static_cast<T*>(terms), stats, a.slabs, a.n, a.d, v.tiles, v.blocks, v.parts, v.lanes, v.stack);
}

}  // namespace

// A launch more than bwd_sums_kernel, whose clusters merge as they end: worth it from 1024 tokens on (64 slabs of 3136 tokens, 49 agents:
// 50 -> 27 + 8 us; 8 of 1457, 144 agents: whole pass 102 -> 87; but 384 of 196: 21 -> 20 + 15, 48 of 784 with 32 channels: whole pass
// 93 -> 95), and where there are several blocks of agents and many tokens (192 slabs of 196 tokens, 81 agents: whole pass 215 -> 200; 64 of
// 196, 196 agents: 128 -> 131).
bool backward_values_eligible(int slabs, int n, int N) { return N > 1024 || (n > 64 && (long long)slabs * N >= 16384); }

size_t backward_values_bytes(int slabs, int n, int N, int sm_count) {
    if (!backward_values_eligible(slabs, n, N)) return 0;
    const Plan v = plan(slabs, n, N, sm_count);
    return (size_t)slabs * v.parts * v.blocks * kState * sizeof(float);
}

cudaError_t launch_backward_values(int dtype, bool full, const BwdCall& c, const void* a_t, void* va_t, float2* stats, const void* padded, void* ws, cudaStream_t st) {
    Args a;
    memset(&a, 0, sizeof(a));
    const int N = c.H * c.W;
    const Plan v = plan(c.slabs, c.n, N, c.sm_count);
    a.slabs = c.slabs; a.heads = c.heads; a.N = N; a.n = c.n; a.d = c.d; a.tiles = v.tiles; a.blocks = v.blocks; a.parts = v.parts;
    a.state = static_cast<float*>(ws);
    a.status = c.status;
    a.scale = c.scale1;
    const bool rows = N % 8 == 0;                       // (TMA takes B1 as it is)
    a.bias = !c.b1 ? 0 : rows ? 2 : 1;
    if (!make_map_3d_u16(&a.tm_k, c.k, c.slabs, N, c.d, kTok) || !make_map_3d_u16(&a.tm_v, c.v, c.slabs, N, c.d, kTok) ||
        !make_map_3d_u16(&a.tm_a, a_t, (full ? 3 : 1) * (uint64_t)c.slabs, c.n, c.d, 64))
        return cudaErrorInvalidValue;
    if (c.b1 && !(rows ? make_map_3d_u16(&a.tm_b, c.b1, c.heads, c.n, N, v.stack ? 64 : 128) : make_map_3d_u16(&a.tm_b, padded, c.heads, N, bias_width(c.n), kTok)))
        return cudaErrorInvalidValue;
    using B = __nv_bfloat16;
    const int grid = v.lanes * v.blocks;
    cudaError_t e;
    if (full) e = v.stack ? launch<B, 3, 3, true>(a, grid, st) : launch<B, 3, 3, false>(a, grid, st);
    else e = dtype == kBF16 ? launch<B, 1, 2, true>(a, grid, st) : launch<__half, 1, 2, true>(a, grid, st);
    if (e != cudaSuccess) return e;
    return full ? merge<B, 3>(a, v, c.ws_va, va_t, stats, st) : dtype == kBF16 ? merge<B, 2>(a, v, c.ws_va, va_t, stats, st) : merge<__half, 2>(a, v, c.ws_va, va_t, stats, st);
}

}  // namespace aa
