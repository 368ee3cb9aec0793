// Short grids (up to 256 tokens, up to 64 agents, up to 64 channels of 16-bit types): the whole forward pass (Eq. 6) of a slab in one
// block on the 5th-generation tensor cores.
//
// One block of sixteen warps per slab, two blocks to an SM so that one works while the other waits for a copy or a product.  The token axis is cut
// in two halves of `ts` tokens (a multiple of 16, at most 128).
//   1. K and V by TMA; meanwhile A = Pooling(Q), the biases B1 and the filter into shared memory.
//   2. S = A K^T: the agents (64 rows, padded) are stacked twice as the A operand in tensor memory, [A; 0] against the first half's keys and
//      [0; A] against the second's into the same columns, so that all 128 lanes carry a row: lane r + 64 h owns agent r and half h.
//   3. Softmax over the tokens: a thread takes 32 of its lane's logits; the maximum of an agent is shared by its eight threads, so their
//      partial sums and products just add up.  Probabilities go back to tensor memory as the A operand of the product with V.
//   4. The halves' products meet in shared memory: V_A.  Meanwhile Q has come in over K, and T = Q A^T is under way.
//   5. Softmax over the agents (thread = token and half of the agents), O = P V_A; the depthwise term by mma.sync with the filter as a diagonal operand (as in
//      broadcast_umma.cu) from the slab's V tokens while the product is in flight; rounded once and stored.
// Normalisers are sums of the rounded weights, so that the two agree.
//
// What bounds it: the chain of copies, products and barriers of a slab, about 14 us with two blocks to an SM (inputs 2.5, either softmax 2, V_A 2,
// depthwise term 2.3), and code that runs once: 384 slabs of 196 tokens, 49 agents of 64 channels 34 us in two waves, register tiles 47.5 us
// (14.3 M warp instructions, here 13 M); 147 slabs 14 us against 34.
#include "dwc_diag.cuh"
#include "stream_common.cuh"
#include "tile_pool.cuh"

#include <algorithm>
#include <cstring>

namespace aa {

namespace {
constexpr int NT = 512;
constexpr int kTimeoutTile = 3, kTimeoutLoads = 4;
constexpr int kMat = 64 * 128;                            // swizzled [64][64] tile of 16-bit elements
constexpr int kExPitch = 68;                              // floats of a row of the exchange of the halves' products

// shared memory: fixed part (bytes from a 1024-aligned base), then K (later Q), V, and a buffer for the biases and the exchange
constexpr int OFF_BAR = 0, OFF_DEAD = 128, OFF_TMEM = 132;
constexpr int OFF_MX = 256;                               // [4 column groups][128 lanes] maxima
constexpr int OFF_SUM = OFF_MX + 4 * 128 * 4;             // the same: sums
constexpr int OFF_ZERO = OFF_SUM + 4 * 128 * 4;           // zeros, as many as the filter
constexpr int OFF_TAB = OFF_ZERO + kFilterWords * 4;      // filter
constexpr int OFF_A = 10 * 1024;                          // agents [64][128 B]
constexpr int OFF_VA = OFF_A + kMat;                      // agent features [64][128 B]
constexpr int OFF_K = OFF_VA + kMat;
static_assert(OFF_ZERO % 128 == 0 && OFF_TAB + kFilterWords * 4 <= OFF_A, "small buffers");

// mbarriers, each used once
constexpr int BAR_K = 0, BAR_V = 1, BAR_Q = 2, BAR_S = 3, BAR_PV = 4, BAR_T = 5, BAR_O = 6, kBars = 7;

// tensor memory columns: logits (then probabilities) 128; the halves' products, later the output tiles, 64 each; the stacked agents
// (32 columns per half) before the products
constexpr uint32_t TM_S = 0, TM_D = 128;

struct SlabArgs {
    const void *q, *a_user, *b1, *b2, *wd;
    void *a, *va, *out;               // A and V_A: workspace [slabs][n][d]
    int slabs, heads, H, W, N, n, d, p, ts, bias_bytes;
    int hf;                           // dimension order of the maps (tma_load_tok)
    float scale1, scale2;
    int* status;
    TokLayout lin, lout;
    alignas(64) CUtensorMap tm_q, tm_k, tm_v;
};

// The bias of a head, [n][N] or [N][n] 2-byte elements wherever they start, as 16-byte vectors of the tensor
struct BiasSpan {
    const uint4* src;
    int first, vecs, left;                                // elements before the head's own in the first vector; vectors; the tensor's elements from src on
    __device__ BiasSpan(const void* base, int head, int heads, int elems) {
        const long long e0 = (long long)head * elems;
        src = static_cast<const uint4*>(base) + (e0 >> 3);
        first = (int)(e0 & 7);
        vecs = (first + elems + 7) >> 3;
        left = (heads - head) * elems + first;
    }
    __device__ uint4 load(int i) const {
        if (8 * i + 8 <= left) return __ldg(src + i);
        uint32_t w[4] = {0u, 0u, 0u, 0u};                 // the tensor's end
        for (int e = 8 * i; e < left; ++e) w[e >> 1 & 3] |= (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(src) + e) << (16 * (e & 1));
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};
// Pairs 4 g .. 4 g + 3 of 2-byte elements at `w` (a word; `sh` = 16: they start in its upper half)
template <typename T> __device__ __forceinline__ void bias8(const uint32_t* w, int g, int sh, float2 (&b)[4]) {
    uint32_t x[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) x[k] = w[4 * g + k];
#pragma unroll
    for (int k = 0; k < 4; ++k) b[k] = unpack2<T>(__funnelshift_r(x[k], x[k + 1], sh));
}
}  // namespace

template <typename T>
__global__ void __launch_bounds__(NT, 2) slab_umma_kernel(const __grid_constant__ SlabArgs p) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int fmt = Elem<T>::kIsBf16 ? 1 : 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int slab = blockIdx.x, head = slab % p.heads;
    const int N = p.N, n = p.n, d = p.d, ts = p.ts;
    const int q = warp & 3, cs = warp >> 2, L = 32 * q + lane;          // tensor-memory lane; group of columns
    const int r = L & 63, h = L >> 6;                                   // agent, token half
    const uint32_t lane_base = (uint32_t)(32 * q) << 16, base = smem_u32(smem);
    const uint32_t sK = base + OFF_K, sV = sK + 2 * ts * 128;
    unsigned char* sB = smem + OFF_K + 4 * ts * 128;                    // biases; exchange of the products
    uint32_t* sTab = reinterpret_cast<uint32_t*>(smem + OFF_TAB);

    Pipe pp;
    pp.status = p.status;
    pp.dead = reinterpret_cast<int*>(smem + OFF_DEAD);
    pp.bars = base + OFF_BAR;
    if (tid == 0) {
        *pp.dead = 0;
        for (int i = 0; i < kBars; ++i) mbar_init(pp.bars + 8 * i, 1u);
        mbar_fence_init();
    }
    for (int e = tid; e < kFilterWords; e += NT) reinterpret_cast<uint32_t*>(smem + OFF_ZERO)[e] = 0u;
    if (warp == 1) tmem_alloc<256>(base + OFF_TMEM);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    pp.tmem = *reinterpret_cast<const volatile uint32_t*>(smem + OFF_TMEM);
    pdl_wait_prior();           // (no early release: blocks of the next call would take the slots that balance this one)

    // ---- 1. inputs
    const uint32_t half_bytes = (uint32_t)ts * 128;
    if (tid == 0) {
        for (int m = 0; m < 2; ++m) {
            const uint32_t bar = pipe_bar(pp, m == 0 ? BAR_K : BAR_V), dst = m == 0 ? sK : sV;
            mbar_arrive_expect_tx(bar, 2 * half_bytes);
            for (int i = 0; i < 2; ++i) tma_load_tok(dst + i * half_bytes, m == 0 ? &p.tm_k : &p.tm_v, p.hf, i * ts, head, slab / p.heads, bar);
        }
    }
    const BiasSpan s1(p.b1, head, p.heads, n * N), s2(p.b2, head, p.heads, n * N);
    if (p.b1)
        for (int i = tid; i < s1.vecs; i += NT) {
            if (8 * i + 8 <= s1.left) cp_async16(reinterpret_cast<uint4*>(sB) + i, s1.src + i, 16);
            else reinterpret_cast<uint4*>(sB)[i] = s1.load(i);
        }
    cp_async_commit();
    if (p.wd) fill_filter(sTab, p.wd, head, d, tid, NT);
    {
        const T* gq = static_cast<const T*>(p.q) + tok_offset(p.lin, slab, p.heads, 0);
        auto put = [&](int agent, int ch, const uint4& v) { *reinterpret_cast<uint4*>(smem + OFF_A + agent * 128 + ((ch ^ (agent & 7)) << 4)) = v; };
        auto mean = [&](int agent, int ch, const float (&f)[8]) {
            const uint4 v = pack16<T>(f);
            *reinterpret_cast<uint4*>(static_cast<T*>(p.a) + ((size_t)slab * n + agent) * d + 8 * ch) = v;
            put(agent, ch, v);
        };
        const bool windows = !p.a_user && N > 16 * n;                   // a warp per window, or (small ones) a thread per 16 bytes of an agent
        if (windows)
            for (int agent = warp; agent < n; agent += NT / 32)
                pool_window<T>(gq, p.lin.st, p.H, p.W, p.p, p.p, agent, d, [&](int ch, const float (&f)[8]) { mean(agent, ch, f); });
#pragma unroll 1
        for (int i = tid; i < 64 * 8; i += NT) {
            const int agent = i >> 3, ch = i & 7;
            if (agent >= n || 8 * ch >= d) put(agent, ch, make_uint4(0u, 0u, 0u, 0u));
            else if (p.a_user) put(agent, ch, __ldg(reinterpret_cast<const uint4*>(static_cast<const T*>(p.a_user) + ((size_t)slab * n + agent) * d + 8 * ch)));
            else if (!windows) pool_chunk<T>(gq + 8 * ch, p.lin.st, p.H, p.W, p.p, p.p, agent, [&](const float (&f)[8]) { mean(agent, ch, f); });
        }
    }
    fence_proxy_async();
    __syncthreads();

    // ---- 2. stacked agents, S = A K^T
    {
        uint32_t ra[16];                                                // part cs / 2, sixteen of its columns
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (h == cs >> 1) v = *reinterpret_cast<const uint4*>(smem + OFF_A + r * 128 + (((4 * (cs & 1) + j) ^ (r & 7)) << 4));
            ra[4 * j] = v.x; ra[4 * j + 1] = v.y; ra[4 * j + 2] = v.z; ra[4 * j + 3] = v.w;
        }
        tmem_st16(pp.tmem + TM_D + 16 * cs + lane_base, ra);
        tmem_st_wait();
    }
    cp_async_wait<0>();
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after_sync();
        wait_par(pp, BAR_K, 0, kTimeoutLoads);
        const uint32_t id = umma_idesc(fmt, 128, ts, 0);
        const uint64_t dk = umma_desc_sw128(sK);
        // descriptor start addresses count 16-byte units: + 2 per K-step of a K-major operand (32 bytes), + 8 per row
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_ts_w(pp.tmem + TM_S, pp.tmem + TM_D + 32 * i + 8 * k, dk + 8 * ts * i + 2 * k, id, i > 0 || k > 0);
        umma_commit_w(pipe_bar(pp, BAR_S));
    }
    __syncwarp();

    // ---- 3. softmax over the tokens
    wait_par(pp, BAR_S, 0, kTimeoutTile);
    tc_fence_after_sync();
    if (tid == 0) {                                                     // K has been read: Q takes its place
        const uint32_t bar = pipe_bar(pp, BAR_Q);
        mbar_arrive_expect_tx(bar, 2 * half_bytes);
        for (int i = 0; i < 2; ++i) tma_load_tok(sK + i * half_bytes, &p.tm_q, p.hf, i * ts, head, slab / p.heads, bar);
    }
    __syncwarp();
    float* s_mx = reinterpret_cast<float*>(smem + OFF_MX);
    float* s_sum = reinterpret_cast<float*>(smem + OFF_SUM);
    float sv[32];
    {
        const int t0 = ts * h + 32 * cs, valid = min(min(32, ts - 32 * cs), N - t0);      // tokens of this thread (may be <= 0)
        if (32 * cs < ts) {
            tmem_ld32(pp.tmem + TM_S + 32 * cs + lane_base, *reinterpret_cast<uint32_t(*)[32]>(sv));
            tmem_ld_wait();
        }
        // (agents past n, and columns past the tokens: anything, of no consequence)
        const int e0 = min(r, n - 1) * N + t0 + s1.first;
        const uint32_t* src = reinterpret_cast<const uint32_t*>(sB) + (e0 >> 1);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            float2 b[4] = {};
            if (p.b1) bias8<T>(src, g, 16 * (e0 & 1), b);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = 4 * g + k;
                const float2 v = ffma2(make_float2(sv[2 * j], sv[2 * j + 1]), make_float2(p.scale1, p.scale1), b[k]);
                sv[2 * j] = v.x; sv[2 * j + 1] = v.y;
            }
        }
        if (valid < 32)
#pragma unroll
            for (int k = 0; k < 32; ++k) if (k >= valid) sv[k] = -INFINITY;
    }
    auto row_max = [&] {
        float m0 = fmaxf(sv[0], sv[1]), m1 = fmaxf(sv[2], sv[3]);
#pragma unroll
        for (int k = 4; k < 32; k += 4) { m0 = max3(m0, sv[k], sv[k + 1]); m1 = max3(m1, sv[k + 2], sv[k + 3]); }
        return fmaxf(m0, m1);
    };
    s_mx[128 * cs + L] = row_max();
    __syncthreads();                                                    // (the logits and the biases have been read, too)
    // probabilities of the first `cols` columns relative to the reference, as packed pairs; returns the sum of the rounded ones
    auto probs = [&](float ref, uint32_t (&pk)[16], int cols) {
        const float nb = -fmaxf(ref, kRefFloor) * kLog2e;
        float2 s0 = make_float2(0.f, 0.f), s1v = s0;
#pragma unroll
        for (int g = 0; g < 4; ++g)
            if (8 * g < cols) {
#pragma unroll
                for (int j = 4 * g; j < 4 * g + 4; ++j) {
                    const float2 x = ffma2(make_float2(sv[2 * j], sv[2 * j + 1]), make_float2(kLog2e, kLog2e), make_float2(nb, nb));
                    pk[j] = pack2<T>(fast_exp2(x.x), fast_exp2(x.y));   // exp2(-inf) = 0
                    if (j & 1) s1v = fadd2(s1v, unpack2<T>(pk[j])); else s0 = fadd2(s0, unpack2<T>(pk[j]));
                }
            } else {
#pragma unroll
                for (int j = 4 * g; j < 4 * g + 4; ++j) pk[j] = 0u;
            }
        return (s0.x + s0.y) + (s1v.x + s1v.y);
    };
    {
        float ref = kRefFloor;
#pragma unroll
        for (int g = 0; g < 8; ++g) ref = fmaxf(ref, s_mx[64 * g + r]);
        uint32_t pk[16];
        s_sum[128 * cs + L] = probs(ref, pk, ts - 32 * cs);
        if (32 * cs < ts) tmem_st16(pp.tmem + TM_S + 16 * cs + lane_base, pk);
        tmem_st_wait();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after_sync();
        wait_par(pp, BAR_V, 0, kTimeoutLoads);
        const uint32_t id = umma_idesc(fmt, 128, 64, 1);
        const uint64_t dv = umma_desc_sw128(sV);
        // + 128 per K-step of an MN-major operand (16 rows of 128 bytes)
        for (int i = 0; i < 2; ++i)
            for (int k = 0; k < ts / 16; ++k) umma_ts_w(pp.tmem + TM_D + 64 * i, pp.tmem + TM_S + 8 * k, dv + 8 * ts * i + 128 * k, id, k > 0);
        umma_commit_w(pipe_bar(pp, BAR_PV));
    }
    __syncwarp();

    // ---- 4. V_A; the other bias; T = Q A^T
    uint4 bw[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) if (p.b2 && tid + NT * j < s2.vecs) bw[j] = s2.load(tid + NT * j);
    uint4 last2 = make_uint4(0u, 0u, 0u, 0u);                           // (256 tokens, 64 agents that start in the middle of a vector)
    if (p.b2 && tid == 0 && 4 * NT < s2.vecs) last2 = s2.load(4 * NT);
    wait_par(pp, BAR_PV, 0, kTimeoutTile);
    tc_fence_after_sync();
    if (warp == 0) {
        wait_par(pp, BAR_Q, 0, kTimeoutLoads);
        const uint32_t id = umma_idesc(fmt, 128, 64, 0);
        const uint64_t dq = umma_desc_sw128(sK), da = umma_desc_sw128(base + OFF_A);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_ss_w(pp.tmem + TM_S + 64 * i, dq + 8 * ts * i + 2 * k, da + 2 * k, id, k > 0);
        umma_commit_w(pipe_bar(pp, BAR_T));
    }
    __syncwarp();
    float* sX = reinterpret_cast<float*>(sB) + r * kExPitch + 16 * cs;
    {
        float o[16];
        tmem_ld16(pp.tmem + TM_D + 64 * h + 16 * cs + lane_base, o);
        tmem_ld_wait();
        tc_fence_before_sync();
        if (h == 1)
#pragma unroll
            for (int k = 0; k < 4; ++k) *reinterpret_cast<float4*>(sX + 4 * k) = make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
        __syncthreads();
        if (h == 0) {
            float l = 0.f;
#pragma unroll
            for (int g = 0; g < 8; ++g) l += s_sum[64 * g + r];
            const float inv = 1.f / l;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float f[8];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float4 x = *reinterpret_cast<const float4*>(sX + 8 * c + 4 * e);
                    f[4 * e] = (o[8 * c + 4 * e] + x.x) * inv; f[4 * e + 1] = (o[8 * c + 4 * e + 1] + x.y) * inv;
                    f[4 * e + 2] = (o[8 * c + 4 * e + 2] + x.z) * inv; f[4 * e + 3] = (o[8 * c + 4 * e + 3] + x.w) * inv;
                }
                const uint4 v = r < n ? pack16<T>(f) : make_uint4(0u, 0u, 0u, 0u);
                const int ch = 2 * cs + c;
                *reinterpret_cast<uint4*>(smem + OFF_VA + r * 128 + ((ch ^ (r & 7)) << 4)) = v;
                if (r < n && 8 * ch < d) *reinterpret_cast<uint4*>(static_cast<T*>(p.va) + ((size_t)slab * n + r) * d + 8 * ch) = v;
            }
        }
    }
    __syncthreads();                                                    // the exchange has been read
    if (p.b2) {
#pragma unroll
        for (int j = 0; j < 4; ++j) if (tid + NT * j < s2.vecs) reinterpret_cast<uint4*>(sB)[tid + NT * j] = bw[j];
        if (tid == 0 && 4 * NT < s2.vecs) reinterpret_cast<uint4*>(sB)[4 * NT] = last2;
    }
    fence_proxy_async();
    __syncthreads();

    // ---- 5. softmax over the agents, O = P V_A, depthwise term
    const int tile = cs & 1, half = cs >> 1, cols = n - 32 * half;      // of the tokens; of the agents, and how many there are
    const int tok = ts * tile + L;                                      // this thread's token; rows ts .. 127 of a tile belong to no token
    const bool ok = L < ts && tok < N;                                  // (others: anything, not stored)
    wait_par(pp, BAR_T, 0, kTimeoutTile);
    tc_fence_after_sync();
    float inv;
    {
        tmem_ld32(pp.tmem + TM_S + 64 * tile + 32 * half + lane_base, *reinterpret_cast<uint32_t(*)[32]>(sv));
        tmem_ld_wait();
        const int e0 = (ok ? tok : 0) * n + 32 * half + s2.first;
        const uint32_t* src = reinterpret_cast<const uint32_t*>(sB) + (e0 >> 1);
#pragma unroll
        for (int g = 0; g < 4; ++g)
            if (8 * g < cols) {
                float2 b[4] = {};
                if (p.b2) bias8<T>(src, g, 16 * (e0 & 1), b);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int j = 4 * g + k;
                    const float2 v = ffma2(make_float2(sv[2 * j], sv[2 * j + 1]), make_float2(p.scale2, p.scale2), b[k]);
                    sv[2 * j] = v.x; sv[2 * j + 1] = v.y;
                }
                if (8 * g + 8 > cols)
#pragma unroll
                    for (int k = 8 * g; k < 8 * g + 8; ++k) if (k >= cols) sv[k] = -INFINITY;
            } else {
#pragma unroll
                for (int k = 8 * g; k < 8 * g + 8; ++k) sv[k] = -INFINITY;
            }
        // the two halves of a row share its maximum (the logits have been read then, too)
        s_mx[128 * cs + L] = row_max();
        asm volatile("bar.sync %0, 64;\n" ::"r"(1 + 4 * tile + q) : "memory");
        const float ref = fmaxf(s_mx[128 * tile + L], s_mx[128 * (tile + 2) + L]);
        uint32_t pk[16];
        s_sum[128 * cs + L] = probs(ref, pk, cols);
        tmem_st16(pp.tmem + TM_S + 64 * tile + 16 * half + lane_base, pk);
        tmem_st_wait();
    }
    tc_fence_before_sync();
    __syncthreads();
    inv = 1.f / (s_sum[128 * tile + L] + s_sum[128 * (tile + 2) + L]);
    if (warp == 0) {
        tc_fence_after_sync();
        const uint32_t id = umma_idesc(fmt, 128, 64, 1);
        const uint64_t dva = umma_desc_sw128(base + OFF_VA);
        const int ks = (n + 15) >> 4;
        for (int i = 0; i < 2; ++i)
            for (int k = 0; k < ks; ++k) umma_ts_w(pp.tmem + TM_D + 64 * i, pp.tmem + TM_S + 64 * i + 8 * k, dva + 128 * k, id, k > 0);
        umma_commit_w(pipe_bar(pp, BAR_O));
    }
    __syncwarp();
    const int lg = lane >> 2;                                           // mma.sync coordinate
    const int row0 = 32 * q;                                            // this warp's rows of the tile
    const int c0 = 32 * half;                                           // and channels
    T* gO = static_cast<T*>(p.out) + tok_offset(p.lout, slab, p.heads, ts * tile + row0);
    const int limit = min(ts - row0, N - ts * tile - row0), t0 = ts * tile + row0 + (lane & 15);       // rows that exist; this lane's token
    const bool active = limit > 0 && c0 < d;
    float o[2][4][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int jj = 0; jj < 4; ++jj)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[mt][jj][e] = 0.f;
    wait_par(pp, BAR_V, 0, kTimeoutLoads);
    if (p.wd && active) {
        uint32_t in[2];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) in[mt] = window_taps(16 * mt + (lane & 15) < limit ? t0 + 16 * mt : N, N, p.H, p.W, 1.f / (float)p.W, lane);
        const uint32_t* tab = filter_lane(sTab + c0, reinterpret_cast<const uint32_t*>(smem + OFF_ZERO), lane);
        dwc_rows<T>(o, sV, t0, 2 * c0, in, base + OFF_ZERO, tab, lane, [&](int u, int v) { return (u - 1) * p.W + v - 1; });
    }
    wait_par(pp, BAR_O, 0, kTimeoutTile);
    tc_fence_after_sync();
    if (active) {
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            float a[16];
            tmem_ld_16x256b_x4(pp.tmem + TM_D + 64 * tile + c0 + lane_base + (16u * mt << 16), a);
            const float w0 = __shfl_sync(0xffffffffu, inv, 16 * mt + lg), w1 = __shfl_sync(0xffffffffu, inv, 16 * mt + 8 + lg);
            tmem_ld_wait();
#pragma unroll
            for (int jj = 0; jj < 4; ++jj)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[mt][jj][e] = fmaf(e < 2 ? w0 : w1, a[4 * jj + e], o[mt][jj][e]);
            const bool have[2] = {16 * mt + lg < limit, 16 * mt + 8 + lg < limit};
            store_rows<T>(o[mt], gO + (size_t)(16 * mt) * p.lout.st, p.lout.st, c0, d, have, lane);
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc<256>(pp.tmem);
}

// ------------------------------------------------------------------------------------- host
namespace {
int half_tokens(int N) { return ((N + 1) / 2 + 15) / 16 * 16; }
int bias_bytes(const TileArgs& a) { return std::max(a.b1 || a.b2 ? (int)(((long long)a.n * a.N * 2 + 14 + 15) / 16 * 16) + 256 : 0, 64 * kExPitch * 4); }
int smem_bytes(const TileArgs& a) { return OFF_K + 4 * half_tokens(a.N) * 128 + bias_bytes(a) + 1024; }

template <typename T> cudaError_t launch(const SlabArgs& g, int smem, cudaStream_t st) {
    static std::atomic<unsigned long long> done;
    cudaError_t e = allow_smem(slab_umma_kernel<T>, done, 227 * 1024);
    if (e != cudaSuccess) return e;
    return launch_dependent(slab_umma_kernel<T>, dim3(g.slabs), NT, smem, st, g);
}
}  // namespace

// Two blocks are resident on an SM, four of the register tiles' (clusters of up to eight a slab where there are fewer slabs; beyond that three
// kernels).  Time of the register tiles over this kernel's, bf16, grids of 20 to 256 tokens, 9 to 64 agents, 1 to 1000 slabs (148 SMs):
//   49 and 64 channels: 16 to 296 slabs of 64 tokens and more 0.92 to 2.4 (under one only with 9 agents or at 256 tokens); 384 slabs of 196
//     tokens 0.97 to 1.39, of 100 tokens 0.80 to 1.07; 600 and 1000 slabs 1.0 to 2.0, of 49 tokens 0.61 to 1.05; up to 12 slabs 0.99 to 1.2 with
//     biases up to 128 tokens (of which each block stages its own; the cluster's blocks read the same rows), 0.75 to 1.19 elsewhere
//   32 and 40 channels, at least 25 agents: 147 slabs 1.5 to 2.0, up to 64 slabs 0.70 to 1.1, 192 and 294 slabs of 155 tokens and more 0.78 to
//     1.36, 384 slabs 0.46 to 1.0, 600 and 1000 slabs 1.0 to 1.95
bool slab_umma_eligible(int dtype, const TileArgs& a, int sm_count) {
    if (!(dtype == kBF16 || dtype == kF16) || a.N > 256 || a.N < 2 || a.n > 64 || a.d > 64 || a.d % 8 || smem_bytes(a) > 113 * 1024 ||
        !tok_map_exists(a.lin, a.slabs / a.heads, a.heads, a.N))
        return false;
    const int wave = 2 * sm_count, tiles = 4 * sm_count;                // slabs resident at once, here and on register tiles
    if (a.d > 48) {
        if (a.slabs < 16) return (a.b1 || a.b2) && a.N >= 32 && a.N <= 128;
        if (a.slabs <= wave) return a.N >= 64 && (a.n >= 16 || a.N >= 128);
        if (a.slabs <= tiles) return a.N >= 176;
        return a.N >= 96 && (a.n >= 16 || a.N >= 128);
    }
    if (a.n < 16) return false;
    if (a.slabs > tiles) return a.N >= 96;
    return a.slabs <= wave && a.slabs > sm_count / 2 && a.N >= (a.slabs <= sm_count ? 96 : 144);
}

// cudaErrorNotSupported: a tensor map could not be encoded.
cudaError_t launch_slab_umma(int dtype, const TileArgs& a, int* status, cudaStream_t st) {
    SlabArgs g;
    memset(&g, 0, sizeof(g));
    g.q = a.q; g.a_user = a.pool ? nullptr : a.a; g.b1 = a.b1; g.b2 = a.b2; g.wd = a.wd;
    g.a = const_cast<void*>(a.a); g.va = a.va; g.out = a.out;
    g.slabs = a.slabs; g.heads = a.heads; g.H = a.H; g.W = a.W; g.N = a.N; g.n = a.n; g.d = a.d; g.p = a.pool;
    g.ts = half_tokens(a.N);
    g.scale1 = a.scale1; g.scale2 = a.scale2; g.status = status; g.lin = a.lin; g.lout = a.lout;
    const int batch = a.slabs / a.heads;
    for (int m = 0; m < 3; ++m)
        if (!make_map_tok_u16(m == 0 ? &g.tm_q : m == 1 ? &g.tm_k : &g.tm_v, &g.hf, m == 0 ? a.q : m == 1 ? a.k : a.v, a.lin, batch, a.heads, a.N, a.d, g.ts, true)) return cudaErrorNotSupported;
    return dtype == kBF16 ? launch<__nv_bfloat16>(g, smem_bytes(a), st) : launch<__half>(g, smem_bytes(a), st);
}

}  // namespace aa
