// The attention stages with fp32 operands on the tensor cores (the gradients, and the forward pass of fp32 tensors): launch plans
// and the small kernels between the stages (term splits, D = dV_A . V_A).
#include "bwd_terms_launch.cuh"
#include "tile_pool.cuh"

#include <algorithm>
#include <cstring>

namespace aa {

namespace {

int dk_of_terms(int d) { return d <= 32 ? 32 : d <= 48 ? 48 : d <= 64 ? 64 : d <= 80 ? 80 : d <= 96 ? 96 : 128; }

cudaError_t stage(int dtype, int d, int st, const BwdTermArgs& a, const BwdTermLaunch& l) {
    switch (dk_of_terms(d)) {
        case 32: return bwd_terms_32(dtype, st, a, l);
        case 48: return bwd_terms_48(dtype, st, a, l);
        case 64: return bwd_terms_64(dtype, st, a, l);
        case 80: return bwd_terms_80(dtype, st, a, l);
        case 96: return bwd_terms_96(dtype, st, a, l);
        default: return bwd_terms_128(dtype, st, a, l);
    }
}

// Buffers that later kernels add to, cleared by extra blocks of the first kernel.
struct ClearList {
    float* p[7];
    size_t words[7];
    int pool_blocks;
};
constexpr int kClearWords = 256 * 32;              // words that a block clears
// Biases as rows of bias_width(n) agents per token [heads][N][width] (zeros past n), by further blocks of the first kernel: B1 transposed, B2.
// (Rows of whole blocks of 64 agents would be four times as much memory at 9 agents.)
struct PadList {
    const void *b1, *b2;
    void *p1, *p2;
    int heads, n, N, width, blocks1, blocks2;
};
PadList pad_list(const void* b1, const void* b2, void* p1, void* p2, int heads, int n, int N) {
    const int width = bias_width(n), blocks = (int)(((size_t)heads * N * (width / 8) + 255) / 256);
    return {b1, b2, p1, p2, heads, n, N, width, b1 && p1 ? blocks : 0, b2 && p2 ? blocks : 0};
}
template <typename T> __device__ __forceinline__ void pad_bias(const T* src, uint4* dst, bool transposed, const PadList& pl, int block) {
    const long long rows = (long long)pl.heads * pl.N, i = (long long)block * 256 + threadIdx.x;
    // neighbouring threads: B1 is read along its tokens, B2 along its agents
    const int chunks = pl.width >> 3;
    const long long row = transposed ? i % rows : i / chunks;
    const int c0 = 8 * (int)(transposed ? i / rows : i % chunks);
    if (c0 >= pl.width || row >= rows) return;
    const int head = (int)(row / pl.N), tok = (int)(row - (long long)head * pl.N);
    __align__(16) T v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int c = c0 + k;
        v[k] = c >= pl.n ? Elem<T>::from_f32(0.f) : transposed ? src[((size_t)head * pl.n + c) * pl.N + tok] : src[(size_t)row * pl.n + c];
    }
    dst[row * chunks + (c0 >> 3)] = *reinterpret_cast<const uint4*>(v);
}

struct PoolArgs8 {
    const void *q, *given;             // tokens, or the caller's agents
    float* plain;                      // the agents in fp32 too, or null
    int slabs, n, H, W, pool, d;
    bool small;
};
// Pooled agents as NT terms of E: a warp per window, or (windows of at most 32 tokens on average) a thread per 8 channels.
template <typename T, typename E, int NT>
__global__ void __launch_bounds__(256) bwd_pool_terms_kernel(PoolArgs8 pa, E* dst, ClearList cl, PadList pl) {
    const T *q = static_cast<const T*>(pa.q), *given = static_cast<const T*>(pa.given);
    const int slabs = pa.slabs, n = pa.n, H = pa.H, W = pa.W, pool = pa.pool, d = pa.d;
    pdl_wait_prior();
    pdl_release_next();
    if ((int)blockIdx.x >= cl.pool_blocks) {
        size_t b = (size_t)(blockIdx.x - cl.pool_blocks) * kClearWords;
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            const size_t room = (cl.words[k] + kClearWords - 1) / kClearWords * kClearWords;
            if (b < room) {
                const size_t e = min(b + kClearWords, cl.words[k]), e4 = b + ((e - b) & ~(size_t)3);
                for (size_t i = b + 4 * threadIdx.x; i < e4; i += 1024) *reinterpret_cast<float4*>(cl.p[k] + i) = make_float4(0.f, 0.f, 0.f, 0.f);
                if (threadIdx.x < e - e4) cl.p[k][e4 + threadIdx.x] = 0.f;
                return;
            }
            b -= room;
        }
        if constexpr (sizeof(T) == 2) {
            const int block = (int)(b / kClearWords);
            if (block < pl.blocks1) pad_bias<T>(static_cast<const T*>(pl.b1), static_cast<uint4*>(pl.p1), true, pl, block);
            else pad_bias<T>(static_cast<const T*>(pl.b2), static_cast<uint4*>(pl.p2), false, pl, block - pl.blocks1);
        }
        return;
    }
    const size_t plane = (size_t)slabs * n * d;
    auto put = [&](size_t off, const float (&f)[8]) {
        if (pa.plain) {
            *reinterpret_cast<float4*>(pa.plain + off) = make_float4(f[0], f[1], f[2], f[3]);
            *reinterpret_cast<float4*>(pa.plain + off + 4) = make_float4(f[4], f[5], f[6], f[7]);
        }
        uint32_t w[4][NT];
#pragma unroll
        for (int i = 0; i < 4; ++i) split_pair<E, NT>(f[2 * i], f[2 * i + 1], w[i]);
#pragma unroll
        for (int k = 0; k < NT; ++k) *reinterpret_cast<uint4*>(dst + k * plane + off) = make_uint4(w[0][k], w[1][k], w[2][k], w[3][k]);
    };
    if (pa.small) {
        const int cpt = d >> 3;
        const long long i = (long long)blockIdx.x * 256 + threadIdx.x, cell = i / cpt;
        if (cell >= (long long)slabs * n) return;
        const int slab = (int)(cell / n), agent = (int)(cell - (long long)slab * n), ch = (int)(i - cell * cpt);
        if (given) {
            float2 a[4] = {};
            add_raw8<T>(a, ld_raw8<T>(given + (size_t)cell * d + ch * 8));
            const float f[8] = {a[0].x, a[0].y, a[1].x, a[1].y, a[2].x, a[2].y, a[3].x, a[3].y};
            put((size_t)cell * d + ch * 8, f);
            return;
        }
        pool_chunk<T>(q + (size_t)slab * H * W * d + ch * 8, d, H, W, pool, pool, agent, [&](const float (&f)[8]) { put((size_t)cell * d + ch * 8, f); });
    } else {
        const long long cell = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
        if (cell >= (long long)slabs * n) return;
        const int slab = (int)(cell / n), agent = (int)(cell - (long long)slab * n);
        pool_window<T>(q + (size_t)slab * H * W * d, d, H, W, pool, pool, agent, d, [&](int ch, const float (&f)[8]) { put((size_t)cell * d + ch * 8, f); });
    }
}

// One warp per agent row: D = dV_A . V_A, and the terms of dV_A.
template <typename E, int NT>
__global__ void __launch_bounds__(256) bwd_dot_split_kernel(const float* va, const float* dva, float2* stats, E* dst, int rows, int d) {
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    pdl_wait_prior();
    pdl_release_next();
    if (r >= rows) return;
    const size_t plane = (size_t)rows * d;
    float acc = 0.f;
    for (int c = 2 * lane; c < d; c += 64) {
        const size_t off = (size_t)r * d + c;
        const float2 a = *reinterpret_cast<const float2*>(va + off), b = *reinterpret_cast<const float2*>(dva + off);
        acc = fmaf(a.x, b.x, fmaf(a.y, b.y, acc));
        uint32_t w[NT];
        split_pair<E, NT>(b.x, b.y, w);
#pragma unroll
        for (int k = 0; k < NT; ++k) *reinterpret_cast<uint32_t*>(dst + k * plane + off) = w[k];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) stats[r].y = acc;
}

struct SumsPlan {
    int rb, rg, kg;
};
SumsPlan sums_plan(int dtype, int n, int d) {
    const int dk = dk_of_terms(d), most = dk <= 64 ? 128 : dk <= 80 ? 64 : 32;       // agent rows of a block: six term tiles of them, and the ring, in shared memory
    SumsPlan s;
    s.rb = (n + most - 1) / most;
    s.rg = ((n + s.rb - 1) / s.rb + 15) / 16;
    s.kg = s.rg <= 2 && dk <= 80 ? 4 : s.rg <= 4 ? 2 : 1;
    // fp32 tokens are three terms: two stages of 32 kg of them, K and V, beside the agents'
    if (dtype == kF32)
        while (s.kg > 1 && (6 * s.rg * 16 + 2 * 6 * 32 * s.kg) * (dk * 2 + 16) + 2 * 32 * s.kg * 8 > 227 * 1024) s.kg /= 2;
    return s;
}
// Parts of the token axis for `slots` resident blocks, of whole units of tokens.  A block takes `pass` tokens at a time, and its start
// (agents' terms into shared memory) costs about 256.
int token_parts(long long others, int N, int unit, int pass, int most, bool pow2, int slots) {
    int best = 1;
    double cost = 0;
    for (int c = 1; c <= most; c = pow2 ? 2 * c : c + 1) {
        const int tokens = ((N + c - 1) / c + unit - 1) / unit * unit;
        if (c > 1 && (long long)tokens * (c - 1) >= N) continue;
        const double k = (double)((others * c + slots - 1) / slots) * ((tokens + pass - 1) / pass * pass + 256);
        if (c == 1 || k < cost) { best = c; cost = k; }
    }
    return best;
}
size_t up256(size_t x) { return (x + 255) / 256 * 256; }

template <typename T, typename E, int NT> cudaError_t launch_pool_terms(PoolArgs8 pa, void* a_t, ClearList cl, PadList pl, cudaStream_t st) {
    pa.small = pa.given || pa.H * pa.W <= 32 * pa.n;
    cl.pool_blocks = (int)(pa.small ? ((long long)pa.slabs * pa.n * (pa.d / 8) + 255) / 256 : ((long long)pa.slabs * pa.n + 7) / 8);
    size_t clear = 0;
    for (size_t w : cl.words) clear += (w + kClearWords - 1) / kClearWords;
    return launch_dependent(bwd_pool_terms_kernel<T, E, NT>, dim3((unsigned)(cl.pool_blocks + clear + pl.blocks1 + pl.blocks2)), 256, 0, st, pa, static_cast<E*>(a_t), cl, pl);
}
// Pooling, and the clearing of the sums that the stages add to.
template <typename T, typename E, int NT> cudaError_t pool_and_clear(const BwdCall& c, void* a_t, bool clear_bias, bool clear_rows, const PadList& pl, cudaStream_t st) {
    const PoolArgs8 pa = {c.q, nullptr, nullptr, c.slabs, c.n, c.H, c.W, c.p, c.d, false};
    ClearList cl = {};
    const size_t bias = clear_bias ? (size_t)c.heads * c.n * c.H * c.W : 0;
    cl.p[0] = c.ws_dva; cl.words[0] = 2 * c.region_bytes / sizeof(float);          // dV_A, dA
    cl.p[1] = c.db1; cl.words[1] = c.db1 ? bias : 0;
    cl.p[2] = c.db2; cl.words[2] = c.db2 ? bias : 0;
    const size_t copies = filter_copy_words(c.heads, c.d);                          // and the word behind them
    cl.p[3] = c.ws_dwd + (c.dwd ? 0 : copies); cl.words[3] = c.wd ? (c.dwd ? copies : 0) + 1 : 0;
    float* const rows[3] = {c.dq, c.dk, c.dv};
    for (int k = 0; k < 3; ++k) { cl.p[4 + k] = rows[k]; cl.words[4 + k] = clear_rows ? (size_t)c.slabs * c.H * c.W * c.d : 0; }
    return launch_pool_terms<T, E, NT>(pa, a_t, cl, pl, st);
}

}  // namespace

bool backward_terms_eligible(int dtype, int n, int d) {
    if (dtype == kF32 && (d % 8 || dk_of_terms(d) > kTermGradientsF32)) return false;
    const int dk = dk_of_terms(d), pitch = dk * 2 + 16, n32 = (n + 31) & ~31;
    return 6 * n32 * pitch + n32 * 8 <= 227 * 1024;
}
size_t backward_terms_bytes(int dtype, int slabs, int heads, int n, int N, int d, int sm_count) {
    return (backward_terms_umma_eligible(dtype, slabs, n, N, d) ? backward_terms_umma_bytes(slabs, heads, n, N) + backward_values_bytes(slabs, n, N, sm_count) : 0) + 3 * up256((size_t)slabs * n * d * 2 * 3) + up256((size_t)slabs * N * 8) + up256((size_t)slabs * n * 8);
}

cudaError_t launch_backward_mixed_forward(int dtype, const BwdCall& c, cudaStream_t st) {
    const int N = c.H * c.W;
    char* padded = static_cast<char*>(c.ws_mixed);                 // (see backward_umma_bytes)
    const PadList pl = pad_list(c.b1, c.b2, padded, c.n % 8 ? padded + padded_bias_bytes(c.heads, c.n, N) : nullptr, c.heads, c.n, N);
    cudaError_t e = dtype == kBF16 ? pool_and_clear<__nv_bfloat16, __nv_bfloat16, 1>(c, c.ws_a, true, false, pl, st) : pool_and_clear<__half, __half, 1>(c, c.ws_a, true, false, pl, st);
    if (e != cudaSuccess) return e;
    if (backward_values_eligible(c.slabs, c.n, N))
        return launch_backward_values(dtype, false, c, c.ws_a, c.ws_part, reinterpret_cast<float2*>(c.ws_lse), padded, padded + backward_umma_bytes(c.heads, c.n, N), st);
    BwdTermArgs a;
    memset(&a, 0, sizeof(a));
    a.slabs = c.slabs; a.heads = c.heads; a.N = N; a.n = c.n; a.d = c.d;
    a.x = c.k; a.y = c.v; a.bias = c.b1; a.scale = c.scale1;
    a.a_t = c.ws_a; a.outer0 = c.ws_va; a.va_t = c.ws_part; a.agent_stats = reinterpret_cast<float2*>(c.ws_lse);
    a.rg = (c.n + 15) / 16;                            // four warps, three blocks on an SM
    BwdTermLaunch l;
    l.stream = st;
    l.kg = a.rg == 1 ? 4 : a.rg == 2 ? 2 : 1;
    const int parts = token_parts(c.slabs, a.N, 64, 64, 8, true, 3 * c.sm_count);
    a.tokens = ((a.N + parts - 1) / parts + 63) / 64 * 64;
    l.grid = dim3(parts, 1, c.slabs);
    l.cluster = parts;
    return bwd_terms_mixed(dtype, a, l);
}

cudaError_t launch_backward_terms(int dtype, const BwdCall& c, void* ws, cudaStream_t st) {
    const int N = c.H * c.W, n = c.n, d = c.d, slabs = c.slabs;
    char* w = static_cast<char*>(ws);
    const size_t terms = up256((size_t)slabs * n * d * 2 * 3);
    void *a_t = w, *va_t = w + terms, *dva_t = w + 2 * terms;
    float2* tok_stats = reinterpret_cast<float2*>(w + 3 * terms);
    float2* agent_stats = reinterpret_cast<float2*>(w + 3 * terms + up256((size_t)slabs * N * 8));
    using B = __nv_bfloat16;
    cudaError_t e;
#define AA_TRY(x) do { e = (x); if (e != cudaSuccess) return e; } while (0)
    const bool umma = backward_terms_umma_eligible(dtype, slabs, n, N, d);
    const UmmaOrder order = umma ? backward_terms_umma_order(slabs, c.heads, n, N, d, c.sm_count) : UmmaOrder{};
    // (a single batch entry stores its bias gradients, and so does the first one of a block that has them all; blocks of 64 agents add to the rows,
    // unless one block has them all)
    const bool clear_bias = slabs != c.heads && !order.stretch, clear_rows = umma && n > 64 && !order.all_agents;
    void *pad1 = nullptr, *pad2 = nullptr, *partial = nullptr;
    char* umma_ws = w + 3 * terms + up256((size_t)slabs * N * 8) + up256((size_t)slabs * n * 8);          // padded biases, partial states of V_A
    if (umma) backward_terms_umma_padded(c.heads, n, N, umma_ws, &pad1, &pad2, &partial);
    AA_TRY(dtype == kBF16 ? (pool_and_clear<B, B, 3>(c, a_t, clear_bias, clear_rows, pad_list(c.b1, c.b2, pad1, pad2, c.heads, n, N), st)) : dtype == kF16 ? (pool_and_clear<__half, B, 3>(c, a_t, clear_bias, clear_rows, PadList{}, st)) : (pool_and_clear<float, B, 3>(c, a_t, clear_bias, clear_rows, PadList{}, st)));

    BwdTermArgs a;
    memset(&a, 0, sizeof(a));
    a.slabs = slabs; a.heads = c.heads; a.N = N; a.n = n; a.d = d;
    a.a_t = a_t; a.tok_stats = tok_stats; a.agent_stats = agent_stats;
    const SumsPlan sp = sums_plan(dtype, n, d);
    a.rg = sp.rg;
    BwdTermLaunch l;
    l.stream = st; l.kg = sp.kg;
    auto sums = [&](int which, bool cluster) {
        const int parts = token_parts((long long)slabs * sp.rb, N, 64, 64, cluster ? 8 : 64, cluster, c.sm_count);
        a.tokens = ((N + parts - 1) / parts + 63) / 64 * 64;
        l.grid = dim3(parts, sp.rb, slabs);
        l.cluster = cluster ? parts : 0;
        return stage(dtype, d, which, a, l);
    };
    auto rows = [&](int which) {
        const int parts = token_parts(slabs, N, 16, 128, 512, false, c.sm_count);
        a.tokens = ((N + parts - 1) / parts + 15) / 16 * 16;
        l.grid = dim3(parts, slabs);
        l.cluster = 0;
        return stage(dtype, d, which, a, l);
    };
    // V_A and the statistics of the aggregation softmax
    a.x = c.k; a.y = c.v; a.bias = c.b1; a.scale = c.scale1; a.outer0 = c.ws_va; a.va_t = va_t;
    if (umma && backward_values_eligible(slabs, n, N)) AA_TRY(launch_backward_values(dtype, true, c, a_t, va_t, agent_stats, pad1, umma_ws + backward_terms_umma_bytes(slabs, c.heads, n, N), st));
    else AA_TRY(sums(kTermForward, true));
    // broadcast stage: token statistics, then dV_A and its share of dA
    a.x = c.q; a.y = c.d_out; a.bias = c.b2; a.scale = a.out_scale = c.scale2; a.m_t = va_t;
    if (umma) {
        AA_TRY(launch_backward_terms_umma(kUmmaStats, c, a_t, va_t, tok_stats, pad2, partial, st));
        AA_TRY(launch_backward_terms_umma(kUmmaBroadcast, c, a_t, va_t, tok_stats, pad2, nullptr, st));
    } else {
        AA_TRY(rows(kTermStats));
        a.outer0 = c.ws_dva; a.outer1 = c.ws_da;
        AA_TRY(sums(kTermBroadcast, false));
        a.row0 = c.dq; a.dbias = c.db2;
        AA_TRY(rows(kTermQuery));
    }
    AA_TRY((launch_dependent(bwd_dot_split_kernel<B, 3>, dim3((slabs * n + 7) / 8), 256, 0, st, (const float*)c.ws_va, (const float*)c.ws_dva, agent_stats, static_cast<B*>(dva_t), slabs * n, d)));
    // aggregation stage
    if (umma) return launch_backward_terms_umma(kUmmaAggregate, c, a_t, dva_t, agent_stats, pad1, nullptr, st);
    a.x = c.k; a.y = c.v; a.bias = c.b1; a.scale = c.scale1; a.out_scale = N == 1 ? 0.f : c.scale1; a.m_t = dva_t; a.dbias = c.db1;
    AA_TRY(sums(kTermAggregate, false));
    a.row0 = c.dk; a.row1 = c.dv; a.dbias = nullptr;
    AA_TRY(rows(kTermKeyValue));
#undef AA_TRY
    return cudaSuccess;
}

// fp32 forward pass: three kernels.  (The CUDA-core kernels took 119 us for one image of 196 tokens, three heads of 64 channels and
// 49 agents.)
bool terms_forward_eligible(int n, int d) {
    const int dk = dk_of_terms(d), n32 = (n + 31) & ~31;
    return d % 8 == 0 && 6 * n32 * (dk * 2 + 16) + 10 * dk * 4 <= 227 * 1024;
}
size_t terms_forward_bytes(int slabs, int n, int d) { return 2 * up256((size_t)slabs * n * d * 2 * 3) + up256((size_t)slabs * n * 8); }

cudaError_t launch_terms_forward(const TermsForward& c, cudaStream_t st) {
    const int N = c.H * c.W;
    char* w = static_cast<char*>(c.ws);
    const size_t terms = up256((size_t)c.slabs * c.n * c.d * 2 * 3);
    const PoolArgs8 pa = {c.q, c.agents, c.agents ? nullptr : c.a_ws, c.slabs, c.n, c.H, c.W, c.p, c.d, false};
    cudaError_t e = launch_pool_terms<float, __nv_bfloat16, 3>(pa, w, ClearList{}, PadList{}, st);
    if (e != cudaSuccess) return e;
    BwdTermArgs a;
    memset(&a, 0, sizeof(a));
    a.slabs = c.slabs; a.heads = c.heads; a.N = N; a.n = c.n; a.d = c.d; a.H = c.H; a.W = c.W;
    a.a_t = w; a.va_t = w + terms; a.agent_stats = reinterpret_cast<float2*>(w + 2 * terms);
    const SumsPlan sp = sums_plan(kF32, c.n, c.d);
    a.rg = sp.rg;
    BwdTermLaunch l;
    l.stream = st; l.kg = sp.kg;
    a.x = c.k; a.y = c.v; a.bias = c.b1; a.scale = c.scale1; a.outer0 = c.va_ws;
    int parts = token_parts((long long)c.slabs * sp.rb, N, 64, 64, 8, true, c.sm_count);
    a.tokens = ((N + parts - 1) / parts + 63) / 64 * 64;
    l.grid = dim3(parts, sp.rb, c.slabs);
    l.cluster = parts;
    e = stage(kF32, c.d, kTermForward, a, l);
    if (e != cudaSuccess) return e;
    a.x = c.q; a.y = c.v; a.bias = c.b2; a.scale = c.scale2; a.m_t = w + terms; a.row0 = c.out; a.wd = c.wd;
    // Fewer groups of 16 tokens than schedulers: two warps each (3 slabs of 196 tokens, 49 agents: whole pass
    // 25.6 -> 22.9 us; 6 of 1200, 196 agents: 75 -> 68; 2 of 3000, 81 agents of 80 channels: 61 -> 55)
    const int dk = dk_of_terms(c.d), n32 = (c.n + 31) & ~31;
    const bool split = c.n > 32 && (long long)c.slabs * ((N + 15) / 16) <= 4 * c.sm_count && 6 * n32 * (dk * 2 + 16) + 10 * dk * 4 + 8 * ((dk / 16 + 1) / 2 * 8 + 4) * 128 <= 227 * 1024;
    parts = token_parts(c.slabs, N, 16, split ? 64 : 128, 512, false, c.sm_count);
    a.tokens = ((N + parts - 1) / parts + 15) / 16 * 16;
    l.grid = dim3(parts, c.slabs);
    l.cluster = 0;
    return stage(kF32, c.d, split ? kTermOutSplit : kTermOut, a, l);
}

}  // namespace aa
