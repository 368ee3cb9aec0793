// Gradients of the attention stages with fp32 operands on the tensor cores: launch plans and the small kernels between the
// stages (term splits, D = dV_A . V_A).
#include "bwd_terms_launch.cuh"

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

// fp32 pairs -> three bf16 terms
__global__ void __launch_bounds__(256) bwd_split_kernel(const float2* src, __nv_bfloat16* dst, size_t pairs) {
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= pairs) return;
    const float2 v = src[i];
    uint32_t w[kTerms];
    split_pair<__nv_bfloat16, kTerms>(v.x, v.y, w);
#pragma unroll
    for (int k = 0; k < kTerms; ++k) reinterpret_cast<uint32_t*>(dst)[k * pairs + i] = w[k];
}

// one warp per agent row: D = dV_A . V_A, and the terms of dV_A
__global__ void __launch_bounds__(256) bwd_dot_split_kernel(const float* va, const float* dva, float2* stats, __nv_bfloat16* dst, int rows, int d) {
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= rows) return;
    const size_t pairs = (size_t)rows * d / 2;
    float acc = 0.f;
    for (int c = 2 * lane; c < d; c += 64) {
        const size_t off = (size_t)r * d + c;
        const float2 a = *reinterpret_cast<const float2*>(va + off), b = *reinterpret_cast<const float2*>(dva + off);
        acc = fmaf(a.x, b.x, fmaf(a.y, b.y, acc));
        uint32_t w[kTerms];
        split_pair<__nv_bfloat16, kTerms>(b.x, b.y, w);
#pragma unroll
        for (int k = 0; k < kTerms; ++k) reinterpret_cast<uint32_t*>(dst)[k * pairs + off / 2] = w[k];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) stats[r].y = acc;
}

struct SumsPlan {
    int rb, rg, kg;
};
SumsPlan sums_plan(int n, int d) {
    const int dk = dk_of_terms(d), most = dk <= 64 ? 128 : dk <= 80 ? 64 : 32;       // agent rows of a block: six term tiles of them, and the ring, in shared memory
    SumsPlan s;
    s.rb = (n + most - 1) / most;
    s.rg = ((n + s.rb - 1) / s.rb + 15) / 16;
    s.kg = s.rg <= 2 && dk <= 80 ? 4 : s.rg <= 4 ? 2 : 1;
    return s;
}
// Parts of the token axis: one block per SM is resident, a block's start (agents' terms into shared memory) costs about 256 tokens.
int token_parts(long long others, int N, int unit, int most, bool pow2, int sm_count) {
    int best = 1;
    double cost = 0;
    for (int c = 1; c <= most; c = pow2 ? 2 * c : c + 1) {
        const int tokens = ((N + c - 1) / c + unit - 1) / unit * unit;
        if (c > 1 && (tokens < 2 * unit || (long long)tokens * (c - 1) >= N)) continue;
        const double k = (double)((others * c + sm_count - 1) / sm_count) * (tokens + 256);
        if (c == 1 || k < cost) { best = c; cost = k; }
    }
    return best;
}

}  // namespace

bool backward_terms_eligible(int dtype, int n, int d) {
    if (dtype != kBF16 && dtype != kF16) return false;
    const int dk = dk_of_terms(d), pitch = dk * 2 + 16, n32 = (n + 31) & ~31;
    return 2 * kTerms * n32 * pitch + n32 * 8 <= 227 * 1024;
}
size_t backward_terms_bytes(int slabs, int n, int N, int d) {
    const size_t terms = ((size_t)slabs * n * d * 2 * kTerms + 255) / 256 * 256;
    return 3 * terms + ((size_t)slabs * N * 8 + 255) / 256 * 256 + ((size_t)slabs * n * 8 + 255) / 256 * 256;
}

cudaError_t launch_backward_terms(int dtype, const BwdCall& c, void* ws, cudaStream_t st) {
    const int N = c.H * c.W, n = c.n, d = c.d, slabs = c.slabs;
    char* w = static_cast<char*>(ws);
    const size_t terms = ((size_t)slabs * n * d * 2 * kTerms + 255) / 256 * 256;
    __nv_bfloat16 *a_t = reinterpret_cast<__nv_bfloat16*>(w), *va_t = reinterpret_cast<__nv_bfloat16*>(w + terms), *dva_t = reinterpret_cast<__nv_bfloat16*>(w + 2 * terms);
    float2* tok_stats = reinterpret_cast<float2*>(w + 3 * terms);
    float2* agent_stats = reinterpret_cast<float2*>(w + 3 * terms + ((size_t)slabs * N * 8 + 255) / 256 * 256);
    const size_t pairs = (size_t)slabs * n * d / 2;
    bwd_split_kernel<<<(unsigned)((pairs + 255) / 256), 256, 0, st>>>(reinterpret_cast<const float2*>(c.ws_a), a_t, pairs);

    BwdTermArgs a;
    memset(&a, 0, sizeof(a));
    a.slabs = slabs; a.heads = c.heads; a.N = N; a.n = n; a.d = d;
    a.a_t = a_t; a.tok_stats = tok_stats; a.agent_stats = agent_stats;
    const SumsPlan sp = sums_plan(n, d);
    a.rg = sp.rg;
    BwdTermLaunch l;
    l.stream = st; l.kg = sp.kg;
    auto sums = [&](int which, bool cluster) {
        const int parts = token_parts((long long)slabs * sp.rb, N, 64, cluster ? 8 : 64, cluster, c.sm_count);
        a.tokens = ((N + parts - 1) / parts + 63) / 64 * 64;
        l.grid = dim3(parts, sp.rb, slabs);
        l.cluster = cluster ? parts : 0;
        return stage(dtype, d, which, a, l);
    };
    auto rows = [&](int which) {
        const int parts = token_parts(slabs, N, 128, 512, false, c.sm_count);
        a.tokens = ((N + parts - 1) / parts + 127) / 128 * 128;
        l.grid = dim3(parts, slabs);
        l.cluster = 0;
        return stage(dtype, d, which, a, l);
    };
    cudaError_t e;
#define AA_TRY(x) do { e = (x); if (e != cudaSuccess) return e; } while (0)
    // V_A and the statistics of the aggregation softmax
    a.x = c.k; a.y = c.v; a.bias = c.b1; a.scale = c.scale1; a.outer0 = c.ws_va; a.va_t = va_t;
    AA_TRY(sums(kTermForward, true));
    // broadcast stage: token statistics, then dV_A and its share of dA
    a.x = c.q; a.y = c.d_out; a.bias = c.b2; a.scale = a.out_scale = c.scale2; a.m_t = va_t;
    AA_TRY(rows(kTermStats));
    a.outer0 = c.ws_dva; a.outer1 = c.ws_da;
    AA_TRY(sums(kTermBroadcast, false));
    a.row0 = c.dq; a.dbias = c.db2;
    AA_TRY(rows(kTermQuery));
    bwd_dot_split_kernel<<<(unsigned)((slabs * n + 7) / 8), 256, 0, st>>>(c.ws_va, c.ws_dva, agent_stats, dva_t, slabs * n, d);
    // aggregation stage
    a.x = c.k; a.y = c.v; a.bias = c.b1; a.scale = c.scale1; a.out_scale = N == 1 ? 0.f : c.scale1; a.m_t = dva_t; a.dbias = c.db1;
    AA_TRY(sums(kTermAggregate, false));
    a.row0 = c.dk; a.row1 = c.dv; a.dbias = nullptr;
    AA_TRY(rows(kTermKeyValue));
#undef AA_TRY
    return cudaGetLastError();
}

}  // namespace aa
