// Gradient kernels on register tiles (mma.sync): operands that carry more than 16 bits are sums of 16-bit terms.
//
// Inputs (Q, K, V, dO) are NX terms of the MMA type E: one where E is their own type, two where fp16 inputs meet bf16 terms (a
// bf16 pair holds all 11 bits).  Derived operands (A, V_A, dV_A: TA, TM terms; P, dS: TP terms) are split when they are made; a
// product keeps the term pairs whose order is below that of the finer operand, so three bf16 terms give fp32 operands.
//
// Two orientations, so that no probability is ever transposed:
//   sums  rows = agents, columns = tokens: everything summed over tokens (V_A, dV_A, dA) and dB1
//   rows  rows = tokens, columns = agents: everything that a token owns (softmax statistics, dQ, dK, dV) and dB2
#pragma once
#include "tile_agg.cuh"

namespace aa {

enum BwdSums { kSumsForward, kSumsBroadcast, kSumsAggregate };
enum BwdRows { kRowsStats, kRowsQuery, kRowsKeyValue, kRowsOut, kRowsOutSplit };       // (split: two warps per 16 tokens, half of the agents each)

// term pairs of a product: i of NA, j of NB with i + j < max(NA, NB)
template <int NA, int NB> struct TermPairs {
    static constexpr int kOrder = NA > NB ? NA : NB;
    __host__ __device__ static constexpr bool keep(int i, int j) { return i + j < kOrder; }
};

// Products of two 8-column tiles (MMA operands A: terms of 16 rows, B: terms of 16 columns).  An mma.sync rounds its sum towards
// zero, so a long chain of them in one accumulator drifts: with chains over a block's whole token range the forward pass of 16384
// tokens was 1.4e-5 off, 1.2e-7 this way (fp32 FMAs: 1.4e-7).  So the pairs of leading terms are kept apart from the small ones, and
// sums over tokens or agents take 32 of them at a time (term_sum) and join in fp32 additions, which round to nearest.
template <typename E> __device__ __forceinline__ void mma_two(float (&c0)[4], float (&c1)[4], const uint32_t (&a)[4], const uint32_t (&b)[4], bool fresh) {
    if (fresh) {
        mma_set<E>(c0, a, b[0], b[1]);
        mma_set<E>(c1, a, b[2], b[3]);
    } else {
        mma_acc<E>(c0, a, b[0], b[1]);
        mma_acc<E>(c1, a, b[2], b[3]);
    }
}
// every pair of A's terms with term k of B, but for that of the leading terms; `fresh`: the first one starts the sum
template <typename E, int NA, int NB> __device__ __forceinline__ void mma_low(float (&c0)[4], float (&c1)[4], const uint32_t (&a)[NA][4], const uint32_t (&b)[4], int k, bool fresh) {
#pragma unroll
    for (int i = NA - 1; i >= 0; --i)
        if (TermPairs<NA, NB>::keep(i, k) && i + k > 0) {
            mma_two<E>(c0, c1, a[i], b, fresh);
            fresh = false;
        }
}
__device__ __forceinline__ void add4(float (&c)[4], const float (&t)[4]) {
#pragma unroll
    for (int e = 0; e < 4; e += 2) {
        const float2 u = fadd2(make_float2(c[e], c[e + 1]), make_float2(t[e], t[e + 1]));
        c[e] = u.x;
        c[e + 1] = u.y;
    }
}
// A product over 32 tokens or agents (two k steps), added to o0 and o1: `load(b, kk, k)` fetches term k of B.  The small pairs come
// first, so that only the two leading ones are rounded at full magnitude.
template <typename E, int NA, int NB, typename F>
__device__ __forceinline__ void term_sum(float (&o0)[4], float (&o1)[4], const uint32_t (&a)[2][NA][4], F&& load) {
    static_assert(NA > 1 || NB > 1, "small pairs start the sum");
    float t[2][4];
    uint32_t b[2][4];
#pragma unroll
    for (int kk = 0; kk < 2; ++kk)
#pragma unroll
        for (int k = NB - 1; k >= 0; --k) {
            load(b[kk], kk, k);
            mma_low<E, NA, NB>(t[0], t[1], a[kk], b[kk], k, kk == 0 && k == NB - 1);
        }
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) mma_two<E>(t[0], t[1], a[kk][0], b[kk], false);
    add4(o0, t[0]);
    add4(o1, t[1]);
}

// pack2 of finite values that never rounds up to infinity (fp32 reaches half a bf16 step past the largest bf16)
template <typename E> __device__ __forceinline__ uint32_t pack2_finite(float lo, float hi) {
    uint32_t w;
    if constexpr (Elem<E>::kIsBf16) asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;\n" : "=r"(w) : "f"(hi), "f"(lo));
    else w = pack2<E>(lo, hi);
    return w;
}
// two fp32 -> NT packed pairs of terms.  Finite values are finite sums of terms; an infinite one has a NaN among its terms.
template <typename E, int NT> __device__ __forceinline__ void split_pair(float a, float b, uint32_t (&w)[NT]) {
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        w[i] = i == 0 && NT > 1 ? pack2_finite<E>(a, b) : pack2<E>(a, b);
        if (i + 1 < NT) {
            const float2 u = unpack2<E>(w[i]);
            a -= u.x;
            b -= u.y;
        }
    }
}
// the same, residuals by packed arithmetic (FINITE: the values may be past the largest E)
template <typename E, int NT, bool FINITE = true> __device__ __forceinline__ void split_pair(float2 v, uint32_t (&w)[NT]) {
    w[0] = FINITE ? pack2_finite<E>(v.x, v.y) : pack2<E>(v.x, v.y);
#pragma unroll
    for (int i = 1; i < NT; ++i) {
        v = ffma2(unpack2<E>(w[i - 1]), make_float2(-1.f, -1.f), v);
        w[i] = pack2<E>(v.x, v.y);
    }
}
__device__ __forceinline__ void bar_named(int id, int threads) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void red_add4(float* p, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1,%2,%3,%4};\n" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
// eight consecutive bias gradients of one row: added, or stored where the batch has one entry
__device__ __forceinline__ void put_dbias8(float* p, const float* v, int cnt, bool aligned, bool store) {
    if (cnt >= 8 && aligned) {
        if (store) {
            *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
        } else {
            red_add4(p, v[0], v[1], v[2], v[3]);
            red_add4(p + 4, v[4], v[5], v[6], v[7]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < cnt) {
                if (store) p[i] = v[i];
                else atomicAdd(p + i, v[i]);
            }
    }
}

// Sum of the infinities and NaNs of a column: what a weighted sum over it comes to (zero: all are finite).  The terms of an infinite value
// hold a NaN, so the forward kernels ask here where a sum is NaN and its weights are not; never on finite inputs.
static __device__ __noinline__ float nonfinite_sum(const float* p, int stride, int count) {
    float s = 0.f;
    for (int i = 0; i < count; ++i) {
        const float v = p[(size_t)i * stride];
        if (!(fabsf(v) < INFINITY)) s += v;
    }
    return s;
}

// A operand (16 rows x 16 channels) from a tile in natural row order
template <int PITCH> __device__ __forceinline__ uint32_t a_lane_offset(int lane) { return (lane & 15) * PITCH + (lane >> 4) * 16; }

// Eight channels of a token row as NX chunks of terms (zeros where there are none)
template <typename T, typename E, int NX> __device__ __forceinline__ void load_terms(const T* src, bool ok, uint4 (&out)[NX]) {
    uint32_t o[NX][4];
    uint4 raw[sizeof(T) / 2];
#pragma unroll
    for (int i = 0; i < (int)sizeof(T) / 2; ++i) raw[i] = ok ? __ldg(reinterpret_cast<const uint4*>(src) + i) : make_uint4(0u, 0u, 0u, 0u);
    float f[8];
    unpack16<T>(raw[0], f);
    if constexpr (sizeof(T) == 4) unpack16<T>(raw[1], f + 4);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t t[NX];
        split_pair<E, NX>(f[2 * i], f[2 * i + 1], t);
#pragma unroll
        for (int k = 0; k < NX; ++k) o[k][i] = t[k];
    }
#pragma unroll
    for (int k = 0; k < NX; ++k) out[k] = make_uint4(o[k][0], o[k][1], o[k][2], o[k][3]);
}
// Two channels of a token row in fp32
template <typename T> __device__ __forceinline__ float2 load_pair(const T* src) {
    if constexpr (sizeof(T) == 4) return __ldg(reinterpret_cast<const float2*>(src));
    else return unpack2<T>(__ldg(reinterpret_cast<const uint32_t*>(src)));
}
// Eight consecutive biases of a row of `row` elements times log2(e); the first `left` exist (the others are not used).
template <typename T> __device__ __forceinline__ void load_bias_row(const T* p, int left, int row, const T* end, float (&bs)[8]) {
    if constexpr (sizeof(T) == 4) {
        if (row % 4 == 0) {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (left > 0) a = __ldg(reinterpret_cast<const float4*>(p));
            if (left > 4) b = __ldg(reinterpret_cast<const float4*>(p) + 1);
            bs[0] = a.x; bs[1] = a.y; bs[2] = a.z; bs[3] = a.w;
            bs[4] = b.x; bs[5] = b.y; bs[6] = b.z; bs[7] = b.w;
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) bs[i] = i < left ? __ldg(p + i) : 0.f;
        }
    } else {
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
        if (left > 0) w = row % 8 == 0 ? __ldg(reinterpret_cast<const uint4*>(p)) : load_bias8_any(p, end);
        unpack16<T>(w, bs);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) bs[i] *= kLog2e;
}

struct BwdTermArgs {
    const void *x, *y, *bias;              // [slabs][N][d] (Q, dO or K, V); B2 [heads][N][n] or B1 [heads][n][N], or null
    const void *a_t, *m_t;                 // terms [terms][slabs][n][d] of A; of V_A or dV_A
    float2* tok_stats;                     // [slabs][N]: (log2-sum-exp, row dot) of the broadcast softmax
    float2* agent_stats;                   // [slabs][n]: (log2-sum-exp, D) of the aggregation softmax
    float *outer0, *outer1;                // fp32 [slabs][n][d]  (rows out: V_A)
    float *row0, *row1;                    // fp32 [slabs][N][d]
    float* dbias;
    void* va_t;                            // forward sums: terms of V_A
    int slabs, heads, N, n, d;
    int rg, tokens;                        // sums: row groups; tokens per block (either kernel)
    const void* wd;                        // rows out: depthwise filter [heads][d][3][3] over y, or null
    int H, W;
    float scale;                           // of the logits
    float out_scale;                       // of dQ, dK and dA: the same; 0 where the softmax has one column (its logit gradients are exactly zero)
};

// ------------------------------------------------------------------------------------------------------------- sums
template <int DK, int NX, int TA, int TM, int KG, int NW, int MODE> struct SumsShape {
    static constexpr int kPitch = DK * 2 + 16;
    static constexpr int kTokens = NX == 1 && KG < 2 ? 64 : 32 * KG;
    static constexpr int kStages = NX == 1 && NW == 8 ? 3 : 2;
    static constexpr int kStats = MODE == kSumsBroadcast ? kTokens * 8 : 0;
    static constexpr int kStage = 2 * NX * kTokens * kPitch + kStats;
    static constexpr int kMats = TA + (MODE == kSumsForward ? 0 : TM);
    static constexpr int kAccPitch = DK + 8;
    static constexpr int kMerge = NW * 16 * (kAccPitch + 2) * 4 + NW * 16 * 8 * KG * 4;        // forward: partial states, over the ring
    __host__ __device__ static constexpr int smem(int rows) {
        const int ring = kStages * kStage, part = MODE == kSumsForward ? kMerge : 0;
        return kMats * rows * kPitch + (ring > part ? ring : part);
    }
};

template <typename T, typename E, int DK, int NX, int TA, int TM, int TP, int KG, int NW, int MODE>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? 1 : 3) bwd_sums_kernel(const __grid_constant__ BwdTermArgs p) {
    using S = SumsShape<DK, NX, TA, TM, KG, NW, MODE>;
    constexpr int PITCH = S::kPitch, KS = DK / 16, NT = DK / 8, TOK = S::kTokens;
    constexpr bool kLow = TA > 1 || NX > 1;            // (mixed precision: the logits have one pair of terms)
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int slab = blockIdx.z, head = slab % p.heads, rows = p.rg * 16, row0 = blockIdx.y * rows;
    const int t0 = min(p.N, (int)blockIdx.x * p.tokens), t1 = min(p.N, t0 + p.tokens);
    const int rgi = warp % p.rg, kgi = warp / p.rg;
    const bool active = kgi < KG;
    const uint32_t sm = smem_u32(smem), ring = sm + S::kMats * rows * PITCH;
    pdl_wait_prior();
    pdl_release_next();
    // agents' terms
    {
        const int chunks = DK / 8;
        for (int i = threadIdx.x; i < S::kMats * rows * chunks; i += NW * 32) {
            const int m = i / (rows * chunks), e = i - m * rows * chunks, r = e / chunks, ch = e - r * chunks;
            const bool ok = row0 + r < p.n && ch * 8 < p.d;
            const E* src = m < TA ? static_cast<const E*>(p.a_t) + (size_t)m * p.slabs * p.n * p.d
                                  : static_cast<const E*>(p.m_t) + (size_t)(m - TA) * p.slabs * p.n * p.d;
            const size_t off = ok ? ((size_t)slab * p.n + row0 + r) * p.d + ch * 8 : 0;
            cp_async16s(sm + (m * rows + r) * PITCH + ch * 16, src + off, ok ? 16 : 0);
        }
        cp_async_commit();
    }
    const T* x = static_cast<const T*>(p.x) + (size_t)slab * p.N * p.d;
    const T* y = static_cast<const T*>(p.y) + (size_t)slab * p.N * p.d;
    auto load = [&](int tok, int stage) {
        const uint32_t dst0 = ring + stage * S::kStage;
        for (int i = threadIdx.x; i < TOK * (DK / 8); i += NW * 32) {
            const int r = i / (DK / 8), ch = i - r * (DK / 8);
            const bool ok = tok + r < t1 && ch * 8 < p.d;
            const size_t off = ok ? (size_t)(tok + r) * p.d + ch * 8 : 0;
            const uint32_t o = col_to_row(r) * PITCH + ch * 16;
            if constexpr (NX == 1) {
                cp_async16s(dst0 + o, x + off, ok ? 16 : 0);
                cp_async16s(dst0 + TOK * PITCH + o, y + off, ok ? 16 : 0);
            } else {
                uint4 a[NX], b[NX];
                load_terms<T, E, NX>(x + off, ok, a);
                load_terms<T, E, NX>(y + off, ok, b);
#pragma unroll
                for (int k = 0; k < NX; ++k) {
                    *reinterpret_cast<uint4*>(smem + (dst0 - sm) + k * TOK * PITCH + o) = a[k];
                    *reinterpret_cast<uint4*>(smem + (dst0 - sm) + (NX + k) * TOK * PITCH + o) = b[k];
                }
            }
        }
        if (MODE == kSumsBroadcast && threadIdx.x < TOK) {
            float2 s = make_float2(INFINITY, 0.f);                    // no such token: its probabilities are zero
            if (tok + (int)threadIdx.x < t1) s = p.tok_stats[(size_t)slab * p.N + tok + threadIdx.x];
            *reinterpret_cast<float2*>(smem + (dst0 - sm) + 2 * NX * TOK * PITCH + threadIdx.x * 8) = s;
        }
    };
    const int tiles = (t1 - t0 + TOK - 1) / TOK;
#pragma unroll
    for (int i = 0; i < S::kStages - 1; ++i) {
        if (i < tiles) load(t0 + i * TOK, i);
        cp_async_commit();
    }
    float o0[NT][4], o1[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) o0[j][e] = o1[j][e] = 0.f;
    const int r0 = row0 + rgi * 16 + g;
    float2 rs[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    if (MODE == kSumsAggregate)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (r0 + h * 8 < p.n) rs[h] = p.agent_stats[(size_t)slab * p.n + r0 + h * 8];
    float ref[2] = {-INFINITY, -INFINITY}, sum[2] = {0.f, 0.f};
    const float c1 = p.scale * kLog2e;
    // bias element (row r, token c): B1 [n][N] in the aggregation, B2 [N][n] in the broadcast
    const T* bias = p.bias ? static_cast<const T*>(p.bias) + (size_t)head * p.n * p.N : nullptr;
    const T* bias_end = p.bias ? static_cast<const T*>(p.bias) + (size_t)p.heads * p.n * p.N : nullptr;
    const uint32_t aoff = sm + rgi * 16 * PITCH + a_lane_offset<PITCH>(lane);
    const uint32_t koff = key_lane_offset<DK>(lane) + kgi * 32 * PITCH, voff = val_lane_offset<DK>(lane) + kgi * 32 * PITCH;
    for (int it = 0; it < tiles; ++it) {
        if (NX == 1) cp_async_wait<S::kStages - 2>();
        else cp_async_wait<0>();
        __syncthreads();
        if (it + S::kStages - 1 < tiles) load(t0 + (it + S::kStages - 1) * TOK, (it + S::kStages - 1) % S::kStages);
        cp_async_commit();
        if (!active) continue;
        const uint32_t st = ring + (it % S::kStages) * S::kStage;
#pragma unroll 1
        for (int sub = 0; sub * 32 * KG < TOK; ++sub) {
            const int tok = t0 + it * TOK + (sub * KG + kgi) * 32;
            if (tok >= t1) break;
            const uint32_t xs = st + sub * KG * 32 * PITCH, ys = xs + NX * TOK * PITCH;
            float s[4][4], dp[4][4], sl[4][4], dl[4][4];                  // leading terms, small ones
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                uint32_t a[TA][4], m[TM][4];
#pragma unroll
                for (int i = 0; i < TA; ++i) ldsm4(a[i], aoff + i * rows * PITCH + ks * 32);
                if (MODE != kSumsForward)
#pragma unroll
                    for (int i = 0; i < TM; ++i) ldsm4(m[i], aoff + (TA + i) * rows * PITCH + ks * 32);
#pragma unroll
                for (int j2 = 0; j2 < 2; ++j2)
#pragma unroll
                    for (int k = 0; k < NX; ++k) {
                        uint32_t b[4];
                        ldsm4(b, xs + koff + k * TOK * PITCH + j2 * 16 * PITCH + ks * 32);
                        if (k == 0) mma_two<E>(s[2 * j2], s[2 * j2 + 1], a[0], b, ks == 0);
                        mma_low<E, TA, NX>(sl[2 * j2], sl[2 * j2 + 1], a, b, k, ks == 0 && k == 0);
                        if (MODE != kSumsForward) {
                            ldsm4(b, ys + koff + k * TOK * PITCH + j2 * 16 * PITCH + ks * 32);
                            if (k == 0) mma_two<E>(dp[2 * j2], dp[2 * j2 + 1], m[0], b, ks == 0);
                            mma_low<E, TM, NX>(dl[2 * j2], dl[2 * j2 + 1], m, b, k, ks == 0 && k == 0);
                        }
                    }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (kLow) add4(s[j], sl[j]);
                if (MODE != kSumsForward) add4(dp[j], dl[j]);
            }
            // logits in log2 units, then probabilities and logit gradients
            const int left = t1 - tok - 8 * t;
            float bs[2][8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = r0 + h * 8;
#pragma unroll
                for (int i = 0; i < 8; ++i) bs[h][i] = 0.f;
                if (bias && r < p.n) {
                    if (MODE == kSumsBroadcast) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (i < left) bs[h][i] = Elem<T>::to_f32(bias[(size_t)(tok + 8 * t + i) * p.n + r]) * kLog2e;
                    } else {
                        load_bias_row<T>(bias + (size_t)r * p.N + tok + 8 * t, left, p.N, bias_end, bs[h]);
                    }
                }
            }
            uint32_t pt[2][TP][4], dt[2][TP][4];
            if constexpr (MODE == kSumsForward) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float mx = -INFINITY;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            float& v = s[j][2 * h + e];
                            v = 2 * j + e < left ? fmaf(v, c1, bs[h][2 * j + e]) : -INFINITY;
                            mx = fmaxf(mx, v);
                        }
                    mx = quad_max(mx);
                    const float nr = fmaxf(ref[h], mx), f = ref[h] == -INFINITY ? 0.f : exp2f(ref[h] - nr);
                    ref[h] = nr;
                    sum[h] *= f;
#pragma unroll
                    for (int j = 0; j < NT; ++j) { o0[j][2 * h] *= f; o0[j][2 * h + 1] *= f; }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float p0 = nr == -INFINITY ? 0.f : fast_exp2(s[j][2 * h] - nr), p1 = nr == -INFINITY ? 0.f : fast_exp2(s[j][2 * h + 1] - nr);
                        sum[h] += p0 + p1;
                        uint32_t w[TP];
                        split_pair<E, TP>(p0, p1, w);
#pragma unroll
                        for (int i = 0; i < TP; ++i) pt[j >> 1][i][(j & 1) * 2 + h] = w[i];
                    }
                }
            } else {
                float2 cs[8];
                if (MODE == kSumsBroadcast)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 v = *reinterpret_cast<const float4*>(smem + (st - sm) + 2 * NX * TOK * PITCH + ((sub * KG + kgi) * 32 + 8 * t + 2 * i) * 8);
                        cs[2 * i] = make_float2(v.x, v.y);
                        cs[2 * i + 1] = make_float2(v.z, v.w);
                    }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float ds[8];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float pv[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int i = 2 * j + e;
                            const float2 q = MODE == kSumsBroadcast ? cs[i] : rs[h];
                            pv[e] = fast_exp2(fmaf(s[j][2 * h + e], c1, bs[h][i] - q.x));
                            if (MODE == kSumsAggregate && (i >= left || p.N == 1)) pv[e] = 0.f;      // (a softmax over one token has no gradient)
                            ds[i] = pv[e] * (dp[j][2 * h + e] - q.y);
                        }
                        uint32_t w[TP];
                        if (MODE == kSumsBroadcast) {
                            split_pair<E, TP>(pv[0], pv[1], w);
#pragma unroll
                            for (int i = 0; i < TP; ++i) pt[j >> 1][i][(j & 1) * 2 + h] = w[i];
                        }
                        split_pair<E, TP>(ds[2 * j], ds[2 * j + 1], w);
#pragma unroll
                        for (int i = 0; i < TP; ++i) dt[j >> 1][i][(j & 1) * 2 + h] = w[i];
                    }
                    if (MODE == kSumsAggregate && p.dbias && r0 + h * 8 < p.n)
                        put_dbias8(p.dbias + ((size_t)head * p.n + r0 + h * 8) * p.N + tok + 8 * t, ds, left, p.N % 4 == 0, p.slabs == p.heads);
                }
            }
#pragma unroll
            for (int c2 = 0; c2 < NT / 2; ++c2) {
                auto rows = [&](uint32_t base) {
                    return [&, base](uint32_t (&b)[4], int kk, int k) { ldsm4t(b, base + voff + k * TOK * PITCH + kk * 16 * PITCH + c2 * 32); };
                };
                if constexpr (MODE != kSumsAggregate) term_sum<E, TP, NX>(o0[2 * c2], o0[2 * c2 + 1], pt, rows(ys));
                if constexpr (MODE != kSumsForward) term_sum<E, TP, NX>(o1[2 * c2], o1[2 * c2 + 1], dt, rows(xs));
            }
        }
    }
    if constexpr (MODE != kSumsForward) {
        if (!active) return;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = r0 + h * 8;
            if (r >= p.n) continue;
            const size_t off = ((size_t)slab * p.n + r) * p.d + 2 * t;
#pragma unroll
            for (int j = 0; j < NT; ++j)
                if (j * 8 + 2 * t < p.d) {
                    if (MODE == kSumsBroadcast) red_add2(p.outer0 + off + j * 8, o0[j][2 * h], o0[j][2 * h + 1]);
                    red_add2(p.outer1 + off + j * 8, o1[j][2 * h] * p.out_scale, o1[j][2 * h + 1] * p.out_scale);
                }
        }
    } else {
        // partial states of the slab's blocks meet in shared memory (as in agg_merge); V_A in fp32 and as terms, and the row statistics
        cp_async_wait<0>();
        __syncthreads();
        const int csize = gridDim.x, crank = blockIdx.x;
        unsigned char* ms = smem + S::kMats * rows * PITCH;
        float* acc = reinterpret_cast<float*>(ms) + warp * 16 * S::kAccPitch;
        float2* ml = reinterpret_cast<float2*>(ms + NW * 16 * S::kAccPitch * 4);
        float* wt = reinterpret_cast<float*>(ms + NW * 16 * (S::kAccPitch + 2) * 4);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float l = quad_sum(sum[h]);
            if (t == 0) ml[warp * 16 + h * 8 + g] = make_float2(ref[h], active ? l : 0.f);
#pragma unroll
            for (int j = 0; j < NT; ++j)
                *reinterpret_cast<float2*>(acc + (h * 8 + g) * S::kAccPitch + j * 8 + 2 * t) = make_float2(o0[j][2 * h], o0[j][2 * h + 1]);
        }
        cluster_sync_all(csize);
        const int nrows = min(rows, p.n - row0), nsrc = csize * KG, share = (nrows - crank + csize - 1) / csize;
        const uint32_t acc0 = smem_u32(ms), ml0 = acc0 + NW * 16 * S::kAccPitch * 4;
        if ((int)threadIdx.x < share) {
            const int r = crank + threadIdx.x * csize;
            float m[8 * KG], l[8 * KG], mm = -INFINITY, tot = 0.f;
#pragma unroll
            for (int q = 0; q < 8 * KG; ++q) {
                m[q] = 0.f; l[q] = 0.f;
                if (q < nsrc) {
                    const float2 v = ld_dsmem_f32x2(ml0 + ((q % KG) * rows + r) * 8, q / KG);
                    m[q] = v.x; l[q] = v.y;
                }
            }
#pragma unroll
            for (int q = 0; q < 8 * KG; ++q)
                if (l[q] > 0.f) mm = fmaxf(mm, m[q]);
#pragma unroll
            for (int q = 0; q < 8 * KG; ++q) {
                m[q] = l[q] > 0.f ? exp2f(m[q] - mm) : (l[q] == 0.f ? 0.f : l[q]);
                tot += l[q] * m[q];
            }
            const float inv = 1.f / tot;
#pragma unroll
            for (int q = 0; q < 8 * KG; ++q)
                if (q < nsrc) wt[threadIdx.x * nsrc + q] = m[q] * inv;
            p.agent_stats[(size_t)slab * p.n + row0 + r].x = mm + log2f(tot);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < share * (DK / 2); i += NW * 32) {
            const int k = i / (DK / 2), ch = 2 * (i - k * (DK / 2)), r = crank + k * csize;
            if (ch >= p.d) continue;
            float2 v = make_float2(0.f, 0.f);
            for (int b = 0; b < csize; ++b)
#pragma unroll
                for (int q = 0; q < KG; ++q) {
                    const float2 w = ld_dsmem_f32x2(acc0 + ((q * rows + r) * S::kAccPitch + ch) * 4, b);
                    const float f = wt[k * nsrc + b * KG + q];
                    v.x = fmaf(w.x, f, v.x);
                    v.y = fmaf(w.y, f, v.y);
                }
            if constexpr (sizeof(T) == 4) {
                if (isnan(v.x) && !isnan(wt[k * nsrc])) { const float f = nonfinite_sum(y + ch, p.d, p.N); if (f != 0.f) v.x = f; }
                if (isnan(v.y) && !isnan(wt[k * nsrc])) { const float f = nonfinite_sum(y + ch + 1, p.d, p.N); if (f != 0.f) v.y = f; }
            }
            const size_t off = ((size_t)slab * p.n + row0 + r) * p.d + ch;
            *reinterpret_cast<float2*>(p.outer0 + off) = v;
            uint32_t w[TM];
            split_pair<E, TM>(v.x, v.y, w);
#pragma unroll
            for (int q = 0; q < TM; ++q)
                *reinterpret_cast<uint32_t*>(static_cast<E*>(p.va_t) + (size_t)q * p.slabs * p.n * p.d + off) = w[q];
        }
        if (csize > 1) cluster_sync_all();
    }
}

// ------------------------------------------------------------------------------------------------------------- rows
template <int DK, int TA, int TM> struct RowsShape {
    static constexpr int kPitch = DK * 2 + 16;
    __host__ __device__ static constexpr int smem(int n) { return (TA + TM) * ((n + 31) & ~31) * kPitch + ((n + 31) & ~31) * 8; }      // (rows out: 9 DK filter words and DK sums)
    __host__ __device__ static constexpr int smem_out(int n) { return (TA + TM) * ((n + 31) & ~31) * kPitch + 10 * DK * 4; }
    // rows out, split: the 8-channel tiles up to kCut are finished by the first warp of a pair; per warp, what it gives away and its sums
    static constexpr int kCut = (DK / 16 + 1) / 2 * 2, kGive = (kCut * 4 + 4) * 128;
    __host__ __device__ static constexpr int smem_split(int n) { return smem_out(n) + 8 * kGive; }
};

template <typename T, typename E, int DK, int NX, int TA, int TM, int TP, int MODE>
__global__ void __launch_bounds__(256, 1) bwd_rows_kernel(const __grid_constant__ BwdTermArgs p) {
    constexpr int PITCH = DK * 2 + 16, KS = DK / 16, NT = DK / 8;
    constexpr bool kRaw = sizeof(T) == 4, kOut = MODE == kRowsOut || MODE == kRowsOutSplit;
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int slab = blockIdx.y, head = slab % p.heads, n32 = (p.n + 31) & ~31;
    const int t0 = min(p.N, (int)blockIdx.x * p.tokens), t1 = min(p.N, t0 + p.tokens);
    const uint32_t sm = smem_u32(smem);
    float2* st_s = reinterpret_cast<float2*>(smem + (TA + TM) * n32 * PITCH);
    float* wt_s = reinterpret_cast<float*>(st_s);
    float* inf_s = wt_s + 9 * DK;                      // (rows out) per channel: nonfinite_sum of V_A
    bool infinite = false;
    pdl_wait_prior();
    pdl_release_next();
    {
        const int chunks = DK / 8;
        for (int i = threadIdx.x; i < (TA + TM) * n32 * chunks; i += 256) {
            const int m = i / (n32 * chunks), e = i - m * n32 * chunks, r = e / chunks, ch = e - r * chunks;
            const bool ok = r < p.n && ch * 8 < p.d;
            const E* src = m < TA ? static_cast<const E*>(p.a_t) + (size_t)m * p.slabs * p.n * p.d
                                  : static_cast<const E*>(p.m_t) + (size_t)(m - TA) * p.slabs * p.n * p.d;
            const size_t off = ok ? ((size_t)slab * p.n + r) * p.d + ch * 8 : 0;
            cp_async16s(sm + (m * n32 + col_to_row(r)) * PITCH + ch * 16, src + off, ok ? 16 : 0);
        }
        if (kOut && p.wd)
            for (int i = threadIdx.x; i < p.d * 9; i += 256) wt_s[(i % 9) * DK + i / 9] = Elem<T>::to_f32(static_cast<const T*>(p.wd)[(size_t)head * p.d * 9 + i]);
        if (MODE == kRowsKeyValue)
            for (int i = threadIdx.x; i < n32; i += 256)                  // (no such agent: its probabilities are zero)
                st_s[i] = i < p.n ? p.agent_stats[(size_t)slab * p.n + i] : make_float2(INFINITY, 0.f);
        cp_async_commit();
        cp_async_wait<0>();
        if constexpr (kOut) {              // a NaN among the last terms of V_A (of those that this thread has copied)
            float2 z = make_float2(0.f, 0.f);
            const int last = (TA + TM - 1) * n32;
            for (int e = (threadIdx.x - last * chunks) & 255; e < n32 * chunks; e += 256) {
                const int r = e / chunks, ch = e - r * chunks;
                const uint4 w = *reinterpret_cast<const uint4*>(smem + (last + col_to_row(r)) * PITCH + ch * 16);
                const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) z = ffma2(unpack2<E>(u[k]), make_float2(0.f, 0.f), z);
            }
            infinite = __syncthreads_or(isnan(z.x + z.y));
            if (infinite) {
                for (int c = threadIdx.x; c < DK; c += 256) inf_s[c] = c < p.d ? nonfinite_sum(p.outer0 + (size_t)slab * p.n * p.d + c, p.d, p.n) : 0.f;
                __syncthreads();
            }
        } else {
            __syncthreads();
        }
    }
    const T* x = static_cast<const T*>(p.x) + (size_t)slab * p.N * p.d;
    const T* y = static_cast<const T*>(p.y) + (size_t)slab * p.N * p.d;
    const T* bias = p.bias ? static_cast<const T*>(p.bias) + (size_t)head * p.n * p.N : nullptr;
    const T* bias_end = p.bias ? static_cast<const T*>(p.bias) + (size_t)p.heads * p.n * p.N : nullptr;
    const float c1 = p.scale * kLog2e;
    const uint32_t koff = sm + key_lane_offset<DK>(lane), voff = sm + val_lane_offset<DK>(lane);
    // Few tokens for the chip: two warps share 16 of them, the blocks of 32 agents in turn, and meet over the running softmax states
    constexpr bool split = MODE == kRowsOutSplit;
    const int side = split ? warp >> 2 : 0, group = split ? warp & 3 : warp;
    constexpr int CUT = RowsShape<DK, TA, TM>::kCut;
    for (int tok = t0 + group * 16; tok < t1; tok += split ? 64 : 128) {
        // operand rows: as terms, or (fp32) as they are, split when they are used: three terms of both do not fit in registers
        uint32_t xf[kRaw ? 1 : NX][kRaw ? 1 : KS][4], yf[kRaw ? 1 : NX][kRaw ? 1 : KS][4];
        float2 xr[kRaw ? KS : 1][4], yr[kRaw ? KS : 1][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const size_t off = (size_t)min(tok + h * 8 + g, t1 - 1) * p.d + 2 * t;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const bool in = ks * 16 + k * 8 + 2 * t < p.d;
                    if constexpr (NX == 1) {
                        xf[0][ks][k * 2 + h] = in ? __ldg(reinterpret_cast<const uint32_t*>(x + off + ks * 16 + k * 8)) : 0u;
                        yf[0][ks][k * 2 + h] = in && !kOut ? __ldg(reinterpret_cast<const uint32_t*>(y + off + ks * 16 + k * 8)) : 0u;
                    } else {
                        float2 fx = make_float2(0.f, 0.f), fy = fx;
                        if (in) fx = load_pair<T>(x + off + ks * 16 + k * 8);
                        if (in && !kOut) fy = load_pair<T>(y + off + ks * 16 + k * 8);
                        if constexpr (kRaw) {
                            xr[ks][k * 2 + h] = fx;
                            yr[ks][k * 2 + h] = fy;
                        } else {
                            uint32_t w[NX];
                            split_pair<E, NX>(fx.x, fx.y, w);
#pragma unroll
                            for (int i = 0; i < NX; ++i) xf[i][ks][k * 2 + h] = w[i];
                            split_pair<E, NX>(fy.x, fy.y, w);
#pragma unroll
                            for (int i = 0; i < NX; ++i) yf[i][ks][k * 2 + h] = w[i];
                        }
                    }
                }
        }
        float o0[NT][4], o1[NT][4];
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) o0[j][e] = o1[j][e] = 0.f;
        float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f}, rd[2] = {0.f, 0.f};
        float2 rs[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        if (MODE == kRowsQuery)
#pragma unroll
            for (int h = 0; h < 2; ++h) rs[h] = p.tok_stats[(size_t)slab * p.N + min(tok + h * 8 + g, t1 - 1)];
#pragma unroll 1
        for (int blk = side * 32; blk < n32; blk += split ? 64 : 32) {
            float bs[2][8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int tk = tok + h * 8 + g, left = p.n - blk - 8 * t;
#pragma unroll
                for (int i = 0; i < 8; ++i) bs[h][i] = 0.f;
                if (bias && tk < t1) {
                    if (MODE == kRowsKeyValue) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (i < left) bs[h][i] = Elem<T>::to_f32(bias[(size_t)(blk + 8 * t + i) * p.N + tk]) * kLog2e;
                    } else {
                        load_bias_row<T>(bias + (size_t)tk * p.n + blk + 8 * t, left, p.n, bias_end, bs[h]);
                    }
                }
            }
            float s[4][4], dp[4][4], sl[4][4], dl[4][4];                  // leading terms, small ones
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                uint32_t xt[NX][4], yt[NX][4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if constexpr (kRaw) {
                        uint32_t w[NX];
                        split_pair<E, NX>(xr[ks][q].x, xr[ks][q].y, w);
#pragma unroll
                        for (int k = 0; k < NX; ++k) xt[k][q] = w[k];
                        if (!kOut) split_pair<E, NX>(yr[ks][q].x, yr[ks][q].y, w);
#pragma unroll
                        for (int k = 0; k < NX; ++k) yt[k][q] = w[k];
                    } else {
#pragma unroll
                        for (int k = 0; k < NX; ++k) { xt[k][q] = xf[k][ks][q]; yt[k][q] = yf[k][ks][q]; }
                    }
                }
#pragma unroll
                for (int j2 = 0; j2 < 2; ++j2) {
#pragma unroll
                    for (int i = 0; i < TA; ++i) {
                        uint32_t b[4];
                        ldsm4(b, koff + (i * n32 + blk + j2 * 16) * PITCH + ks * 32);
                        if (i == 0) mma_two<E>(s[2 * j2], s[2 * j2 + 1], xt[0], b, ks == 0);
                        mma_low<E, NX, TA>(sl[2 * j2], sl[2 * j2 + 1], xt, b, i, ks == 0 && i == (NX == 1));
                    }
                    if (!kOut)
#pragma unroll
                        for (int i = 0; i < TM; ++i) {
                            uint32_t b[4];
                            ldsm4(b, koff + ((TA + i) * n32 + blk + j2 * 16) * PITCH + ks * 32);
                            if (i == 0) mma_two<E>(dp[2 * j2], dp[2 * j2 + 1], yt[0], b, ks == 0);
                            mma_low<E, NX, TM>(dl[2 * j2], dl[2 * j2 + 1], yt, b, i, ks == 0 && i == (NX == 1));
                        }
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                add4(s[j], sl[j]);
                if (!kOut) add4(dp[j], dl[j]);
            }
            const int left = p.n - blk - 8 * t;
            if constexpr (MODE == kRowsStats) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {          // every thread keeps its own reference; the quad meets at the end
                    float mx = m[h];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float& v = s[i >> 1][2 * h + (i & 1)];
                        v = i < left ? fmaf(v, c1, bs[h][i]) : -INFINITY;
                        mx = fmaxf(mx, v);
                    }
                    const float base = mx == -INFINITY ? 0.f : mx, f = exp2f(m[h] - base);
                    m[h] = mx;
                    l[h] *= f;
                    rd[h] *= f;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float e = fast_exp2(s[i >> 1][2 * h + (i & 1)] - base);
                        l[h] += e;
                        rd[h] = fmaf(e, dp[i >> 1][2 * h + (i & 1)], rd[h]);
                    }
                }
            } else if constexpr (kOut) {
                uint32_t pt[2][TP][4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float mx = m[h];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float& v = s[i >> 1][2 * h + (i & 1)];
                        v = i < left ? fmaf(v, c1, bs[h][i]) : -INFINITY;
                        mx = fmaxf(mx, v);
                    }
                    mx = quad_max(mx);
                    const float base = mx == -INFINITY ? 0.f : mx, f = exp2f(m[h] - base);      // (every agent so far may be masked)
                    m[h] = mx;
                    l[h] *= f;
#pragma unroll
                    for (int j = 0; j < NT; ++j) { o0[j][2 * h] *= f; o0[j][2 * h + 1] *= f; }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float p0 = fast_exp2(s[j][2 * h] - base), p1 = fast_exp2(s[j][2 * h + 1] - base);
                        l[h] += p0 + p1;
                        uint32_t w[TP];
                        split_pair<E, TP>(p0, p1, w);
#pragma unroll
                        for (int i = 0; i < TP; ++i) pt[j >> 1][i][(j & 1) * 2 + h] = w[i];
                    }
                }
#pragma unroll
                for (int c2 = 0; c2 < NT / 2; ++c2)
                    term_sum<E, TP, TM>(o0[2 * c2], o0[2 * c2 + 1], pt, [&](uint32_t (&b)[4], int kk, int i) { ldsm4t(b, voff + ((TA + i) * n32 + blk + kk * 16) * PITCH + c2 * 32); });
            } else {
                uint32_t pt[2][TP][4], dt[2][TP][4];
                float2 cs[8];
                if (MODE == kRowsKeyValue)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 v = *reinterpret_cast<const float4*>(st_s + blk + 8 * t + 2 * i);
                        cs[2 * i] = make_float2(v.x, v.y);
                        cs[2 * i + 1] = make_float2(v.z, v.w);
                    }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float ds[8];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float pv[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int i = 2 * j + e;
                            const float2 q = MODE == kRowsKeyValue ? cs[i] : rs[h];
                            pv[e] = fast_exp2(fmaf(s[j][2 * h + e], c1, bs[h][i] - q.x));
                            if (MODE == kRowsQuery && i >= left) pv[e] = 0.f;
                            ds[i] = pv[e] * (dp[j][2 * h + e] - q.y);
                        }
                        uint32_t w[TP];
                        if (MODE == kRowsKeyValue) {
                            split_pair<E, TP>(pv[0], pv[1], w);
#pragma unroll
                            for (int i = 0; i < TP; ++i) pt[j >> 1][i][(j & 1) * 2 + h] = w[i];
                        }
                        split_pair<E, TP>(ds[2 * j], ds[2 * j + 1], w);
#pragma unroll
                        for (int i = 0; i < TP; ++i) dt[j >> 1][i][(j & 1) * 2 + h] = w[i];
                    }
                    if (MODE == kRowsQuery && p.dbias && tok + h * 8 + g < t1)
                        put_dbias8(p.dbias + ((size_t)head * p.N + tok + h * 8 + g) * p.n + blk + 8 * t, ds, left, p.n % 4 == 0, p.slabs == p.heads);
                }
#pragma unroll
                for (int c2 = 0; c2 < NT / 2; ++c2) {
                    term_sum<E, TP, TA>(o0[2 * c2], o0[2 * c2 + 1], dt, [&](uint32_t (&b)[4], int kk, int i) { ldsm4t(b, voff + (i * n32 + blk + kk * 16) * PITCH + c2 * 32); });
                    if (MODE == kRowsKeyValue)
                        term_sum<E, TP, TM>(o1[2 * c2], o1[2 * c2 + 1], pt, [&](uint32_t (&b)[4], int kk, int i) { ldsm4t(b, voff + ((TA + i) * n32 + blk + kk * 16) * PITCH + c2 * 32); });
                }
            }
        }
        if constexpr (kOut) {
            // neighbouring threads swap halves of two 8-channel tiles: then a thread has four channels of tile j + (t & 1) of both rows,
            // and the eighteen 16-byte loads of its two depthwise windows are in flight at once
            const bool odd = t & 1;
            bool in[2][9];
            if (split) {                               // (the partner's elements belong to the same lane)
                float* mine = reinterpret_cast<float*>(smem + RowsShape<DK, TA, TM>::smem_out(p.n) + warp * RowsShape<DK, TA, TM>::kGive) + lane;
                const float* other = reinterpret_cast<const float*>(smem + RowsShape<DK, TA, TM>::smem_out(p.n) + (warp ^ 4) * RowsShape<DK, TA, TM>::kGive) + lane;
#pragma unroll
                for (int j = 0; j < NT; ++j)
                    if ((j >= CUT) != side)
#pragma unroll
                        for (int e = 0; e < 4; ++e) mine[((j >= CUT ? j - CUT : j) * 4 + e) * 32] = o0[j][e];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    mine[(CUT * 4 + h) * 32] = m[h];
                    mine[(CUT * 4 + 2 + h) * 32] = l[h];
                }
                bar_named(1 + group, 64);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float om = other[(CUT * 4 + h) * 32], ol = other[(CUT * 4 + 2 + h) * 32], mm = fmaxf(m[h], om), base = mm == -INFINITY ? 0.f : mm;
                    const float f = exp2f(m[h] - base), fo = exp2f(om - base);
                    l[h] = l[h] * f + ol * fo;
#pragma unroll
                    for (int j = 0; j < NT; ++j)
                        if ((j >= CUT) == side)
#pragma unroll
                            for (int e = 0; e < 2; ++e) o0[j][2 * h + e] = o0[j][2 * h + e] * f + other[((j >= CUT ? j - CUT : j) * 4 + 2 * h + e) * 32] * fo;
                }
                bar_named(1 + group, 64);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float inv = 1.f / quad_sum(l[h]);
#pragma unroll
                for (int j = 0; j < NT; ++j) { o0[j][2 * h] *= inv; o0[j][2 * h + 1] *= inv; }
                if (infinite && !isnan(inv))
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int c = 0; c < 2; ++c)
                            if (inf_s[j * 8 + 2 * t + c] != 0.f) o0[j][2 * h + c] = inf_s[j * 8 + 2 * t + c];
                const int tk = tok + h * 8 + g, gy = tk / p.W, gx = tk - gy * p.W;
#pragma unroll
                for (int k = 0; k < 9; ++k) in[h][k] = p.wd && tk < t1 && (unsigned)(gy + k / 3 - 1) < (unsigned)p.H && (unsigned)(gx + k % 3 - 1) < (unsigned)p.W;
            }
#pragma unroll
            for (int j = 0; j < NT; j += 2) {
                if (split && (j >= CUT) != side) continue;
                const int ch = 8 * (j + (t & 1)) + 4 * (t >> 1);
                const bool live = ch < p.d;
                float4 u[2][9];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int k = 0; k < 9; ++k) {
                        u[h][k] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (in[h][k] && live) u[h][k] = __ldg(reinterpret_cast<const float4*>(y + (size_t)(tok + h * 8 + g + (k / 3 - 1) * p.W + k % 3 - 1) * p.d + ch));
                    }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float sx = odd ? o0[j][2 * h] : o0[j + 1][2 * h], sy = odd ? o0[j][2 * h + 1] : o0[j + 1][2 * h + 1];
                    const float rx = __shfl_xor_sync(0xffffffffu, sx, 1), ry = __shfl_xor_sync(0xffffffffu, sy, 1);
                    float4 v = odd ? make_float4(rx, ry, o0[j + 1][2 * h], o0[j + 1][2 * h + 1]) : make_float4(o0[j][2 * h], o0[j][2 * h + 1], rx, ry);
                    if (p.wd)
#pragma unroll
                        for (int k = 0; k < 9; ++k) {
                            const float4 w = *reinterpret_cast<const float4*>(wt_s + k * DK + ch);
                            v.x = fmaf(u[h][k].x, w.x, v.x);
                            v.y = fmaf(u[h][k].y, w.y, v.y);
                            v.z = fmaf(u[h][k].z, w.z, v.z);
                            v.w = fmaf(u[h][k].w, w.w, v.w);
                        }
                    if (live && tok + h * 8 + g < t1) *reinterpret_cast<float4*>(p.row0 + ((size_t)slab * p.N + tok + h * 8 + g) * p.d + ch) = v;
                }
            }
            continue;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int tk = tok + h * 8 + g;
            if constexpr (MODE == kRowsStats) {
                const float mm = quad_max(m[h]), f = m[h] == -INFINITY ? 0.f : exp2f(m[h] - mm);
                const float tot = quad_sum(l[h] * f), dot = quad_sum(rd[h] * f);
                if (t == 0 && tk < t1) p.tok_stats[(size_t)slab * p.N + tk] = make_float2(mm + log2f(tot), dot / tot);
            } else if (tk < t1) {
                const size_t off = ((size_t)slab * p.N + tk) * p.d + 2 * t;
#pragma unroll
                for (int j = 0; j < NT; ++j)
                    if (j * 8 + 2 * t < p.d) {
                        *reinterpret_cast<float2*>(p.row0 + off + j * 8) = make_float2(o0[j][2 * h] * p.out_scale, o0[j][2 * h + 1] * p.out_scale);
                        if (MODE == kRowsKeyValue) *reinterpret_cast<float2*>(p.row1 + off + j * 8) = make_float2(o1[j][2 * h], o1[j][2 * h + 1]);
                    }
            }
        }
    }
}

}  // namespace aa
