// Aggregation on register tiles: V_A = softmax(scale1 A K^T + B1) V (Eq. 3 inner attention, bias of Eq. 5).
//
// A block of NW warps owns up to 16 NW agent rows of a slab and a range of its tokens: rg row groups of 16 agents times KG key
// groups that take alternate 32-token blocks.  Keys and values stream through a cp.async ring; the blocks of a slab form a
// thread-block cluster and merge their softmax states through distributed shared memory at the end.
#pragma once
#include "tile.cuh"

namespace aa {

constexpr int kAggStages = 3;

template <int DK, int KG, int NW> struct AggShape {
    using G = TileGeom<DK>;
    static constexpr int kThreads = NW * 32;
    static constexpr int kTokens = KG == 1 || KG * NW == 8 ? 64 : 128;                 // tokens of a stage
    static constexpr int kStage = 2 * kTokens * G::kPitch;             // K rows, then V rows
    static constexpr int kAccPitch = DK + 8;                           // fp32 words between the rows of a partial state
    static constexpr int kPart = NW * 16 * (kAccPitch + 2) * 4;         // partial states of the warps (over the ring, after the loop)
    static constexpr int kMerge = kPart + NW * 16 * 8 * KG * 4;            // and the merge weights
    static constexpr int kSmem = kAggStages * kStage > kMerge ? kAggStages * kStage : kMerge;
    // copies: a thread keeps its 16-byte channel chunk and steps by kRowStep rows
    static constexpr int kChunks = DK / 8;
    static constexpr int kRowStep = (kChunks <= 4 ? 64 : kChunks <= 8 ? 32 : 16) * NW / 8;
};

template <typename T> struct AggCta {
    const T *a, *k, *v, *b1;      // slab's agents [n][d], keys and values (token stride kst), head's bias [n][N] or null
    T* va;                        // slab's agent features [n][d]
    long long kst;
    int N, n, d, t0, t1;          // token range of this block
    int row0, rg;                 // first agent row of this block, row groups
    float c1;                     // logit scale in log2 units
    const T* b1_end;              // end of the bias tensor
};

// Eight bias elements from element address p of a tensor whose rows have no alignment: five aligned words, funnel-shifted.
template <typename T> __device__ __forceinline__ uint4 load_bias8_any(const T* p, const T* end) {
    uint32_t w[5];
    const uintptr_t u = reinterpret_cast<uintptr_t>(p);
    if (p + 9 < end) {
        const uint32_t* q = reinterpret_cast<const uint32_t*>(u & ~(uintptr_t)3);
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = __ldg(q + i);
        w[4] = (u & 2) ? __ldg(q + 4) : 0u;
        const int sh = (int)(u & 2) * 8;
        return make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh), __funnelshift_r(w[2], w[3], sh), __funnelshift_r(w[3], w[4], sh));
    }
    const unsigned short* s = reinterpret_cast<const unsigned short*>(p);
    const int cnt = p < end ? (int)(end - p) : 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = (2 * i < cnt ? s[2 * i] : 0u) | ((2 * i + 1 < cnt ? s[2 * i + 1] : 0u) << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// One stage of keys and values: token rows in block order, channels past d and tokens past the range zero.
template <typename T, int DK, int KG, int NW>
__device__ __forceinline__ void agg_load(const AggCta<T>& c, uint32_t dst, const T* kp, const T* vp, int left) {
    using G = TileGeom<DK>;
    using S = AggShape<DK, KG, NW>;
    const long long step = S::kRowStep * c.kst;
    if (left >= S::kTokens) {
#pragma unroll
        for (int i = 0; i < S::kTokens / S::kRowStep; ++i) {
            constexpr int R = S::kRowStep;
            const int off = ((i * R & ~31) + ((i * R >> 2) & 6)) * G::kPitch;          // col_to_row(i * R): R is 8, 16, 32 or 64
            cp_async16s(dst + off, kp + i * step, 16);
            cp_async16s(dst + S::kTokens * G::kPitch + off, vp + i * step, 16);
        }
    } else {
        const int r0 = threadIdx.x / S::kChunks;
        for (int i = 0; i < S::kTokens / S::kRowStep; ++i) {
            const int r = i * S::kRowStep, off = ((r & ~31) + ((r >> 2) & 6)) * G::kPitch;
            const bool ok = r0 + r < left;
            cp_async16s(dst + off, kp + (ok ? i * step : -(long long)r0 * c.kst), ok ? 16 : 0);
            cp_async16s(dst + S::kTokens * G::kPitch + off, vp + (ok ? i * step : -(long long)r0 * c.kst), ok ? 16 : 0);
        }
    }
}

// Aggregation over the block's token range; leaves the warps' partial states in `smem`.  `wait_agents` runs after the first
// copies have been issued.  BIAS: 0 none, 1 rows of 16-byte pieces (N a multiple of 8), 2 any row length.
template <typename T, int DK, int KG, int NW, int BIAS, typename F>
__device__ __forceinline__ void agg_phase(const AggCta<T>& c, unsigned char* smem, F&& wait_agents) {
    using G = TileGeom<DK>;
    using S = AggShape<DK, KG, NW>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    int rgi = warp, kgi = 0;
    if (KG > 1 && rgi >= c.rg) { rgi -= c.rg; ++kgi; }
    if (KG > 2 && rgi >= c.rg) { rgi -= c.rg; ++kgi; }
    if (KG > 2 && rgi >= c.rg) { rgi -= c.rg; ++kgi; }
    const bool active = rgi < c.rg;                          // the other warps only copy
    const uint32_t sm = smem_u32(smem);
    const int tiles = (c.t1 - c.t0 + S::kTokens - 1) / S::kTokens;
    const int lr = threadIdx.x / S::kChunks, lch = threadIdx.x - lr * S::kChunks;
    const bool loader = lr < S::kRowStep && lch * 8 < c.d;
    const uint32_t ldst = sm + col_to_row(lr) * G::kPitch + lch * 16;
    const T* kp = c.k + (long long)(c.t0 + lr) * c.kst + lch * 8;
    const T* vp = c.v + (long long)(c.t0 + lr) * c.kst + lch * 8;
    if (lr < S::kRowStep && lch * 8 >= c.d) {                // channels past d: cleared once
        for (int r = 0; r < kAggStages * S::kTokens * 2; r += S::kRowStep)
            *reinterpret_cast<uint4*>(smem + (size_t)(r + lr) * G::kPitch + lch * 16) = make_uint4(0u, 0u, 0u, 0u);
    }
    const long long tile_step = (long long)S::kTokens * c.kst;
#pragma unroll
    for (int i = 0; i < kAggStages - 1; ++i) {
        if (loader && i < tiles) agg_load<T, DK, KG, NW>(c, ldst + i * S::kStage, kp + i * tile_step, vp + i * tile_step, c.t1 - c.t0 - i * S::kTokens);
        cp_async_commit();
    }
    kp += (kAggStages - 1) * tile_step;
    vp += (kAggStages - 1) * tile_step;
    wait_agents();
    uint32_t a[G::kKS][4];
    const int r0 = c.row0 + rgi * 16 + g;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const bool ok = active && r0 + h * 8 < c.n;
        const T* ap = c.a + (size_t)(ok ? r0 + h * 8 : 0) * c.d + 2 * t;
#pragma unroll
        for (int ks = 0; ks < G::kKS; ++ks)
#pragma unroll
            for (int q = 0; q < 2; ++q)
                a[ks][q * 2 + h] = (ok && ks * 16 + q * 8 + 2 * t < c.d) ? *reinterpret_cast<const uint32_t*>(ap + ks * 16 + q * 8) : 0u;
    }
    float o[G::kNT][4];
#pragma unroll
    for (int j = 0; j < G::kNT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[j][e] = 0.f;
    SoftRows st;
    st.init();
    uint4 bias[2];
    // rows past n read the last row's bias (their results are not stored); columns past the end are masked, their loads clamped
    const T* brow = c.b1 + (size_t)min(r0, c.n - 1) * c.N;
    const long long brow8 = (long long)(min(r0 + 8, c.n - 1) - min(r0, c.n - 1)) * c.N;
    auto fetch_bias = [&](int tok) {
        if constexpr (BIAS == 1) {
            const int col = min(tok + 8 * t, c.N - 8);
            bias[0] = __ldg(reinterpret_cast<const uint4*>(brow + col));
            bias[1] = __ldg(reinterpret_cast<const uint4*>(brow + brow8 + col));
        } else if constexpr (BIAS == 2) {
            const int col = min(tok + 8 * t, c.N - 1);
            bias[0] = load_bias8_any(brow + col, c.b1_end);
            bias[1] = load_bias8_any(brow + brow8 + col, c.b1_end);
        }
    };
    int tok = c.t0 + kgi * 32;
    if (active) fetch_bias(tok);
    const uint32_t koff = key_lane_offset<DK>(lane) + kgi * 32 * G::kPitch;
    const uint32_t voff = val_lane_offset<DK>(lane) + (S::kTokens + kgi * 32) * G::kPitch;
    uint32_t rd = 0u, wr = (kAggStages - 1) * S::kStage;      // offsets of the stage being read / filled
    int left = c.t1 - c.t0 - (kAggStages - 1) * S::kTokens;
    for (int it = 0; it < tiles; ++it) {
        cp_async_wait<kAggStages - 2>();
        __syncthreads();
        if (loader && left > 0) agg_load<T, DK, KG, NW>(c, ldst + wr, kp, vp, left);
        cp_async_commit();
        kp += tile_step; vp += tile_step; left -= S::kTokens;
        if (active) {
#pragma unroll
            for (int sub = 0; sub < S::kTokens / (32 * KG); ++sub) {
                if (tok < c.t1) {
                    const uint32_t so = sm + rd + sub * KG * 32 * G::kPitch;
                    float s[4][4];
                    uint32_t p[2][4];
                    tile_logits<T, DK>(s, a, so + koff);
                    tile_softmax<T, DK, BIAS>(s, bias, c.c1, c.t1 - tok, t, st, o, p);
                    tok += 32 * KG;
                    fetch_bias(tok);
                    tile_values<T, DK>(o, p, so + voff);
                }
            }
        }
        rd = rd + S::kStage == kAggStages * S::kStage ? 0u : rd + S::kStage;
        wr = wr + S::kStage == kAggStages * S::kStage ? 0u : wr + S::kStage;
    }
    cp_async_wait<0>();
    __syncthreads();
    float* acc = reinterpret_cast<float*>(smem) + warp * 16 * S::kAccPitch;
    float2* ml = reinterpret_cast<float2*>(smem + NW * 16 * S::kAccPitch * 4) + warp * 16;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = h * 8 + g;
        const float l = st.total(h);
        if (t == 0) ml[r] = make_float2(st.ref[h], l);
#pragma unroll
        for (int j = 0; j < G::kNT; ++j)
            *reinterpret_cast<float2*>(acc + r * S::kAccPitch + j * 8 + 2 * t) = make_float2(o[j][2 * h], o[j][2 * h + 1]);
    }
}

// Merge of the partial states of the `csize` blocks of a cluster (KG states per row each): block `crank` writes its share of the
// agent rows (r = crank, crank + csize, ...).  A thread per row turns (reference, sum) pairs into weights, then a thread per two
// channels adds up: loads of different sources are independent, so the latency is that of two of them.  Fixed order:
// bit-reproducible.
template <typename T, int DK, int KG, int NW>
__device__ __forceinline__ void agg_merge(const AggCta<T>& c, unsigned char* smem, int crank, int csize) {
    using S = AggShape<DK, KG, NW>;
    const int rows = min(c.rg * 16, c.n - c.row0);
    const uint32_t acc0 = smem_u32(smem), ml0 = acc0 + NW * 16 * S::kAccPitch * 4;
    float* wt = reinterpret_cast<float*>(smem + S::kPart);                    // [share][csize * KG], normalised
    const int nsrc = csize * KG, share = (rows - crank + csize - 1) / csize;
    if ((int)threadIdx.x < share) {
        const int r = crank + threadIdx.x * csize;
        constexpr int kSrc = KG == 1 ? 16 : 32;                               // at most
        float m[kSrc], l[kSrc], mm = -INFINITY, tot = 0.f;
#pragma unroll
        for (int q = 0; q < kSrc; ++q) {
            m[q] = 0.f; l[q] = 0.f;
            if (q < nsrc) {
                const float2 v = ld_dsmem_f32x2(ml0 + ((q % KG) * c.rg * 16 + r) * 8, q / KG);
                m[q] = v.x; l[q] = v.y;
            }
        }
#pragma unroll
        for (int q = 0; q < kSrc; ++q)
            if (l[q] > 0.f) mm = fmaxf(mm, m[q]);
#pragma unroll
        for (int q = 0; q < kSrc; ++q) {
            m[q] = l[q] > 0.f ? fast_exp2(m[q] - mm) : (l[q] == 0.f ? 0.f : l[q]);      // (a NaN sum stays one)
            tot += l[q] * m[q];
        }
        const float inv = 1.f / tot;
#pragma unroll
        for (int q = 0; q < kSrc; ++q)
            if (q < nsrc) wt[threadIdx.x * nsrc + q] = m[q] * inv;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < share * (DK / 2); i += S::kThreads) {
        const int k = i / (DK / 2), ch = 2 * (i - k * (DK / 2)), r = crank + k * csize;
        if (ch >= c.d) continue;
        const uint32_t src = acc0 + (r * S::kAccPitch + ch) * 4;
        const float* w = wt + k * nsrc;
        float2 sum = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int b = 0; b < csize; ++b)
#pragma unroll
            for (int g = 0; g < KG; ++g) {
                const float2 v = ld_dsmem_f32x2(src + g * c.rg * 16 * S::kAccPitch * 4, b);
                const float f = w[b * KG + g];
                sum.x = fmaf(v.x, f, sum.x);
                sum.y = fmaf(v.y, f, sum.y);
            }
        *reinterpret_cast<uint32_t*>(c.va + (size_t)(c.row0 + r) * c.d + ch) = pack2<T>(sum.x, sum.y);
    }
}

}  // namespace aa
