// Broadcast on register tiles: O = softmax(scale2 Q A^T + B2) V_A + DWC(V) (Eq. 3 outer attention, Eq. 6).
//
// A block keeps the slab's agents and agent features in shared memory and walks a run of tokens, 16 per warp and pass.  The depthwise
// 3x3 term is added by MMAs into the same accumulators: k = (tap of a pair, channel of an 8-channel tile), the V rows of a tap come from
// a halo tile through ldmatrix (whose row addresses are free, so zero padding is the address of a zero row), and the filter is a
// diagonal operand.
#pragma once
#include "tile_agg.cuh"

namespace aa {

template <int DK> struct BcShape {
    using G = TileGeom<DK>;
    static constexpr int kChunks = DK / 8;
    static constexpr int kTab = 5 * G::kNT * 32 * 8;                  // filter operands: [tap pair][8-channel tile][lane] of two words
    __host__ __device__ static constexpr int rows(int n) { return (n + 31) & ~31; }
    __host__ __device__ static constexpr bool staged(int n) { return n % 8 != 0 && n <= 64; }   // bias rows go through shared memory
    __host__ __device__ static constexpr int bias_bytes(int n) { return staged(n) ? ((16 * n * 2 + 16 + 15) & ~15) : 0; }
    // rows of V around T tokens: the run of T + 2 W + 2, or (wide grids) three runs of T + 2, one per grid row of the window
    __host__ __device__ static constexpr int halo_rows(int tokens, int W) { return W <= tokens + 2 ? tokens + 2 * W + 2 : 3 * (tokens + 2); }
    __host__ __device__ static constexpr int v_bytes(int warps, int W, bool dwc) {      // (the outputs are staged in the same memory)
        return (dwc ? (halo_rows(warps * 16, W) > warps * 16 ? halo_rows(warps * 16, W) + 1 : warps * 16) : warps * 16) * G::kPitch;
    }
    __host__ __device__ static constexpr int smem_bytes(int n, int warps, int W, bool dwc) {
        return 2 * rows(n) * G::kPitch + v_bytes(warps, W, dwc) + (dwc ? kTab : 0) + warps * bias_bytes(n);
    }
};

template <typename T> struct BcCta {
    const T *q, *a, *va, *v, *b2, *wd;    // slab bases; b2 and wd: the head's, or null
    T* out;
    long long qst, ost;                   // token strides (Q and V share theirs)
    int N, n, d, H, W, t0, t1;
    float c1;
    const T* b2_end;                      // end of the bias tensor
};

// Agents and agent features: 16-byte copies in block order.
template <typename T, int DK>
__device__ __forceinline__ void bc_fill(const BcCta<T>& c, unsigned char* smem) {
    using G = TileGeom<DK>;
    using S = BcShape<DK>;
    const int rows = S::rows(c.n);
    const uint32_t sa = smem_u32(smem), sv = sa + rows * G::kPitch;
    for (int i = threadIdx.x; i < rows * S::kChunks; i += blockDim.x) {
        const int r = i / S::kChunks, ch = i - r * S::kChunks;
        const bool ok = r < c.n && ch * 8 < c.d;
        const size_t off = ok ? (size_t)r * c.d + ch * 8 : 0;
        const uint32_t dst = col_to_row(r) * G::kPitch + ch * 16;
        cp_async16s(sa + dst, c.a + off, ok ? 16 : 0);
        cp_async16s(sv + dst, c.va + off, ok ? 16 : 0);
    }
}
// Filter operands and the zero row of the halo tile; channels past d of the halo rows are cleared too.
template <typename T, int DK>
__device__ __forceinline__ void bc_fill_filter(const BcCta<T>& c, unsigned char* vtile, unsigned char* tab, int halo) {
    using G = TileGeom<DK>;
    using S = BcShape<DK>;
    const unsigned short* w = reinterpret_cast<const unsigned short*>(c.wd);
    // lane (g, t) of tile j has weights where t == g / 2: a thread fetches the nine taps of one (tile, lane), all at once
    for (int i = threadIdx.x; i < G::kNT * 32; i += blockDim.x) {
        const int ln = i & 31, j = i >> 5, col = ln >> 2, ch = 8 * j + col;
        const bool on = (ln & 3) == (col >> 1) && ch < c.d;
        uint32_t x[10];
#pragma unroll
        for (int u = 0; u < 9; ++u) x[u] = on ? (uint32_t)__ldg(w + ch * 9 + u) << ((col & 1) * 16) : 0u;
        x[9] = 0u;
#pragma unroll
        for (int pr = 0; pr < 5; ++pr) *reinterpret_cast<uint2*>(tab + (size_t)(pr * G::kNT * 32 + i) * 8) = make_uint2(x[2 * pr], x[2 * pr + 1]);
    }
    for (int i = threadIdx.x; i < S::kChunks; i += blockDim.x)
        *reinterpret_cast<uint4*>(vtile + (size_t)halo * G::kPitch + i * 16) = make_uint4(0u, 0u, 0u, 0u);
    if (c.d < DK)
        for (int i = threadIdx.x; i < halo; i += blockDim.x)
            for (int ch = c.d / 8; ch < S::kChunks; ++ch)
                *reinterpret_cast<uint4*>(vtile + (size_t)i * G::kPitch + ch * 16) = make_uint4(0u, 0u, 0u, 0u);
}

// V rows around the tokens [tok, tok + tokens).
template <typename T, int DK>
__device__ __forceinline__ void bc_load_halo(const BcCta<T>& c, uint32_t vtile, int tok, int tokens) {
    using G = TileGeom<DK>;
    using S = BcShape<DK>;
    const int step = blockDim.x / S::kChunks, r0 = threadIdx.x / S::kChunks, ch = threadIdx.x - r0 * S::kChunks;
    if (r0 >= step || ch * 8 >= c.d) return;
    const bool flat = c.W <= tokens + 2;
    const int run = flat ? tokens + 2 * c.W + 2 : tokens + 2, runs = flat ? 1 : 3;
    const int last = min(c.N, c.t1 + c.W + 1);
    for (int k = 0; k < runs; ++k) {
        const int first = flat ? tok - c.W - 1 : tok + (k - 1) * c.W - 1;
        const int lo = max(0, -first), hi = min(run, last - first);
        const uint32_t base = vtile + k * run * G::kPitch + ch * 16;
        for (int i = r0; i < hi; i += step)
            if (i >= lo) cp_async16s(base + i * G::kPitch, c.v + (long long)(first + i) * c.qst + ch * 8, 16);
    }
}

__device__ __forceinline__ void stsm4(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};\n" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}

// The whole phase for the tokens [t0, t1) of a block.
template <typename T, int DK, int BIAS>
__device__ __forceinline__ void bc_phase(const BcCta<T>& c, unsigned char* smem, int warps) {
    using G = TileGeom<DK>;
    using S = BcShape<DK>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int rows = S::rows(c.n), tokens = warps * 16, halo = S::halo_rows(tokens, c.W);
    const bool dwc = c.wd != nullptr, staged = BIAS == 2 && c.b2 && S::staged(c.n);
    unsigned char* vtile = smem + 2 * rows * G::kPitch;
    unsigned char* tab = vtile + S::v_bytes(warps, c.W, dwc);
    unsigned char* bstage = tab + (dwc ? S::kTab : 0) + warp * S::bias_bytes(c.n);
    const uint32_t ka = smem_u32(smem) + key_lane_offset<DK>(lane);
    const uint32_t vb = smem_u32(smem) + rows * G::kPitch + val_lane_offset<DK>(lane);
    const uint32_t vt = smem_u32(vtile);
    if (dwc) bc_fill_filter<T, DK>(c, vtile, tab, halo);

    const bool full = c.d == DK;
    uint32_t a[G::kKS][4];
    uint4 bias[2];
    auto fetch_q = [&](int tok) {                      // tokens past the range read its last row (results not stored)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const T* q = c.q + (long long)min(tok + h * 8 + g, c.t1 - 1) * c.qst + 2 * t;
#pragma unroll
            for (int ks = 0; ks < G::kKS; ++ks)
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    a[ks][k * 2 + h] = (full || ks * 16 + k * 8 + 2 * t < c.d) ? __ldg(reinterpret_cast<const uint32_t*>(q + ks * 16 + k * 8)) : 0u;
        }
    };
    int shift = 0;
    auto stage_bias = [&](int tok) {                   // the warp's bias rows are one run: copied in whole 16-byte pieces around it
        if (BIAS == 2 && staged && tok < c.t1) {
            const uintptr_t src = reinterpret_cast<uintptr_t>(c.b2 + (size_t)tok * c.n);
            shift = (int)(src & 15u);
            const int bytes = min(16, c.t1 - tok) * c.n * 2 + shift;
            __syncwarp();
            for (int i = lane * 16; i < bytes; i += 512)
                cp_async16s(smem_u32(bstage) + i, reinterpret_cast<const void*>(src - shift + i), min(16, bytes - i));
        }
        cp_async_commit();
    };
    auto fetch_bias = [&](int tok, int blk) {
        if constexpr (BIAS != 0) {
            const int col = blk + 8 * t;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = min(tok + h * 8 + g, c.t1 - 1);
                if constexpr (BIAS == 1) {
                    bias[h] = __ldg(reinterpret_cast<const uint4*>(c.b2 + (size_t)r * c.n + min(col, c.n - 8)));
                } else if (staged) {
                    const unsigned short* u = reinterpret_cast<const unsigned short*>(bstage + shift) + (r - tok) * c.n;
                    uint32_t w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[i] = u[min(col + 2 * i, c.n - 1)] | ((uint32_t)u[min(col + 2 * i + 1, c.n - 1)] << 16);
                    bias[h] = make_uint4(w[0], w[1], w[2], w[3]);
                } else {
                    bias[h] = load_bias8_any(c.b2 + (size_t)r * c.n + min(col, c.n - 1), c.b2_end);
                }
            }
        }
    };
    int tok = c.t0 + warp * 16;
    fetch_q(tok);
    stage_bias(tok);
    if (!staged) fetch_bias(tok, 0);
    for (int base = c.t0; base < c.t1; base += tokens, tok += tokens) {
        if (dwc) bc_load_halo<T, DK>(c, vt, base, tokens);
        cp_async_commit();
        float o[G::kNT][4];
        if (tok < c.t1) {
            SoftRows st;
            st.init();
#pragma unroll
            for (int j = 0; j < G::kNT; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[j][e] = 0.f;
            if (BIAS == 2 && staged) {
                cp_async_wait<1>();
                __syncwarp();
                fetch_bias(tok, 0);
            }
            for (int blk = 0; blk < rows; blk += 32) {
                float s[4][4];
                uint32_t p[2][4];
                tile_logits<T, DK>(s, a, ka + blk * G::kPitch);
                tile_softmax<T, DK, BIAS>(s, bias, c.c1, c.n - blk, t, st, o, p);
                if (blk + 32 < rows) fetch_bias(tok, blk + 32);
                tile_values<T, DK>(o, p, vb + blk * G::kPitch);
            }
            fetch_q(tok + tokens);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float inv = 1.f / st.total(h);
#pragma unroll
                for (int j = 0; j < G::kNT; ++j) { o[j][2 * h] *= inv; o[j][2 * h + 1] *= inv; }
            }
        }
        stage_bias(tok + tokens);
        if (!staged) fetch_bias(tok + tokens, 0);
        cp_async_wait<1>();
        __syncthreads();                               // the halo tile has arrived
        if (dwc) {
            if (tok < c.t1) {
                const int tk = tok + (lane & 15), y = (int)((unsigned)tk / (unsigned)c.W), x = tk - y * c.W;
                const bool flat = c.W <= tokens + 2;
                const int dyr = flat ? c.W : tokens + 2;
                const uint32_t row = vt + (tk - base + dyr + 1) * G::kPitch, zero = vt + halo * G::kPitch;
                const uint2* tp = reinterpret_cast<const uint2*>(tab) + lane;
#pragma unroll
                for (int pr = 0; pr < 5; ++pr) {
                    const int dy = lane < 16 ? (2 * pr) / 3 - 1 : (2 * pr + 1) / 3 - 1, dx = lane < 16 ? (2 * pr) % 3 - 1 : (2 * pr + 1) % 3 - 1;
                    const bool ok = (unsigned)(y + dy) < (unsigned)c.H && (unsigned)(x + dx) < (unsigned)c.W;      // (tap 9: dy = 2, weight 0)
                    const uint32_t addr = ok && (pr < 4 || lane < 16) ? row + (dy * dyr + dx) * G::kPitch : zero;
#pragma unroll
                    for (int j = 0; j < G::kNT; ++j) {
                        uint32_t f[4];
                        ldsm4(f, addr + j * 16);
                        const uint2 w = tp[(pr * G::kNT + j) * 32];
                        mma_acc<T>(o[j], f, w.x, w.y);
                    }
                }
            }
            __syncthreads();                           // the halo tile makes room for the outputs
        }
        if (tok < c.t1) {
            const uint32_t os = vt + warp * 16 * G::kPitch;
#pragma unroll
            for (int j = 0; j < G::kNT; j += 2)
                stsm4(os + (lane & 15) * G::kPitch + (j + (lane >> 4)) * 16, pack2<T>(o[j][0], o[j][1]), pack2<T>(o[j][2], o[j][3]),
                      pack2<T>(o[j + 1][0], o[j + 1][1]), pack2<T>(o[j + 1][2], o[j + 1][3]));
            __syncwarp();
            const unsigned char* op = vtile + warp * 16 * G::kPitch;
#pragma unroll
            for (int i = 0; i < (16 * S::kChunks + 31) / 32; ++i) {
                const int e = i * 32 + lane, r = e / S::kChunks, ch = e - r * S::kChunks;
                if (r < 16 && tok + r < c.t1 && ch * 8 < c.d)
                    *reinterpret_cast<uint4*>(c.out + (long long)(tok + r) * c.ost + ch * 8) = *reinterpret_cast<const uint4*>(op + r * G::kPitch + ch * 16);
            }
        }
        if (base + tokens < c.t1) __syncthreads();     // before the next halo tile
    }
    cp_async_wait<0>();
}

}  // namespace aa
