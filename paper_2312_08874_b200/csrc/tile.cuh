// Building blocks of the register-tiled attention kernels (mma.sync m16n8k16, 16-bit operands, fp32 accumulators).
//
// A warp owns 16 rows of one softmax attention and walks its columns in blocks of 32: logits (16 x 32) and outputs (16 x DK)
// stay in registers (with 128 channels at 128 registers a thread the compiler spills 96 to 644 bytes).  Rows are agents and columns tokens in the aggregation (Eq. 3, inner
// attention); rows are tokens and columns agents in the broadcast (outer attention).
//
// Column order: inside a block, thread t of a quad owns columns 8 t .. 8 t + 7 (so its biases are one 16-byte load):
// MMA column (j, 2 t + e), j = n-tile, stands for column 8 t + 2 j + e.  Key and value rows are put into shared memory in
// that order (col_to_row), so the permutation costs nothing afterwards.
#pragma once
#include "common.cuh"
#include "kernels.h"

namespace aa {

template <int DK> struct TileGeom {
    static constexpr int kPitch = DK * 2 + 16;      // bytes between rows in shared memory: ldmatrix without bank conflicts
    static constexpr int kKS = DK / 16;             // k steps of the logits
    static constexpr int kNT = DK / 8;              // 8-channel tiles of the output
};

__device__ __forceinline__ int col_to_row(int c) { return (c & ~31) | ((c & 6) << 2) | ((c >> 2) & 6) | (c & 1); }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// D = A B (+ D): pure functions of their registers, so the compiler may interleave them with the softmax arithmetic.
template <typename T> __device__ __forceinline__ void mma_acc(float* c, const uint32_t* a, uint32_t b0, uint32_t b1);
template <typename T> __device__ __forceinline__ void mma_set(float* c, const uint32_t* a, uint32_t b0, uint32_t b1);
#define AA_MMA_FORMS(TYPE, NAME)                                                                                          \
    template <> __device__ __forceinline__ void mma_acc<TYPE>(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {      \
        asm("mma.sync.aligned.m16n8k16.row.col.f32." NAME "." NAME ".f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n" \
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1)); \
    }                                                                                                                     \
    template <> __device__ __forceinline__ void mma_set<TYPE>(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {      \
        asm("mma.sync.aligned.m16n8k16.row.col.f32." NAME "." NAME ".f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};\n" \
            : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])                                                              \
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));                                    \
    }
AA_MMA_FORMS(__nv_bfloat16, "bf16")
AA_MMA_FORMS(__half, "f16")
#undef AA_MMA_FORMS
__device__ __forceinline__ void cp_async16s(uint32_t dst, const void* src, int src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_sync_all(int csize) {
    if (csize == 1) __syncthreads();
    else cluster_sync_all();
}
__device__ __forceinline__ float2 ld_dsmem_f32x2(uint32_t addr, uint32_t rank) {
    uint32_t a;
    float2 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(a) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float quad_max(float v) {
    v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
    return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Byte offset (inside a block of key or value rows) that a lane hands to ldmatrix.
template <int DK> __device__ __forceinline__ uint32_t key_lane_offset(int lane) {
    return ((lane & 7) + ((lane >> 4) & 1) * 8) * TileGeom<DK>::kPitch + ((lane >> 3) & 1) * 16;
}
template <int DK> __device__ __forceinline__ uint32_t val_lane_offset(int lane) {
    return (lane & 15) * TileGeom<DK>::kPitch + (lane >> 4) * 16;
}

// s = rows . keys^T for one block of 32 key rows at `kb` (lane offset included).
template <typename T, int DK> __device__ __forceinline__ void tile_logits(float (&s)[4][4], const uint32_t (&a)[TileGeom<DK>::kKS][4], uint32_t kb) {
    using G = TileGeom<DK>;
#pragma unroll
    for (int ks = 0; ks < G::kKS; ++ks)
#pragma unroll
        for (int j2 = 0; j2 < 2; ++j2) {
            uint32_t b[4];
            ldsm4(b, kb + j2 * 16 * G::kPitch + ks * 32);
            if (ks == 0) {
                mma_set<T>(s[2 * j2], a[ks], b[0], b[1]);
                mma_set<T>(s[2 * j2 + 1], a[ks], b[2], b[3]);
            } else {
                mma_acc<T>(s[2 * j2], a[ks], b[0], b[1]);
                mma_acc<T>(s[2 * j2 + 1], a[ks], b[2], b[3]);
            }
        }
}

// o += p . values for one block of 32 value rows at `vb` (lane offset included).
template <typename T, int DK> __device__ __forceinline__ void tile_values(float (&o)[TileGeom<DK>::kNT][4], const uint32_t (&p)[2][4], uint32_t vb) {
    using G = TileGeom<DK>;
#pragma unroll
    for (int ks = 0; ks < 2; ++ks)
#pragma unroll
        for (int c2 = 0; c2 < G::kNT / 2; ++c2) {
            uint32_t b[4];
            ldsm4t(b, vb + ks * 16 * G::kPitch + c2 * 32);
            mma_acc<T>(o[2 * c2], p[ks], b[0], b[1]);
            mma_acc<T>(o[2 * c2 + 1], p[ks], b[2], b[3]);
        }
}

// Running state of the softmax of a thread's two rows.  `ref` is the exponent reference in log2 units, taken from the row's first
// block; it moves only when a logit exceeds it by more than 8 (so the products are rescaled rarely, and probabilities stay below 2^8:
// inside fp16).  `lim` is that 8, or -inf while the row has no weight.  The sums of the rounded probabilities come out of one more MMA
// per k step, against ones (every column of it holds them): weights and normaliser agree, as they do not where the sums take the
// probabilities before rounding (2^-9 / sqrt(agents) apart in bf16), at the same time.
struct SoftRows {
    float ref[2], lim[2], sum[4];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int h = 0; h < 2; ++h) { ref[h] = 0.f; lim[h] = -INFINITY; sum[2 * h] = sum[2 * h + 1] = 0.f; }
    }
    __device__ __forceinline__ float total(int h) const { return sum[2 * h]; }
    template <typename T> __device__ __forceinline__ void add(const uint32_t (&p)[2][4]) {
        constexpr uint32_t kOnes = Elem<T>::kIsBf16 ? 0x3f803f80u : 0x3c003c00u;
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) mma_acc<T>(sum, p[ks], kOnes, kOnes);
    }
};

// Logits of one block -> probabilities as MMA operands.  x = s * c1 + bias * log2(e) - ref; columns at and past `valid`
// (counted inside the block) are removed.
template <typename T, int DK, int BIAS>
__device__ __forceinline__ void tile_softmax(float (&s)[4][4], const uint4 (&bias)[2], float c1, int valid, int t, SoftRows& st,
                                             float (&o)[TileGeom<DK>::kNT][4], uint32_t (&p)[2][4]) {
    using G = TileGeom<DK>;
    float2 x[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float2 nref = make_float2(-st.ref[h], -st.ref[h]);
        const uint32_t w[4] = {bias[h].x, bias[h].y, bias[h].z, bias[h].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float2 y = nref;
            if constexpr (BIAS != 0) y = ffma2(unpack2<T>(w[j]), make_float2(kLog2e, kLog2e), nref);
            x[h][j] = ffma2(make_float2(s[j][2 * h], s[j][2 * h + 1]), make_float2(c1, c1), y);
        }
    }
    if (valid < 32) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = 8 * t + 2 * j;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (c >= valid) x[h][j].x = -INFINITY;
                if (c + 1 >= valid) x[h][j].y = -INFINITY;
            }
        }
    }
    float mx[2];
    bool grow = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float m = fmaxf(x[h][0].x, x[h][0].y);
#pragma unroll
        for (int j = 1; j < 4; ++j) m = max3(m, x[h][j].x, x[h][j].y);
        mx[h] = m;
        grow |= m > st.lim[h];
    }
    if (__any_sync(0xffffffffu, grow)) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float m = quad_max(mx[h]);
            const bool first = st.lim[h] < 0.f;                           // then nothing is accumulated yet
            const float by = m > st.lim[h] ? m : 0.f;
            const float f = first ? 1.f : fast_exp2(-by);
            if (m > -INFINITY) st.lim[h] = 8.f;
            st.ref[h] += by;
            st.sum[2 * h] *= f;
            st.sum[2 * h + 1] *= f;
#pragma unroll
            for (int c = 0; c < G::kNT; ++c) { o[c][2 * h] *= f; o[c][2 * h + 1] *= f; }
#pragma unroll
            for (int j = 0; j < 4; ++j) { x[h][j].x -= by; x[h][j].y -= by; }
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j >> 1][(j & 1) * 2 + h] = pack2<T>(fast_exp2(x[h][j].x), fast_exp2(x[h][j].y));
    st.add<T>(p);
}

}  // namespace aa
