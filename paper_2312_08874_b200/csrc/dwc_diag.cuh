// The depthwise 3x3 term (Eq. 6) by mma.sync with the filter as a diagonal operand, and the end of an output tile in that layout, for the
// tensor-memory kernels that keep V tokens as 128-byte rows in shared memory (128-byte swizzle).
#pragma once
#include "common.cuh"

namespace aa {

// Filter table: [10 taps][64 channels] words, the weight in the half that the channel has in a pair; the tenth tap weighs nothing.
constexpr int kFilterWords = 10 * 64;
__device__ __forceinline__ void fill_filter(uint32_t* tab, const void* filter, int head, int d, int tid, int threads) {
    const uint16_t* w = static_cast<const uint16_t*>(filter) + (size_t)head * d * 9;
#pragma unroll 2
    for (int e = tid; e < kFilterWords; e += threads) {
        const int tap = e >> 6, ch = e & 63;
        tab[e] = tap < 9 && ch < d ? (uint32_t)__ldg(w + ch * 9 + tap) << (16 * (ch & 1)) : 0u;
    }
}
// This lane's words of it: those of its channels on the operand's diagonal, zeros (a table of them) elsewhere.
__device__ __forceinline__ const uint32_t* filter_lane(const uint32_t* tab, const uint32_t* zeros, int lane) {
    return (lane & 3) == (lane >> 3) ? tab + (lane >> 2) : zeros;
}

// Window positions (bit 3 u + v) of the token at (x, y) that lie in the grid; with `lane`'s half of the tap pairs: bit 2 k is the tap that the lane
// addresses for pair k (lanes 0-15 the even taps, lanes 16-31 the odd ones).
__device__ __forceinline__ uint32_t grid_taps(int x, int y, int H, int W, int lane) {
    uint32_t in = 0x1ffu;
    if (x == 0) in &= ~0x49u;
    if (x == W - 1) in &= ~0x124u;
    if (y == 0) in &= ~7u;
    if (y == H - 1) in &= ~0x1c0u;
    return lane < 16 ? in : in >> 1;
}
// The same for token `tok` of a short grid (none from N on).
__device__ __forceinline__ uint32_t window_taps(int tok, int N, int H, int W, float inv_w, int lane) {
    int y = (int)((float)tok * inv_w), x = tok - y * W;                 // the quotient is off by one at most
    if (x < 0) { x += W; --y; }
    if (x >= W) { x -= W; ++y; }
    return tok >= N ? 0u : grid_taps(x, y, H, W, lane);
}

// o[mt][j] += the term of rows 16 mt .. + 15 and channels 8 j .. + 7 (mma.sync accumulator layout), k = (tap of a pair, channel of eight).
// Row `row0` + off(u, v) of `buf` holds the token at window position (u, v) of this lane's row (lane & 15); `chunk` is the byte offset of the
// first channel in an unswizzled row (a multiple of 64); the rows of mt = 1 are the next sixteen; rows outside the grid are read from `zeros`
// (128 bytes, 128-byte aligned).
template <typename T, typename Off>
__device__ __forceinline__ void dwc_rows(float (&o)[2][4][4], uint32_t buf, int row0, uint32_t chunk, const uint32_t (&in)[2], uint32_t zeros,
                                         const uint32_t* tab, int lane, Off&& off) {
#pragma unroll
    for (int pr = 0; pr < 5; ++pr) {
        const int ka = 2 * pr, kb = pr < 4 ? 2 * pr + 1 : 8;
        const int row = row0 + (lane < 16 ? off(ka / 3, ka % 3) : off(kb / 3, kb % 3));
        uint32_t w[4][2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            w[j][0] = tab[2 * pr * 64 + 8 * j];
            w[j][1] = tab[(2 * pr + 1) * 64 + 8 * j];
        }
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {
            const int r = row + 16 * mt;
            // (zeros at the same offset in their row, so that the eight rows of a matrix stay in different banks)
            const uint32_t src = (in[mt] & (1u << (2 * pr)) ? buf + r * 128 : zeros) + (chunk ^ ((r & 7) << 4));
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t f[4];
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                             : "=r"(f[0]), "=r"(f[1]), "=r"(f[2]), "=r"(f[3]) : "r"(src ^ (j << 4)) : "memory");
                mma16816<T>(o[mt][j], f, w[j][0], w[j][1]);
            }
        }
    }
}

// The same for two rows of a patch (mt: one of them) in a window of PITCH tokens a row, zeros included: the twelve operands (window row, shift) of both
// are read once, six instructions per 8-channel tile instead of ten.  `at`: see patch_offsets, plus the window's address.
template <int PITCH> __device__ __forceinline__ void patch_offsets(uint32_t (&at)[6], int row0, uint32_t chunk, int lane) {
#pragma unroll
    for (int i = 0; i < 6; ++i) {                                      // lanes 0-15 address operand 2 i, lanes 16-31 operand 2 i + 1
        const int f = 2 * i + (lane >> 4), r = row0 + f / 3 * PITCH + f % 3 + (lane & 15);
        at[i] = r * 128 + (chunk ^ ((r & 7) << 4));
    }
}
template <typename T>
__device__ __forceinline__ void dwc_patch(float (&o)[2][4][4], const uint32_t (&at)[6], uint32_t buf, const uint32_t* tab) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t f[6][4], w[10];
#pragma unroll
        for (int k = 0; k < 10; ++k) w[k] = tab[k * 64 + 8 * j];
#pragma unroll
        for (int i = 0; i < 6; ++i)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                         : "=r"(f[i][0]), "=r"(f[i][1]), "=r"(f[i][2]), "=r"(f[i][3]) : "r"((buf + at[i]) ^ (j << 4)) : "memory");
#pragma unroll
        for (int pr = 0; pr < 5; ++pr)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const int a = 3 * mt + 2 * pr, b = pr < 4 ? a + 1 : 0;
                uint32_t k[4] = {f[a >> 1][2 * (a & 1)], f[a >> 1][2 * (a & 1) + 1], f[b >> 1][2 * (b & 1)], f[b >> 1][2 * (b & 1) + 1]};
                if (pr == 4) k[2] = k[3] = 0u;                         // the tenth tap: no token (nothing times an infinity is NaN)
                mma16816<T>(o[mt][j], k, w[2 * pr], w[2 * pr + 1]);
            }
    }
}

// 16 rows x 32 channels in accumulator layout -> 16-bit rows at `out` (row stride in elements), channels c0 ..: neighbouring threads swap the channels
// of one 8-channel tile: eight bytes a thread, a row's 32 bytes a store.  Rows g and g + 8 exist where `ok`.
template <typename T>
__device__ __forceinline__ void store_rows(const float (&o)[4][4], T* out, size_t stride, int c0, int d, const bool (&ok)[2], int lane) {
    const int lg = lane >> 2, lt = lane & 3;
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        T* dst = out + (size_t)(8 * hh + lg) * stride;
#pragma unroll
        for (int jp = 0; jp < 2; ++jp) {
            const int ch = c0 + 16 * jp + 8 * (lt & 1) + 4 * (lt >> 1);
            const uint32_t wa = pack2<T>(o[2 * jp][2 * hh], o[2 * jp][2 * hh + 1]), wb = pack2<T>(o[2 * jp + 1][2 * hh], o[2 * jp + 1][2 * hh + 1]);
            const uint32_t got = __shfl_xor_sync(0xffffffffu, (lt & 1) ? wa : wb, 1);
            if (ok[hh] && ch < d) *reinterpret_cast<uint2*>(dst + ch) = (lt & 1) ? make_uint2(got, wb) : make_uint2(wa, got);
        }
    }
}

}  // namespace aa
