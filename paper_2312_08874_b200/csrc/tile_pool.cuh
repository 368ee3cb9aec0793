// Agent tokens by average pooling (text under Eq. 6): means of eight channels handed to the caller.
#pragma once
#include "tile.cuh"

namespace aa {

// Eight channels as loaded, and added to four pairs of sums.
template <typename T> struct Raw8 { uint4 w[sizeof(T) / 2]; };
template <typename T> __device__ __forceinline__ Raw8<T> ld_raw8(const T* p) {
    Raw8<T> r;
#pragma unroll
    for (int i = 0; i < (int)sizeof(T) / 2; ++i) r.w[i] = __ldg(reinterpret_cast<const uint4*>(p) + i);
    return r;
}
template <typename T> __device__ __forceinline__ void add_raw8(float2 (&acc)[4], const Raw8<T>& r) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            acc[2 * i] = fadd2(acc[2 * i], make_float2(__uint_as_float(r.w[i].x), __uint_as_float(r.w[i].y)));
            acc[2 * i + 1] = fadd2(acc[2 * i + 1], make_float2(__uint_as_float(r.w[i].z), __uint_as_float(r.w[i].w)));
        }
    } else {
        acc[0] = fadd2(acc[0], unpack2<T>(r.w[0].x));
        acc[1] = fadd2(acc[1], unpack2<T>(r.w[0].y));
        acc[2] = fadd2(acc[2], unpack2<T>(r.w[0].z));
        acc[3] = fadd2(acc[3], unpack2<T>(r.w[0].w));
    }
}

// One warp (of `parts` that take turns; the shares add up): mean of the window of agent (ay, ax) -> put(chunk, eight means) for every 8-channel chunk (fixed order, fp32).
template <typename T, typename F>
__device__ __forceinline__ void pool_window(const T* q, long long qst, int H, int W, int ph, int pw, int agent, int d, F&& put, int part = 0, int parts = 1) {
    const int lane = threadIdx.x & 31;
    const int ay = agent / pw, ax = agent - ay * pw;
    const int y0 = (ay * H) / ph, y1 = ((ay + 1) * H + ph - 1) / ph, x0 = (ax * W) / pw, x1 = ((ax + 1) * W + pw - 1) / pw;
    const int ww = x1 - x0, cnt = (y1 - y0) * ww;
    // lanes = (token sub-lane, 8-channel chunk): a power of two of chunks, so that shuffles reduce over the sub-lanes
    const int cpt = d / 8, cp2 = cpt <= 1 ? 1 : cpt <= 2 ? 2 : cpt <= 4 ? 4 : cpt <= 8 ? 8 : 16, tpl = 32 / cp2;
    const int ch = lane & (cp2 - 1), ts = lane / cp2, step = tpl * parts, t0 = ts + part * tpl;
    float2 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = make_float2(0.f, 0.f);
    int wy = t0 / ww, wx = t0 - wy * ww;
    const T* base = q + ((size_t)y0 * W + x0) * qst + ch * 8;
    for (int i = t0; i < cnt; i += 8 * step) {
        Raw8<T> raw[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            raw[u] = Raw8<T>{};
            if (i + u * step < cnt && ch < cpt) raw[u] = ld_raw8<T>(base + ((size_t)wy * W + wx) * qst);
            wx += step;
            while (wx >= ww) { wx -= ww; ++wy; }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) add_raw8<T>(acc, raw[u]);
    }
    for (int o = cp2; o < 32; o <<= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            acc[k].x += __shfl_xor_sync(0xffffffffu, acc[k].x, o);
            acc[k].y += __shfl_xor_sync(0xffffffffu, acc[k].y, o);
        }
    if (ts == 0 && ch < cpt) {
        const float inv = 1.f / (float)cnt;
        const float f[8] = {acc[0].x * inv, acc[0].y * inv, acc[1].x * inv, acc[1].y * inv,
                            acc[2].x * inv, acc[2].y * inv, acc[3].x * inv, acc[3].y * inv};
        put(ch, f);
    }
}

// One thread: eight channels of one agent, for small windows (independent loads, no shuffles; fixed order, fp32).
template <typename T, typename F>
__device__ __forceinline__ void pool_chunk(const T* q, long long qst, int H, int W, int ph, int pw, int agent, F&& put) {
    const int ay = agent / pw, ax = agent - ay * pw;
    const int y0 = (ay * H) / ph, y1 = ((ay + 1) * H + ph - 1) / ph, x0 = (ax * W) / pw, x1 = ((ax + 1) * W + pw - 1) / pw;
    float2 acc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[k] = make_float2(0.f, 0.f);
    for (int y = y0; y < y1; ++y) {
        const T* row = q + (long long)(y * W) * qst;
#pragma unroll 4
        for (int x = x0; x < x1; ++x) add_raw8<T>(acc, ld_raw8<T>(row + x * qst));
    }
    const float inv = 1.f / (float)((y1 - y0) * (x1 - x0));
    const float f[8] = {acc[0].x * inv, acc[0].y * inv, acc[1].x * inv, acc[1].y * inv,
                        acc[2].x * inv, acc[2].y * inv, acc[3].x * inv, acc[3].y * inv};
    put(f);
}

}  // namespace aa
