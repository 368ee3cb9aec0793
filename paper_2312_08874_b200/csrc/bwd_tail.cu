// Token-wise tail of the backward pass:
//   dQ  += Pooling^T(dA)   a window spreads its agent's gradient evenly over its tokens
//   dV  += DWC^T(dO)       tap (u, v) of output token (y - u + 1, x - v + 1) read V[y][x]
//   dWd += corr(dO, V)     dWd[c][u][v] = sum over tokens of dO[y - u + 1][x - v + 1][c] V[y][x][c]
// The first two are one pass with a thread per token and four channels and all its loads in flight at once (dQ and dV are read and
// written in fp32: that traffic is the bound).  The third is a pass of its own: its 36 sums per thread would halve the threads of
// the first.  64 slabs of a 56 x 56 grid: one pass for all three 156 us, these two 74 + 31 us.
#include "common.cuh"
#include "kernels.h"

namespace aa {

namespace {

struct TailArgs {
    const void *v, *go, *wd;
    const float* da;
    float *dq, *dv, *dwd;
    int heads, H, W, d, n, p, strip;
};

// Four channels of a token, as loaded; channel pairs in fp32 on use.
template <typename T> struct Raw4 { uint2 w; };
template <> struct Raw4<float> { float4 w; };
template <typename T> __device__ __forceinline__ Raw4<T> ld_raw4(const T* p) {
    Raw4<T> r;
    if constexpr (sizeof(T) == 4) r.w = __ldg(reinterpret_cast<const float4*>(p));
    else r.w = __ldg(reinterpret_cast<const uint2*>(p));
    return r;
}
template <typename T> __device__ __forceinline__ Raw4<T> zero_raw4() {
    Raw4<T> r;
    if constexpr (sizeof(T) == 4) r.w = make_float4(0.f, 0.f, 0.f, 0.f);
    else r.w = make_uint2(0u, 0u);
    return r;
}
template <typename T> __device__ __forceinline__ float2 pair(const Raw4<T>& r, int q) {
    if constexpr (sizeof(T) == 4) return q == 0 ? make_float2(r.w.x, r.w.y) : make_float2(r.w.z, r.w.w);
    else return unpack2<T>(q == 0 ? r.w.x : r.w.y);
}

// Pooling windows over position i of an axis of L positions and p cells: first cell, and the lengths of it and of the next
// (0: it does not contain i).  At most two windows overlap, since p <= L.
struct Windows {
    int first, len0, len1;
};
__device__ __forceinline__ Windows windows_of(int i, int L, int p) {
    Windows w = {0, 0, 0};
    int c = (i * p) / L;
    for (int k = 0; k < 2 && c < p; ++k, ++c) {
        const int lo = (c * L) / p, hi = ((c + 1) * L + p - 1) / p;
        if (i < lo || i >= hi) continue;
        if (w.len0 == 0) { w.first = c; w.len0 = hi - lo; }
        else w.len1 = hi - lo;
    }
    return w;
}

constexpr int kAxis = 512;         // positions of an axis whose windows are kept in shared memory

template <typename T, bool DWC>
__global__ void __launch_bounds__(256, DWC ? 3 : 4) bwd_tail_kernel(const TailArgs a, int tokens) {
    __shared__ __align__(16) float wt[DWC ? 9 * 128 : 4];
    __shared__ Windows yw[kAxis], xw[kAxis];
    const int d = a.d, H = a.H, W = a.W, p = a.p, N = H * W, slab = blockIdx.y;
    const int t0 = blockIdx.x * tokens, t1 = min(N, t0 + tokens);
    const int groups = d >> 2, cols = 256 / groups;               // d <= 128: at least eight tokens at once
    const int cg = threadIdx.x % groups, cl = threadIdx.x / groups;
    pdl_wait_prior();
    pdl_release_next();
    const int ylo = t0 / W, rows = (t1 - 1) / W - ylo + 1;
    for (int i = threadIdx.x; i < min(rows, kAxis); i += 256) yw[i] = windows_of(ylo + i, H, p);
    for (int i = threadIdx.x; i < min(W, kAxis); i += 256) xw[i] = windows_of(i, W, p);
    if (DWC) {
        const T* w = static_cast<const T*>(a.wd) + (size_t)(slab % a.heads) * d * 9;
        for (int i = threadIdx.x; i < d * 9; i += 256) wt[(i % 9) * d + i / 9] = Elem<T>::to_f32(w[i]);
    }
    __syncthreads();
    if (cl >= cols) return;
    const size_t base = (size_t)slab * N * d + 4 * cg;
    const T* go = static_cast<const T*>(a.go) + base;
    const float* da = a.da + (size_t)slab * a.n * d + 4 * cg;
    int tok = t0 + cl, y = tok / W, x = tok - y * W;
    for (; tok < t1; tok += cols) {
        float4 q = *reinterpret_cast<const float4*>(a.dq + base + (size_t)tok * d), o = make_float4(0.f, 0.f, 0.f, 0.f);
        Raw4<T> win[9];
        if (DWC) {
            o = *reinterpret_cast<const float4*>(a.dv + base + (size_t)tok * d);
#pragma unroll
            for (int k = 0; k < 9; ++k) {                         // window position k: token (y + k / 3 - 1, x + k % 3 - 1)
                const int dy = k / 3 - 1, dx = k % 3 - 1;
                win[k] = zero_raw4<T>();
                if ((unsigned)(y + dy) < (unsigned)H && (unsigned)(x + dx) < (unsigned)W) win[k] = ld_raw4<T>(go + (long long)(tok + dy * W + dx) * d);
            }
        }
        const Windows wy = y - ylo < kAxis ? yw[y - ylo] : windows_of(y, H, p), wx = x < kAxis ? xw[x] : windows_of(x, W, p);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int area = (i ? wy.len1 : wy.len0) * (k ? wx.len1 : wx.len0);
                if (area == 0) continue;
                const float4 g = __ldg(reinterpret_cast<const float4*>(da + (size_t)((wy.first + i) * p + wx.first + k) * d));
                const float inv = 1.f / (float)area;
                q.x = fmaf(g.x, inv, q.x); q.y = fmaf(g.y, inv, q.y);
                q.z = fmaf(g.z, inv, q.z); q.w = fmaf(g.w, inv, q.w);
            }
        *reinterpret_cast<float4*>(a.dq + base + (size_t)tok * d) = q;
        if (DWC) {
            float2 c[2] = {make_float2(o.x, o.y), make_float2(o.z, o.w)};
#pragma unroll
            for (int k = 0; k < 9; ++k) {                         // window position k meets tap 8 - k
                const float4 f = *reinterpret_cast<const float4*>(wt + (8 - k) * d + 4 * cg);
                c[0] = ffma2(pair<T>(win[k], 0), make_float2(f.x, f.y), c[0]);
                c[1] = ffma2(pair<T>(win[k], 1), make_float2(f.z, f.w), c[1]);
            }
            *reinterpret_cast<float4*>(a.dv + base + (size_t)tok * d) = make_float4(c[0].x, c[0].y, c[1].x, c[1].y);
        }
        x += cols;
        while (x >= W) { x -= W; ++y; }
    }
}

// A thread owns four channels of a grid column and slides down a strip of rows, three rows at a time: twelve loads in flight, and
// the window rows above come from registers.
template <typename T>
__global__ void __launch_bounds__(256, 2) bwd_filter_kernel(const TailArgs a) {
    __shared__ float2 red[256][9][2];
    const int d = a.d, H = a.H, W = a.W, slab = blockIdx.y;
    const int y0 = blockIdx.x * a.strip, y1 = min(H, y0 + a.strip);
    const int groups = d >> 2, cols = 256 / groups;
    const int cg = threadIdx.x % groups, cl = threadIdx.x / groups;
    const size_t base = (size_t)slab * H * W * d + 4 * cg;
    const T* v = static_cast<const T*>(a.v) + base;
    const T* go = static_cast<const T*>(a.go) + base;
    float2 acc[9][2];
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[k][0] = acc[k][1] = make_float2(0.f, 0.f);
    if (cl < cols)
        for (int x = cl; x < W; x += cols) {
            Raw4<T> win[5][3], t[3];                              // dO rows y - 1 .. y + 3 around V rows y .. y + 2
            auto row = [&](Raw4<T> (&r)[3], int y) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    r[c] = zero_raw4<T>();
                    if ((unsigned)y < (unsigned)H && (unsigned)(x + c - 1) < (unsigned)W) r[c] = ld_raw4<T>(go + (long long)(y * W + x + c - 1) * d);
                }
            };
            row(win[0], y0 - 1);
            row(win[1], y0);
            for (int y = y0; y < y1; y += 3) {
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    row(win[2 + i], y + 1 + i);
                    t[i] = zero_raw4<T>();
                    if (y + i < y1) t[i] = ld_raw4<T>(v + (long long)((y + i) * W + x) * d);
                }
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float2 s = pair<T>(t[i], q);
#pragma unroll
                        for (int u = 0; u < 3; ++u)
#pragma unroll
                            for (int w = 0; w < 3; ++w) acc[3 * u + w][q] = ffma2(pair<T>(win[i + 2 - u][2 - w], q), s, acc[3 * u + w][q]);
                    }
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    win[0][c] = win[3][c];
                    win[1][c] = win[4][c];
                }
            }
        }
#pragma unroll
    for (int k = 0; k < 9; ++k)
#pragma unroll
        for (int q = 0; q < 2; ++q) red[threadIdx.x][k][q] = acc[k][q];
    __syncthreads();
    pdl_wait_prior();                                             // (before that: inputs only)
    for (int o = threadIdx.x; o < d * 9; o += 256) {              // o = channel * 9 + tap
        const int c = o / 9, k = o - c * 9;
        float s = 0.f;
        for (int l = 0; l < cols; ++l) {
            const float2 t = red[l * groups + (c >> 2)][k][(c >> 1) & 1];
            s += (c & 1) ? t.y : t.x;
        }
        atomicAdd(a.dwd + (size_t)(slab % a.heads) * d * 9 + o, s);
    }
}

template <typename T> cudaError_t launch_tail(TailArgs a, int slabs, int sm_count, cudaStream_t st) {
    const int N = a.H * a.W, cols = 256 / (a.d / 4);
    // runs of tokens: three blocks per SM are resident; at least eight passes of a block, for its tables and taps
    const long long want = 3LL * sm_count;
    long long tokens = ((long long)N * slabs + want - 1) / want;
    tokens = tokens < 8 * cols ? 8 * cols : tokens;
    const int parts = (int)((N + tokens - 1) / tokens);
    tokens = (N + parts - 1) / parts;
    const dim3 grid(parts, slabs);
    cudaError_t e = launch_dependent(a.wd ? bwd_tail_kernel<T, true> : bwd_tail_kernel<T, false>, grid, 256, 0, st, a, (int)tokens);
    if (e != cudaSuccess || !a.dwd) return e;
    // strips: two blocks per SM are resident, at least six rows each (a strip reads two more)
    const int strip = (int)(((long long)a.H * slabs + 2LL * sm_count - 1) / (2LL * sm_count));
    a.strip = ((strip < 6 ? 6 : strip) + 2) / 3 * 3;
    return launch_dependent(bwd_filter_kernel<T>, dim3((a.H + a.strip - 1) / a.strip, slabs), 256, 0, st, a);
}

}  // namespace

cudaError_t launch_backward_tail(int dtype, const BwdCall& c, cudaStream_t st) {
    TailArgs a;
    a.v = c.v; a.go = c.d_out; a.wd = c.wd; a.da = c.ws_da; a.dq = c.dq; a.dv = c.dv; a.dwd = c.dwd;
    a.heads = c.heads; a.H = c.H; a.W = c.W; a.d = c.d; a.n = c.n; a.p = c.p; a.strip = 0;
    switch (dtype) {
        case kF32:  return launch_tail<float>(a, c.slabs, c.sm_count, st);
        case kBF16: return launch_tail<__nv_bfloat16>(a, c.slabs, c.sm_count, st);
        default:    return launch_tail<__half>(a, c.slabs, c.sm_count, st);
    }
}

}  // namespace aa
