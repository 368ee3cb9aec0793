// Token-wise tail of the backward pass:
//   dQ  += Pooling^T(dA)   a window spreads its agent's gradient evenly over its tokens
//   dV  += DWC^T(dO)       tap (u, v) of output token (y - u + 1, x - v + 1) read V[y][x]
//   dWd += corr(dO, V)     dWd[c][u][v] = sum over tokens of dO[y - u + 1][x - v + 1][c] V[y][x][c]
// Two kernels of threads that slide down a strip of rows of a grid column.  bwd_conv_tail does dV and dWd, two channels a thread: a row
// brings three new window entries, the other six come from registers, an entry serves both its tap and its sum, and dO is requested two
// rows ahead.  (Four channels a thread need twice the registers for taps and sums: with the taps in shared memory and two blocks of
// eight warps an SM 60 us; a spill of 100 bytes in the loop costs 26 us, so tokens are addressed by one offset.)  Its blocks add their
// share of dWd to one of kFilterCopies copies, which the second kernel adds up: relative error 1.4e-7, against 5e-7 in a single copy.
// A block goes through several batch entries of its head where that fills one wave of blocks (384 slabs of a 14 x 14 grid: 24.3 -> 20.5 us;
// 64 slabs of 56 x 56: 43 -> 39 us).
// bwd_pool_tail is a stream over dQ, four rows in flight, beside the blocks of the other (64 slabs of 56 x 56, whole pass: 177.6 -> 174.4 us).  dQ and dV are read and written in fp32, which is the bound.  64 slabs of a
// 56 x 56 grid: 39 us (154 MB, 24 us at the copy bandwidth) and 16 us (103 MB, 16 us); one kernel for dQ and dV with all nine window
// loads of a token, and one for dWd, took 74 and 31.
#include "common.cuh"
#include "kernels.h"

#include <algorithm>
#include <cmath>

namespace aa {

namespace {

struct TailArgs {
    const void *v, *go, *wd;
    const float* da;
    float *dq, *dv, *dwd, *dwd_copies;
    unsigned* handed;                  // nonzero once the gradient stages' results are there for bwd_pool_tail (zero on entry)
    int heads, H, W, d, n, p, strip, strips, passes, batch;
};

__device__ __forceinline__ void store_release(unsigned* p, unsigned v) { asm volatile("st.release.gpu.global.u32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory"); }
__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Two channels of a token as loaded (zeros where there is no token; volatile: left to itself the compiler gathers the loads of several
// rows and spills), and in fp32 on use.
template <typename T> struct Raw2 { uint32_t w; };
template <> struct Raw2<float> { float2 w; };
template <typename T> __device__ __forceinline__ Raw2<T> ld_raw2(const T* p, bool ok) {
    Raw2<T> r;
    if constexpr (sizeof(T) == 4)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.b32 %0, 0f00000000;\n\tmov.b32 %1, 0f00000000;\n\t@p ld.global.nc.v2.f32 {%0,%1}, [%2];\n\t}\n"
                     : "=&f"(r.w.x), "=&f"(r.w.y) : "l"(p), "r"((int)ok));
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\tmov.b32 %0, 0;\n\t@p ld.global.nc.u32 %0, [%1];\n\t}\n" : "=&r"(r.w) : "l"(p), "r"((int)ok));
    return r;
}
__device__ __forceinline__ float2 ld_pair(const float* p, bool ok) {
    float2 r;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.b32 %0, 0f00000000;\n\tmov.b32 %1, 0f00000000;\n\t@p ld.global.v2.f32 {%0,%1}, [%2];\n\t}\n"
                 : "=&f"(r.x), "=&f"(r.y) : "l"(p), "r"((int)ok) : "memory");
    return r;
}
template <typename T> __device__ __forceinline__ float2 pair(const Raw2<T>& r) {
    if constexpr (sizeof(T) == 4) return r.w;
    else return unpack2<T>(r.w);
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

constexpr int kAxis = 512;         // rows whose windows are kept in shared memory
constexpr int kThreadsQ = 256, kThreadsV = 128;
constexpr int kStartV = 8;         // the start and the end of a bwd_conv_tail block cost about so many rows

// Columns of a slab's strips, one after the other: a block takes `passes` times `cols` of them.
struct Column {
    int x, y0, y1;
};
__device__ __forceinline__ Column column_of(const TailArgs& a, int i) {
    const int s = i / a.W;
    return {i - s * a.W, s * a.strip, min(a.H, (s + 1) * a.strip)};
}

// BESIDE: the kernel before is bwd_conv_tail, whose blocks touch nothing that this one does and release it once the gradient stages are complete;
// so it runs beside them, and waits for their end before its own (what comes next waits for this kernel alone).  A release of the launch orders
// no memory: bwd_conv_tail, which has waited for the stages, says so in `handed` with a release, every block here reads that with an acquire, and
// one that finds nothing waits for the kernel before after all.  What the stages wrote is read past L1, which was not emptied since.
template <bool BESIDE>
__global__ void __launch_bounds__(kThreadsQ, 4) bwd_pool_tail_kernel(const TailArgs a) {
    __shared__ Windows yw[kAxis];
    const int d = a.d, H = a.H, W = a.W, p = a.p, slab = blockIdx.y;
    if (a.dwd && blockIdx.x == gridDim.x - 1) {                   // the last column of blocks: the filter gradient's copies
        pdl_wait_prior();
        pdl_release_next();
        const int words = a.heads * d * 9;
        for (int o = slab * kThreadsQ + threadIdx.x; o < words; o += gridDim.y * kThreadsQ) {
            float c[kFilterCopies];
#pragma unroll
            for (int k = 0; k < kFilterCopies; ++k) c[k] = a.dwd_copies[(size_t)k * words + o];
#pragma unroll
            for (int h = kFilterCopies / 2; h; h >>= 1)
#pragma unroll
                for (int k = 0; k < h; ++k) c[k] += c[k + h];
            a.dwd[o] = c[0];
        }
        return;
    }
    const int groups = d >> 2, cols = kThreadsQ / groups;         // d <= 128: at least eight columns at once
    const int cg = threadIdx.x % groups, cl = threadIdx.x / groups;
    for (int i = threadIdx.x; i < min(H, kAxis); i += kThreadsQ) yw[i] = windows_of(i, H, p);
    if (!BESIDE) {
        pdl_wait_prior();
        pdl_release_next();
        __syncthreads();
    } else if (!__syncthreads_or(threadIdx.x == 0 && load_acquire(a.handed))) {
        pdl_wait_prior();
    }
    if (cl < cols) {
    const float* da = a.da + (size_t)slab * a.n * d + 4 * cg;
    const int first = blockIdx.x * a.passes * cols, last = min(first + a.passes * cols, a.strips * W);
    for (int i = first + cl; i < last; i += cols) {
        const Column c = column_of(a, i);
        const Windows wx = windows_of(c.x, W, p);
        float* dq = a.dq + ((size_t)slab * H * W + (size_t)c.y0 * W + c.x) * d + 4 * cg;
        float4 pooled = make_float4(0.f, 0.f, 0.f, 0.f);
        Windows wy = {-1, 0, 0};
        for (int y = c.y0; y < c.y1; y += 4) {
            float4 q[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (y + k < c.y1) q[k] = __ldcg(reinterpret_cast<const float4*>(dq + (size_t)k * W * d));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (y + k >= c.y1) break;
                const Windows w = y + k < kAxis ? yw[y + k] : windows_of(y + k, H, p);
                if (w.first != wy.first || w.len0 != wy.len0 || w.len1 != wy.len1) {       // another window row: its agents' gradients
                    wy = w;
                    pooled = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int l = 0; l < 2; ++l) {
                            const int area = (j ? wy.len1 : wy.len0) * (l ? wx.len1 : wx.len0);
                            if (area == 0) continue;
                            const float4 g = __ldcg(reinterpret_cast<const float4*>(da + (size_t)((wy.first + j) * p + wx.first + l) * d));
                            const float inv = 1.f / (float)area;
                            pooled.x = fmaf(g.x, inv, pooled.x); pooled.y = fmaf(g.y, inv, pooled.y);
                            pooled.z = fmaf(g.z, inv, pooled.z); pooled.w = fmaf(g.w, inv, pooled.w);
                        }
                }
                q[k].x += pooled.x; q[k].y += pooled.y; q[k].z += pooled.z; q[k].w += pooled.w;
                *reinterpret_cast<float4*>(dq + (size_t)k * W * d) = q[k];
            }
            dq += (size_t)4 * W * d;
        }
    }
    }
    if (BESIDE) {
        pdl_release_next();
        pdl_wait_prior();
    }
}

template <typename T, bool DWD>
__global__ void __launch_bounds__(kThreadsV, sizeof(T) == 4 ? 4 : 5) bwd_conv_tail_kernel(const TailArgs a) {
    __shared__ float2 red[DWD ? kThreadsV : 1][9];
    const int d = a.d, H = a.H, W = a.W, head = blockIdx.y % a.heads;
    const int groups = d >> 1, cols = kThreadsV / groups;         // d <= 128: at least two columns at once
    const int cg = threadIdx.x % groups, cl = threadIdx.x / groups;
    float2 tap[9], acc[DWD ? 9 : 1];
    {
        const T* w = static_cast<const T*>(a.wd) + ((size_t)head * d + 2 * cg) * 9;
#pragma unroll
        for (int k = 0; k < 9; ++k) tap[k] = make_float2(Elem<T>::to_f32(w[k]), Elem<T>::to_f32(w[9 + k]));
    }
    pdl_wait_prior();                                             // (before that: inputs only)
    if (blockIdx.x + blockIdx.y + threadIdx.x == 0) store_release(a.handed, 1u);
    pdl_release_next();
    if (DWD)
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[k] = make_float2(0.f, 0.f);
    const int first = blockIdx.x * a.passes * cols, last = min(first + a.passes * cols, a.strips * W);
    const size_t pitch = (size_t)W * d;
    // its columns in every so many batch entries of one head: the filter and its gradient's sums stay in registers
    for (int e = blockIdx.y / a.heads, step = gridDim.y / a.heads; e < a.batch; e += step) {
        const int slab = e * a.heads + head;
        if (cl < cols)
        for (int i = first + cl; i < last; i += cols) {
            const Column c = column_of(a, i);
            const bool left = c.x > 0, right = c.x + 1 < W;
            size_t off = ((size_t)slab * H * W + (size_t)c.y0 * W + c.x) * d + 2 * cg;       // of row y + k
            const T *v = static_cast<const T*>(a.v), *go = static_cast<const T*>(a.go);
            // rings of three rows: dO in fp32 (y - 1 .. y + 1), the dO rows on their way (y + 2, y + 3), dV and V (y, y + 1)
            float2 win[3][3], o[3];
            Raw2<T> raw[3][3], rv[3];
            auto row = [&](Raw2<T> (&r)[3], size_t at, int y) {
                const bool in = (unsigned)y < (unsigned)H;
                r[0] = ld_raw2<T>(go + at - d, in && left);
                r[1] = ld_raw2<T>(go + at, in);
                r[2] = ld_raw2<T>(go + at + d, in && right);
            };
            auto convert = [&](float2 (&f)[3], const Raw2<T> (&r)[3]) {
#pragma unroll
                for (int k = 0; k < 3; ++k) f[k] = pair<T>(r[k]);
            };
            row(raw[2], off - pitch, c.y0 - 1);
            row(raw[0], off, c.y0);
            o[0] = ld_pair(a.dv + off, true);
            if (DWD) rv[0] = ld_raw2<T>(v + off, true);
            row(raw[1], off + pitch, c.y0 + 1);
            convert(win[2], raw[2]);
            convert(win[0], raw[0]);
            row(raw[2], off + 2 * pitch, c.y0 + 2);
            for (int y = c.y0; y < c.y1; y += 3)
#pragma unroll
                for (int k = 0; k < 3; ++k) {                     // row y + k (rows past the strip: zeros, not stored)
                    const bool more = y + k + 1 < c.y1;
                    row(raw[k], off + 3 * pitch, y + k + 3);
                    o[(k + 1) % 3] = ld_pair(a.dv + off + pitch, more);
                    if (DWD) rv[(k + 1) % 3] = ld_raw2<T>(v + off + pitch, more);
                    convert(win[(k + 1) % 3], raw[(k + 1) % 3]);
                    float2 s = o[k];
                    const float2 t = DWD ? pair<T>(rv[k]) : make_float2(0.f, 0.f);
#pragma unroll
                    for (int j = 0; j < 9; ++j) {                 // window position j = token (y + j / 3 - 1, x + j % 3 - 1) meets tap 8 - j
                        const float2 g = win[(k + j / 3 + 2) % 3][j % 3];
                        s = ffma2(g, tap[8 - j], s);
                        if (DWD) acc[8 - j] = ffma2(g, t, acc[8 - j]);
                    }
                    if (y + k < c.y1) *reinterpret_cast<float2*>(a.dv + off) = s;
                    off += pitch;
                }
        }
    }
    if (DWD) {
#pragma unroll
        for (int k = 0; k < 9; ++k) red[threadIdx.x][k] = acc[k];
        __syncthreads();
        // one of several copies, by the block's rank in its head: a sum of all blocks' shares in one word would round as often as there are
        // blocks
        const unsigned rank = blockIdx.x + gridDim.x * (blockIdx.y / a.heads);
        float* copy = a.dwd_copies + ((size_t)(rank % kFilterCopies) * a.heads + head) * d * 9;
        for (int o = threadIdx.x; o < d * 9; o += kThreadsV) {    // o = channel * 9 + tap
            const int c = o / 9, k = o - c * 9;
            float s = 0.f;
            for (int l = 0; l < cols; ++l) {
                const float2 t = red[l * groups + (c >> 1)][k];
                s += (c & 1) ? t.y : t.x;
            }
            atomicAdd(copy + o, s);
        }
    }
}

// Strips of rows, passes of a block over `cols` columns, and (`most` > 1) batch entries of a block: the least rows that a slot (a resident
// block) goes through, when a strip costs `halo` rows more than it has and a block `start` rows.
dim3 plan_strips(TailArgs* a, int most, int cols, int slots, int halo, int start) {
    double best = 0;
    int blocks = 1, groups = a->batch, tried = 0;
    for (int strips = 1; strips <= 32 && (strips == 1 || strips * 4 <= a->H); ++strips) {
        const int rows = (a->H + strips - 1) / strips;
        if (rows == tried) continue;                              // (this runs on every call: no plan twice, few divisions)
        tried = rows;
        const int used = (a->H + rows - 1) / rows;
        const long long columns = ((long long)used * a->W + cols - 1) / cols;
        for (int passes = 1; passes <= 8 && passes <= columns; ++passes) {
            const int per_slab = (int)((columns + passes - 1) / passes);
            auto consider = [&](int entries, int gy) {
                const double cost = ceil((double)gy * a->heads * per_slab / slots) * ((double)entries * passes * (rows + halo) + start);
                if (best == 0 || cost < best) { best = cost; blocks = per_slab; groups = gy; a->strip = rows; a->strips = used; a->passes = passes; }
            };
            consider(1, a->batch);
            // or as many batch entries as leave a single wave of blocks
            const double wave = (double)per_slab * a->heads;
            if (most > 1 && wave * a->batch > slots) {
                const int room = wave >= slots ? 1 : (int)(slots / wave), entries = std::min(most, (a->batch + room - 1) / room);
                consider(entries, (a->batch + entries - 1) / entries);
            }
        }
    }
    return dim3(blocks, groups * a->heads);
}

template <typename T> cudaError_t launch_tail(TailArgs a, int sm_count, cudaStream_t st) {
    // dV first: the stage before has just written it
    if (a.wd) {
        const dim3 grid = plan_strips(&a, a.batch, kThreadsV / (a.d / 2), (sizeof(T) == 4 ? 4 : 5) * sm_count, 2, kStartV);
        const cudaError_t e = launch_dependent(a.dwd ? bwd_conv_tail_kernel<T, true> : bwd_conv_tail_kernel<T, false>, grid, kThreadsV, 0, st, a);
        if (e != cudaSuccess) return e;
    }
    dim3 grid = plan_strips(&a, 1, kThreadsQ / (a.d / 4), 4 * sm_count, 0, 4);
    if (a.dwd) ++grid.x;
    return launch_dependent(a.wd ? bwd_pool_tail_kernel<true> : bwd_pool_tail_kernel<false>, grid, kThreadsQ, 0, st, a);
}

}  // namespace

cudaError_t launch_backward_tail(int dtype, const BwdCall& c, cudaStream_t st) {
    TailArgs a;
    a.v = c.v; a.go = c.d_out; a.wd = c.wd; a.da = c.ws_da; a.dq = c.dq; a.dv = c.dv; a.dwd = c.dwd; a.dwd_copies = c.ws_dwd;
    a.handed = reinterpret_cast<unsigned*>(c.ws_dwd) + filter_copy_words(c.heads, c.d);
    a.heads = c.heads; a.H = c.H; a.W = c.W; a.d = c.d; a.n = c.n; a.p = c.p; a.strip = a.strips = a.passes = 0; a.batch = c.slabs / c.heads;
    switch (dtype) {
        case kF32:  return launch_tail<float>(a, c.sm_count, st);
        case kBF16: return launch_tail<__nv_bfloat16>(a, c.sm_count, st);
        default:    return launch_tail<__half>(a, c.sm_count, st);
    }
}

}  // namespace aa
