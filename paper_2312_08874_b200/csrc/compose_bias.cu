// Dense agent bias from its three components (App. B): B = (B'_c + B'_r + B'_b).reshape(n, N), with
// the column bias repeated over rows, the row bias repeated over columns and the block bias resized
// to the token grid by bilinear interpolation (half-pixel centres, edge clamp).  fp32 arithmetic, one rounding to the storage type.
// A block takes 32 tokens of a head and all its agents: lanes are tokens, so a token's place in the block bias is found once for all
// agents and the components are read along their rows; the transposed layout goes through shared memory, from where the block's outputs
// are one contiguous run.  256 agents on a 128 x 210 grid: 31 us, and 62 us transposed, with eight consecutive outputs a thread (a
// transposed thread's agents are rows apart); 19 us (31 us) this way.
#include "common.cuh"
#include "kernels.h"

namespace aa {

constexpr int kComposeTokens = 32;

template <typename T, bool TRANSPOSE>
__global__ void __launch_bounds__(256) compose_bias_kernel(ComposeArgs p) {
    extern __shared__ __align__(16) unsigned char smem[];
    pdl_wait_prior();
    pdl_release_next();
    const int N = p.h * p.w, head = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = blockIdx.x * kComposeTokens, t = t0 + lane;
    const bool live = t < N;
    const int y = live ? t / p.w : 0, x = live ? t - y * p.w : 0;
    const float sy = fmaxf(0.f, ((float)y + 0.5f) * (float)p.h0 / (float)p.h - 0.5f), sx = fmaxf(0.f, ((float)x + 0.5f) * (float)p.w0 / (float)p.w - 0.5f);
    const int y0 = min((int)sy, p.h0 - 1), x0 = min((int)sx, p.w0 - 1), y1 = min(y0 + 1, p.h0 - 1), x1 = min(x0 + 1, p.w0 - 1);
    const float ly = fminf(sy - (float)y0, 1.f), lx = fminf(sx - (float)x0, 1.f);
    const int area = p.h0 * p.w0, o00 = y0 * p.w0 + x0, o01 = y0 * p.w0 + x1, o10 = y1 * p.w0 + x0, o11 = y1 * p.w0 + x1;
    const T *col = static_cast<const T*>(p.col), *row = static_cast<const T*>(p.row), *blk = static_cast<const T*>(p.blk);
    T* out = static_cast<T*>(p.out) + (size_t)head * p.n * N;
    T* tile = reinterpret_cast<T*>(smem);                         // TRANSPOSE: [32 tokens][n]
    const int pitch = p.n + (p.n % 2 ? 0 : 1);                    // odd: lanes write different banks
    // four weights: (1 - ly) ((1 - lx) b00 + lx b01) + ly ((1 - lx) b10 + lx b11)
    const float w00 = (1.f - ly) * (1.f - lx), w01 = (1.f - ly) * lx, w10 = ly * (1.f - lx), w11 = ly * lx;
    const size_t ha = (size_t)head * p.n;
    const T *cp = col ? col + ha * p.w + x : nullptr, *rp = row ? row + ha * p.h + y : nullptr, *bp = blk ? blk + ha * area : nullptr;
    for (int a0 = warp; a0 < p.n; a0 += 32) {                     // four agents of this warp at a time: all their loads in flight
        T c[4], r[4], b[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int a = min(a0 + 8 * i, p.n - 1);
            if (cp) c[i] = cp[a * p.w];
            if (rp) r[i] = rp[a * p.h];
            if (bp) {
                const T* u = bp + a * area;
                b[i][0] = u[o00]; b[i][1] = u[o01]; b[i][2] = u[o10]; b[i][3] = u[o11];
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int a = a0 + 8 * i;
            if (a >= p.n) break;
            float v = 0.f;
            if (cp) v += Elem<T>::to_f32(c[i]);
            if (rp) v += Elem<T>::to_f32(r[i]);
            if (bp) v += w00 * Elem<T>::to_f32(b[i][0]) + w01 * Elem<T>::to_f32(b[i][1]) + w10 * Elem<T>::to_f32(b[i][2]) + w11 * Elem<T>::to_f32(b[i][3]);
            if (TRANSPOSE) tile[lane * pitch + a] = Elem<T>::from_f32(v);
            else if (live) out[(size_t)a * N + t] = Elem<T>::from_f32(v);
        }
    }
    if constexpr (TRANSPOSE) {
        __syncthreads();
        out += (size_t)t0 * p.n;
        // one contiguous run of outputs; a warp copies whole token rows
        for (int tk = warp; tk < min(kComposeTokens, N - t0); tk += 8)
            for (int a = lane; a < p.n; a += 32) out[tk * p.n + a] = tile[tk * pitch + a];
    }
}

template <typename T> static cudaError_t launch_compose(const ComposeArgs& p, cudaStream_t st) {
    const dim3 grid((p.h * p.w + kComposeTokens - 1) / kComposeTokens, p.heads);
    if (p.transpose) return launch_dependent(compose_bias_kernel<T, true>, grid, 256, kComposeTokens * (p.n + 1) * sizeof(T), st, p);
    return launch_dependent(compose_bias_kernel<T, false>, grid, 256, 0, st, p);
}

cudaError_t launch_compose_bias(int dtype, const ComposeArgs& p, cudaStream_t st) {
    switch (dtype) {
        case kF32:  return launch_compose<float>(p, st);
        case kBF16: return launch_compose<__nv_bfloat16>(p, st);
        case kF16:  return launch_compose<__half>(p, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace aa
