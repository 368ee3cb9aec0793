// Instantiations of the term-split gradient kernels: a translation unit per head size.
#pragma once
#include "bwd_terms.cuh"
#include "tile_launch.cuh"

namespace aa {

struct BwdTermLaunch {
    dim3 grid;
    int cluster, kg;
    cudaStream_t stream;
};

template <typename K> inline cudaError_t bwd_launch(K kern, std::atomic<unsigned long long>& done, const BwdTermArgs& a, const BwdTermLaunch& l, int threads, int smem) {
    cudaError_t e = tile_allow_smem(kern, done);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = l.grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = l.stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = l.cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = l.cluster > 0 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

// How many 16-bit terms the operands carry.  Full: fp32 operands as three bf16 terms, eight warps on an SM.  Mixed (the forward
// sums of up to 64 agents of 64 channels): A rounded once to the element type, the probabilities and V_A two terms of it.
template <typename T> struct TermsFull {
    using E = __nv_bfloat16;
    static constexpr int NX = sizeof(T) == 4 ? 3 : Elem<T>::kIsBf16 ? 1 : 2, TA = 3, TM = 3, TP = 3, NW = 8;
};
template <typename T> struct TermsMixed {
    using E = T;
    static constexpr int NX = 1, TA = 1, TM = 2, TP = 2, NW = 4;
};

template <typename T, typename C, int DK, int KG, int MODE> cudaError_t bwd_sums_kg(const BwdTermArgs& a, const BwdTermLaunch& l) {
    static std::atomic<unsigned long long> done;
    return bwd_launch(bwd_sums_kernel<T, typename C::E, DK, C::NX, C::TA, C::TM, C::TP, KG, C::NW, MODE>, done, a, l, C::NW * 32,
                      SumsShape<DK, C::NX, C::TA, C::TM, KG, C::NW, MODE>::smem(a.rg * 16));
}
template <typename T, typename C, int DK, int MODE> cudaError_t bwd_sums(const BwdTermArgs& a, const BwdTermLaunch& l) {
    return l.kg == 1 ? bwd_sums_kg<T, C, DK, 1, MODE>(a, l) : l.kg == 2 ? bwd_sums_kg<T, C, DK, 2, MODE>(a, l) : bwd_sums_kg<T, C, DK, 4, MODE>(a, l);
}
template <typename T, int DK, int MODE> cudaError_t bwd_rows(const BwdTermArgs& a, const BwdTermLaunch& l) {
    using C = TermsFull<T>;
    static std::atomic<unsigned long long> done;
    return bwd_launch(bwd_rows_kernel<T, typename C::E, DK, C::NX, C::TA, C::TM, C::TP, MODE>, done, a, l, 256, MODE == kRowsOutSplit ? RowsShape<DK, C::TA, C::TM>::smem_split(a.n) : MODE == kRowsOut ? RowsShape<DK, C::TA, C::TM>::smem_out(a.n) : RowsShape<DK, C::TA, C::TM>::smem(a.n));
}

enum BwdTermStage { kTermForward, kTermStats, kTermBroadcast, kTermAggregate, kTermKeyValue, kTermQuery, kTermOut, kTermOutSplit };
constexpr int kTermGradientsF32 = 80;      // fp32 inputs: the gradient kernels' accumulators and operand rows fit in registers up to here
template <typename T, int DK> cudaError_t bwd_terms_stage(int stage, const BwdTermArgs& a, const BwdTermLaunch& l) {
    if (stage == kTermForward) return bwd_sums<T, TermsFull<T>, DK, kSumsForward>(a, l);
    if constexpr (sizeof(T) == 4) {
        if (stage == kTermOut) return bwd_rows<T, DK, kRowsOut>(a, l);
        if (stage == kTermOutSplit) return bwd_rows<T, DK, kRowsOutSplit>(a, l);
    }
    if constexpr (sizeof(T) == 2 || DK <= kTermGradientsF32) {
        switch (stage) {
            case kTermStats:     return bwd_rows<T, DK, kRowsStats>(a, l);
            case kTermBroadcast: return bwd_sums<T, TermsFull<T>, DK, kSumsBroadcast>(a, l);
            case kTermAggregate: return bwd_sums<T, TermsFull<T>, DK, kSumsAggregate>(a, l);
            case kTermKeyValue:  return bwd_rows<T, DK, kRowsKeyValue>(a, l);
            case kTermQuery:     return bwd_rows<T, DK, kRowsQuery>(a, l);
        }
    }
    return cudaErrorInvalidValue;
}
#define AA_BWD_TERMS_DECLARE(DK) cudaError_t bwd_terms_##DK(int dtype, int stage, const BwdTermArgs& a, const BwdTermLaunch& l)
#define AA_BWD_TERMS_DEFINE(DK)                                                                            \
    AA_BWD_TERMS_DECLARE(DK) {                                                                             \
        return dtype == kBF16 ? bwd_terms_stage<__nv_bfloat16, DK>(stage, a, l)                            \
               : dtype == kF16 ? bwd_terms_stage<__half, DK>(stage, a, l) : bwd_terms_stage<float, DK>(stage, a, l); \
    }
AA_BWD_TERMS_DECLARE(32); AA_BWD_TERMS_DECLARE(48); AA_BWD_TERMS_DECLARE(64); AA_BWD_TERMS_DECLARE(80); AA_BWD_TERMS_DECLARE(96); AA_BWD_TERMS_DECLARE(128);
cudaError_t bwd_terms_mixed(int dtype, const BwdTermArgs& a, const BwdTermLaunch& l);         // forward sums

}  // namespace aa
