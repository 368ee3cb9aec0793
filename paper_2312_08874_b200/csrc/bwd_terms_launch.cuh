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

template <typename K> inline cudaError_t bwd_launch(K kern, std::atomic<unsigned long long>& done, const BwdTermArgs& a, const BwdTermLaunch& l, int smem) {
    cudaError_t e = tile_allow_smem(kern, done);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = l.grid;
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = l.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = l.cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = l.cluster > 0 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

constexpr int kTerms = 3;          // bf16 terms of an fp32 operand

template <typename T, int DK, int KG, int MODE> cudaError_t bwd_sums_kg(const BwdTermArgs& a, const BwdTermLaunch& l) {
    constexpr int NX = sizeof(T) == 2 && Elem<T>::kIsBf16 ? 1 : 2;
    static std::atomic<unsigned long long> done;
    return bwd_launch(bwd_sums_kernel<T, __nv_bfloat16, DK, NX, kTerms, kTerms, kTerms, KG, MODE>, done, a, l,
                      SumsShape<DK, NX, kTerms, kTerms, KG, MODE>::smem(a.rg * 16));
}
template <typename T, int DK, int MODE> cudaError_t bwd_sums(const BwdTermArgs& a, const BwdTermLaunch& l) {
    return l.kg == 1 ? bwd_sums_kg<T, DK, 1, MODE>(a, l) : l.kg == 2 ? bwd_sums_kg<T, DK, 2, MODE>(a, l) : bwd_sums_kg<T, DK, 4, MODE>(a, l);
}
template <typename T, int DK, int MODE> cudaError_t bwd_rows(const BwdTermArgs& a, const BwdTermLaunch& l) {
    constexpr int NX = Elem<T>::kIsBf16 ? 1 : 2;
    static std::atomic<unsigned long long> done;
    return bwd_launch(bwd_rows_kernel<T, __nv_bfloat16, DK, NX, kTerms, kTerms, kTerms, MODE>, done, a, l, RowsShape<DK, kTerms, kTerms>::smem(a.n));
}

enum BwdTermStage { kTermForward, kTermStats, kTermBroadcast, kTermAggregate, kTermKeyValue, kTermQuery };
template <typename T, int DK> cudaError_t bwd_terms_stage(int stage, const BwdTermArgs& a, const BwdTermLaunch& l) {
    switch (stage) {
        case kTermForward:   return bwd_sums<T, DK, kSumsForward>(a, l);
        case kTermStats:     return bwd_rows<T, DK, kRowsStats>(a, l);
        case kTermBroadcast: return bwd_sums<T, DK, kSumsBroadcast>(a, l);
        case kTermAggregate: return bwd_sums<T, DK, kSumsAggregate>(a, l);
        case kTermKeyValue:  return bwd_rows<T, DK, kRowsKeyValue>(a, l);
        default:             return bwd_rows<T, DK, kRowsQuery>(a, l);
    }
}
#define AA_BWD_TERMS_DECLARE(DK) cudaError_t bwd_terms_##DK(int dtype, int stage, const BwdTermArgs& a, const BwdTermLaunch& l)
#define AA_BWD_TERMS_DEFINE(DK)                                                                            \
    AA_BWD_TERMS_DECLARE(DK) {                                                                             \
        return dtype == kBF16 ? bwd_terms_stage<__nv_bfloat16, DK>(stage, a, l) : bwd_terms_stage<__half, DK>(stage, a, l); \
    }
AA_BWD_TERMS_DECLARE(32); AA_BWD_TERMS_DECLARE(48); AA_BWD_TERMS_DECLARE(64); AA_BWD_TERMS_DECLARE(80); AA_BWD_TERMS_DECLARE(96); AA_BWD_TERMS_DECLARE(128);

}  // namespace aa
