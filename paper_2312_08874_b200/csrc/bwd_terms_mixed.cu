// Forward sums of the backward pass for up to 64 agents of 64 channels: mixed precision (see TermsMixed).
#include "bwd_terms_launch.cuh"

namespace aa {
cudaError_t bwd_terms_mixed(int dtype, const BwdTermArgs& a, const BwdTermLaunch& l) {
    return dtype == kBF16 ? bwd_sums<__nv_bfloat16, TermsMixed<__nv_bfloat16>, 64, kSumsForward>(a, l) : bwd_sums<__half, TermsMixed<__half>, 64, kSumsForward>(a, l);
}
}  // namespace aa
