// Term-split gradient kernels for head sizes padded to 80 channels.
#include "bwd_terms_launch.cuh"

namespace aa {
AA_BWD_TERMS_DEFINE(80)
}  // namespace aa
