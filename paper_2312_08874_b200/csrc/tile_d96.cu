// Register-tiled forward kernels for head sizes padded to 96 channels.
#include "tile_launch.cuh"

namespace aa {
AA_TILE_DECLARE(96) { return tile_dispatch_dk<96>(k, dtype, bias, a, l); }
}  // namespace aa
