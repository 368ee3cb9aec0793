// Register-tiled forward kernels for head sizes padded to 64 channels.
#include "tile_launch.cuh"

namespace aa {
AA_TILE_DECLARE(64) { return tile_dispatch_dk<64>(k, dtype, bias, a, l); }
}  // namespace aa
