// Register-tiled forward kernels for head sizes padded to 32 channels.
#include "tile_launch.cuh"

namespace aa {
AA_TILE_DECLARE(32) { return tile_dispatch_dk<32>(k, dtype, bias, a, l); }
}  // namespace aa
