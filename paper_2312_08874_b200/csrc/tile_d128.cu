// Register-tiled forward kernels for head sizes padded to 128 channels.
#include "tile_launch.cuh"

namespace aa {
AA_TILE_DECLARE(128) { return tile_dispatch_dk<128>(k, dtype, bias, a, l); }
}  // namespace aa
