// Register-tiled forward kernels for head sizes padded to 80 channels.
#include "tile_launch.cuh"

namespace aa {
AA_TILE_DECLARE(80) { return tile_dispatch_dk<80>(k, dtype, bias, a, l); }
}  // namespace aa
