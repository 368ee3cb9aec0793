// Register-tiled forward kernels for head sizes padded to 48 channels.
#include "tile_launch.cuh"

namespace aa {
AA_TILE_DECLARE(48) { return tile_dispatch_dk<48>(k, dtype, bias, a, l); }
}  // namespace aa
