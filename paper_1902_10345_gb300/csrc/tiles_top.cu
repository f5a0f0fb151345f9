// Register-tile kernels of 16 warps with bands of 14 to 18 rows.
#include "tiles.cuh"

namespace sdfg {
const void *tile_fn_top(int rb, int dtype) {
    return rb == 14 ? tile_fn_of<16, 14>(dtype)
         : rb == 16 ? tile_fn_of<16, 16>(dtype)
         : rb == 17 ? tile_fn_of<16, 17>(dtype)
         : tile_fn_of<16, 18>(dtype);
}
}  // namespace sdfg
