// Register-tile kernels of 16 warps with bands of 4 to 9 rows.
#include "tiles.cuh"

namespace sdfg {
const void *tile_fn_mid(int rb, int dtype) {
    return rb == 4 ? tile_fn_of<16, 4>(dtype)
         : rb == 5 ? tile_fn_of<16, 5>(dtype)
         : rb == 6 ? tile_fn_of<16, 6>(dtype)
         : rb == 7 ? tile_fn_of<16, 7>(dtype)
         : rb == 8 ? tile_fn_of<16, 8>(dtype)
         : tile_fn_of<16, 9>(dtype);
}
}  // namespace sdfg
