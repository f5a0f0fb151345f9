// Register-tile kernels of 16 warps with bands of 10 to 12 rows.
#include "tiles.cuh"

namespace sdfg {
const void *tile_fn_tall(int rb, int dtype) {
    return rb == 10 ? tile_fn_of<16, 10>(dtype)
         : rb == 11 ? tile_fn_of<16, 11>(dtype)
         : tile_fn_of<16, 12>(dtype);
}
}  // namespace sdfg
