// Register-tile kernels for red-black SOR: 16 warps with 10 rows and more.
#include "tiles.cuh"

namespace sdfg {
const void *sor_tile_fn_tall(TileShape v, int dtype) {
    return v.rb == 10   ? tile_fn_of<16, 10, true>(dtype)
           : v.rb == 12 ? tile_fn_of<16, 12, true>(dtype)
           : v.rb == 14 ? tile_fn_of<16, 14, true>(dtype)
                        : tile_fn_of<16, 17, true>(dtype);
}
}  // namespace sdfg
