// Register-tile kernels for red-black SOR: 8 warps, and 16 with up to 8 rows.
#include "tiles.cuh"

namespace sdfg {
const void *sor_tile_fn(TileShape v, int dtype) {
    if (v.nw == 8) return v.rb == 4 ? tile_fn_of<8, 4, true>(dtype) : tile_fn_of<8, 6, true>(dtype);
    return v.rb == 4   ? tile_fn_of<16, 4, true>(dtype)
           : v.rb == 6 ? tile_fn_of<16, 6, true>(dtype)
                       : tile_fn_of<16, 8, true>(dtype);
}
}  // namespace sdfg
