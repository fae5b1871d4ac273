// Tiled passes of the D1Q3 lattice (two to four species in float, two and three in double).
#include "tile.cuh"

namespace lbms {

template <>
cudaError_t dispatch_tile_lattice<LBMS_D1Q3>(int dtype, const KArgs& a)
{
    return dtype == LBMS_F64 ? launch_tile_species<LBMS_D1Q3, double>(a) : launch_tile_species<LBMS_D1Q3, float>(a);
}

}  // namespace lbms
