// Tiled passes of the D2Q4 lattice (two to four species in float, two and three in double).
#include "tile.cuh"

namespace lbms {

template <>
cudaError_t dispatch_tile_lattice<LBMS_D2Q4>(int dtype, const KArgs& a)
{
    return dtype == LBMS_F64 ? launch_tile_species<LBMS_D2Q4, double>(a) : launch_tile_species<LBMS_D2Q4, float>(a);
}

}  // namespace lbms
