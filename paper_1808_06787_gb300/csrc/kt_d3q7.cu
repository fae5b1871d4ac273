// Tiled passes of the D3Q7 lattice (two and three species, float).
#include "tile.cuh"

namespace lbms {

template <>
cudaError_t dispatch_tile_lattice<LBMS_D3Q7>(int dtype, const KArgs& a)
{
    return dtype == LBMS_F64 ? cudaErrorInvalidValue : launch_tile_species<LBMS_D3Q7, float>(a);
}

}  // namespace lbms
