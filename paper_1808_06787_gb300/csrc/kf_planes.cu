// Fused passes of the 1D and 2D lattices (two to five species, float).
#include "fused.cuh"

namespace lbms {

namespace {

template <int LAT>
cudaError_t run(const KArgs& a)
{
    switch (a.n_species) {
        case 2: return launch_fused<LAT, 1>(a);
        case 3: return launch_fused<LAT, 2>(a);
        case 4: return launch_fused<LAT, 3>(a);
        case 5: return launch_fused<LAT, 4>(a);
        default: return cudaErrorInvalidValue;
    }
}

template <int LAT>
int limit(int n)
{
    switch (n) {
        case 2: return fused_limit<LAT, 1>();
        case 3: return fused_limit<LAT, 2>();
        case 4: return fused_limit<LAT, 3>();
        case 5: return fused_limit<LAT, 4>();
        default: return 1;
    }
}

}  // namespace

int fused_limit_of(int lattice, int n_species)
{
    switch (lattice) {
        case LBMS_D1Q3: return limit<LBMS_D1Q3>(n_species);
        case LBMS_D2Q4: return limit<LBMS_D2Q4>(n_species);
        case LBMS_D2Q5: return limit<LBMS_D2Q5>(n_species);
        case LBMS_D2Q9: return limit<LBMS_D2Q9>(n_species);
        default: return 1;
    }
}

cudaError_t dispatch_fused(int lattice, const KArgs& a)
{
    switch (lattice) {
        case LBMS_D1Q3: return run<LBMS_D1Q3>(a);
        case LBMS_D2Q4: return run<LBMS_D2Q4>(a);
        case LBMS_D2Q5: return run<LBMS_D2Q5>(a);
        case LBMS_D2Q9: return run<LBMS_D2Q9>(a);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbms
