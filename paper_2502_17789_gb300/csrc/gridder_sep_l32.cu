// Separable-phasor gridder kernels for subgrid size 32 (templates in gridder_sep_kernels.cuh).
#include "gridder_sep_kernels.cuh"

namespace idg {

template int configure_gridder_sep_l<32>(int*);
template int launch_gridder_sep_l<32>(const GridArgs&, int, int, void*);
template int launch_gridder_sep_multi_l<32>(const GridArgs*, const int2*, int, int, void*);

}  // namespace idg
