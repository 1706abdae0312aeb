// Separable-phasor gridder kernels for subgrid size 128 (templates in gridder_sep_kernels.cuh).
#include "gridder_sep_kernels.cuh"

namespace idg {

template int configure_gridder_sep_l<128>(int*);
template int launch_gridder_sep_l<128>(const GridArgs&, int, int, void*);
template int launch_gridder_sep_multi_l<128>(const GridArgs*, const int2*, int, int, void*);

}  // namespace idg
