// Separable-phasor degridder kernels for subgrid size 128 (templates in degridder_sep_kernels.cuh).
#include "degridder_sep_kernels.cuh"

namespace idg {

template int configure_degridder_sep_l<128>(int*);
template int degridder_sep_vis_l<128>(int);
template int launch_degridder_sep_l<128>(const DegridArgs&, int, int, bool, void*);
template int launch_degridder_sep_multi_l<128>(const DegridArgs*, const int2*, int, int, bool, void*);

}  // namespace idg
