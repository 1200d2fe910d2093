// lines3_f64_b.cu -- float64 instantiations of the 1D/3D/sine line kernels.
#include "lines3.cuh"

namespace gpe {
template gpe_status launch_axis_x<double, EPI_HESS>(const GridHost&, const GridDev<double>&, const PassData<double>&, cudaStream_t);
template gpe_status launch_axis_x<double, EPI_RATIO>(const GridHost&, const GridDev<double>&, const PassData<double>&, cudaStream_t);
}  // namespace gpe
