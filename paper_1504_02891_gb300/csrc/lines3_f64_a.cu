// lines3_f64_a.cu -- float64 instantiations of the 1D/3D/sine line kernels.
#include "prolong.cuh"

namespace gpe {
template gpe_status launch_axis_s<double>(const GridHost&, const GridDev<double>&, int, const PassData<double>&, cudaStream_t);
template gpe_status launch_axis_x<double, EPI_GRAD>(const GridHost&, const GridDev<double>&, const PassData<double>&, cudaStream_t);
template gpe_status launch_prolong_line<double>(const GridHost&, int, const PassGeom<double>&, const void*, void*, const double*,
                                            const GridDev<double>&, cudaStream_t);
}  // namespace gpe
