// lines3_f32_b.cu -- float32 instantiations of the 1D/3D/sine line kernels.
#include "lines3.cuh"

namespace gpe {
template gpe_status launch_axis_x<float, EPI_HESS>(const GridHost&, const GridDev<float>&, const PassData<float>&, cudaStream_t);
template gpe_status launch_axis_x<float, EPI_RATIO>(const GridHost&, const GridDev<float>&, const PassData<float>&, cudaStream_t);
}  // namespace gpe
