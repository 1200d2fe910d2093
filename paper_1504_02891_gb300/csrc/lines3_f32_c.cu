// lines3_f32_c.cu -- float32 instantiations of the 1D/3D/sine line kernels.
#include "lines3.cuh"

namespace gpe {
template gpe_status launch_axis_x<float, EPI_F>(const GridHost&, const GridDev<float>&, const PassData<float>&, cudaStream_t);
template gpe_status launch_axis_x<float, EPI_WS>(const GridHost&, const GridDev<float>&, const PassData<float>&, cudaStream_t);
}  // namespace gpe
