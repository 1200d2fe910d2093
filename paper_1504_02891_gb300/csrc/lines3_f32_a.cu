// lines3_f32_a.cu -- float32 instantiations of the 1D/3D/sine line kernels.
#include "lines3.cuh"

namespace gpe {
template gpe_status launch_axis_s<float>(const GridHost&, const GridDev<float>&, int, const PassData<float>&, cudaStream_t);
}  // namespace gpe
