// lines3_f32_a.cu -- float32 instantiations of the 1D/3D/sine line kernels.
#include "prolong.cuh"

namespace gpe {
template gpe_status launch_axis_s<float>(const GridHost&, const GridDev<float>&, int, const PassData<float>&, cudaStream_t);
template gpe_status launch_prolong_line<float>(const GridHost&, int, const PassGeom<float>&, const void*, void*, const double*,
                                            const GridDev<float>&, cudaStream_t);
}  // namespace gpe
