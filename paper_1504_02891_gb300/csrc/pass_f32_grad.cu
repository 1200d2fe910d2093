// pass_f32_grad.cu -- float32 axis passes of known length, EPI_GRAD.
#include "pass_f32.cuh"

namespace gpe {
template gpe_status launch_pass_s<true, EPI_GRAD>(const PassGeom<float>&, int, const PassData<float>&, size_t, cudaStream_t);
template gpe_status launch_pass_s<false, EPI_GRAD>(const PassGeom<float>&, int, const PassData<float>&, size_t, cudaStream_t);
}  // namespace gpe
