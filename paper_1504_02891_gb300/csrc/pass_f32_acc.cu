// pass_f32_acc.cu -- float32 axis passes of known length, EPI_ACC.
#include "pass_f32.cuh"

namespace gpe {
template gpe_status launch_pass_s<true, EPI_ACC>(const PassGeom<float>&, int, const PassData<float>&, size_t, cudaStream_t);
template gpe_status launch_pass_s<false, EPI_ACC>(const PassGeom<float>&, int, const PassData<float>&, size_t, cudaStream_t);
}  // namespace gpe
