// Instantiations of the small-tile kernels for BF16 and TF32 inputs on the NVIDIA models (T-FDPA).
#include "mmasim_direct.cuh"
namespace mmasim { namespace direct {
cudaError_t launch_bf16(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t st) {
    if (m.L == 8) return launch<FAM_T, fast::EK_BF16, 8, RHO_RZ_FP32>(m, g, size, st);
    if (m.L == 16 && g.redo) return launch_rest<FAM_T, fast::EK_BF16, 16, RHO_RZ_FP32>(m, g, st);
    if (m.L == 16) return launch<FAM_T, fast::EK_BF16, 16, RHO_RZ_FP32>(m, g, size, st);
    return cudaErrorInvalidValue;
}
cudaError_t launch_tf32(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t st) {
    if (m.L == 4) return launch<FAM_T, fast::EK_TF32, 4, RHO_RZ_FP32>(m, g, size, st);
    if (m.L == 8 && g.redo) return launch_rest<FAM_T, fast::EK_TF32, 8, RHO_RZ_FP32>(m, g, st);
    if (m.L == 8) return launch<FAM_T, fast::EK_TF32, 8, RHO_RZ_FP32>(m, g, size, st);
    return cudaErrorInvalidValue;
}
}}
