// Instantiations of the small-tile kernels for the CDNA1 (E-FDPA) and CDNA3 (TR-, GTR-FDPA) models.
#include "mmasim_direct.cuh"
namespace mmasim { namespace direct {
cudaError_t launch_tr(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t st) {
    if (m.family == FAM_GTR) return launch<FAM_GTR, fast::EK_LUT8, 16, RHO_RNE_FP32>(m, g, size, st);
    if (m.fmt_a == EF_F16) return launch<FAM_TR, fast::EK_F16, 8, RHO_RNE_FP32>(m, g, size, st);
    if (m.fmt_a == EF_BF16) return launch<FAM_TR, fast::EK_BF16, 8, RHO_RNE_FP32>(m, g, size, st);
    if (m.fmt_a == EF_TF32) return launch<FAM_TR, fast::EK_TF32, 4, RHO_RNE_FP32>(m, g, size, st);
    return cudaErrorInvalidValue;
}
cudaError_t launch_e(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t st) {
    if (m.fmt_a == EF_F16) return launch<FAM_E, fast::EK_F16, 4, RHO_RNE_FP32>(m, g, size, st);
    return launch<FAM_E, fast::EK_BF16, 2, RHO_RNE_FP32>(m, g, size, st);
}
}}
